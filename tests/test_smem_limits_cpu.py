"""Source check of the kernels' shared-memory limits (no GPU): the limit belongs
to a device, so no flag that is kept for the process may decide whether it is
raised.  Only two places raise it: the helper, which keeps a limit for every
kernel and device, and the resident median/MAD, which raises it on every call."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2509_21754_gb300", "csrc")


def functions_with(call):
    """(file, function body up to the call) of every place that makes the call."""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as fh:
                text = fh.read()
            for m in re.finditer(re.escape(call) + r"\(", text):
                start = max((h.start() for h in re.finditer(r"\n[A-Za-z][^\n;]*\([^;{]*\)\s*\{", text[:m.start()])),
                            default=0)
                yield f, text[start:m.start()]


def test_limits_are_raised_for_the_device():
    places = list(functions_with("cudaFuncSetAttribute"))
    assert sorted(f for f, _ in places) == ["k_noise.cu", "plan.cu"]
    for f, body in places:
        if f == "plan.cu":
            assert "allow_smem_limit" in body and "cudaGetDevice" in body and "std::mutex" in body
        else:
            assert "launch_medmad_small" in body and "static bool" not in body and "if (" not in body
