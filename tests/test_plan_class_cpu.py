"""A plan that the library refuses to configure is destroyed once (no GPU: the
entry points are stand-ins)."""
import gc

import pytest

from paper_2509_21754_gb300 import fitrig as F


def test_refused_plan_is_destroyed_once(monkeypatch):
    destroyed = []

    def refuse(handle, option, value):
        raise F.FitrigError(F.EINVAL, "fitrig_plan_set")

    monkeypatch.setattr(F, "fitrig_plan_create", lambda *a: "handle")
    monkeypatch.setattr(F, "fitrig_plan_set", refuse)
    monkeypatch.setattr(F, "fitrig_plan_destroy", destroyed.append)
    with pytest.raises(F.FitrigError):
        F.Plan(32, 32, 5, 4, 3.0, stride=F.STRIDE_SLIDING)
    gc.collect()
    assert destroyed == ["handle"]
