// Column march (k_col.cuh) of FP32 stacks, and its geometry.
#include "k_col.cuh"

namespace fitrig {

template <int W>
static bool col_shape(int elem_bytes, StackGeom* g) {
  using S = ColShape<W>;
  g->w = W;
  g->R = S::kR;
  g->nseg = S::kSeg;
  g->TBX = S::kTBX;
  g->TBY = S::kTBY;
  g->BW = S::kBW;
  g->BH = S::kTBY * W;
  g->boxW = g->BW;
  g->aligned = true;
  g->col = true;
  g->threads = S::kThreads;
  g->stage_bytes = ((size_t)g->BW * g->BH * elem_bytes + 127) / 128 * 128;
  // about 40 KB of ring: with the partials, three to five CTAs per SM
  g->stages = std::max(3, std::min(6, (int)(40960 / g->stage_bytes)));
  g->smem_bytes = g->stages * g->stage_bytes +
                  (size_t)2 * g->TBX * g->TBY * S::kStride * sizeof(float4) + 8 * g->stages;
  return true;
}

bool col_geometry(int w, int elem_bytes, StackGeom* g) {
  switch (w) {
    case 7: return col_shape<7>(elem_bytes, g);
    case 9: return col_shape<9>(elem_bytes, g);
    case 10: return col_shape<10>(elem_bytes, g);
    case 11: return col_shape<11>(elem_bytes, g);
    case 12: return col_shape<12>(elem_bytes, g);
    case 13: return col_shape<13>(elem_bytes, g);
    case 14: return col_shape<14>(elem_bytes, g);
    case 15: return col_shape<15>(elem_bytes, g);
    default: return false;
  }
}

template cudaError_t launch_col<float, false>(const CUtensorMap*, const StackArgs&, cudaStream_t);
template cudaError_t launch_col<float, true>(const CUtensorMap*, const StackArgs&, cudaStream_t);

}  // namespace fitrig
