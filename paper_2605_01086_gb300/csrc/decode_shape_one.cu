// The shape kernel (decode_shape.cuh) of plans whose domains all have one compiled
// form: 16 warps, 12 for N = 128 (whose larger transforms would spill 132 and 440
// bytes a thread at 16; at 12 (128, 64) spills 24), two output tiles per warp.
#include "decode_shape.cuh"

namespace fptc {

void *shape_kernel_one(uint32_t form) {
#define FPTC_ONE(N, K) \
  case (N << 8 | K): \
    return reinterpret_cast<void *>(&k_decode_shape<N == 128 ? 12 : 16, 2, kShapeCompiled, (N << 8 | K)>);
  switch (form) {
    FPTC_ONE(4, 4)
    FPTC_ONE(8, 8)
    FPTC_ONE(16, 4)
    FPTC_ONE(16, 8)
    FPTC_ONE(16, 16)
    FPTC_ONE(32, 8)
    FPTC_ONE(32, 16)
    FPTC_ONE(32, 32)
    FPTC_ONE(64, 16)
    FPTC_ONE(64, 32)
    FPTC_ONE(64, 64)
    FPTC_ONE(128, 32)
    FPTC_ONE(128, 64)
  }
#undef FPTC_ONE
  return nullptr;
}

}  // namespace fptc
