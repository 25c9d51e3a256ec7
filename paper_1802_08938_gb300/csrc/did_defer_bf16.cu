// Instantiations of the read-only sweep kernel: bfloat16 residual.
#include "did_defer_kernel.cuh"

namespace did {
namespace defer_impl {

template <int NR>
static const void* pick(int CW) {
  if (NR <= 4) {
    if (CW == 4) return reinterpret_cast<const void*>(&defer_kernel<NR, NR <= 4 ? 4 : 1, true>);
    if (CW == 2) return reinterpret_cast<const void*>(&defer_kernel<NR, NR <= 4 ? 2 : 1, true>);
  }
  return CW == 1 ? reinterpret_cast<const void*>(&defer_kernel<NR, 1, true>) : nullptr;
}

const void* defer_func_bf16(int NR, int CW) {
  switch (NR) {
    case 1: return pick<1>(CW);
    case 2: return pick<2>(CW);
    case 3: return pick<3>(CW);
    case 4: return pick<4>(CW);
    case 5: return pick<5>(CW);
  }
  return nullptr;
}

}  // namespace defer_impl
}  // namespace did
