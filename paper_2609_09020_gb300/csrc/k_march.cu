// k_march.cu -- instantiations of the row-marching tcgen05 decode kernel
// (k_tcmarch.cuh): the 64-wide nets, int32 latent symbols.
#include "k_tcmarch.cuh"

namespace pic {
namespace {
const int d_c3[] = {14, 64, 64, 3};
const int d_c4[] = {16, 64, 64, 64, 3};
const int d_c5[] = {7, 64, 64, 3};
const int d_w64[] = {8, 64, 64, 64, 3};
}  // namespace

int march_kernels(KernelInfo* out, int cap) {
  const KernelInfo list[] = {
      make_march<7, 1, 3, ACT_RELU>("tc05_7x64x64x3_relu", d_c5),
      make_march<7, 2, 3, ACT_RELU>("tc05_14x64x64x3_relu", d_c3),
      make_march<8, 2, 4, ACT_GELU>("tc05_16x64x64x64x3_gelu", d_c4),
      make_march<8, 1, 4, ACT_RELU>("tc05_8x64x64x64x3_relu", d_w64),
  };
  const int n = static_cast<int>(sizeof(list) / sizeof(list[0]));
  int k = 0;
  for (; k < n && k < cap; ++k) out[k] = list[k];
  return k;
}

}  // namespace pic
