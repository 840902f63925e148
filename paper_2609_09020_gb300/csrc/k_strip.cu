// k_strip.cu -- instantiations of the narrow nets' decode kernel
// (k_strip.cuh): the decode workloads' 16- and 40-wide nets, both latent
// formats, and the width ablation's 8-w-w-w-3 for w = 8, 16, 32 (Sec. 4.3).
#include "k_strip.cuh"

namespace pic {
namespace {
const int d_c1[] = {4, 16, 16, 3};
const int d_c2[] = {7, 40, 40, 3};
const int d_w8[] = {8, 8, 8, 8, 3};
const int d_w16[] = {8, 16, 16, 16, 3};
const int d_w32[] = {8, 32, 32, 32, 3};
}  // namespace

int strip_kernels(KernelInfo* out, int cap) {
  const KernelInfo list[] = {
      make_strip<4, 1, 3, 16, ACT_RELU>("tc05_4x16x16x3_relu", d_c1),
      make_strip<7, 1, 3, 40, ACT_GELU>("tc05_7x40x40x3_gelu", d_c2),
      make_strip<4, 1, 3, 16, ACT_RELU, true>("tc05_4x16x16x3_relu_f32lat", d_c1),
      make_strip<7, 1, 3, 40, ACT_GELU, true>("tc05_7x40x40x3_gelu_f32lat", d_c2),
      make_strip<8, 1, 4, 8, ACT_RELU>("tc05_8x8x8x8x3_relu", d_w8),
      make_strip<8, 1, 4, 16, ACT_RELU>("tc05_8x16x16x16x3_relu", d_w16),
      make_strip<8, 1, 4, 32, ACT_RELU>("tc05_8x32x32x32x3_relu", d_w32),
  };
  const int n = static_cast<int>(sizeof(list) / sizeof(list[0]));
  int k = 0;
  for (; k < n && k < cap; ++k) out[k] = list[k];
  return k;
}

}  // namespace pic
