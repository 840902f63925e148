// k_march_f32lat.cu -- the row-marching tcgen05 decode kernel
// (k_tcmarch.cuh) for fp32 latents (PIC_LATENT_FP32, the inverse DCT stage's
// output).
#include "k_tcmarch.cuh"

namespace pic {
namespace {
const int d_c3[] = {14, 64, 64, 3};
const int d_c4[] = {16, 64, 64, 64, 3};
const int d_c5[] = {7, 64, 64, 3};
}  // namespace

int march_kernels_f32lat(KernelInfo* out, int cap) {
  const KernelInfo list[] = {
      make_march<7, 1, 3, ACT_RELU, true>("tc05_7x64x64x3_relu_f32lat", d_c5),
      make_march<7, 2, 3, ACT_RELU, true>("tc05_14x64x64x3_relu_f32lat", d_c3),
      make_march<8, 2, 4, ACT_GELU, true>("tc05_16x64x64x64x3_gelu_f32lat", d_c4),
  };
  const int n = static_cast<int>(sizeof(list) / sizeof(list[0]));
  int k = 0;
  for (; k < n && k < cap; ++k) out[k] = list[k];
  return k;
}

}  // namespace pic
