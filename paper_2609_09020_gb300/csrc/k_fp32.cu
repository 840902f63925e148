// k_fp32.cu -- instantiations of the fp32 CUDA-core decode kernel
// (k_fp32.cuh) for the decode workloads' architectures and the registry
// of all fp32 kernels that have one of their own.
#include "k_fp32.cuh"

namespace pic {

// Instantiations: the decode workloads' architectures, specialised at compile
// time; anything else runs on the generic kernel.
int fp32_kernels(KernelInfo* out, int cap) {
  const KernelInfo list[] = {
      make_fp32<1, 3, 4, 16, 16, 3, 0, ACT_RELU>("fp32_4x16x16x3_relu"),
      make_fp32<1, 3, 7, 40, 40, 3, 0, ACT_GELU>("fp32_7x40x40x3_gelu"),
      make_fp32<2, 3, 14, 64, 64, 3, 0, ACT_RELU>("fp32_14x64x64x3_relu"),
      make_fp32<2, 4, 16, 64, 64, 64, 3, ACT_GELU>("fp32_16x64x64x64x3_gelu"),
      make_fp32<1, 3, 7, 64, 64, 3, 0, ACT_RELU>("fp32_7x64x64x3_relu"),
      make_fp32<1, 3, 7, 64, 64, 3, 0, ACT_RELU, true>("fp32_7x64x64x3_relu_f32lat"),
  };
  const int n = static_cast<int>(sizeof(list) / sizeof(list[0]));
  int k = 0;
  for (; k < n && k < cap; ++k) out[k] = list[k];
  if (k < cap) k += fp32_kernels_sweep(out + k, cap - k);
  return k;
}

}  // namespace pic
