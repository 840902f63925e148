// k_fp32_any.cu -- the fp32 CUDA-core kernels for nets without one of their own
// (k_fp32.cuh), in a module of their own: a process that decodes other nets
// does not load them.
#include "k_fp32.cuh"

namespace pic {

namespace {
template <bool FL>
const void* any_fn(int t2) {
  if (t2 <= 2) return reinterpret_cast<const void*>(&fp32_any_kernel<2, FL>);
  if (t2 <= 5) return reinterpret_cast<const void*>(&fp32_any_kernel<5, FL>);
  if (t2 <= 8) return reinterpret_cast<const void*>(&fp32_any_kernel<8, FL>);
  return reinterpret_cast<const void*>(&fp32_any_kernel<16, FL>);
}
}  // namespace

KernelInfo fp32_generic_kernel_info(int latent_format, int n_layers, const int* dims, long long params, int max_smem) {
  KernelInfo k{};
  k.name = latent_format ? "fp32_generic_f32lat" : "fp32_generic";
  k.precision = 0;
  k.latent_format = latent_format ? 1 : 0;
  k.generic = 1;
  k.threads = kThreads;
  k.tile_px = kThreads;
  int t2 = 1;
  const long long tiled = 4 * any_smem_floats(n_layers, dims, &t2);
  if (tiled <= max_smem) {
    k.smem_bytes = static_cast<int>(tiled);
    k.fn = latent_format ? any_fn<true>(t2) : any_fn<false>(t2);
  } else {
    k.smem_bytes = params * 4 <= max_smem ? static_cast<int>(params * 4) : max_smem + 1;  // refused by the caller
    k.fn = latent_format ? reinterpret_cast<const void*>(&fp32_flat_kernel<true>)
                        : reinterpret_cast<const void*>(&fp32_flat_kernel<false>);
  }
  k.smem_attr = max_smem;  // one function serves nets of many sizes
  return k;
}

}  // namespace pic
