// k_tcmarch.cuh -- the decode kernel for 64-wide nets (PIC_PREC_FP16_TC): the
// row-marching feature pass of march.cuh in warps of its own, and the MLP g_s
// (Sec. 4.1) as a chain of tcgen05 MMAs over tiles of 128 pixels of one image
// row, operands and accumulators in tensor memory.
//
// Precision: fp16 weights as given, every activation (feature or hidden
// value) that an MMA reads as hi + lo fp16 terms (hi = truncated, lo = rounded
// remainder, ~22 bits, values below 131,008), fp32 accumulation; the output
// layer of nets with four layers on fp32 hidden values.
//
// Warps 0-15: four decoding groups of four, one tile at a time each (thread =
// pixel = tensor-memory lane): accumulator -> activation -> hi/lo split ->
// the next layer's operand, and RGB at the end.  Warps 16-23: two feature
// sets of four (one 32-column strip per warp); set s marches down its own
// run of tiles and hands them in turn to groups 2s and 2s + 1 through a
// shared-memory operand per group.  Warps 24-27: one MMA-issuing warp per
// group.
//
// Tensor memory: two 64-column regions per group.  An epilogue replaces each
// 16 accumulator columns it reads by the 8 columns of hi pairs and 8 of lo
// pairs made from them, so a layer's operand lies where its input's
// accumulator was, and the layer accumulates into the other region.  The
// next tile's layer 0 (operand from shared memory) goes into the region whose
// operand a tile's last layer reads, as soon as that layer is complete; its
// latency disappears behind the decoding warps' RGB.  (Queued right behind the
// last layer, without the wait, it would rest on issue order alone, which
// tensor-memory MMAs keep only with the same accumulator and shape; the wait
// costs 1 %: 64 images of 768x512 660 -> 668 us, 16-64-64-64-3 at 3840x2160
// 789 -> 795 us.)
//
// What bounds it: the chain of a tile's two (or more) remaining round trips
// with four tiles in flight -- tensor memory holds no more -- and, next to
// it, the splits.  An SM finishes a 7-64-64-3 tile every 1,070 cycles.
// Uncontended, a tile's chain is 200 (wait for layer 0) + 410 (epilogue) + 745
// (hidden layer, nine MMAs) + 340 + 395 (output layer) + 265 cycles; four
// of them share one tensor pipe (about 540 cycles a tile in such small
// batches) and the issue slots (720 warp instructions per 32 pixels, 0.73
// a cycle).  64 images of 768x512: 701 us with the per-tile kernel, whose
// decoding warps also staged and interpolated the features, 668 us here;
// 14-64-64-3 at 1361x2041, two images: 228 -> 175 us; 16-64-64-64-3 GELU at
// 3840x2160, bound by the GELUs: 1021 -> 789 us (990 without the GELU of
// pic_common.cuh and the operands in two parts).
// Both thin layers, or the output layer alone, by warp-level mma.sync on
// accumulator fragments (one round trip less) measured 740 and 779 us:
// mma.sync shares the tensor pipe with tcgen05, waits whenever that is busy,
// and takes about 6 cycles of the FMA pipe per instruction besides.  The
// output layer on the FP32 pipe: 762 us.
//
// Every wait is bounded; on timeout the status word is raised, the rest is
// skipped and tensor memory is still freed.
#pragma once

#include "march.cuh"
#include "pic_kernels.h"

namespace pic {
namespace {

constexpr int kGroups = 4;
constexpr int kSets = 2;  // feature sets
constexpr int kDecWarps = 4 * kGroups, kFeatWarps = 4 * kSets;

template <int L_, int C_, int NL_, int ACT_>
struct MarchNet {
  static constexpr int L = L_, C = C_, NL = NL_, N = 64, ACT = ACT_;
  using F = FeatLayout<L, C>;
  static constexpr int K1 = F::K1, HID = NL - 2;
  // Output layer of deep nets in fp32 by the decoding warps (output_layer),
  // inside the last hidden layer's epilogue: one round trip less, 192 FMAs a
  // pixel more.  16-64-64-64-3 GELU at 3840x2160: 795 -> 789 us; 8-64-64-64-3,
  // 24 images of 768x512: 366 -> 383 us; both keep the hidden values' range and
  // bits, as the per-tile kernels do.  (7-64-64-3 in fp32 measured 762 us with
  // 657 on the tensor pipe, where the per-tile kernel has it too.)
  static constexpr bool OUT_FP32 = NL >= 4;
  static constexpr int MMA_LAYERS = OUT_FP32 ? NL - 1 : NL;
  // An operand is handed to the tensor pipe in two parts, its first 16 columns
  // ahead of the rest: the MMAs of the first part, and the better part of
  // their round trip, run beside the rest of the epilogue.  16-64-64-64-3 GELU
  // at 3840x2160: 836 us in one part, 789 cut after 16 columns, 825 after 32,
  // 890 after 48; 7-64-64-3, one 768x512 image 20.4 -> 18.8 us, 64 of them
  // the same; 14-64-64-3, one image of 1361x2041 70.0 -> 66.7 us (all before
  // layer 0 waited for the last layer).
  static constexpr int CUT = 1;
  static constexpr int THREADS = 32 * (kDecWarps + kFeatWarps + kGroups);
  // 896 threads x 72 registers at launch, moved between the roles'
  // warpgroups (within the launch's total; below 96 the feature warps spill,
  // at 64 the decoding ones do not).
  static constexpr int MAXREG = 72, REG_ISSUE = 56, REG_FEAT = 96, REG_DECODE = 64;
  static_assert(32 * (REG_DECODE * kDecWarps + REG_FEAT * kFeatWarps + REG_ISSUE * kGroups) <= MAXREG * THREADS,
                "within the launch budget");
  static constexpr int CTRL = 512;
  // K-major operand tiles in the canonical no-swizzle layout (core matrices of
  // 8 rows x 16 bytes): layer 0's W, the hidden layers' W, the output's W
  // (16 rows, 3 used), and per layer a [rows][16] bias tile (b, 0..0) that
  // meets a constant A tile of rows (1, 0..0).
  static constexpr int B1_BYTES = N * K1 * 2, BH_BYTES = N * N * 2, BO_BYTES = OUT_FP32 ? 3 * N * 4 : 16 * N * 2, BB_BYTES = N * 16 * 2;
  static constexpr int OFF_ONES = CTRL;
  static constexpr int OFF_B1 = OFF_ONES + 128 * 16 * 2;
  static constexpr int OFF_BH = OFF_B1 + B1_BYTES;
  static constexpr int OFF_BO = OFF_BH + HID * BH_BYTES;
  static constexpr int OFF_BB = OFF_BO + BO_BYTES;  // bias tiles of layer 0 (unused with BIASCOL) and the hidden ones
  static constexpr int OFF_BOUT = OFF_BB + (1 + HID) * BB_BYTES;  // the output's 3 biases, fp32
  static constexpr int A1_BYTES = 128 * K1 * 2;
  static constexpr int PARAMS = N * (F::D0 + 1) + HID * N * (N + 1) + 3 * (N + 1);
  static constexpr int OFF_RAW = OFF_BOUT + 128;  // the weights as given (copy_raw)
  static constexpr int OFF_A1 = OFF_RAW + raw_bytes(PARAMS);
  static constexpr int OFF_FEAT = OFF_A1 + kGroups * A1_BYTES;
  static constexpr int SMEM = OFF_FEAT + kFeatWarps * F::FEAT_BYTES;
  static_assert(HID >= 1 && SMEM <= 227 * 1024, "shared memory of one CTA per SM");
};

// Byte offset of 16-byte chunk kc of row r in such a tile with K columns.
__host__ __device__ constexpr uint32_t kmaj_chunk(int r, int kc, int K) {
  return static_cast<uint32_t>((r >> 3) * (16 * K) + kc * 128 + (r & 7) * 16);
}

// Fills a [rows][K] tile; val(n, k).
template <int K, class V>
__device__ __forceinline__ void fill_tile(uint8_t* tile, int rows, int tid, int nthr, V val) {
  for (int e = tid; e < rows * (K / 2); e += nthr) {  // a pair of columns each
    const int n = e / (K / 2), k = 2 * (e - n * (K / 2));
    *reinterpret_cast<__half2*>(tile + kmaj_chunk(n, k >> 3, K) + (k & 7) * 2) =
        __halves2half2(val(n, k), val(n, k + 1));
  }
}

template <class Net>
__device__ __forceinline__ void load_weights_march(uint8_t* smem, const __half* w, int tid, int nthr) {
  using F = typename Net::F;
  constexpr int N = Net::N, D0 = F::D0;
  const __half zero = __float2half_rn(0.0f);
  const __half* b0 = w + N * D0;
  fill_tile<Net::K1>(smem + Net::OFF_B1, N, tid, nthr, [&](int n, int k) {
    const int i = F::input_of(k);
    return i >= 0 ? w[n * D0 + i] : (i == -1 && F::BIASCOL ? b0[n] : zero);
  });
  if constexpr (!F::BIASCOL)
    fill_tile<16>(smem + Net::OFF_BB, N, tid, nthr, [&](int n, int k) { return k == 0 ? b0[n] : zero; });
  const __half* p = b0 + N;
#pragma unroll
  for (int h = 0; h < Net::HID; ++h) {
    fill_tile<N>(smem + Net::OFF_BH + h * Net::BH_BYTES, N, tid, nthr,
                 [&](int n, int k) { return p[n * N + k]; });
    fill_tile<16>(smem + Net::OFF_BB + (1 + h) * Net::BB_BYTES, N, tid, nthr,
                  [&](int n, int k) { return k == 0 ? p[N * N + n] : zero; });
    p += N * N + N;
  }
  if constexpr (Net::OUT_FP32) {  // four inputs' weights of each colour in turn
    float* wo = reinterpret_cast<float*>(smem + Net::OFF_BO);
    for (int e = tid; e < 3 * N; e += nthr) {
      const int q = e / 12, c = (e - 12 * q) >> 2;
      wo[e] = __half2float(p[c * N + 4 * q + (e & 3)]);
    }
  } else {
    fill_tile<N>(smem + Net::OFF_BO, 16, tid, nthr, [&](int n, int k) { return n < 3 ? p[n * N + k] : zero; });
  }
  if (tid < 3) reinterpret_cast<float*>(smem + Net::OFF_BOUT)[tid] = __half2float(p[3 * N + tid]);
}

// Bounded mbarrier wait (as in k_tc.cuh): false if the phase does not
// complete within `limit` polls or another thread has given up.
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                           uint32_t limit) {
  if (tc::mbar_test_wait(bar, parity)) return true;
  for (uint32_t i = 0; i < limit; ++i) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 63u) {
      if (*abort_flag) return false;
      if (i > 4096) __nanosleep(64);
    }
  }
  *abort_flag = 1;
  atomicOr(status, 1);
  return false;
}

// One pixel's accumulator row in region t -> activation, hi/lo split -> the
// next layer's operand in place (per 16 columns: 8 of hi pairs, 8 of lo).
template <class Net, class Part>
__device__ __forceinline__ void epilogue(uint32_t t, Part part_done) {
  uint32_t acc[2][16];
  tc::tmem_ld16(t, acc[0]);
#pragma unroll
  for (int c = 0; c < Net::N / 16; ++c) {
    tc::tmem_ld_wait();
    if (c + 1 < Net::N / 16) tc::tmem_ld16(t + 16 * (c + 1), acc[(c + 1) & 1]);
    uint32_t hl[16];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      act_split<Net::ACT>(__uint_as_float(acc[c & 1][2 * q]), __uint_as_float(acc[c & 1][2 * q + 1]), hl[q], hl[8 + q]);
    tc::tmem_st16(t + 16 * c, hl);
    if (c + 1 == Net::CUT || c + 1 == Net::N / 16) {
      tc::tmem_st_wait();
      part_done(c + 1 == Net::CUT);
    }
  }
}

// One pixel's accumulator row in region t -> activation and output layer, in
// fp32 throughout: the hidden values stay as wide as the accumulators they come
// from (an fp16 pair would end at 131,008 and lose bits below 2^-3).
template <class Net>
__device__ __forceinline__ void output_layer(uint32_t t, const float4* wo, float (&rgb)[3]) {
  uint32_t acc[2][16];
  unsigned long long s[3] = {0ull, 0ull, 0ull};
  tc::tmem_ld16(t, acc[0]);
#pragma unroll
  for (int c = 0; c < Net::N / 16; ++c) {
    tc::tmem_ld_wait();
    if (c + 1 < Net::N / 16) tc::tmem_ld16(t + 16 * (c + 1), acc[(c + 1) & 1]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      unsigned long long h[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float a = __uint_as_float(acc[c & 1][4 * q + 2 * i]), b = __uint_as_float(acc[c & 1][4 * q + 2 * i + 1]);
        if constexpr (Net::ACT == ACT_GELU) h[i] = gelu_approx2(pack2(a, b));
        else h[i] = pack2(fmaxf(a, 0.0f), fmaxf(b, 0.0f));
      }
#pragma unroll
      for (int o = 0; o < 3; ++o) {
        const ulonglong2 w = reinterpret_cast<const ulonglong2*>(wo)[3 * (4 * c + q) + o];
        s[o] = fma2(w.y, h[1], fma2(w.x, h[0], s[o]));
      }
    }
  }
#pragma unroll
  for (int o = 0; o < 3; ++o) {
    const float2 v = unpack2(s[o]);
    rgb[o] = v.x + v.y;
  }
}

template <class Net, bool FL>
__global__ void __launch_bounds__(Net::THREADS) __maxnreg__(Net::MAXREG)
    march_decode_kernel(const DecodeParams p) {
  using F = typename Net::F;
  using namespace tc;
  constexpr int NL = Net::NL, N = Net::N, K1 = Net::K1;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = smem_addr(smem);
  // mbarriers, 8 bytes each, per group: feat_full (layer 0's operand written;
  // one arrival per feature warp), feat_free (read), acc0_full (layer 0
  // done), acc_full (another layer done), a_full and a2_full (the first and
  // second part of a hidden operand written; one arrival per decoding warp;
  // two barriers, since a warp may finish both parts before the issuing warp
  // looks for the first), drain (the issuing warp's end).
  const uint32_t bar_ff = sbase, bar_fe = sbase + 8 * kGroups, bar_c0 = sbase + 16 * kGroups,
                 bar_c = sbase + 24 * kGroups, bar_a = sbase + 32 * kGroups, bar_a2 = sbase + 40 * kGroups,
                 bar_drain = sbase + 48 * kGroups;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + 56 * kGroups);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 2);
  static_assert(56 * kGroups + 16 <= Net::CTRL, "control block");

  if (threadIdx.x == 0) {
    for (int w = 0; w < kGroups; ++w) {
      mbar_init(bar_ff + 8 * w, 4);
      mbar_init(bar_fe + 8 * w, 1);
      mbar_init(bar_c0 + 8 * w, 1);
      mbar_init(bar_c + 8 * w, 1);
      mbar_init(bar_a + 8 * w, 4);
      mbar_init(bar_a2 + 8 * w, 4);
      mbar_init(bar_drain + 8 * w, 1);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kDecWarps + kFeatWarps) {
    tmem_alloc(smem_addr(tmem_slot), 512);
    tmem_relinquish();
  }
  if (threadIdx.x < 256) {
    const int row = threadIdx.x >> 1, kc = threadIdx.x & 1;
    sts128(sbase + Net::OFF_ONES + kmaj_chunk(row, kc, 16), kc == 0 ? 0x00003C00u : 0u, 0u, 0u, 0u);
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // Balanced contiguous ranges of tiles (image, column block, row; rows
  // fastest); within an image, each feature set takes half of the range and
  // its two groups every other tile of that.
  const long long t_begin = blockIdx.x * p.total_tiles / gridDim.x;
  const long long t_end = (blockIdx.x + 1LL) * p.total_tiles / gridDim.x;
  auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
    return __all_sync(0xffffffffu, wait_phase(bar, parity, abort_flag, p.status, p.spin_limit));
  };

  if (warp < kDecWarps) {
    setmaxnreg_dec<Net::REG_DECODE>();
    const __half* wts = static_cast<const __half*>(p.weights);
    const float* bout = reinterpret_cast<const float*>(smem + Net::OFF_BOUT);
    const int w = warp >> 2, par = w & 1;
    // the two regions of this warp's lanes, XORed by 64 columns
    const uint32_t t_base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + static_cast<uint32_t>(w * 2 * N);
    const uint32_t my_c0 = bar_c0 + 8 * w, my_c = bar_c + 8 * w, my_a = bar_a + 8 * w, my_a2 = bar_a2 + 8 * w;
    uint32_t c0_phase = 0, c_phase = 0, reg = 0;

    for (long long seg = t_begin; seg < t_end;) {
      const int b = static_cast<int>(seg / p.tiles_per_image);
      const long long first = static_cast<long long>(b) * p.tiles_per_image;
      const long long seg_end = min(t_end, first + p.tiles_per_image);
      __syncthreads();  // all MMAs and reads of the previous image's weights are done
      const __half* const wimg = wts + b * p.params_per_image;
      copy_raw(smem + Net::OFF_RAW, wimg, Net::PARAMS, threadIdx.x, 32 * kDecWarps);
      cp_async_wait_all();
      named_bar(1, 32 * kDecWarps);  // the decoding warps: every copy has landed
      load_weights_march<Net>(smem, reinterpret_cast<const __half*>(smem + Net::OFF_RAW) + raw_skip(wimg),
                              threadIdx.x, 32 * kDecWarps);
      fence_async_smem();
      __syncthreads();
      float* const out_img = static_cast<float*>(p.out) + static_cast<long long>(b) * 3 * p.H * p.W;
      const long long n = seg_end - seg;
      const long long s0 = n * (w >> 1) / kSets;
      const int tiles = (static_cast<int>(n * ((w >> 1) + 1) / kSets - s0) + 1 - par) / 2;
      // the tile being decoded: row y, this lane's column x
      int y, x;
      {
        const long long t = seg - first + s0 + par;
        const int col = static_cast<int>(t / p.H);
        y = static_cast<int>(t - static_cast<long long>(col) * p.H);
        x = col * 128 + (warp & 3) * 32 + lane;
      }
      bool ok = true;
      for (int i = 0; i < tiles; ++i) {
#pragma unroll
        for (int k = 0; k < Net::MMA_LAYERS - 1; ++k) {
          ok = k == 0 ? wait(my_c0, c0_phase) : wait(my_c, c_phase);
          if (!ok) break;
          if (k == 0) c0_phase ^= 1u;
          else c_phase ^= 1u;
          tc_fence_after();
          epilogue<Net>(t_base + reg, [&](bool first) {
            tc_fence_before();
            __syncwarp();
            // p.test_fault (tests of the bounded waits only): one warp of each
            // of CTA 0's groups withholds its first arrival
            if (lane == 0 &&
                !(p.test_fault && blockIdx.x == 0 && (warp & 3) == 0 && seg == t_begin && i == 0 && k == 0 && first))
              mbar_arrive(first ? my_a : my_a2);
          });
          reg ^= N;
        }
        if (!ok) break;
        ok = wait(my_c, c_phase);
        if (!ok) break;
        c_phase ^= 1u;
        tc_fence_after();
        float rgb[3];
        if constexpr (Net::OUT_FP32) {
          output_layer<Net>(t_base + reg, reinterpret_cast<const float4*>(smem + Net::OFF_BO), rgb);
        } else {
          uint32_t o[4];
          tmem_ld4(t_base + reg, o);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 3; ++c) rgb[c] = __uint_as_float(o[c]);
        }
        tc_fence_before();
        reg ^= N;  // the next tile's layer 0 goes to the other region
        write_rgb(p, out_img, b, y, x, rgb[0] + bout[0], rgb[1] + bout[1], rgb[2] + bout[2]);
        y += 2;
        while (y >= p.H) {
          y -= p.H;
          x += 128;
        }
      }
      seg = seg_end;
    }
  } else if (warp < kDecWarps + kFeatWarps) {
    setmaxnreg_inc<Net::REG_FEAT>();
    const int set = (warp - kDecWarps) >> 2, strip = warp & 3;
    Strip<Net::L, Net::C, FL> st;
    st.init(sbase + Net::OFF_FEAT + (warp - kDecWarps) * F::FEAT_BYTES, lane);
    uint32_t free_phase = 3;  // bit q: parity of feat_free of the set's group q (both start free)
    for (long long seg = t_begin; seg < t_end;) {
      const int b = static_cast<int>(seg / p.tiles_per_image);
      const long long first = static_cast<long long>(b) * p.tiles_per_image;
      const long long seg_end = min(t_end, first + p.tiles_per_image);
      const long long n = seg_end - seg;
      long long t = seg - first + n * set / kSets;
      const long long te = seg - first + n * (set + 1) / kSets;
      st.lat = p.latents + b * p.lat_per_image;
      st.steps = p.steps + b * Net::L;
      int rows = 0, q = 0;
      auto start_run = [&]() {
        const int col = static_cast<int>(t / p.H);
        const int y0 = static_cast<int>(t - static_cast<long long>(col) * p.H);
        rows = static_cast<int>(min(static_cast<long long>(p.H - y0), te - t));
        cp_async_wait_all();  // the copies of the run before
        st.start(p, col * 128 + strip * 32 + lane, y0, lane);
      };
      __syncthreads();
      if (t < te) start_run();  // while the decoding warps load the weights
      __syncthreads();
      for (; t < te; ++t, q ^= 1) {
        if (rows == 0) start_run();
        --rows;
        const int g = 2 * set + q;
        if (!wait(bar_fe + 8 * g, (free_phase >> q) & 1u)) break;
        free_phase ^= 1u << q;
        const uint32_t a1 = sbase + Net::OFF_A1 + g * Net::A1_BYTES;
        st.features(p, [&](int kc) { return a1 + kmaj_chunk(strip * 32 + lane, kc, K1); }, lane, rows > 0);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_ff + 8 * g);
      }
      seg = seg_end;
    }
    cp_async_wait_all();  // copies still in flight land before shared memory goes
  } else {
    setmaxnreg_dec<Net::REG_ISSUE>();
    const int w = warp - kDecWarps - kFeatWarps, par = w & 1;
    const uint32_t t_base = tmem + static_cast<uint32_t>(w * 2 * N);
    const uint64_t dA1 = smem_desc(sbase + Net::OFF_A1 + w * Net::A1_BYTES, 128, 16 * K1);
    const uint64_t dB1 = smem_desc(sbase + Net::OFF_B1, 128, 16 * K1);
    const uint64_t dBH = smem_desc(sbase + Net::OFF_BH, 128, 16 * N);
    const uint64_t dBO = smem_desc(sbase + Net::OFF_BO, 128, 16 * N);
    const uint64_t dBB = smem_desc(sbase + Net::OFF_BB, 128, 16 * 16);
    const uint64_t dONES = smem_desc(sbase + Net::OFF_ONES, 128, 16 * 16);
    constexpr uint32_t id_hidden = idesc_f16(128, N), id_out = idesc_f16(128, 16);
    constexpr uint64_t kStep = 256 >> 4;  // one K step (16 fp16)
    const uint32_t my_ff = bar_ff + 8 * w, my_fe = bar_fe + 8 * w, my_c0 = bar_c0 + 8 * w, my_c = bar_c + 8 * w,
                   my_a = bar_a + 8 * w, my_a2 = bar_a2 + 8 * w;
    uint32_t a_phase = 0, c_phase = 0, ff_phase = 0, reg = 0;
    // layer 0 of the group's next tile into region reg
    auto first_layer = [&]() -> bool {
      if (!wait(my_ff, ff_phase)) return false;
      ff_phase ^= 1u;
      if (elect_one()) {
        tc_fence_after();
        if constexpr (!F::BIASCOL) mma_f16(t_base + reg, dONES, dBB, id_hidden, 0);
#pragma unroll
        for (int s = 0; s < K1 / 16; ++s)
          mma_f16(t_base + reg, dA1 + s * kStep, dB1 + s * kStep, id_hidden, s > 0 || !F::BIASCOL);
        mma_commit(my_fe);
        mma_commit(my_c0);
      }
      __syncwarp();
      return true;
    };
    for (long long seg = t_begin; seg < t_end;) {
      const int b = static_cast<int>(seg / p.tiles_per_image);
      const long long seg_end = min(t_end, (b + 1LL) * p.tiles_per_image);
      __syncthreads();  // all MMAs of the previous image are complete
      __syncthreads();  // the decoding warps have loaded this image's weights
      const long long n = seg_end - seg;
      const long long s0 = n * (w >> 1) / kSets;
      const int tiles = (static_cast<int>(n * ((w >> 1) + 1) / kSets - s0) + 1 - par) / 2;
      bool ok = tiles > 0 && first_layer();
      for (int i = 0; i < tiles && ok; ++i) {
        for (int k = 1; k < Net::MMA_LAYERS; ++k) {
          const uint32_t ta = t_base + reg, d = t_base + (reg ^ N);
          reg ^= N;
          const bool out_layer = k == NL - 1;
          const uint64_t db = out_layer ? dBO : dBH + (k - 1) * (Net::BH_BYTES >> 4);
          const uint32_t id = out_layer ? id_out : id_hidden;
#pragma unroll
          for (int part = 0; part < 2; ++part) {
            ok = wait(part == 0 ? my_a : my_a2, a_phase);
            if (!ok) break;
            if (elect_one()) {
              tc_fence_after();
              // bias: [1 0..0] x [b 0..0]
              if (part == 0 && !out_layer) mma_f16(d, dONES, dBB + k * (Net::BB_BYTES >> 4), id, 0);
              // the lo terms first: each MMA rounds the running sum, which is
              // small until the hi terms come
#pragma unroll
              for (int s = part ? Net::CUT : 0; s < (part ? N / 16 : Net::CUT); ++s)
                mma_f16_ta(d, ta + 16 * s + 8, db + s * kStep, id, s > 0 || !out_layer);
#pragma unroll
              for (int s = part ? Net::CUT : 0; s < (part ? N / 16 : Net::CUT); ++s)
                mma_f16_ta(d, ta + 16 * s, db + s * kStep, id, 1);
              if (part == 1) mma_commit(my_c);
            }
            __syncwarp();
          }
          if (!ok) break;
          a_phase ^= 1u;
          c_phase ^= 1u;
        }
        reg ^= N;  // the region of the last layer's operand, free once that layer is complete
        if (ok && i + 1 < tiles) ok = wait(my_c, c_phase ^ 1u) && first_layer();
      }
      seg = seg_end;
    }
    if (elect_one()) {  // every MMA this thread issued completes before the memory goes
      const uint32_t drain = bar_drain + 8 * w;
      mma_commit(drain);
      int dummy = 0;
      wait_phase(drain, 0, reinterpret_cast<volatile int*>(&dummy), p.status, kWaitPolls);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kDecWarps + kFeatWarps) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <int L, int C, int NL, int ACT, bool FL = false>
KernelInfo make_march(const char* name, const int* dims) {
  using Net = MarchNet<L, C, NL, ACT>;
  KernelInfo k{};
  k.name = name;
  k.precision = 1;
  k.latent_format = FL ? 1 : 0;
  k.C = C;
  k.n_layers = NL;
  for (int i = 0; i <= NL; ++i) k.dims[i] = dims[i];
  k.act = ACT;
  k.threads = Net::THREADS;
  k.regs_at_launch = Net::MAXREG;
  k.tile_px = kTcTile;
  k.smem_bytes = Net::SMEM;
  k.march = 1;
  k.fn = reinterpret_cast<const void*>(&march_decode_kernel<Net, FL>);
  return k;
}

}  // namespace
}  // namespace pic
