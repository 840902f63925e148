// k_strip.cuh -- the decode kernel for narrow nets (every hidden layer at
// most 40 wide), PIC_PREC_FP16_TC: one warp decodes a strip of 32 pixel
// columns row after row (march.cuh), the whole MLP g_s (Sec. 4.1) with
// warp-level mma.sync whose accumulators stay in registers: the accumulator
// fragment of one layer is, after activation and hi/lo split, the operand
// fragment of the next.
//
// Nothing is handed from warp to warp, so a row has no barrier and no round
// trip through tensor memory, which is what bounded the per-tile tcgen05
// kernel on these nets (two to four dependent round trips of 360 cycles and
// more per tile, four tiles in flight).  mma.sync runs at a quarter of
// tcgen05's rate (8.2 cycles per m16n8k16 and sub-partition) and each one
// takes about 6 cycles of the FMA pipe besides, so its share grows with the
// square of the width; up to 40 it pays.  64 images of 768x512, the per-tile
// kernel's time first: 8-8-8-8-3 573 -> 283 us, 8-16-16-16-3 636 -> 403 us,
// 8-32-32-32-3 790 -> 771 us; one 7-40-40-3 GELU image with L2 flushed 37.5 ->
// 31.4 us, one 256x256 4-16-16-3 image 10.9 -> 8.8 us.  Bound by issue, latency
// and the L1 data pipe (74 % of its rate): 364 warp instructions per 32 pixels
// of the 16-wide net at 0.60 a cycle.
//
// Precision is that of the per-tile tcgen05 kernels: fp16 weights as given, every
// activation that an MMA reads as hi + lo fp16 terms (~22 bits, values below
// 131,008), fp32 accumulation, and the output layer of all but 7-40-40-3 on
// fp32 hidden values; biases enter as the accumulators' start values or, where operand A has room, as
// the weight of a constant-1 column.
#pragma once

#include "march.cuh"
#include "pic_kernels.h"

namespace pic {
namespace {

constexpr int kStripWarps = 4;
constexpr int kStripThreads = 32 * kStripWarps;

constexpr int kOutRow = 12;  // output weights of a lane's two neurons of a tile: 2 x 3, each twice

template <int L_, int C_, int NL_, int N_, int ACT_>
struct StripNet {
  static constexpr int L = L_, C = C_, NL = NL_, N = N_, ACT = ACT_;
  using F = FeatLayout<L, C>;
  static constexpr int J = N / 8;            // output tiles of a hidden layer = blocks of the next
  static constexpr int NB1 = F::K1 / 8;
  static constexpr int HID = NL - 2;         // hidden x hidden layers
  static constexpr int W1_WORDS = frag_words(J, NB1);
  static constexpr int WH_WORDS = frag_words(J, J);
  // Output layer in fp32 (output_layer), as the per-tile kernels have it for
  // nets at most 32 wide or with four layers; 7-40-40-3 alone is left, whose
  // hidden values go to the tensor pipe as pairs there too (24 images of
  // 768x512: 476 us, 490 in fp32).
  static constexpr bool OUT_FP32 = N <= 32 || NL >= 4;
  static constexpr int WO_WORDS = OUT_FP32 ? 4 * J * kOutRow + 4 : frag_words(1, J);
  static constexpr int OFF_H = W1_WORDS, OFF_O = OFF_H + HID * WH_WORDS, OFF_B = OFF_O + WO_WORDS;
  // Weight fragments, two registers a lane each.  Up to width 16 they fit into
  // registers for an image's rows (24 images of 768x512: width 8 109 -> 104
  // us, width 16 144 -> 139.5 us with the output layer among them, of shared
  // memory's 102 wavefronts a row 14); the next wider net has 20, which spill.
  static constexpr int FRAGS = OFF_O / 64;
  static constexpr bool HELD = FRAGS <= 8;
  // bias tables (load_bias): layer 0 (BIASCOL nets: zeros), hidden layers, output (unless in fp32)
  static constexpr int B_WORDS = ((1 + HID) * J + (OUT_FP32 ? 0 : 1)) * 16;
  static constexpr int PARAMS = N * (F::D0 + 1) + HID * N * (N + 1) + 3 * (N + 1);
  static constexpr int OFF_RAW = round_to((OFF_B + B_WORDS) * 4, 128);  // the weights as given (copy_raw)
  static constexpr int W_BYTES = OFF_RAW + raw_bytes(PARAMS);
  static constexpr int OFF_A = F::FEAT_BYTES, OFF_OUT = OFF_A + F::A_BYTES;
  static constexpr int WARP_BYTES = OFF_OUT + (OUT_FP32 ? 0 : kOutBytes);
  static constexpr int SMEM = W_BYTES + kStripWarps * WARP_BYTES;
  // CTAs per SM: five hide more latency where their 96 registers do (width
  // 8: 301 -> 274 us); wider nets spill there (width 16 equal, 32 and 40
  // 6 % slower).
  static constexpr int MINB = N <= 8 ? 5 : 4;
  static_assert(N % 8 == 0 && N <= 40 && NL >= 3, "narrow nets with at least two hidden layers");
};

template <class Net>
__device__ __forceinline__ void load_weights_strip(uint32_t* sm, const __half* w, int tid) {
  using F = typename Net::F;
  constexpr int N = Net::N, D0 = F::D0;
  const __half zero = __float2half_rn(0.0f);
  const __half* b0 = w + N * D0;
  fill_frags<Net::J, Net::NB1>(sm, tid, kStripThreads, [&](int n, int k) {
    const int i = F::input_of(k);
    return i >= 0 ? w[n * D0 + i] : (i == -1 && F::BIASCOL ? b0[n] : zero);
  });
  float* bias = reinterpret_cast<float*>(sm + Net::OFF_B);
  fill_bias(bias, Net::J, tid, kStripThreads,
            [&](int n) { return F::BIASCOL ? 0.0f : __half2float(b0[n]); });
  const __half* p = b0 + N;
#pragma unroll
  for (int h = 0; h < Net::HID; ++h) {
    fill_frags<Net::J, Net::J>(sm + Net::OFF_H + h * Net::WH_WORDS, tid, kStripThreads,
                               [&](int n, int k) { return p[n * N + k]; });
    fill_bias(bias + (1 + h) * 16 * Net::J, Net::J, tid, kStripThreads,
              [&](int n) { return __half2float(p[N * N + n]); });
    p += N * N + N;
  }
  if constexpr (Net::OUT_FP32) {  // [tile j][t][neuron 8j + 2t, the next][r r g g b b], then the biases
    float* wo = reinterpret_cast<float*>(sm + Net::OFF_O);
    for (int e = tid; e < 4 * Net::J * kOutRow; e += kStripThreads) {
      const int jt = e / kOutRow, q = e - jt * kOutRow, h = q / 6;
      wo[e] = __half2float(p[(q - 6 * h) / 2 * N + 2 * jt + h]);
    }
    if (tid < 3) wo[4 * Net::J * kOutRow + tid] = __half2float(p[3 * N + tid]);
  } else {
    fill_frags<1, Net::J>(sm + Net::OFF_O, tid, kStripThreads,
                          [&](int n, int k) { return n < 3 ? p[n * N + k] : zero; });
    fill_bias(bias + (1 + Net::HID) * 16 * Net::J, 1, tid, kStripThreads,
              [&](int n) { return n < 3 ? __half2float(p[3 * N + n]) : 0.0f; });
  }
}

// d = A B + bias for both pixel halves, A the hi and lo fragments of the previous
// layer's J tiles (blocks 0 .. J-1 hi, J .. 2J-1 lo, both against the same
// weights), B the fragments from the f0-th on (JO output tiles of J blocks).
template <int J, int JO, class Frag>
__device__ __forceinline__ void layer(const Frag& frag, int f0, const float* bias4, int lane, const uint32_t (&hi)[2][J][2],
                                      const uint32_t (&lo)[2][J][2], float (&d)[2][JO][4]) {
  constexpr int NB2 = (J + 1) / 2;
#pragma unroll
  for (int j = 0; j < JO; ++j) {
    uint32_t b[2 * NB2];
    float c[4];
    load_bias(bias4, j, lane, c);
#pragma unroll
    for (int i2 = 0; i2 < NB2; ++i2) {
      const uint2 v = frag(f0 + j * NB2 + i2);
      b[2 * i2] = v.x;
      b[2 * i2 + 1] = v.y;
    }
#pragma unroll
    for (int s = J - 1; s >= 0; --s) {  // K steps of 16 = 2 blocks: the lo terms first (see k_tcmarch.cuh)
      const int p = 2 * s, q = 2 * s + 1;
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const uint32_t a[4] = {p < J ? hi[m][p % J][0] : lo[m][p % J][0], p < J ? hi[m][p % J][1] : lo[m][p % J][1],
                               q < J ? hi[m][q % J][0] : lo[m][q % J][0], q < J ? hi[m][q % J][1] : lo[m][q % J][1]};
        if (s == J - 1) hmma(d[m][j], a, b[p % J], b[q % J], c);
        else hmma(d[m][j], a, b[p % J], b[q % J], d[m][j]);
      }
    }
  }
}

template <int ACT, int J>
__device__ __forceinline__ void split_acc(const float (&d)[2][J][4], uint32_t (&hi)[2][J][2],
                                          uint32_t (&lo)[2][J][2]) {
#pragma unroll
  for (int j = 0; j < J; ++j)
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int h = 0; h < 2; ++h) act_split<ACT>(d[m][j][2 * h], d[m][j][2 * h + 1], hi[m][j][h], lo[m][j][h]);
}

// Activation and output layer in fp32: the hidden values stay as wide as the
// accumulators they come from (an fp16 pair would end at 131,008 and lose bits
// below 2^-3).  Each lane sums over its neurons (8j + 2t, 8j + 2t + 1 with t =
// lane % 4) for its four pixels, in pairs of the two pixel rows of a fragment;
// two exchanges add up the four lanes' sums and leave lane 4g + t with pixel
// out_pixel(lane) = 16 (t & 1) + 8 (t >> 1) + g of the strip.  Against split
// pairs and one MMA a tile, which cost no exchange, 24 images of 768x512:
// 8-8-8-8-3 104 -> 112 us, 8-16-16-16-3 143 -> 159 us, 8-32-32-32-3 285 -> 297
// us.  The exchanges are 8 us of it; weights in registers, sums in pairs of
// neurons, or the exchanges finished beside the next row's features are within
// 2 % of this.
__device__ __forceinline__ int out_pixel(int lane) { return 16 * (lane & 1) + 4 * (lane & 2) + (lane >> 2); }

template <class Net>
__device__ __forceinline__ void output_layer(const float* wo, int lane, const float (&d)[2][Net::J][4], float (&rgb)[3]) {
  constexpr int J = Net::J;
  auto act = [](float a, float b) {
    if constexpr (Net::ACT == ACT_GELU) return gelu_approx2(pack2(a, b));
    else return pack2(fmaxf(a, 0.0f), fmaxf(b, 0.0f));
  };
  unsigned long long s[2][3];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const ulonglong2* w = reinterpret_cast<const ulonglong2*>(wo + (4 * j + (lane & 3)) * kOutRow);
    const ulonglong2 w0 = w[0], w1 = w[1], w2 = w[2];
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const unsigned long long a = act(d[m][j][0], d[m][j][2]), b = act(d[m][j][1], d[m][j][3]);
      s[m][0] = fma2(w1.y, b, j == 0 ? mul2(w0.x, a) : fma2(w0.x, a, s[m][0]));
      s[m][1] = fma2(w2.x, b, j == 0 ? mul2(w0.y, a) : fma2(w0.y, a, s[m][1]));
      s[m][2] = fma2(w2.y, b, j == 0 ? mul2(w1.x, a) : fma2(w1.x, a, s[m][2]));
    }
  }
  const float* bias = wo + 4 * J * kOutRow;
#pragma unroll
  for (int o = 0; o < 3; ++o) {
    const unsigned long long keep = lane & 1 ? s[1][o] : s[0][o], send = lane & 1 ? s[0][o] : s[1][o];
    const float2 v = unpack2(add2(keep, __shfl_xor_sync(0xffffffffu, send, 1)));
    rgb[o] = (lane & 2 ? v.y : v.x) + __shfl_xor_sync(0xffffffffu, lane & 2 ? v.x : v.y, 2) + bias[o];
  }
}

template <class Net, bool FL>
__global__ void __launch_bounds__(kStripThreads, Net::MINB) strip_decode_kernel(const DecodeParams p) {
  using F = typename Net::F;
  constexpr int J = Net::J, HID = Net::HID;
  extern __shared__ __align__(128) uint8_t smem[];
  uint32_t* const sw = reinterpret_cast<uint32_t*>(smem);
  const float* const bias = reinterpret_cast<const float*>(sw + Net::OFF_B);
  const float* const wo = reinterpret_cast<const float*>(sw + Net::OFF_O);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t mine = tc::smem_addr(smem) + Net::W_BYTES + warp * Net::WARP_BYTES;
  Strip<Net::L, Net::C, FL> st;
  st.init(mine, lane);

  // balanced contiguous ranges of strip rows (image, strip, row; rows fastest)
  const long long t_begin = blockIdx.x * p.total_tiles / gridDim.x;
  const long long t_end = (blockIdx.x + 1LL) * p.total_tiles / gridDim.x;
  const __half* wts = static_cast<const __half*>(p.weights);

  for (long long seg = t_begin; seg < t_end;) {
    const int b = static_cast<int>(seg / p.tiles_per_image);
    const long long first = static_cast<long long>(b) * p.tiles_per_image;
    const long long seg_end = min(t_end, first + p.tiles_per_image);
    st.lat = p.latents + b * p.lat_per_image;
    st.steps = p.steps + b * Net::L;
    float* const out_img = static_cast<float*>(p.out) + static_cast<long long>(b) * 3 * p.H * p.W;
    // this warp's share of the segment
    const long long n = seg_end - seg;
    long long t = seg - first + n * warp / kStripWarps;
    const long long te = seg - first + n * (warp + 1) / kStripWarps;
    int col = 0, y0 = 0;
    auto start_run = [&]() {
      col = static_cast<int>(t / p.H);
      y0 = static_cast<int>(t - static_cast<long long>(col) * p.H);
      st.start(p, col * 32 + lane, y0, lane);
    };
    // the weights' copy and the first run's loads are in flight together
    tc::cp_async_wait_all();
    __syncthreads();  // the previous image's weights have been read
    const __half* const w = wts + b * p.params_per_image;
    copy_raw(smem + Net::OFF_RAW, w, Net::PARAMS, threadIdx.x, kStripThreads);
    if (t < te) start_run();
    tc::cp_async_wait_all();
    __syncthreads();
    load_weights_strip<Net>(sw, reinterpret_cast<const __half*>(smem + Net::OFF_RAW) + raw_skip(w), threadIdx.x);
    __syncthreads();
    uint2 held[Net::HELD ? Net::FRAGS : 1];
    if constexpr (Net::HELD) {
#pragma unroll
      for (int f = 0; f < Net::FRAGS; ++f) held[f] = *reinterpret_cast<const uint2*>(sw + f * 64 + 2 * lane);
    }
    auto frag = [&](int f) {
      if constexpr (Net::HELD) return held[f];
      else return *reinterpret_cast<const uint2*>(sw + f * 64 + 2 * lane);
    };
    for (bool started = true; t < te; started = false) {
      if (!started) {
        tc::cp_async_wait_all();
        start_run();
      }
      const int rows = static_cast<int>(min(static_cast<long long>(p.H - y0), te - t));
      for (int r = 0; r < rows; ++r) {
        st.features(p, [&](int kc) { return mine + Net::OFF_A + F::chunk(lane, kc); }, lane, r + 1 < rows);
        float d[2][J][4];
#pragma unroll
        for (int s = 0; s < F::K1 / 16; ++s) {
          uint32_t a[2][4];
          load_a<F>(mine + Net::OFF_A, lane, 0, s, a[0]);
          load_a<F>(mine + Net::OFF_A, lane, 1, s, a[1]);
#pragma unroll
          for (int j = 0; j < J; ++j) {
            const uint2 v = frag(j * (Net::NB1 / 2) + s);
            if (s == 0) {
              float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
              if constexpr (!F::BIASCOL) load_bias(bias, j, lane, c);
              hmma(d[0][j], a[0], v.x, v.y, c);
              hmma(d[1][j], a[1], v.x, v.y, c);
            } else {
              hmma(d[0][j], a[0], v.x, v.y, d[0][j]);
              hmma(d[1][j], a[1], v.x, v.y, d[1][j]);
            }
          }
        }
        uint32_t hi[2][J][2], lo[2][J][2];
#pragma unroll
        for (int h = 0; h < HID; ++h) {
          split_acc<Net::ACT, J>(d, hi, lo);
          layer<J, J>(frag, (Net::OFF_H + h * Net::WH_WORDS) / 64, bias + (1 + h) * 16 * J, lane, hi, lo, d);
        }
        float rgb[3];
        int x = st.x;
        if constexpr (Net::OUT_FP32) {
          output_layer<Net>(wo, lane, d, rgb);
          x = col * 32 + out_pixel(lane);
        } else {
          split_acc<Net::ACT, J>(d, hi, lo);
          float o[2][1][4];
          layer<J, 1>(frag, Net::OFF_O / 64, bias + (1 + HID) * 16 * J, lane, hi, lo, o);
          const float both[2][4] = {{o[0][0][0], o[0][0][1], o[0][0][2], o[0][0][3]},
                                    {o[1][0][0], o[1][0][1], o[1][0][2], o[1][0][3]}};
          put_rgb(mine + Net::OFF_OUT, lane, both);
          get_rgb(mine + Net::OFF_OUT, lane, rgb[0], rgb[1], rgb[2]);
        }
        write_rgb(p, out_img, b, y0 + r, x, rgb[0], rgb[1], rgb[2]);
      }
      t += rows;
    }
    seg = seg_end;
  }
  tc::cp_async_wait_all();  // copies still in flight land before shared memory goes
}

template <int L, int C, int NL, int N, int ACT, bool FL = false>
KernelInfo make_strip(const char* name, const int* dims) {
  using Net = StripNet<L, C, NL, N, ACT>;
  KernelInfo k{};
  k.name = name;
  k.precision = 1;
  k.latent_format = FL ? 1 : 0;
  k.C = C;
  k.n_layers = NL;
  for (int i = 0; i <= NL; ++i) k.dims[i] = dims[i];
  k.act = ACT;
  k.threads = kStripThreads;
  k.tile_px = 32;
  k.smem_bytes = Net::SMEM;
  k.march = 1;
  k.fn = reinterpret_cast<const void*>(&strip_decode_kernel<Net, FL>);
  return k;
}

}  // namespace
}  // namespace pic
