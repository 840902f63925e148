// march.cuh -- what the row-marching decode kernels (k_strip.cuh,
// k_tcmarch.cuh) share: above all the latent side, dequantisation, bilinear upsampling and
// concatenation of the pyramid levels (Sec. 3.1, Eq. 1) for one warp's strip
// of 32 pixel columns, row after row downwards.
//
// Lane = pixel column.  Per interpolated feature (level l >= 1, channel) a
// lane keeps the horizontally interpolated, dequantised value of its lower
// source row (v, row i1) and its difference to the upper one (d) in
// registers.  Going down one image row moves level l's source row by at most
// one, on average by 2^-l, so all levels together need about one new source
// row per image row (two texels and a lerp), and the vertical interpolation
// is one packed FMA per two features.
//
// The vertical weights and the levels that move are the same for the whole
// warp: every 32 rows, lane r works them out for the r-th row and leaves them
// in a small shared table, from which each row is two broadcast loads.
//
// Texels come by 4-byte asynchronous copies into the lane's own shared slots:
// level 0 one row ahead, the next source row of a coarser level as soon as
// the one before it has been taken up, so nothing waits on memory within a
// row and no register is held meanwhile.
#pragma once

#include "pic_common.cuh"
#include "tc_ptx.cuh"

namespace pic {
namespace {

__host__ __device__ constexpr int round_to(int v, int m) { return (v + m - 1) / m * m; }

// Operand A of the first layer: one row of K1 fp16 per pixel.  Words (pairs
// of fp16) 0 .. NPAIR-1 are the hi terms of the feature pairs, the next
// NPAIR the lo terms.  Feature order along K: the interpolated ones
// (level-major from level 1, channel-minor), then level 0's; an odd count is
// filled up with the constant 1 (hi word only), an even one leaves room for
// the constant in the word after the lo terms, or not (BIASCOL = false).
template <int L_, int C_>
struct FeatLayout {
  static constexpr int L = L_, C = C_, D0 = L * C;
  static constexpr int NS = (L - 1) * C;          // interpolated features
  static constexpr int NP = (NS + 1) / 2;         // their register pairs
  static constexpr int NPAIR = (D0 + 1) / 2;
  static constexpr int K1 = round_to(4 * NPAIR, 16);
  static constexpr bool BIASCOL = (D0 & 1) || 4 * NPAIR < K1;
  static constexpr int CHUNKS = K1 / 8;           // 16-byte chunks per row
  // Table row: NS weights (C copies each), then the mask word.
  static constexpr int TABW = round_to(NS + 1, 4);
  static constexpr int SLOTS = C + 2 * NS;        // staged words per lane
  static constexpr int A_BYTES = 32 * K1 * 2;
  static constexpr int STAGE_BYTES = SLOTS * 128;
  static constexpr int TAB_BYTES = 32 * TABW * 4;
  static constexpr int XTAB_BYTES = (L - 1) * 256; // per level and lane: next texel's offset, weight
  // shared memory of one strip's feature pass (operand A lives elsewhere)
  static constexpr int OFF_TAB = STAGE_BYTES, OFF_X = OFF_TAB + TAB_BYTES, FEAT_BYTES = OFF_X + XTAB_BYTES;
  static_assert(L >= 2, "at least one interpolated level");
  static_assert(CHUNKS == 2 || CHUNKS == 4, "swizzle below");

  // The weight that column k of operand A meets: >= 0 an input of W_0,
  // -1 the bias, -2 nothing.
  __host__ __device__ static constexpr int input_of(int k) {
    const int w = k >> 1, h = k & 1;
    const int kf = 2 * (w < NPAIR ? w : w - NPAIR) + h;  // feature in K order
    if (w < 2 * NPAIR) {
      if (kf < NS) return C + kf;
      if (kf < D0) return kf - NS;
      return w < NPAIR ? -1 : -2;  // the odd count's filler
    }
    return (w == 2 * NPAIR && h == 0 && !(D0 & 1)) ? -1 : -2;
  }
  // Byte offset of 16-byte chunk kc of row r: chunks XORed so that 8
  // consecutive rows' equal chunks fall into the 8 different 16-byte bank
  // groups (stores by row and ldmatrix).
  __device__ static __forceinline__ uint32_t chunk(int r, int kc) {
    const int x = CHUNKS == 2 ? (r >> 2) & 1 : (r >> 1) & 3;
    return static_cast<uint32_t>(r * (K1 * 2) + ((kc ^ x) << 4));
  }
};

__device__ __forceinline__ int lds32(uint32_t a) {
  int v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

template <int L, int C, bool FL>
struct Strip {
  using F = FeatLayout<L, C>;
  float v[2 * F::NP], d[2 * F::NP];  // row i1, and row i1 - row i0
  const int32_t* lat;   // the image's latents
  const float* steps;   // its steps (unused for real latents)
  uint32_t mine;        // the strip's shared memory (FeatLayout offsets)
  uint32_t slot;        // this lane's staging slots (128 bytes apart)
  int x, xc;            // this lane's column, and clamped to the image
  int y;                // row the next features() call decodes
  uint32_t tab;         // its table row
  float st0;            // level 0's step

  __device__ __forceinline__ void init(uint32_t warp_smem, int lane) {
    mine = warp_smem;
    slot = warp_smem + 4 * lane;
  }
  __device__ __forceinline__ uint32_t xtab(int l, int lane) const {
    return mine + F::OFF_X + (l - 1) * 256 + 8 * lane;
  }
  __device__ __forceinline__ float step_of(int l) const { return FL ? 1.0f : __ldg(steps + l); }

  // Table of rows y .. y + 31: the weights frac - 1 of the upper source rows
  // (f = v + (frac - 1) d) and the levels whose source row moves on the way
  // to the row.  A run's first row starts from the state start() makes.
  __device__ __forceinline__ void build_table(const DecodeParams& p, int lane, bool first) {
    unsigned m = 0;
    const uint32_t row = mine + F::OFF_TAB + lane * (F::TABW * 4);
#pragma unroll
    for (int l = 1; l < L; ++l) {
      const LevelGeom& g = p.lv[l];
      const Tap t = bilinear_tap(y + lane, g.sy, g.H);
      const Tap b = bilinear_tap(max(y + lane - 1, 0), g.sy, g.H);
      m |= b.i0 != t.i0 ? 1u << l : 0u;
#pragma unroll
      for (int c = 0; c < C; ++c) sts32(row + 4 * ((l - 1) * C + c), __float_as_uint(t.frac - 1.0f));
    }
    sts32(row + 4 * F::NS, first && lane == 0 ? 0u : m);
    __syncwarp();
    tab = mine + F::OFF_TAB;
  }

  __device__ __forceinline__ void copy_level0(const DecodeParams& p, int row) {
    const int32_t* q = lat + (static_cast<long long>(row) * p.W + xc);
#pragma unroll
    for (int c = 0; c < C; ++c)
      tc::cp_async4(slot + c * 128, q + c * (static_cast<long long>(p.H) * p.W));
  }
  // Texel pair at element offset off of level l's planes -> the level's slots.
  __device__ __forceinline__ void copy_pair(const DecodeParams& p, int l, unsigned off, unsigned du) {
    const LevelGeom& g = p.lv[l];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int32_t* q = lat + g.off + static_cast<long long>(c) * g.H * g.W + off;
      const int i = (l - 1) * C + c;
      tc::cp_async4(slot + (C + 2 * i) * 128, q);
      tc::cp_async4(slot + (C + 2 * i + 1) * 128, q + du);
    }
  }

  // Starts a run at column x_ (this lane's) and row y_: both source rows of
  // every level, the first table, level 0 of row y_, the next source rows.
  // The caller has waited for the copies of the run before.
  __device__ __forceinline__ void start(const DecodeParams& p, int x_, int y_, int lane) {
    x = x_;
    y = y_;
    xc = min(x_, p.W - 1);
    copy_level0(p, y);
    st0 = step_of(0);
    float nv[F::NS], up[F::NS];
#pragma unroll
    for (int l = 1; l < L; ++l) {
      const LevelGeom& g = p.lv[l];
      const Tap tx = bilinear_tap(xc, g.sx, g.W);
      const Tap ty = bilinear_tap(y, g.sy, g.H);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const int i = (l - 1) * C + c;
        const int32_t* q = lat + g.off + static_cast<long long>(c) * g.H * g.W;
        const int32_t* r0 = q + static_cast<unsigned>(ty.i0 * g.W);
        const int32_t* r1 = q + static_cast<unsigned>(ty.i1 * g.W);
        up[i] = lat_lerp<FL>(__ldg(r0 + tx.i0), __ldg(r0 + tx.i1), tx.frac);
        nv[i] = lat_lerp<FL>(__ldg(r1 + tx.i0), __ldg(r1 + tx.i1), tx.frac);
      }
      const unsigned off = static_cast<unsigned>(min(ty.i1 + 1, g.H - 1) * g.W + tx.i0);
      const unsigned du = tx.i1 - tx.i0;
      copy_pair(p, l, off, du);
      // the weight's sign bit: the pair is one texel (right edge)
      sts32(xtab(l, lane), off);
      sts32(xtab(l, lane) + 4, __float_as_uint(tx.frac) | (du ? 0u : 0x80000000u));
    }
    tc::cp_async_commit();
#pragma unroll
    for (int i = 0; i < F::NS; ++i) {
      const float st = step_of(1 + i / C);
      const float a = st * nv[i];
      v[i] = a;
      d[i] = a - st * up[i];
    }
    if constexpr (F::NS & 1) {  // the last pair's unused half
      v[F::NS] = 0.0f;
      d[F::NS] = 0.0f;
    }
    build_table(p, lane, true);
  }

  // Level l moves to its next source row (staged), and the one after that is
  // fetched.
  __device__ __forceinline__ void move_level(const DecodeParams& p, int l, int lane) {
    const LevelGeom& g = p.lv[l];
    unsigned off, fb;
    const uint32_t xt = xtab(l, lane);
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(off), "=r"(fb) : "r"(xt));
    const float fx = fabsf(__uint_as_float(fb));
    const float st = step_of(l);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int i = (l - 1) * C + c;
      const uint32_t s = slot + (C + 2 * i) * 128;
      const float nv = st * lat_lerp<FL>(lds32(s), lds32(s + 128), fx);
      d[i] = nv - v[i];
      v[i] = nv;
    }
    const unsigned next = off + g.W;
    off = next < static_cast<unsigned>(g.H) * static_cast<unsigned>(g.W) ? next : off;
    sts32(xt, off);
    __syncwarp();  // the staged texels have been read: their slots may be refilled
    copy_pair(p, l, off, (fb >> 31) ^ 1u);
  }

  // Features of row y -> this lane's row of operand A, whose 16-byte chunk kc
  // goes to shared address at(kc), and level 0 of row y + 1 if `more`; then y
  // moves on.
  template <class At>
  __device__ __forceinline__ void features(const DecodeParams& p, At at, int lane, bool more) {
    tc::cp_async_wait_all();
    if (tab == mine + F::OFF_TAB + F::TAB_BYTES) {
      __syncwarp();  // every lane has read the old table
      build_table(p, lane, false);
    }
    float w[F::TABW];
#pragma unroll
    for (int q = 0; q < F::TABW / 4; ++q)
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(w[4 * q]), "=f"(w[4 * q + 1]), "=f"(w[4 * q + 2]), "=f"(w[4 * q + 3])
                   : "r"(tab + 16 * q));
    tab += F::TABW * 4;
    const unsigned mask = __float_as_uint(w[F::NS]);
    float f0[C];
#pragma unroll
    for (int c = 0; c < C; ++c) f0[c] = lat_value<FL>(lds32(slot + c * 128));
    if constexpr (!FL) {
#pragma unroll
      for (int c = 0; c < C; ++c) f0[c] *= st0;
    }
    // one level moves in most rows: the two finest are tested for alone
#pragma unroll
    for (int l = 1; l < L && l < 3; ++l)
      if ((mask >> l) & 1u) move_level(p, l, lane);
    if (mask >> 3) {
#pragma unroll
      for (int l = 3; l < L; ++l)
        if ((mask >> l) & 1u) move_level(p, l, lane);
    }
    uint32_t hw[F::K1 / 2];  // this pixel's row of A
#pragma unroll
    for (int q = 0; q < F::K1 / 2; ++q) hw[q] = 0u;
#pragma unroll
    for (int q = 0; q < F::NPAIR; ++q) {
      float a, b;
      if (q < F::NP) {
        // (the odd count's second half: the mask's bits * 0 + 0)
        const float2 f = unpack2(fma2(pack2(w[2 * q], w[2 * q + 1]), pack2(d[2 * q], d[2 * q + 1]), pack2(v[2 * q], v[2 * q + 1])));
        a = f.x;
        b = 2 * q + 1 < F::NS ? f.y : f0[0];
      } else {
        const int i = 2 * q - F::NS;
        a = f0[i];
        b = i + 1 < C ? f0[i + 1 < C ? i + 1 : 0] : 1.0f;
      }
      tc::split_pair<false>(a, b, hw[q], hw[F::NPAIR + q]);
    }
    if constexpr (!(F::D0 & 1) && F::BIASCOL) hw[2 * F::NPAIR] = 0x00003C00u;
#pragma unroll
    for (int kc = 0; kc < F::CHUNKS; ++kc)
      tc::sts128(at(kc), hw[4 * kc], hw[4 * kc + 1], hw[4 * kc + 2], hw[4 * kc + 3]);
    __syncwarp();  // A is complete, and level 0's slots may be refilled
    ++y;
    if (more) copy_level0(p, y);
    tc::cp_async_commit();
  }
};

// ---- warp-level tensor-core pieces ------------------------------------------
// D (16 pixels x 8 neurons, fp32) = A (16 x 16 fp16) B (16 x 8 fp16) + C.
__device__ __forceinline__ void hmma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1,
                                     const float (&c)[4]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%10, %11, %12, %13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
// The accumulator start of output tile j: the biases of this lane's two
// neurons, for both pixel rows of a fragment; one 16-byte load from the
// [tile][4][b0 b1 b0 b1] table, shared by both halves of the strip.
__device__ __forceinline__ void load_bias(const float* bias4, int j, int lane, float (&c)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(bias4 + 16 * j + 4 * (lane & 3));
  c[0] = q.x;
  c[1] = q.y;
  c[2] = q.z;
  c[3] = q.w;
}
// Fills it: entry e of J * 16 floats is the bias of neuron 8 j + 2 t + (e & 1).
template <class V>
__device__ __forceinline__ void fill_bias(float* bias4, int J, int tid, int nthr, V val) {
  for (int e = tid; e < 16 * J; e += nthr) bias4[e] = val(8 * (e >> 4) + 2 * ((e >> 2) & 3) + (e & 1));
}

// Operand A of 16 pixels (m-th half of the strip), 16 columns from 16 s on.
template <class F>
__device__ __forceinline__ void load_a(uint32_t a_s, int lane, int m, int s, uint32_t (&a)[4]) {
  const int r = 16 * m + (lane & 7) + ((lane >> 3) & 1) * 8, kc = 2 * s + (lane >> 4);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
               : "r"(a_s + F::chunk(r, kc))
               : "memory");
}

// Activation of a pair and its hi/lo split into two f16x2.
template <int ACT>
__device__ __forceinline__ void act_split(float a, float b, uint32_t& hi, uint32_t& lo) {
  if constexpr (ACT == ACT_GELU) {
    const float2 g = unpack2(gelu_approx2(pack2(a, b)));
    tc::split_pair<false>(g.x, g.y, hi, lo);
  } else {
    tc::split_pair<true>(a, b, hi, lo);
  }
}

// The n fp16 weights of one image -> shared memory at dst (raw_bytes(n)),
// as asynchronous copies of the words that cover them, so that the layouts
// below are made from shared memory: one global latency instead of one per
// layout (a small image's decode is a few microseconds, of which the
// dependent 2-byte loads of five layouts took two).  The first weight is
// half `raw_skip(src)` of the copy.
__host__ __device__ constexpr int raw_bytes(int n) { return round_to(2 * n + 4, 128); }
__device__ __forceinline__ int raw_skip(const __half* src) {
  return static_cast<int>((reinterpret_cast<uintptr_t>(src) >> 1) & 1u);
}
__device__ __forceinline__ void copy_raw(uint8_t* dst, const __half* src, int n, int tid, int nthr) {
  const int skip = raw_skip(src), words = (skip + n) >> 1;  // whole words: no read past the weights
  const char* base = reinterpret_cast<const char*>(src - skip);
  const uint32_t d = tc::smem_addr(dst);
  for (int i = tid; i < words; i += nthr) tc::cp_async4(d + 4 * i, base + 4 * i);
  if (tid == 0 && ((skip + n) & 1)) reinterpret_cast<__half*>(dst)[2 * words] = src[n - 1];
  tc::cp_async_commit();
}

// B fragments of one layer in shared memory: word [(j * NB2 + i / 2) * 64 +
// 2 lane + (i & 1)] holds, for output tile j (8 neurons) and block i (8
// inputs), the weights of neuron 8j + lane / 4 for inputs 8i + 2 (lane % 4)
// and the next one, so that two blocks are one conflict-free 8-byte load.
__host__ __device__ constexpr int frag_words(int J, int NB) { return J * ((NB + 1) / 2) * 64; }

// Fills them; val(n, k) is the weight of neuron n for column k (0 outside).
template <int J, int NB, class V>
__device__ __forceinline__ void fill_frags(uint32_t* sm, int tid, int nthr, V val) {
  constexpr int NB2 = (NB + 1) / 2;
  for (int e = tid; e < frag_words(J, NB); e += nthr) {
    const int lane = (e & 63) >> 1, ji = e >> 6;
    const int j = ji / NB2, i = 2 * (ji - j * NB2) + (e & 1);
    const int n = 8 * j + (lane >> 2), k = 8 * i + 2 * (lane & 3);
    __half2 v = __floats2half2_rn(0.0f, 0.0f);
    if (i < NB) v = __halves2half2(val(n, k), val(n, k + 1));
    sm[e] = *reinterpret_cast<uint32_t*>(&v);
  }
}

// The strip's RGB from the output tiles' fragments (lane 4g: r, g of pixels
// g, g + 8, 16 + g, 24 + g; lane 4g + 1: their b) to lane = pixel, through
// the warp's transpose buffer: [32 pixels][4], kOutBytes.
constexpr int kOutBytes = 512;
__device__ __forceinline__ void put_rgb(uint32_t out_s, int lane, const float (&d)[2][4]) {
  const int g = lane >> 2, t = lane & 3;
  __syncwarp();  // the previous row's values have been read
  if (t < 2) {
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(out_s + (16 * m + 8 * h + g) * 16 + 8 * t),
                     "f"(d[m][2 * h]), "f"(d[m][2 * h + 1])
                     : "memory");
  }
  __syncwarp();
}
__device__ __forceinline__ void get_rgb(uint32_t out_s, int lane, float& r, float& g, float& bl) {
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r), "=f"(g) : "r"(out_s + lane * 16));
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(bl) : "r"(out_s + lane * 16 + 8));
}

// Step 5 for pixel (x, y) of image b, whose planes start at out_img.
__device__ __forceinline__ void write_rgb(const DecodeParams& p, float* out_img, int b, int y, int x, float r,
                                          float g, float bl) {
  if (x >= p.W) return;
  if (p.out_format == OUT_F32_CHW) {  // the default, with few 64-bit operations
    if (p.clamp) {
      r = __saturatef(r);
      g = __saturatef(g);
      bl = __saturatef(bl);
    }
    float* o = out_img + (static_cast<unsigned>(y) * static_cast<unsigned>(p.W) + x);
    const long long plane = static_cast<long long>(p.H) * p.W;
    o[0] = r;
    o[plane] = g;
    o[2 * plane] = bl;
  } else {
    store_rgb(p, b, y, x, r, g, bl);
  }
}

}  // namespace
}  // namespace pic
