// k_huffman.cu -- Huffman decoding of B image-specific streams on the GPU
// (include/pic_huffman.h; Sec. 3.3 and Sec. 4.1 of the paper, which adapts
// GPUHD, Weissenberger & Schmidt 2018: self-synchronising parallel decoding).
//
// One cooperative launch (every CTA resident, grid-wide barriers between the
// phases):
//    0. tables (for more images than CTAs by a launch of their own): the CTAs
//       expand the stored tables, up to kMaxParts CTAs to an image.  A table -- values and lengths in canonical order -- is the
//       run-length code of the 2^p-entry lookup table: symbol k covers
//       2^(p - len_k) consecutive entries.  Expanding the runs gives the table,
//       so one lookup of the next p bits decodes a symbol.  A 16-bit entry is
//       value << 4 | length; where a value takes more than 12 bits the image's
//       entries are row << 4 | length, the row in the stored table, whose value
//       is then read when it is written out.  Kraft's inequality is checked
//       here.  A second table holds, for every p-bit window, how many codewords
//       lie wholly inside it and the bits they take (one byte: 2.4 codewords on
//       average where one takes 4.3 bits), which is all that counting needs.
//    a. each thread decodes its 256-bit subsequences speculatively from their
//       first bit, which may lie inside a codeword, until it passes the
//       subsequence's end; it records how far past the end the first
//       codeword boundary lies (the overshoot, below 12 bits);
//    b. synchronisation passes: a subsequence whose predecessor's overshoot
//       differs from the one it was decoded with is decoded again from there
//       (in the first pass every one is, and counts its codewords).
//       Codes of different lengths resynchronise within a few codewords, so a
//       pass seldom changes an overshoot, and the passes end with the first that
//       changes none (usually the first); pass i has made subsequence i exact,
//       and after 64 passes without convergence (codewords of one length that
//       does not divide 256) the status word says so.  Each
//       pass also leaves the CTAs' codeword totals, from which
//    c. every CTA takes its output position (the total must equal the symbol
//       offsets');
//    d. every subsequence is decoded from its final start, writing values
//       through per-warp staging rows, so that a warp store writes a run of
//       one subsequence's values instead of 32 scattered words.
// Each CTA holds its images' tables in shared memory; each warp goes through
// groups of 32 subsequences of its own, whose stream words it stages in
// shared memory (9 words apart: equal words of neighbouring subsequences fall
// into different banks, and the ninth is the word that follows) without a CTA
// barrier.
//
// What bounds it: for one image latency -- 3 grid barriers, the tables, and a
// subsequence's serial chain (window, lookup, shift) three times; for a batch
// the instructions of the chains (half the issue slots, mostly shifts, which
// issue at half rate).  So a chain's step is branch-free and has two lookups
// per 32-bit window, every phase runs without divergence, and the groups are
// dealt out so that the fewest warps do a group more than the others.  Before,
// a branch per lookup reloaded words from conflicting banks (230 cycles a step
// against the lookup's 30), the tables came from a launch of their own and a
// memset, CTA barriers held every warp to the slowest, and the passes kept 36
// bytes a subsequence instead of 5.  Measured, before and now (768x512, 6,800
// subsequences an image, the streams of perf/cases.py's distribution; the 24 of
// another seed, with a few more, 48 us): 1 image 54.3 -> 24.8 us, 24 images 100.2 -> 45.4 us,
// 64 images 163 -> 96.5 us; 256 images of 64x64 108 -> 38.4 us.
#include <algorithm>
#include <atomic>
#include <cstdint>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "pic_decode.h"
#include "pic_huffman.h"

namespace cg = cooperative_groups;

namespace {

constexpr int kQ = PIC_HUFF_WORDS_PER_SUBSEQ;  // words per subsequence
constexpr int kS = 32 * kQ;                     // bits per subsequence
// Warps of a CTA: 8, or 9 where that saves a round of groups (24 images of
// 768x512, 5,129 groups on 152 SMs: 45.4 us in one round, 64 in two).  Nine
// warps of 56 registers on each of four CTAs fill an SM; ten, at 48
// registers, spill (69 us).  Held to eight warps and 64 registers, 1 and 64
// images take the same time within 1 %, and 24 images 55.6 us.  Fewer than 8 make the tables too slowly (one
// image: 33 us with 2, 26.9 with 4, 25.9 with 8).
constexpr int kMaxWarps = 9;
constexpr int kMinWarps = 8;
constexpr int kCtasPerSm = 4;
constexpr int kMaxParts = 8;  // CTAs that share one image's tables (one 100x100 image: 27.0 us with 1, 22.4 with 8)
constexpr int kMaxPasses = 64;
constexpr int kHead = 16 + 4 * 68;  // workspace bytes before block_sum (a multiple of 16)
static_assert(kHead >= 16 + 4 * kMaxPasses && kHead % 16 == 0, "status, pass counters");
constexpr int kMaxTable = 4096;
constexpr int kMaxGrid = 4096;
constexpr int kWords = 32 * kQ + 2;                  // stream words of a warp's 32 subsequences (two past the last)
constexpr int kWrow = kQ + 1;                        // a subsequence's staged words, and the one that follows
constexpr int kWbuf = 32 * kWrow + 2;
constexpr int kRound = 32;                           // symbols a thread decodes between two warp stores
constexpr int kStep = 8;                             // symbols between two looks at whether any thread goes on
constexpr int kRow = kRound + 2;                     // staging row, 16-bit entries (odd number of words)
enum : int { kBadCode = 1, kBadCount = 2, kNoSync = 4, kBadTable = 8 };

struct Ws {
  int* status;           // [4]
  int* changed;          // [kMaxPasses]
  long long* block_sum;  // [kMaxGrid]: codewords of each CTA's range
  uint16_t* lut;         // [B][2^p]
  uint16_t* cnt;         // [n_sub]: codewords
  uint8_t* over0;        // [n_sub]: overshoot, double-buffered over the passes
  uint8_t* over1;        // [n_sub]
  uint8_t* start;        // [n_sub]: the overshoot it was decoded from
  uint8_t* multi;        // [B][2^p]: codewords inside the window << 4 | their bits (small workspace: none)
  uint8_t* direct;       // [B]: the lookup table holds values, not rows (small workspace: none, all hold rows)
};

__host__ __device__ inline Ws ws_view(void* w, long long n_sub, int B, int p, bool small, long long* bytes = nullptr) {
  char* c = static_cast<char*>(w);
  const long long tab = static_cast<long long>(B) << p;
  Ws v;
  v.status = reinterpret_cast<int*>(c);
  v.changed = reinterpret_cast<int*>(c + 16);
  v.block_sum = reinterpret_cast<long long*>(c + kHead);
  long long o = kHead + kMaxGrid * 8;
  v.lut = reinterpret_cast<uint16_t*>(c + o);
  o += tab * 2;
  v.cnt = reinterpret_cast<uint16_t*>(c + o);
  o += (n_sub * 2 + 15) / 16 * 16;
  o = (o + 15) / 16 * 16;
  v.multi = small ? nullptr : reinterpret_cast<uint8_t*>(c + o);
  o += small ? 0 : tab;
  v.over0 = reinterpret_cast<uint8_t*>(c + o);
  v.over1 = v.over0 + n_sub;
  v.start = v.over1 + n_sub;
  o += 3 * n_sub;
  v.direct = small ? nullptr : reinterpret_cast<uint8_t*>(c + o);
  o += small ? 0 : B;
  if (bytes) *bytes = (o + 15) / 16 * 16;
  return v;
}

long long ws_size(long long n_sub, int B, int p) {
  long long b = 0;
  ws_view(nullptr, n_sub, B, p, false, &b);
  return b;
}

// The other size that is accepted, 36 bytes a subsequence and 2 a table entry:
// what was asked for before the multi tables, and less than they need where
// images average fewer than about 132 subsequences (at p = 12).  In it every
// CTA works the multi tables out for its own images, and a table's values are
// all looked up by row: 256 images of 64x64 take 53 us in it, 39 in the other.  (The small layout
// takes 5 bytes a subsequence, so it always fits.)
long long ws_size_small(long long n_sub, int B, int p) {
  const long long b = (16 + 4 * kMaxPasses + 8 * 8192 + (2LL * B << p) + 15) / 16 * 16;
  return (b + 36 * n_sub + 15) / 16 * 16;
}

struct DecodeParams {
  const uint32_t* words;
  long long n_words;
  const long long* word_off;
  const long long* n_bits;
  int B;
  int p;
  const long long* sym_off;
  const int32_t* tab_value;  // [B][max_table]: a row entry's high 12 bits index it
  const int32_t* tab_len;    // [B][max_table]
  int max_table;
  int32_t* out;
  Ws ws;
  long long n_sub;
  // groups of 32 subsequences, dealt out to the CTAs in contiguous ranges
  // (groups_base each, the first groups_more CTAs one more), and there to the warps
  long long groups_base;
  int groups_more;
  int parts;            // CTAs that share the making of one image's tables (0: huff_tables has made them)
};

// Dynamic shared memory: two images' tables, the warps' words,
// staging rows and row descriptors.  (Phase 0 works in the same memory: run starts, then a table.)
__host__ __device__ constexpr size_t smem_bytes(int p, int warps) {
  return (size_t{2} * 3 << p) + 16 + size_t(warps) * (4 * (kWbuf + 32) + 2 * 32 * kRow);
}

__device__ __forceinline__ uint32_t* words_of(uint8_t* s_dyn, int p) {
  return reinterpret_cast<uint32_t*>(s_dyn + (((size_t{6} << p) + 4 + 15) & ~size_t{15}));
}

// ---------------------------------------------------------------- 0. tables
// Codewords that lie wholly inside p-bit window i << 4 | the bits they take; a
// window that starts with no codeword counts as one of 1 bit (the final decode
// reports it).
__device__ __forceinline__ int codewords_in(const uint16_t* lut, int i, int p) {
  int pos = 0, c = 0;
  while (pos < p) {
    const int l = lut[(i << pos) & ((1 << p) - 1)] & 15;
    if (l == 0 || pos + l > p) break;
    pos += l;
    ++c;
  }
  return c == 0 ? 1 << 4 | 1 : c << 4 | pos;
}

// The part-th of P.parts pieces of image b's lookup and multi tables -> global
// memory (the whole CTA; the pieces' run starts are worked out by each, the
// windows' codewords, three quarters of the time, only for the piece).
// Returns true if the stored table is bad (then every entry is "no codeword").
__device__ bool build_tables(const DecodeParams& P, int b, int part, void* scratch) {
  __shared__ int s_warp[kMaxWarps];
  __shared__ int s_m;
  const int p = P.p, size = 1 << p;
  uint32_t* s_start = static_cast<uint32_t*>(scratch);                // [2^p + 1]: value << 16 | run start
  uint16_t* s_lut = reinterpret_cast<uint16_t*>(s_start + size + 1);  // [2^p]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, n_threads = blockDim.x, n_warps = n_threads >> 5;
  const int32_t* tl = P.tab_len + static_cast<long long>(b) * P.max_table;
  const int32_t* tv = P.tab_value + static_cast<long long>(b) * P.max_table;
  // the table ends at its first zero length
  __syncthreads();  // (the memory and s_m are free)
  if (t == 0) s_m = P.max_table;
  __syncthreads();
  bool wide = false;  // values past 12 bits (or such rows behind the table's end: then it is read like one that has)
#pragma unroll 2
  for (int k = t; k < P.max_table; k += n_threads) {
    const int l = __ldg(tl + k), v = __ldg(tv + k);
    if (l == 0) atomicMin(&s_m, k);
    wide |= v < -2048 || v > 2047;
  }
  const bool direct = !__syncthreads_or(wide) && P.ws.direct;
  const int m = s_m;
  // run sizes 2^(p - len) scanned into run starts, 256 entries at a time; more
  // than 2^p entries cannot be a code
  bool bad = m > size;
  int carry = 0;
  for (int k0 = 0; k0 < m && m <= size; k0 += n_threads) {
    const int k = k0 + t;
    int run = 0;
    if (k < m) {
      const int l = __ldg(tl + k);
      if (l < 1 || l > p) bad = true;
      else run = 1 << (p - l);
    }
    int x = run;  // inclusive warp scan, then across the warps
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int i = 0; i < kMaxWarps; ++i) {
      if (i >= n_warps) break;
      before += i < warp ? s_warp[i] : 0;
      total += s_warp[i];
    }
    if (k < m) {
      s_start[k] = static_cast<uint32_t>(__ldg(tv + k)) << 16 | static_cast<uint32_t>(min(carry + before + x - run, size));
    }
    carry = min(carry + total, size + 1);  // capped: runs may sum past 2^p only in bad tables
    __syncthreads();
  }
  bad = __syncthreads_or(bad) || carry > size;  // a bad length, or Kraft's inequality violated
  const int fill = bad ? 0 : carry;  // a bad table decodes nothing
  if (t == 0 && m <= size) s_start[m] = fill;
  if (t == 0 && P.ws.direct) P.ws.direct[b] = direct;
  __syncthreads();
  auto entry = [&](int k, int& next) {  // and where symbol k's run ends
    const uint32_t v = s_start[k];
    next = s_start[k + 1] & 0xFFFF;
    const int len = p - (31 - __clz(next - static_cast<int>(v & 0xFFFF)));
    return static_cast<int>((direct ? v >> 16 : static_cast<uint32_t>(k)) << 4) | len;
  };
  // each thread finds the run of its first entry and walks on from there
  const int per = (size + n_threads - 1) / n_threads;
  uint16_t* lut = P.ws.lut + (static_cast<long long>(b) << p);
  uint8_t* multi = P.ws.multi + (static_cast<long long>(b) << p);
  const int i0 = t * per;
  if (i0 < size) {
    int lo = 0, e = 0, next = 0;
    if (i0 < fill) {
      int hi = m - 1;  // last k with s_start[k] <= i0
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (static_cast<int>(s_start[mid] & 0xFFFF) <= i0) lo = mid;
        else hi = mid - 1;
      }
      e = entry(lo, next);
    }
    for (int i = i0; i < min(i0 + per, size); ++i) {
      if (i >= fill) {
        e = 0;  // no codeword
      } else if (i >= next) {
        e = entry(++lo, next);
      }
      s_lut[i] = static_cast<uint16_t>(e);
    }
  }
  __syncthreads();
  const int piece = size / max(P.parts, 1);
  for (int i = part * piece + t; i < (part + 1) * piece; i += n_threads) {
    lut[i] = s_lut[i];
    if (P.ws.multi) multi[i] = static_cast<uint8_t>(codewords_in(s_lut, i, p));
  }
  return bad;
}

// --------------------------------------------------------------- 1. decode
// The image of stream word `word`, among images lo .. hi.
__device__ __forceinline__ int image_of(const DecodeParams& P, long long word, int lo, int hi) {
  while (lo < hi) {  // last b with word_off[b] <= word
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(P.word_off + mid) <= word) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// An image's tables for the decode loops: in shared memory (SH), or in global
// memory for the images that lie strictly inside a CTA's range.
template <bool SH>
struct Tables {
  uint32_t lut_s, multi_s;  // shared addresses
  const uint16_t* lut_g;
  const uint8_t* multi_g;
  __device__ __forceinline__ int lut(uint32_t w) const {
    if (SH) {
      unsigned short v;
      asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(lut_s + 2 * w));
      return v;
    }
    return lut_g[w];
  }
  __device__ __forceinline__ int multi(uint32_t w) const {
    if (SH) {
      unsigned short v;
      asm volatile("{\n\t.reg .b32 t;\n\tld.shared.u8 t, [%1];\n\tcvt.u16.u32 %0, t;\n\t}" : "=h"(v) : "r"(multi_s + w));
      return v;
    }
    if (multi_g) return multi_g[w];
    return 1 << 4 | max(lut_g[w] & 15, 1);  // none was made: one codeword at a time
  }
};

// The 32 bits at bit `pos` of a subsequence's staged words: two codewords.
__device__ __forceinline__ uint32_t window(const uint32_t* row, int pos) {
  const uint32_t* w = row + (pos >> 5);
  return __funnelshift_l(w[1], w[0], pos);
}

// Counts the codewords that start at bits pos .. end - 1 of a subsequence's
// staged words, the first at pos; pos becomes the first codeword boundary at
// or after end.  The whole warp goes through it together, without divergence;
// lanes with pos >= end take no part.
template <bool SH>
__device__ __forceinline__ int count_span(const uint32_t* row, int& pos, int end, const Tables<SH>& tab, int p) {
  const int shr = 32 - p, begin = pos;
  int sum = 0;  // of the windows' entries: 16 x codewords + bits
  // whole windows: every codeword inside one that ends by `end` starts before it
  while (__any_sync(0xffffffffu, pos + p <= end)) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint32_t w = window(row, pos);
      const int e0 = tab.multi(w >> shr);
      const int e1 = tab.multi(w << (e0 & 15) >> shr);
      if (pos + p <= end) {
        sum += e0;
        pos += e0 & 15;
      }
      if (pos + p <= end) {
        sum += e1;
        pos += e1 & 15;
      }
    }
  }
  int c = (sum - (pos - begin)) >> 4;
  while (__any_sync(0xffffffffu, pos < end)) {
    const uint32_t w = window(row, pos);
    const int l0 = max(tab.lut(w >> shr) & 15, 1);
    const int l1 = max(tab.lut(w << l0 >> shr) & 15, 1);
    if (pos < end) {
      ++c;
      pos += l0;
    }
    if (pos < end) {
      ++c;
      pos += l1;
    }
  }
  return c;
}

__device__ long long block_sum_ll(long long v, long long* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  long long t = 0;
#pragma unroll
  for (int i = 0; i < kMaxWarps; ++i) t += i < static_cast<int>(blockDim.x >> 5) ? red[i] : 0;
  return t;
}

// 32 subsequences' stream words -> shared memory (a warp; coalesced), so that
// no global load sits inside a decode chain.
__device__ __forceinline__ void stage(const DecodeParams& P, uint32_t* s_words, long long k0) {
  const int lane = threadIdx.x & 31;
  const long long w0 = k0 * kQ;
#pragma unroll
  for (int j = 0; j < (kWords + 31) / 32; ++j) {
    const int i = lane + 32 * j, at = i + i / kQ;
    if (i < kWords) {
      const uint32_t w = w0 + i < P.n_words ? __ldg(P.words + w0 + i) : 0u;
      s_words[at] = w;
      if (i % kQ == 0 && i > 0) s_words[at - 1] = w;
    }
  }
}

// Phases a to d, with every image's tables in shared memory (SH) or not, for
// subsequences [k_begin, k_end) of this warp.
template <bool SH>
__device__ __forceinline__ void decode_phases(const DecodeParams& P, cg::grid_group& grid, uint8_t* s_dyn, int b_first,
                                              int b_last, long long k_begin, long long k_end) {
  __shared__ long long red[kMaxWarps];
  __shared__ long long wsum[kMaxWarps];
  const Ws& ws = P.ws;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, size = 1 << P.p;
  const int n_threads = blockDim.x, n_warps = n_threads >> 5;
  uint32_t* const all_words = words_of(s_dyn, P.p);
  uint32_t* const s_words = all_words + warp * kWbuf;
  uint32_t* const s_desc = all_words + n_warps * kWbuf + warp * 32;
  uint16_t* const wbuf = reinterpret_cast<uint16_t*>(all_words + n_warps * (kWbuf + 32)) + warp * 32 * kRow;
  const uint32_t lut_s = static_cast<uint32_t>(__cvta_generic_to_shared(s_dyn)), multi_s = lut_s + 4 * size;
  auto tables = [&](int b) {
    Tables<SH> t;
    if (SH) {
      t.lut_s = lut_s + (b == b_first ? 0 : 2 * size);
      t.multi_s = multi_s + (b == b_first ? 0 : size);
    } else {
      t.lut_g = ws.lut + (static_cast<long long>(b) << P.p);
      t.multi_g = ws.multi ? ws.multi + (static_cast<long long>(b) << P.p) : nullptr;
    }
    return t;
  };
  long long held = k_begin;  // first subsequence of the words held: staged before the tables were made
  auto stage_words = [&](long long k0) {
    if (k0 == held) return;
    held = k0;
    __syncwarp();  // the words before have been read
    stage(P, s_words, k0);
    __syncwarp();
  };
  // Subsequence k: its image, whether it is the image's first or last, its
  // bits (0: past the image's last bit).
  auto locate = [&](long long k, int& b, bool& first, bool& last) -> int {
    b = image_of(P, k * kQ, b_first, b_last);
    const long long ks = (k * kQ - __ldg(P.word_off + b)) * 32, left = __ldg(P.n_bits + b) - ks;
    first = ks == 0;
    last = left <= kS;
    return static_cast<int>(max(min(static_cast<long long>(kS), left), 0LL));
  };
  const uint32_t* const row = s_words + lane * kWrow;  // this lane's subsequence

  // a. speculative decode of every subsequence from its first bit
  for (long long k0 = k_begin; k0 < k_end; k0 += 32) {
    stage_words(k0);
    const long long k = k0 + lane;
    int b = b_first, bits = 0;
    bool first, last;
    if (k < k_end) bits = locate(k, b, first, last);
    int pos = 0;
    count_span<SH>(row, pos, bits, tables(b), P.p);
    if (k < k_end) ws.over0[k] = static_cast<uint8_t>(max(pos - kS, 0));
  }
  grid.sync();

  // b. synchronisation passes
  bool stable = false;
  for (int pass = 0; pass < kMaxPasses; ++pass) {
    const uint8_t* in = (pass & 1) ? ws.over1 : ws.over0;
    uint8_t* out = (pass & 1) ? ws.over0 : ws.over1;
    bool changed = false;
    long long total = 0;
    for (long long k0 = k_begin; k0 < k_end; k0 += 32) {
      const long long k = k0 + lane;
      int b = b_first, bits = 0, st = 0, c = 0, over = 0;
      bool redo = false;
      if (k < k_end) {
        bool first, last;
        bits = locate(k, b, first, last);
        st = first || bits == 0 || k == 0 ? 0 : __ldcg(in + k - 1);
        redo = pass == 0 || st != ws.start[k];
        if (pass > 0) c = ws.cnt[k];
        over = in[k];
        if (!redo) out[k] = static_cast<uint8_t>(over);
      }
      if (__any_sync(0xffffffffu, redo)) {
        stage_words(k0);
        int pos = st;
        const int c_now = count_span<SH>(row, pos, redo ? bits : 0, tables(b), P.p);
        if (redo) {
          c = c_now;
          const int over_now = max(pos - kS, 0);
          changed |= over_now != over;
          out[k] = static_cast<uint8_t>(over_now);
          ws.start[k] = static_cast<uint8_t>(st);
          ws.cnt[k] = static_cast<uint16_t>(c);
        }
      }
      total += c;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    if (lane == 0) wsum[warp] = total;
    if (__syncthreads_or(changed) && tid == 0) atomicAdd(ws.changed + pass, 1);
    if (tid == 0) {
      long long all = 0;
#pragma unroll
      for (int i = 0; i < kMaxWarps; ++i) all += i < n_warps ? wsum[i] : 0;
      ws.block_sum[blockIdx.x] = all;
    }
    grid.sync();
    if (*reinterpret_cast<volatile int*>(ws.changed + pass) == 0) {
      stable = true;
      break;
    }
  }
  if (!stable && blockIdx.x == 0 && tid == 0) atomicOr(ws.status, kNoSync);

  // c. this warp's output position
  long long carry = 0;
  for (int j = tid; j < static_cast<int>(blockIdx.x); j += n_threads) carry += __ldcg(ws.block_sum + j);
  carry = block_sum_ll(carry, red);
  for (int i = 0; i < warp; ++i) carry += wsum[i];

  // d. final decode from the synchronised starts.  Each lane decodes its
  // subsequence in rounds of up to kRound symbols into its row of the warp's
  // buffer; the warp then stores the rows, one per instruction, instead of 32
  // scattered words.
  const int shr = 32 - P.p;
  bool bad = false;
  for (long long k0 = k_begin; k0 < k_end; k0 += 32) {
    stage_words(k0);
    const long long k = k0 + lane;
    int b = b_first, end = 0, pos = 0, n_mine = 0;
    bool first = false, last = false;
    if (k < k_end) {
      end = locate(k, b, first, last);
      pos = ws.start[k];
      n_mine = ws.cnt[k];
    }
    const bool some = end > 0;
    // output positions: exclusive scan of the counts
    int x = n_mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    int32_t* const dst = P.out + carry + lane;
    int at = x - n_mine;  // this lane's next symbol, from carry on: at most 32 x (256 + kRound)
    int room = 0;         // and how many it may still write
    if (k < k_end) {
      const long long o = carry + at, img_end = __ldg(P.sym_off + b + 1);
      if (first && o != __ldg(P.sym_off + b)) atomicOr(ws.status, kBadCount);
      room = static_cast<int>(max(min(img_end - o, 1LL << 16), 0LL));
    }
    carry += __shfl_sync(0xffffffffu, x, 31);
    const Tables<SH> tab = tables(b);
    // this lane's rows in the value table (at most 2^28); -1: its entries are values
    const int vals = ws.direct && __ldcg(ws.direct + b) ? -1 : b * P.max_table;
    const bool direct = __all_sync(0xffffffffu, vals < 0);
    while (__any_sync(0xffffffffu, pos < end)) {
      int n = 0;
#pragma unroll
      for (int u0 = 0; u0 < kRound; u0 += kStep) {
        int len = 1;
#pragma unroll
        for (int u = u0; u < u0 + kStep; u += 2) {  // the whole warp, without divergence
          const uint32_t w = window(row, pos);
          const int e0 = tab.lut(w >> shr), l0 = e0 & 15;
          const int e1 = tab.lut(w << l0 >> shr);
          len = e1 & 15;
          wbuf[lane * kRow + u] = static_cast<uint16_t>(e0);
          wbuf[lane * kRow + u + 1] = static_cast<uint16_t>(e1);
          if (pos < end) {
            pos += l0;
            ++n;
          }
          if (pos < end) {
            pos += len;
            ++n;
          }
        }
        if (len == 0 && pos < end) {  // stuck at a bit pattern that is no codeword
          bad = true;
          pos = end;
        }
        if (!__any_sync(0xffffffffu, pos < end)) break;
      }
      // one word describes a lane's row: where it goes, and how much of it
      s_desc[lane] = static_cast<unsigned>(at) << 6 | static_cast<unsigned>(max(min(n, room), 0));
      at += n;
      room -= n;  // (negative: more symbols than the image has)
      __syncwarp();
      // eight rows' loads ahead of their stores (which the compiler cannot
      // tell from the shared memory they come from)
#pragma unroll
      for (int j0 = 0; j0 < 32; j0 += 8) {
        unsigned pk[8];
        int q[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          pk[j] = s_desc[j0 + j];
          q[j] = static_cast<int16_t>(wbuf[(j0 + j) * kRow + lane]) >> 4;
        }
        if (!direct) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int v = __shfl_sync(0xffffffffu, vals, j0 + j);
            if (v >= 0 && lane < static_cast<int>(pk[j] & 63u)) q[j] = __ldg(P.tab_value + v + (q[j] & 0xFFF));
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (lane < static_cast<int>(pk[j] & 63u)) dst[pk[j] >> 6] = q[j];
      }
      __syncwarp();
    }
    if (some) {
      if (room < 0) atomicOr(ws.status, kBadCount);
      if (last && pos != end) atomicOr(ws.status, kBadCode);  // the image's last codeword overruns
    }
  }
  if (blockIdx.x == gridDim.x - 1 && tid == n_threads - 1 && carry != __ldg(P.sym_off + P.B))
    atomicOr(ws.status, kBadCount);
  if (bad) atomicOr(ws.status, kBadCode);
}

__global__ void __launch_bounds__(kMaxWarps * 32, kCtasPerSm) huff_decode(const DecodeParams P) {
  cg::grid_group grid = cg::this_grid();
  extern __shared__ __align__(16) uint8_t s_dyn[];
  const Ws& ws = P.ws;
  const int tid = threadIdx.x, n_threads = blockDim.x, n_warps = n_threads >> 5;

  // this CTA's groups, and this warp's among them
  const int cta = blockIdx.x, warp = tid >> 5;
  const long long g_cta = P.groups_base + (cta < P.groups_more), g0 = cta * P.groups_base + min(cta, P.groups_more);
  const int g_warp = static_cast<int>(g_cta / n_warps), g_more = static_cast<int>(g_cta % n_warps);
  const long long gw = g0 + warp * static_cast<long long>(g_warp) + min(warp, g_more);
  const long long c_begin = min(32 * g0, P.n_sub), c_end = min(32 * (g0 + g_cta), P.n_sub);
  const long long k_begin = min(32 * gw, P.n_sub), k_end = min(32 * (gw + g_warp + (warp < g_more)), P.n_sub);
  // the first words, which the making of the tables leaves alone
  stage(P, words_of(s_dyn, P.p) + (tid >> 5) * kWbuf, k_begin);

  // 0. tables
  if (P.parts > 0) {
    if (blockIdx.x == 0 && tid < 4 + kMaxPasses) ws.status[tid] = 0;  // and the pass counters behind it
    bool bad_table = false;
    for (int u = blockIdx.x; u < P.B * P.parts; u += gridDim.x)
      bad_table |= build_tables(P, u / P.parts, u % P.parts, s_dyn);
    grid.sync();
    if (bad_table && tid == 0) atomicOr(ws.status, kBadTable);
  }

  // every lookup is a dependent load in a decode chain: the tables of the
  // CTA's first and last image go to shared memory.  A range with images in
  // between (only tiny streams produce one) reads all of its from global.
  const int size = 1 << P.p;
  const int b_first = image_of(P, c_begin * kQ, 0, P.B - 1);
  const int b_last = image_of(P, (c_end - 1) * kQ, b_first, P.B - 1);
  if (b_last - b_first > 1) {
    decode_phases<false>(P, grid, s_dyn, b_first, b_last, k_begin, k_end);
    return;
  }
  for (int q = 0; q <= b_last - b_first; ++q) {
    const uint16_t* gl = ws.lut + (static_cast<long long>(b_first + q) << P.p);
    const uint8_t* gm = ws.multi + (static_cast<long long>(b_first + q) << P.p);
    uint8_t* sl = s_dyn + q * 2 * size;
    uint8_t* sm = s_dyn + (4 + q) * size;
    if (P.p >= 4) {
#pragma unroll 2
      for (int i = tid; i < size / 8; i += n_threads)
        reinterpret_cast<uint4*>(sl)[i] = __ldcg(reinterpret_cast<const uint4*>(gl) + i);
      for (int i = tid; ws.multi && i < size / 16; i += n_threads)
        reinterpret_cast<uint4*>(sm)[i] = __ldcg(reinterpret_cast<const uint4*>(gm) + i);
    } else if (tid < size) {
      reinterpret_cast<uint16_t*>(sl)[tid] = __ldcg(gl + tid);
      if (ws.multi) sm[tid] = __ldcg(gm + tid);
    }
  }
  __syncthreads();
  if (!ws.multi) {
    for (int i = tid; i < (b_last - b_first + 1) * size; i += n_threads)
      s_dyn[4 * size + i] = static_cast<uint8_t>(
          codewords_in(reinterpret_cast<const uint16_t*>(s_dyn) + (i & -size), i & (size - 1), P.p));
    __syncthreads();
  }
  decode_phases<true>(P, grid, s_dyn, b_first, b_last, k_begin, k_end);
}

// Phase 0 alone, a CTA per image, for batches of more images than huff_decode
// has CTAs: 2,048 threads of an SM make tables instead of 1,024 (3,000 images of
// 300 symbols at p = 12 128 -> 125 us, 10,000 of 20 at p = 6 89 -> 72 us).
constexpr int kTableThreads = 256;
__global__ void __launch_bounds__(kTableThreads) huff_tables(const DecodeParams P) {
  extern __shared__ __align__(16) uint8_t s_dyn[];
  if (build_tables(P, blockIdx.x, 0, s_dyn) && threadIdx.x == 0) atomicOr(P.ws.status, kBadTable);
}

bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Resident CTAs of huff_decode on the current device with `smem` bytes of
// lookup tables each (the cooperative grid), per device and precision.
int decode_grid(int p, int* grid) {
  constexpr int kMaxDev = 64;
  static std::atomic<int> cached[kMaxDev][PIC_HUFF_MAX_PRECISION + 1];  // (first calls may come from several threads)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
    cudaGetLastError();
    return PIC_ERR_CUDA;
  }
  if (cached[dev][p] == 0) {
    int coop = 0, sms = 0, per_sm = 0;
    // the attribute is the function's, for every precision: set it to the largest
    if (cudaFuncSetAttribute(huff_decode, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem_bytes(PIC_HUFF_MAX_PRECISION, kMaxWarps))) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, huff_decode, 32 * kMaxWarps,
                                                      smem_bytes(p, kMaxWarps)) != cudaSuccess) {
      cudaGetLastError();
      return PIC_ERR_CUDA;
    }
    if (!coop || per_sm < 1) return PIC_ERR_UNSUPPORTED;
    cached[dev][p] = sms * per_sm < kMaxGrid ? sms * per_sm : kMaxGrid;
  }
  *grid = cached[dev][p];
  return PIC_OK;
}

}  // namespace

extern "C" {

int64_t pic_huffman_workspace_bytes(int64_t n_words, int B, int p) {
  if (n_words < 0 || n_words % kQ != 0 || B < 1 || p < 1 || p > PIC_HUFF_MAX_PRECISION) return -1;
  return ws_size(n_words / kQ, B, p);
}

int pic_huffman_decode(const uint32_t* words, int64_t n_words, const int64_t* word_off,
                       const int64_t* n_bits, int B, const int32_t* tab_value, const int32_t* tab_len,
                       int max_table, int p, const int64_t* sym_off, int32_t* out, void* workspace,
                       size_t workspace_bytes, void* stream) {
  if (n_words < 1 || n_words % kQ != 0 || B < 1 || B > 65536 || p < 1 || p > PIC_HUFF_MAX_PRECISION ||
      max_table < 1 || max_table > kMaxTable)
    return PIC_ERR_INVALID_ARG;
  if (!words || !word_off || !n_bits || !tab_value || !tab_len || !sym_off || !out || !workspace ||
      !aligned(words, 16) || !aligned(workspace, 16) || !aligned(word_off, 8) || !aligned(n_bits, 8) ||
      !aligned(sym_off, 8) || !aligned(tab_value, 4) || !aligned(tab_len, 4) || !aligned(out, 4))
    return PIC_ERR_INVALID_ARG;
  const long long n_sub = n_words / kQ;
  const bool small = static_cast<long long>(workspace_bytes) < ws_size(n_sub, B, p);
  if (small && static_cast<long long>(workspace_bytes) < ws_size_small(n_sub, B, p)) return PIC_ERR_INVALID_ARG;
  int grid = 0;
  int rc = decode_grid(p, &grid);
  if (rc != PIC_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  DecodeParams P{};
  P.words = words;
  P.n_words = n_words;
  P.word_off = reinterpret_cast<const long long*>(word_off);
  P.n_bits = reinterpret_cast<const long long*>(n_bits);
  P.B = B;
  P.p = p;
  P.sym_off = reinterpret_cast<const long long*>(sym_off);
  P.tab_value = tab_value;
  P.tab_len = tab_len;
  P.max_table = max_table;
  P.out = out;
  P.ws = ws_view(workspace, n_sub, B, p, small);
  P.n_sub = n_sub;
  const long long groups = (n_sub + 31) / 32;
  // the fewest rounds that the resident warps can do the groups in, and the
  // warps per CTA that it takes
  const long long rounds = (groups + kMaxWarps * grid - 1) / (kMaxWarps * grid);
  const long long per = (groups + rounds * grid - 1) / (rounds * grid);
  const int warps = static_cast<int>(per < kMinWarps ? kMinWarps : per);
  // at least the CTAs that the tables can be made by: small images then have
  // CTAs of their own, whose shared memory holds their tables (256 images of
  // 64x64: 86 us packed, 38 us spread)
  const long long g = std::min<long long>(std::max<long long>((groups + warps - 1) / warps, kMaxParts * (long long)B), grid);
  P.groups_base = groups / g;
  P.groups_more = static_cast<int>(groups % g);
  P.parts = 1;
  while (P.parts < kMaxParts && p >= 8 && 2LL * P.parts * B <= g) P.parts *= 2;
  if (B > grid) {
    P.parts = 0;
    // images of less than 2^(p - 2) bits do not repay the 2^p steps that a table of
    // their windows' codewords takes (3,000 images of 30 symbols 136 -> 95 us)
    if (128 * n_words < static_cast<long long>(B) << p) P.ws.multi = nullptr;
    if (cudaMemsetAsync(workspace, 0, kHead, s) != cudaSuccess) {  // status, pass counters
      cudaGetLastError();
      return PIC_ERR_CUDA;
    }
    huff_tables<<<B, kTableThreads, (size_t{6} << p) + 4, s>>>(P);
  }
  void* args[] = {&P};
  if (cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(huff_decode), dim3(static_cast<unsigned>(g)),
                                  dim3(32 * warps), args, smem_bytes(p, warps), s) != cudaSuccess) {
    cudaGetLastError();
    return PIC_ERR_CUDA;
  }
  if (cudaGetLastError() != cudaSuccess) return PIC_ERR_CUDA;
  return PIC_OK;
}

int pic_huffman_status(const void* workspace, void* stream) {
  if (!workspace) return PIC_ERR_INVALID_ARG;
  int st = 0;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemcpyAsync(&st, workspace, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return PIC_ERR_CUDA;
  }
  return st == 0 ? PIC_OK : PIC_ERR_INVALID_ARG;
}

}  // extern "C"
