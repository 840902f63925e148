// k_izpr.cu -- inverse ZpR on the GPU (Sec. 3.3, Fig. 2; App. B, Algorithm 1),
// behind the C ABI of include/pic_izpr.h.
//
// Algorithm 1 expands each block from its end-of-block marker offsets, which
// the paper finds beforehand by a stream compaction.  Here, with the stream
// cut into 2048-symbol chunks:
// 1. izpr_count: the eob markers of each group of 4 chunks, and before each
//    chunk within its group.
// 2. izpr_expand: persistent CTAs do the compaction and the expansion
//    together, chunk by chunk, as a segmented scan; a CTA takes every
//    gridDim-th chunk and adds up the groups that it passes over, which gives
//    it the chunk's first block.  Each thread holds 16
//    consecutive symbols of the chunk in registers (loaded while the CTA
//    expanded its previous chunk) and reduces them to (markers, positions
//    covered since its last marker); warp 0 reads the 96 symbols before the
//    chunk (a block has at most 64 symbols before its marker, so the marker
//    ending the previous block is in that halo); a CTA-wide scan gives each
//    thread the block and zigzag position of its first symbol, and each
//    thread walks its symbols as Algorithm 1 walks a block: a literal goes to
//    the next zigzag position, a run code of n zeros skips n positions, a
//    marker closes the block (its stream index is Algorithm 1's offset).  The
//    blocks, assembled in shared memory, leave as whole 256-byte blocks.
// The stream is read twice; nothing else touches HBM but the coefficients and
// offsets written.
//
// What bounds it: small streams, the launches -- two, where a memset of the
// status word and a scan of the counts by one CTA made it four -- and large
// ones, the instructions of the walks (66 for 32 symbols).
// Measured, with four launches and now: one 768x512 image (407 k symbols) 16.7
// -> 10.6 us, the 64-image batch (26 M symbols) 100 -> 96 us, one symbol 15.2 ->
// 9.9 us.
// Chunks differ in cost: one of 2,048 empty blocks writes 512 KB in 22 passes,
// one of long blocks 10 KB in one.  Dealt out in turn, a flat stretch of the
// stream is shared by all CTAs; in contiguous ranges, one per CTA, a few CTAs
// get it whole.  64 images, the first 32 flat: 82 us in turn, 200 us in ranges,
// which take 92 us on the even batch.
#include <algorithm>
#include <atomic>
#include <cstdint>

#include <cuda_runtime.h>

#include "pic_decode.h"
#include "pic_izpr.h"

namespace pic {
namespace {

constexpr int kThreads = 128;
constexpr int kPerThread = 16;
constexpr int kChunk = kThreads * kPerThread;  // symbols per compaction chunk

enum : int { kBadBlock = 1, kBadCount = 2 };

constexpr int kGroup = 4;  // chunks whose markers one CTA counts
// CTAs of izpr_expand: its threads load at most three groups' counts each from
// one of a CTA's chunks to the next
constexpr int kMaxGrid = (3 * kThreads - 1) * kGroup;

// Workspace: status word, each group's markers, and before each chunk those of
// its group.  What callers provide is 5.5 bytes a chunk, as it was with groups
// of 8 and their first blocks beside the counts: no less than these 5 take.
struct Workspace {
  int* status;
  int* gcount;
  int* local;
};
__host__ __device__ inline long long n_chunks_of(long long n) { return (n + kChunk - 1) / kChunk; }
__host__ __device__ inline long long n_groups_of(long long n) { return (n_chunks_of(n) + kGroup - 1) / kGroup; }
__host__ __device__ inline long long align16(long long b) { return (b + 15) / 16 * 16; }
__host__ __device__ inline long long ws_bytes(long long n) {
  const long long c = n_chunks_of(n), eights = (c + 7) / 8;
  return 32 + align16(4 * eights) + align16(4 * c) + 8 * eights;
}
__host__ __device__ inline Workspace ws_view(void* w, long long n) {
  char* p = static_cast<char*>(w);
  return Workspace{reinterpret_cast<int*>(p), reinterpret_cast<int*>(p + 32),
                   reinterpret_cast<int*>(p + 32 + align16(4 * n_groups_of(n)))};
}

// Zigzag order of an 8x8 block (raster index of the k-th zigzag position):
// anti-diagonal d = row + col, row falling for even d, rising for odd d.
struct ZigzagTable {
  int v[64];
};
constexpr ZigzagTable make_zigzag() {
  ZigzagTable t{};
  int k = 0;
  for (int d = 0; d < 15; ++d) {
    const int first = d < 8 ? 0 : d - 7;
    const int last = d < 8 ? d : 7;
    for (int s = 0; s <= last - first; ++s) {
      const int row = (d & 1) ? first + s : last - s;
      t.v[k++] = row * 8 + (d - row);
    }
  }
  return t;
}

// 16 consecutive symbols from stream index i0 into r; positions past the
// end read as `fill`.  16-byte loads when the stream is 16-byte aligned.
__device__ __forceinline__ void load16(const int32_t* __restrict__ sym, long long n, long long i0,
                                       bool vec, int fill, int (&r)[16]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long i = i0 + 4 * q;
    if (vec && i + 3 < n) {
      const int4 v = __ldg(reinterpret_cast<const int4*>(sym + i));
      r[4 * q] = v.x;
      r[4 * q + 1] = v.y;
      r[4 * q + 2] = v.z;
      r[4 * q + 3] = v.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) r[4 * q + u] = i + u < n ? __ldg(sym + i + u) : fill;
    }
  }
}

// The markers of group blockIdx.x, and before each of its chunks.  What bounds
// it is DRAM for large streams (6 TB/s) and one load's latency for small ones:
// thread t loads symbols 4t .. 4t + 3 of all four chunks at once (groups of 8:
// the same, and one image 5.0 instead of 3.4 us).
constexpr int kCountThreads = kChunk / 4;
__global__ void __launch_bounds__(kCountThreads) izpr_count(const int32_t* __restrict__ sym, long long n, int32_t eob,
                                                            long long n_chunks, Workspace ws) {
  constexpr int kWarps = kCountThreads / 32;
  __shared__ unsigned s_cnt[kWarps];
  const int t = threadIdx.x, lane = t & 31;
  const long long c0 = static_cast<long long>(blockIdx.x) * kGroup, i0 = c0 * kChunk + 4 * t;
  const bool vec = (reinterpret_cast<uintptr_t>(sym) & 15u) == 0;
  static_assert(kGroup == 4 && kWarps <= 32, "a byte per chunk, a lane per warp");
  unsigned cnt = 0u;  // a byte per chunk: at most 4 a thread, 128 a warp
  if (vec && (c0 + kGroup) * kChunk <= n) {
    int4 v[kGroup];
#pragma unroll
    for (int k = 0; k < kGroup; ++k) v[k] = __ldg(reinterpret_cast<const int4*>(sym + i0 + k * kChunk));
#pragma unroll
    for (int k = 0; k < kGroup; ++k)
      cnt += static_cast<unsigned>((v[k].x == eob) + (v[k].y == eob) + (v[k].z == eob) + (v[k].w == eob)) << 8 * k;
  } else {
#pragma unroll
    for (int k = 0; k < kGroup; ++k) {
      const long long i = i0 + k * kChunk;
#pragma unroll
      for (int u = 0; u < 4; ++u) cnt += static_cast<unsigned>(i + u < n && __ldg(sym + i + u) == eob) << 8 * k;
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) s_cnt[t / 32] = cnt;
  __syncthreads();
  if (t >= 32) return;
  const unsigned x = lane < kWarps ? s_cnt[lane] : 0u;
  const unsigned even = __reduce_add_sync(0xffffffffu, x & 0x00FF00FFu), odd = __reduce_add_sync(0xffffffffu, x >> 8 & 0x00FF00FFu);
  if (lane == 0) {
    const int m[4] = {static_cast<int>(even & 0xFFFF), static_cast<int>(odd & 0xFFFF), static_cast<int>(even >> 16), static_cast<int>(odd >> 16)};
    int run = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (c0 + k < n_chunks) ws.local[c0 + k] = run;
      run += m[k];
    }
    ws.gcount[blockIdx.x] = run;
  }
  if (t == 0 && blockIdx.x == 0) *ws.status = 0;
}

// Compaction and expansion in one pass over the stream, as a segmented scan.
// A block holds at most 64 symbols before its marker, so the marker that
// precedes a chunk's first block lies within the kHalo symbols before the
// chunk (or the block is malformed).  CTAs take chunks c, c + grid, ...; for each:
//  - every thread holds 16 consecutive symbols of the chunk in registers
//    (loaded while the CTA worked on its previous chunk) and reduces them to
//    (markers, positions covered since its last marker);
//  - warp 0 finds the halo's last marker and the positions of the part of
//    the chunk's first block that lies in the halo (they carry in);
//  - a CTA-wide segmented scan of the (markers, positions) pairs gives each
//    thread the block of its first symbol (block q of the chunk = block
//    gb0 + q of the stream) and the zigzag position reached in it;
//  - each thread walks its symbols: a literal goes to the block's next
//    zigzag position, a run code of n zeros skips n positions, a marker
//    closes the block (its stream index is Algorithm 1's offset);
//  - the blocks, assembled in shared memory, leave as whole 256-byte blocks
//    in raster order.
// Symbols after the chunk's last marker belong to the next chunk's first
// block; here they land in a spare block slot that is cleared, not written
// out.  A chunk with more than kMaxBlk blocks (only possible with very short
// blocks) is expanded in several passes over its block range.
constexpr int kHalo = 96;                   // 3 symbols per lane of warp 0
constexpr int kMaxBlk = 96;                 // blocks assembled per pass
constexpr int kBlkStride = 68;              // words per block slot: equal raster
                                            // entries of neighbouring blocks
                                            // fall 4 banks apart
constexpr int kExpandSmem = (kMaxBlk + 1) * kBlkStride * 4  // block slots + spare
                            + 64 * 4                        // scan scratch
                            + 64 + 16;                      // zigzag table, halo carry

// Segmented-scan combine: (m1, s1) then (m2, s2) -> markers m1 + m2, and
// the positions covered since the last marker.
struct Seg {
  int m, s;
};
__device__ __forceinline__ Seg seg_cat(Seg a, Seg b) { return Seg{a.m + b.m, b.m > 0 ? b.s : a.s + b.s}; }

__global__ void __launch_bounds__(kThreads, 8) izpr_expand(const int32_t* __restrict__ sym,
                                                        long long n, int32_t eob,
                                                        long long n_chunks, const int* __restrict__ gcount,
                                                        const int* __restrict__ local, long long n_blocks,
                                                        int32_t* __restrict__ coeffs,
                                                        int64_t* __restrict__ offsets, int* status) {
  extern __shared__ __align__(16) unsigned char smem[];
  int* s_buf = reinterpret_cast<int*>(smem);
  int* s_scan = s_buf + (kMaxBlk + 1) * kBlkStride;
  unsigned char* s_zz = reinterpret_cast<unsigned char*>(s_scan + 64);
  int* s_carry = reinterpret_cast<int*>(s_zz + 64);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  constexpr int kWarps = kThreads / 32;
  if (t < 64) s_zz[t] = static_cast<unsigned char>(make_zigzag().v[t]);
  if (blockIdx.x == 0 && t == 0) {
    if (__ldg(sym + n - 1) != eob) atomicOr(status, kBadCount);  // symbols after the last marker
  }
  for (int j = t; j < (kMaxBlk + 1) * kBlkStride / 4; j += kThreads)
    reinterpret_cast<int4*>(s_buf)[j] = make_int4(0, 0, 0, 0);
  const bool vec = (reinterpret_cast<uintptr_t>(sym) & 15u) == 0;
  const uint32_t ueob16 = static_cast<uint32_t>(eob) - 16u;  // first run code
  // Past the end of the stream the symbols read as a literal (eob - 17):
  // never a marker, and only ever in the spare slot.
  const int fill = static_cast<int>(static_cast<uint32_t>(eob) - 17u);

  // The halo of chunk c for warp 0 (lane l: symbols c0 - kHalo + 3 l .. + 2);
  // before the stream they act as markers.
  auto load_halo = [&](long long c, int (&h)[3]) {
    const long long hi = c * kChunk - kHalo + 3 * lane;
#pragma unroll
    for (int u = 0; u < 3; ++u) h[u] = (warp != 0 || hi + u < 0) ? eob : __ldg(sym + hi + u);
  };

  // the blocks before group g: the counts of the groups passed over, up to three a thread
  int* const s_sum = s_scan + 2 * kWarps;
  int passed[3];
  auto load_passed = [&](long long g, long long g_next) {
    const int* const from = gcount + g + t;
    const int left = static_cast<int>(g_next - g) - t;
    passed[0] = left > 0 ? __ldg(from) : 0;
    passed[1] = left > kThreads ? __ldg(from + kThreads) : 0;
    passed[2] = left > 2 * kThreads ? __ldg(from + 2 * kThreads) : 0;
  };
  auto put_passed = [&]() {
    const int sum = __reduce_add_sync(0xffffffffu, passed[0] + passed[1] + passed[2]);
    if (lane == 0) s_sum[warp] = sum;
  };
  long long group_base = 0;
  auto add_passed = [&]() {
    static_assert(kWarps == 4, "one word per warp");
    const int4 q = *reinterpret_cast<const int4*>(s_sum);
    group_base += q.x + q.y + q.z + q.w;
  };

  // the next chunk's symbols, halo and first block, loaded one chunk ahead
  int cur[16], hcur[3], lcur = 0;
  const long long grid = gridDim.x;
  load16(sym, n, blockIdx.x * static_cast<long long>(kChunk) + 16 * t, vec, fill, cur);
  load_halo(blockIdx.x, hcur);
  lcur = __ldg(local + blockIdx.x);
  load_passed(0, blockIdx.x / kGroup);
  put_passed();
  __syncthreads();
  add_passed();
  for (long long c = blockIdx.x; c < n_chunks; c += grid) {
    const long long gb0 = group_base + lcur;
    const long long c0 = c * kChunk;
    int x16[16], h[3];
#pragma unroll
    for (int i = 0; i < 16; ++i) x16[i] = cur[i];
#pragma unroll
    for (int u = 0; u < 3; ++u) h[u] = hcur[u];
    const bool more = c + grid < n_chunks;
    if (more) {  // next chunk, in flight meanwhile
      load16(sym, n, (c + grid) * kChunk + 16 * t, vec, fill, cur);
      load_halo(c + grid, hcur);
      lcur = __ldg(local + c + grid);
      load_passed(c / kGroup, (c + grid) / kGroup);
    }

    // this thread's markers (bit i: symbol i) and positions since its last one
    unsigned mk = 0;
    int s = 0, vmax = x16[0];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int x = x16[i];
      const uint32_t d = static_cast<uint32_t>(x) - ueob16;
      const bool m = x == eob;
      mk |= m ? 1u << i : 0u;
      s = m ? 0 : s + (d < 16u ? static_cast<int>(d) + 1 : 1);
      vmax = max(vmax, x);
    }
    bool bad = vmax > eob;
    // warp-inclusive segmented scan
    Seg inc{__popc(mk), s};
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const Seg y{__shfl_up_sync(0xffffffffu, inc.m, o), __shfl_up_sync(0xffffffffu, inc.s, o)};
      if (lane >= o) inc = seg_cat(y, inc);
    }
    if (lane == 31) {
      s_scan[2 * warp] = inc.m;
      s_scan[2 * warp + 1] = inc.s;
    }
    // the halo (warp 0): its last marker, and the positions of the part of
    // the chunk's first block that lies in it
    int halo_pos = 0;
    if (warp == 0) {
      int last = -1;
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (h[u] == eob) last = 3 * lane + u;
      last = __reduce_max_sync(0xffffffffu, last);
      int sum = 0;
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        if (3 * lane + u <= last || last < 0) h[u] = eob;  // not part of the first block
        const uint32_t d = static_cast<uint32_t>(h[u]) - ueob16;
        sum += h[u] == eob ? 0 : (d < 16u ? static_cast<int>(d) + 1 : 1);
      }
      int x = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      halo_pos = x - sum;  // zigzag position of this lane's first halo symbol
      // a block with no marker in the halo has more than 64 symbols
      if (lane == 31) *s_carry = last < 0 ? 65 : x;
    }
    __syncthreads();  // warp totals and the halo carry

    // exclusive prefix of this thread: (block of its first symbol, position)
    Seg pre{0, *s_carry};
    int tot = 0;
#pragma unroll
    for (int w2 = 0; w2 < kWarps; ++w2) {
      const Seg v{s_scan[2 * w2], s_scan[2 * w2 + 1]};
      if (w2 < warp) pre = seg_cat(pre, v);
      tot += v.m;  // blocks of this chunk
    }
    {
      const Seg y{__shfl_up_sync(0xffffffffu, inc.m, 1), __shfl_up_sync(0xffffffffu, inc.s, 1)};
      if (lane > 0) pre = seg_cat(pre, y);
    }
    // offsets (Algorithm 1): the stream index of each marker
    {
      int q = pre.m;
      for (unsigned b = mk; b; b &= b - 1u, ++q) {
        const long long gb = gb0 + q;
        if (gb < n_blocks) offsets[gb] = c0 + 16 * t + (__ffs(b) - 1);
        else atomicOr(status, kBadCount);
      }
    }

    // expansion, kMaxBlk blocks of the chunk per pass; in a pass the blocks
    // outside it (and the next chunk's first block) go to the spare slot
    for (int p0 = 0; p0 < tot; p0 += kMaxBlk) {
      const int p1 = min(tot, p0 + kMaxBlk);
      const bool one_pass = tot <= kMaxBlk;  // then q - p0 never leaves [0, kMaxBlk]
      if (p0 == 0 && warp == 0) {  // the first block's literals from the halo
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const uint32_t d = static_cast<uint32_t>(h[u]) - ueob16;
          if (h[u] != eob && d > 16u && halo_pos < 64) s_buf[s_zz[halo_pos]] = h[u];
          halo_pos += h[u] == eob ? 0 : (d < 16u ? static_cast<int>(d) + 1 : 1);
        }
      }
      int q = pre.m, pos = pre.s;
      auto slot = [&](int qq) {
        return one_pass ? qq * kBlkStride : ((qq >= p0 && qq < p1) ? qq - p0 : kMaxBlk) * kBlkStride;
      };
      int qb = slot(q);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int x = x16[i];
        const uint32_t d = static_cast<uint32_t>(x) - ueob16;  // < 16: run code, 16: marker
        const int zz = s_zz[pos & 63];
        if (d > 16u) s_buf[qb + zz] = x;  // a literal (or a malformed value)
        if (d == 16u) {
          if (pos > 64) bad = true;
          ++q;
          pos = 0;
          qb = slot(q);
        } else {
          pos += d < 16u ? static_cast<int>(d) + 1 : 1;
        }
      }
      __syncthreads();  // the pass's blocks are assembled
      // copy-out: two blocks per warp instruction, 16 bytes per lane; every
      // slot used (the spare one too) is cleared for the next pass
      const int last_slot = one_pass ? p1 - p0 : kMaxBlk;
      for (int b = 2 * warp + (lane >> 4); b <= last_slot; b += 2 * kWarps) {
        int4* src = reinterpret_cast<int4*>(s_buf + b * kBlkStride) + (lane & 15);
        const int4 v = *src;
        *src = make_int4(0, 0, 0, 0);
        const long long gb = gb0 + p0 + b;
        if (b < p1 - p0 && gb < n_blocks) reinterpret_cast<int4*>(coeffs + gb * 64)[lane & 15] = v;
      }
      __syncthreads();  // the slots are clear again
    }
    if (bad) atomicOr(status, kBadBlock);
    if (c + 1 == n_chunks && t == 0 && gb0 + tot != n_blocks) atomicOr(status, kBadCount);
    if (more) put_passed();
    __syncthreads();  // the scan scratch and the halo carry are free again
    if (more) add_passed();
  }
}

__global__ void izpr_flag(int* status, int bits) { *status = bits; }

bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Resident CTAs of izpr_expand on the current device, set up once per device.
int expand_grid(int* grid) {
  constexpr int kMaxDev = 64;
  static std::atomic<int> cached[kMaxDev];  // (first calls may come from several threads at once)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
    cudaGetLastError();
    return PIC_ERR_CUDA;
  }
  if (cached[dev] == 0) {
    int sms = 0, per_sm = 0;
    if (cudaFuncSetAttribute(izpr_expand, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kExpandSmem) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, izpr_expand, kThreads,
                                                      kExpandSmem) != cudaSuccess ||
        per_sm < 1) {
      cudaGetLastError();
      return PIC_ERR_CUDA;
    }
    cached[dev] = std::min(sms * per_sm, kMaxGrid);
  }
  *grid = cached[dev];
  return PIC_OK;
}

}  // namespace
}  // namespace pic

extern "C" {

int64_t pic_izpr_workspace_bytes(int64_t n_symbols) {
  if (n_symbols < 0) return -1;
  return pic::ws_bytes(n_symbols);
}

int pic_izpr_decode(const int32_t* symbols, int64_t n_symbols, int32_t eob, int64_t n_blocks,
                    int32_t* coeffs, int64_t* offsets, void* workspace, size_t workspace_bytes,
                    void* stream) {
  using namespace pic;
  if (n_symbols < 0 || n_blocks < 0) return PIC_ERR_INVALID_ARG;
  if (!workspace || !aligned(workspace, 16)) return PIC_ERR_INVALID_ARG;
  if (static_cast<long long>(workspace_bytes) < ws_bytes(n_symbols)) return PIC_ERR_INVALID_ARG;
  if ((n_symbols > 0 && (!symbols || !aligned(symbols, 4))) ||
      (n_blocks > 0 && (!coeffs || !offsets || !aligned(coeffs, 16) || !aligned(offsets, 8))))
    return PIC_ERR_INVALID_ARG;
  if (eob < INT32_MIN + 17) return PIC_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Workspace ws = ws_view(workspace, n_symbols);
  const long long chunks = n_chunks_of(n_symbols);
  if (chunks > 0) {
    int grid = 0;
    if (expand_grid(&grid) != PIC_OK) return PIC_ERR_CUDA;
    izpr_count<<<static_cast<unsigned>(n_groups_of(n_symbols)), kCountThreads, 0, s>>>(symbols, n_symbols, eob, chunks,
                                                                                     ws);
    izpr_expand<<<static_cast<unsigned>(std::min<long long>(chunks, grid)), kThreads, kExpandSmem, s>>>(
        symbols, n_symbols, eob, chunks, ws.gcount, ws.local, n_blocks, coeffs, offsets, ws.status);
  } else {
    izpr_flag<<<1, 1, 0, s>>>(ws.status, n_blocks > 0 ? kBadCount : 0);  // no symbols, hence no markers
  }
  if (cudaGetLastError() != cudaSuccess) return PIC_ERR_CUDA;
  return PIC_OK;
}

int pic_izpr_status(const void* workspace, void* stream) {
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
