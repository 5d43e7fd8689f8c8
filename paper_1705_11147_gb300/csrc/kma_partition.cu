// Partitioned mode of the counting passes: the paper's owner-computes scheme (Section 5.1: a
// deterministic k-mer -> owner map, every owner counting in a table of its own) applied on one
// GPU, with owners small enough to count in one SM's shared memory.
//
//   part_scatter_kernel  every window becomes a record (key hash, rest of the key, extension
//                        outcomes); each tile of 8192 window starts is sorted by bucket (the top
//                        bits of the key hash) in shared memory and written out as it lies, with
//                        a row of bucket offsets
//   part_split_kernel    gathers a bucket's runs from many scatter tiles, orders them by sub-bucket
//                        (the next part of the hash) and appends each run to its sub-bucket
//   part_count_kernel    brings a sub-bucket into shared memory: all occurrences of a few hundred
//                        to a few thousand k-mers, counted there; only k-mers seen at least twice
//                        (every k-mer without the singleton filter) are listed
//   part_large_kernel    the same for sub-buckets that do not fit (very frequent k-mers)
//   part_build_kernel    the listed keys with their counters into the table, a range of slots at a
//                        time
//   part_insert_kernel   the output records, and the keys that left their range
//
// Why two sorts and no filter in front of the table: a Bloom test-and-set plus table atomics in
// L2 took 4.6 L2 requests per window, 21 ns per 1000 windows, and a second pass over the first
// sightings another 8 ns. A sort pass reads and writes 8 or 16 bytes per window in whole lines,
// and with all occurrences of a k-mer in one shared memory the singletons (error k-mers) are known
// exactly, so they cost no memory traffic outside the SM. 2.4 G windows, k = 51: 110 ms -> 78 ms
// from reads to answers, 166 M windows, k = 51: 8.2 ms -> 5.7 ms.
#include <mutex>
#include <utility>
#include <vector>

#include "kma_device.cuh"

namespace kma {

// ------------------------------------------------------------------ records
//
// A record keeps the key in hashed form: h = key_hash(lo, hi) is a bijection of lo for a given
// hi, so (h, hi) identifies the key and lo is recomputed only for the k-mers that reach the
// table. The top kInfoBits of h are implied by the bucket (at least 2^6 buckets) and make room
// for the two extension outcomes. 8 bytes for k <= 32 (hi = 0), 16 above.
//   word 0   left outcome (bits 58..60: 0-3 base, 4 none) | right outcome (61..63) | h bits 0..57
//   word 1   hi (k > 32)

constexpr unsigned kInfoBits = 6;
constexpr u64 kHashMask = (1ull << (64 - kInfoBits)) - 1;

__device__ __forceinline__ unsigned left_outcome(u64 r) { return (unsigned)(r >> 58) & 7u; }
__device__ __forceinline__ unsigned right_outcome(u64 r) { return (unsigned)(r >> 61); }

__device__ __forceinline__ u64 unxorshift33(u64 x) { return x ^ (x >> 33); }
// Inverse of key_hash in lo: fmix64 backwards (its shifts are involutions, its multipliers odd,
// the constants are their inverses modulo 2^64).
__device__ __forceinline__ u64 key_lo(u64 h, u64 hi) {
  u64 x = unxorshift33(h) * 0x9cb4b2f8129337dbull;
  x = unxorshift33(x) * 0x4f74430c22a54005ull;
  return unxorshift33(x) ^ (hi * 0x9e3779b97f4a7c15ull + 0x632be59bd9b4e019ull);
}

// Sub-bucket of a record inside its bucket: the 32 hash bits after the bucket's, scaled to n.
__device__ __forceinline__ unsigned sub_of(u64 r, unsigned log_b, unsigned n) {
  return __umulhi((unsigned)((r << log_b) >> 32), n);
}

// Sub-buckets per bucket, from the windows counted so far (the same value in every kernel of
// one finalize): `avg` records each on average.
__device__ __forceinline__ unsigned sub_buckets(const PartGeom& G) {
  const u64 per = (u64)G.avg << G.log_b;
  const u64 n = (__ldcg(&G.status->valid_windows) + per - 1) / per;
  return n < 1 ? 1u : n > G.sub_max ? G.sub_max : (unsigned)n;
}

// ------------------------------------------------------------------ small block helpers

template <int BYTES>
__device__ __forceinline__ void cp_async(unsigned dst, const void* src) {
  if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// 1-D bulk copy shared -> global (16-byte aligned, a multiple of 16 bytes).
__device__ __forceinline__ void tma_store_1d(void* dst, unsigned src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Until the committed stores have read their shared memory / are complete.
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Exclusive scan of one value per thread over the block; `total` is the block's sum. wsum: one
// word per warp (32). One block barrier inside, after which wsum may be read by other warps: a
// second call needs a barrier in between.
template <int THREADS>
__device__ __forceinline__ unsigned block_scan(unsigned v, unsigned* wsum, unsigned& total) {
  constexpr int kWarps = THREADS / 32;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (unsigned)o) incl += x;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  const unsigned ws = lane < kWarps ? wsum[lane] : 0u;
  unsigned wi = ws;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned x = __shfl_up_sync(0xffffffffu, wi, o);
    if (lane >= (unsigned)o) wi += x;
  }
  total = __shfl_sync(0xffffffffu, wi, 31);
  return __shfl_sync(0xffffffffu, wi - ws, warp) + incl - v;
}

// ------------------------------------------------------------------ scatter
//
// One tile = 8192 consecutive window starts; thread t takes the kScatterWpt consecutive starts
// t * kScatterWpt + j.
//  1. extract the windows (WindowRun), stage the records in shared memory, rank each inside its
//     bucket for this tile (shared-memory atomics);
//  2. exclusive scan of the bucket counts: the tile's offset row;
//  3. the staged records into bucket order (through registers, in place), and the sorted tile to
//     HBM with bulk copies.
// The tile keeps a fixed place (tile number * 8192 records), so nothing is reserved: no global
// atomics, no bucket capacities and no overflow, whatever the skew of the keys.

constexpr int kScatterThreads = 1024;
constexpr int kScatterWpt = 8;
constexpr int kScatterTile = kScatterThreads * kScatterWpt;
static_assert(kScatterTile == kPartTile && kScatterTile <= 8192, "ranks are 13 bits");
constexpr int kScatterMaxPer = (1 << kMaxLogBuckets) / kScatterThreads;  // buckets per thread

// The packed reads of the next tile are brought into shared memory while this one is sorted (as
// loads from L2 they took a third of a tile's time): the tile's positions with up to 256 before
// and 384 behind, in words of 128 positions from a multiple of 128 on.
constexpr unsigned kArenaPositions = kScatterTile + 256 + 384;
constexpr size_t kArenaStage = kArenaPositions / 4 * 2 + kArenaPositions / 8 * 2;  // codes, rcodes, inv, hq
static_assert(kArenaPositions % 128 == 0, "every staged array starts on 16 bytes");

__host__ __device__ constexpr size_t scatter_smem(unsigned log_b, int kw) {
  return (size_t)kScatterTile * kw * 8 + 2 * kArenaStage + ((size_t)4 << log_b) + 32 * 4;
}

template <int KW>
__global__ void __launch_bounds__(kScatterThreads, 1) part_scatter_kernel(const __grid_constant__ PartGeom G,
                                                                          const __grid_constant__ PartWindows W,
                                                                          const __grid_constant__ PartTiles T) {
  extern __shared__ __align__(128) unsigned char s_raw[];
  const unsigned B = 1u << G.log_b;
  __shared__ __align__(8) unsigned long long s_bar[2];
  __shared__ unsigned s_lost;
  u64* s_rec = reinterpret_cast<u64*>(s_raw);                                  // [tile * KW]
  unsigned char* s_arena = s_raw + (size_t)kScatterTile * KW * 8;              // [2][codes, rcodes, inv, hq]
  unsigned* s_bin = reinterpret_cast<unsigned*>(s_arena + 2 * kArenaStage);    // [B] counts, then offsets
  unsigned* s_wsum = s_bin + B;                                                // [32]
  const unsigned tid = threadIdx.x, lane = tid & 31;
  const unsigned n_tiles = (unsigned)((W.q1 - W.q0 + kScatterTile - 1) / kScatterTile);
  const unsigned per = (B + kScatterThreads - 1) / kScatterThreads;
  // first staged position of tile t, and (thread 0) its copies into buffer `buf`
  auto stage_from = [&](unsigned t) -> u64 {
    const u64 q = W.q0 + (u64)t * kScatterTile;
    return (q > 128 ? q - 128 : 0) & ~127ull;
  };
  auto issue = [&](unsigned t, unsigned buf) {
    const u64 q = W.q0 + (u64)t * kScatterTile, from = stage_from(t);
    const u64 end = ((q + kScatterTile < W.q1 ? q + kScatterTile : W.q1) + 256 + 127) & ~127ull;
    const unsigned n = (unsigned)(end - from);  // a multiple of 128, at most kArenaPositions
    const unsigned bar = smem_u32(&s_bar[buf]), dst = smem_u32(s_arena) + buf * (unsigned)kArenaStage;
    fence_proxy_async_smem();
    mbar_expect_tx(bar, n / 4 * 2 + n / 8 * 2);
    tma_load_1d(dst, W.codes + from / 32, n / 4, bar);
    tma_load_1d(dst + kArenaPositions / 4, W.rcodes + from / 32, n / 4, bar);
    tma_load_1d(dst + kArenaPositions / 2, W.inv + from / 64, n / 8, bar);
    tma_load_1d(dst + kArenaPositions / 2 + kArenaPositions / 8, W.hq + from / 64, n / 8, bar);
  };
  if (tid == 0) {
    s_lost = 0;
    mbar_init(smem_u32(&s_bar[0]), 1);
    mbar_init(smem_u32(&s_bar[1]), 1);
    if (blockIdx.x < n_tiles) issue(blockIdx.x, 0);
  }
  __syncthreads();
  unsigned acc_valid = 0, phases = 0, buf = 0;
  unsigned acc_bucket[kScatterMaxPer] = {};  // records of this thread's buckets, over the CTA's tiles
  for (unsigned t = blockIdx.x; t < n_tiles; t += gridDim.x, buf ^= 1) {
    // everyone is done with the other buffer: the previous tile was extracted some barriers ago
    if (tid == 0 && t + gridDim.x < n_tiles) issue(t + gridDim.x, buf ^ 1);
    if (!mbar_wait_bounded(smem_u32(&s_bar[buf]), (phases >> buf) & 1u, kWaitPolls)) s_lost = 1;
    const u64 q = W.q0 + (u64)t * kScatterTile + (u64)tid * kScatterWpt;
    WindowRun<KW> win;
    win.valid = 0;
    if (q < W.q1) {  // q1 - q0 is a multiple of 64: all kScatterWpt starts are inside
      const unsigned char* a = s_arena + buf * kArenaStage;
      win.init(reinterpret_cast<const u64*>(a), reinterpret_cast<const u64*>(a + kArenaPositions / 4),
               reinterpret_cast<const u64*>(a + kArenaPositions / 2),
               reinterpret_cast<const u64*>(a + kArenaPositions / 2 + kArenaPositions / 8), G.k, q - stage_from(t),
               q == 0, true);
    }
    if (tid == 0) tma_store_wait_read();  // the previous tile has left shared memory
    for (unsigned p = tid; p < B; p += kScatterThreads) s_bin[p] = 0;
    __syncthreads();
    if (s_lost) {  // uniform: a copy did not land. Report; those in flight land now (bounded)
      if (tid == 0) {
        atomicOr(&G.status->flags, kFlagTimeout);
        mbar_drain(smem_u32(&s_bar[buf]), (phases >> buf) & 1u, kWaitPolls);
        if (t + gridDim.x < n_tiles) mbar_drain(smem_u32(&s_bar[buf ^ 1]), (phases >> (buf ^ 1)) & 1u, kWaitPolls);
      }
      break;
    }
    phases ^= 1u << buf;
    unsigned pr[kScatterWpt];  // bucket << 13 | rank, or ~0u
#pragma unroll
    for (int j = 0; j < kScatterWpt; ++j) pr[j] = 0xFFFFFFFFu;
#pragma unroll
    for (int j = 0; j < kScatterWpt; ++j) {
      if (!((win.valid >> j) & 1u)) continue;
      u64 lo, hi;
      const bool forward = win.key(j, G.canonical, lo, hi);
      const u64 h = key_hash(lo, hi);
      if (G.n_parts > 1 && owner_of(h, G.n_parts) != G.part) continue;
      ++acc_valid;
      const unsigned slot = j * kScatterThreads + tid, top = (unsigned)(h >> 32);
      const unsigned p = top >> (32 - G.log_b);
      pr[j] = (p << 13) | atomicAdd(&s_bin[p], 1u);
      const u64 r = ((u64)((top & (unsigned)(kHashMask >> 32)) | win.info(j, forward)) << 32) | (unsigned)h;
      if (KW == 1) s_rec[slot] = r;
      else reinterpret_cast<ulonglong2*>(s_rec)[slot] = make_ulonglong2(r, hi);
    }
    __syncthreads();
    // bucket offsets (thread t: buckets t * per ..), written as the tile's row
    unsigned c[kScatterMaxPer];
    unsigned local = 0;
#pragma unroll
    for (unsigned x = 0; x < kScatterMaxPer; ++x) {
      const unsigned p = tid * per + x;
      c[x] = x < per && p < B ? s_bin[p] : 0u;
      local += c[x];
      acc_bucket[x] += c[x];
    }
    unsigned total;
    unsigned run = block_scan<kScatterThreads>(local, s_wsum, total);
    unsigned short* row = T.offs + (T.tile0 + t) * T.stride;
#pragma unroll
    for (unsigned x = 0; x < kScatterMaxPer; ++x) {
      const unsigned p = tid * per + x;
      if (x < per && p < B) {
        s_bin[p] = run;
        row[p] = (unsigned short)run;
        run += c[x];
      }
    }
    if (tid == 0) row[B] = (unsigned short)total;
    // own records back into registers, then to their sorted places
    u64 r0[kScatterWpt], r1[kScatterWpt];
#pragma unroll
    for (int j = 0; j < kScatterWpt; ++j) {
      const unsigned slot = j * kScatterThreads + tid;
      if (pr[j] != 0xFFFFFFFFu) {
        if (KW == 1) {
          r0[j] = s_rec[slot];
        } else {
          const ulonglong2 v = reinterpret_cast<const ulonglong2*>(s_rec)[slot];
          r0[j] = v.x;
          r1[j] = v.y;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kScatterWpt; ++j) {
      if (pr[j] == 0xFFFFFFFFu) continue;
      const unsigned at = s_bin[pr[j] >> 13] + (pr[j] & 8191u);
      if (KW == 1) s_rec[at] = r0[j];
      else reinterpret_cast<ulonglong2*>(s_rec)[at] = make_ulonglong2(r0[j], r1[j]);
    }
    fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0 && total) {
      unsigned char* dst = reinterpret_cast<unsigned char*>(T.recs) + (T.tile0 + t) * (u64)(kScatterTile * KW * 8);
      const unsigned bytes = (total * KW * 8 + 15u) & ~15u;
      for (unsigned o = 0; o < bytes; o += 16384u)
        tma_store_1d(dst + o, smem_u32(s_rec) + o, bytes - o < 16384u ? bytes - o : 16384u);
      tma_store_commit();
    }
  }
  if (tid == 0) tma_store_wait();  // complete before the CTA may leave
#pragma unroll
  for (unsigned x = 0; x < kScatterMaxPer; ++x)
    if (acc_bucket[x]) atomicAdd(&T.totals[tid * per + x], (u64)acc_bucket[x]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc_valid += __shfl_down_sync(0xffffffffu, acc_valid, o);
  if (lane == 0 && acc_valid) atomicAdd(&G.status->valid_windows, (u64)acc_valid);
}

// ------------------------------------------------------------------ split
//
// One work item = a chunk of scatter tiles x kSplitBuckets adjacent buckets. The offset rows of
// the chunk's tiles are read once for all of the item's buckets (adjacent entries of a row).
// Per bucket: the lengths of its runs are scanned, the records gathered into shared memory (a
// few lanes per run, 8- or 16-byte asynchronous copies) and ordered by sub-bucket (a list of
// record numbers: the records stay where they are), at most kPartSubTile at a time (a chunk is
// sized so that one such sub-tile is the rule).
// Each sub-bucket's run then takes the next places of its sub-bucket (one atomic per run) and is
// written there, so that the count kernel finds a sub-bucket in one piece: gathering it there, a
// handful of records per run, took more instructions than the counting. Items go through the
// buckets in order, so the pieces of one line meet in L2. A sub-bucket has room for G.cap
// records; what does not fit (very frequent k-mers) goes to an overflow segment of the bucket.
//
// Bound by the waits on shared memory between its steps (134 instructions a record, 46 % of the
// issue slots used, DRAM at 4.3 TB/s); a third and a fourth CTA per SM (40 and 32 registers) and
// sub-tiles of 3072, 6144 or 8192 records were slower. 134 M records of 16 bytes: 0.94 ms; 2.4 G
// of them: 25 ms (1.17 and 27 ms when the records were moved to their sorted places, from and to
// registers).

constexpr int kSplitThreads = 512;
constexpr int kSplitItems = kPartSubTile / kSplitThreads;
constexpr int kSplitMaxPer = kMaxSubBuckets / kSplitThreads;  // sub-buckets per thread
static_assert(kPartSubTile <= 8192, "ranks are 13 bits");

// Where sub-bucket p of n comes in a sorted sub-tile: thread t sorts p = t, t + kSplitThreads, ..
__device__ __forceinline__ unsigned sub_order(unsigned p, unsigned n) {
  return (p % kSplitThreads) * ((n + kSplitThreads - 1) / kSplitThreads) + p / kSplitThreads;
}

// First overflow segment of each bucket of [b0, b1): a sub-tile makes one at most.
constexpr int kBaseThreads = 1024;
__global__ void __launch_bounds__(kBaseThreads) part_base_kernel(const u64* totals, unsigned b0, unsigned b1,
                                                                 unsigned n_chunks, unsigned* seg_base) {
  __shared__ unsigned s_sum[32];
  constexpr unsigned kPer = (1u << kMaxLogBuckets) / kBaseThreads;
  unsigned v[kPer], local = 0, total;
#pragma unroll
  for (unsigned x = 0; x < kPer; ++x) {
    const unsigned b = b0 + threadIdx.x * kPer + x;
    v[x] = b < b1 ? (unsigned)(totals[b] / kPartSubTile) + n_chunks : 0u;
    local += v[x];
  }
  unsigned run = block_scan<kBaseThreads>(local, s_sum, total);
#pragma unroll
  for (unsigned x = 0; x < kPer; ++x) {
    const unsigned b = b0 + threadIdx.x * kPer + x;
    if (b < b1) seg_base[b - b0] = run;
    run += v[x];
  }
}

__host__ __device__ constexpr size_t split_smem(unsigned chunk_tiles, unsigned sub_max, int kw) {
  return (size_t)kPartSubTile * (kw * 8 + 2) + (size_t)sub_max * (4 + 4 + 2) + 32 * 4 + (size_t)chunk_tiles * 4 +
         (((size_t)chunk_tiles * (kSplitBuckets + 1) * 2 + 15) & ~(size_t)15);
}

template <int KW>
__global__ void __launch_bounds__(kSplitThreads, 2) part_split_kernel(const __grid_constant__ PartGeom G,
                                                                      const __grid_constant__ PartTiles T,
                                                                      const __grid_constant__ PartSplit S) {
  extern __shared__ __align__(128) unsigned char s_raw[];
  __shared__ u64 s_over;
  u64* s_rec = reinterpret_cast<u64*>(s_raw);                                  // [sub-tile * KW]
  unsigned short* s_ord = reinterpret_cast<unsigned short*>(s_rec + kPartSubTile * KW);  // [sub-tile] record at a sorted place
  unsigned* s_bin = reinterpret_cast<unsigned*>(s_ord + kPartSubTile);         // [sub_max] counts, then offsets
  unsigned* s_to = s_bin + G.sub_max;                                          // [sub_max] place minus sorted position
  unsigned* s_wsum = s_to + G.sub_max;                                         // [32]
  unsigned* s_dst = s_wsum + 32;                                               // [chunk tiles] first record of the run
  unsigned short* s_lim = reinterpret_cast<unsigned short*>(s_dst + S.chunk_tiles);  // [sub_max] end of what fits
  unsigned short* s_off = s_lim + G.sub_max;                                   // [chunk tiles][buckets + 1]
  const unsigned tid = threadIdx.x;
  const unsigned n_sub = sub_buckets(G);
  const unsigned per_sub = (n_sub + kSplitThreads - 1) / kSplitThreads;
  const unsigned n_blocks = (S.b1 - S.b0 + kSplitBuckets - 1) / kSplitBuckets;
  const unsigned n_chunks = (T.n_tiles + S.chunk_tiles - 1) / S.chunk_tiles;
  const u64 n_items = (u64)n_chunks * n_blocks;
  const unsigned glanes = 1u << S.log_lanes, gl = tid & (glanes - 1), gi = tid >> S.log_lanes,
                 gn = kSplitThreads >> S.log_lanes;
  for (u64 item = blockIdx.x; item < n_items; item += gridDim.x) {
    const unsigned chunk = (unsigned)(item % n_chunks);
    const unsigned bb = S.b0 + (unsigned)(item / n_chunks) * kSplitBuckets;
    const unsigned nb = S.b1 - bb < kSplitBuckets ? S.b1 - bb : kSplitBuckets;
    const unsigned t0 = chunk * S.chunk_tiles;
    const unsigned nt = T.n_tiles - t0 < S.chunk_tiles ? T.n_tiles - t0 : S.chunk_tiles;
    __syncthreads();  // the previous item's offsets are no longer read
    for (unsigned i = tid; i < nt; i += kSplitThreads) {
      // eight entries in one load (groups of buckets start at multiples of 8, rows are padded), and the next one
      static_assert(kSplitBuckets == 8, "an item's offsets are one 16-byte load");
      const unsigned short* row = T.offs + (u64)(t0 + i) * T.stride + bb;
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(row));
      const unsigned next = __ldg(row + kSplitBuckets);  // inside the row's padding for the last buckets
      unsigned short* o = s_off + i * (kSplitBuckets + 1);
      o[0] = (unsigned short)v.x, o[1] = (unsigned short)(v.x >> 16);
      o[2] = (unsigned short)v.y, o[3] = (unsigned short)(v.y >> 16);
      o[4] = (unsigned short)v.z, o[5] = (unsigned short)(v.z >> 16);
      o[6] = (unsigned short)v.w, o[7] = (unsigned short)(v.w >> 16);
      o[8] = (unsigned short)next;
    }
    __syncthreads();
    const unsigned per = (nt + kSplitThreads - 1) / kSplitThreads;  // runs per thread
    for (unsigned j = 0; j < nb; ++j) {
      unsigned local = 0, total;
      for (unsigned x = 0; x < per; ++x) {
        const unsigned i = tid * per + x;
        if (i < nt) local += s_off[i * (kSplitBuckets + 1) + j + 1] - s_off[i * (kSplitBuckets + 1) + j];
      }
      unsigned run = block_scan<kSplitThreads>(local, s_wsum, total);
      for (unsigned x = 0; x < per; ++x) {
        const unsigned i = tid * per + x;
        if (i < nt) {
          s_dst[i] = run;
          run += s_off[i * (kSplitBuckets + 1) + j + 1] - s_off[i * (kSplitBuckets + 1) + j];
        }
      }
      const u64 sub0 = (u64)(bb + j - S.b0) * n_sub;  // the bucket's first sub-bucket
      u64* out = S.recs + sub0 * G.cap * KW;
      for (unsigned w0 = 0; w0 < total; w0 += kPartSubTile) {
        const unsigned n = total - w0 < kPartSubTile ? total - w0 : kPartSubTile;
        for (unsigned p = tid; p < n_sub; p += kSplitThreads) s_bin[p] = 0;
        __syncthreads();  // also: s_dst is set, the previous sub-tile has been written
        // gather the window [w0, w0 + n) of the bucket's records
        if (total <= kPartSubTile) {
          for (unsigned i = gi; i < nt; i += gn) {
            const unsigned a = s_off[i * (kSplitBuckets + 1) + j], len = s_off[i * (kSplitBuckets + 1) + j + 1] - a;
            const u64* src = T.recs + ((u64)(t0 + i) * kPartTile + a + gl) * KW;
            unsigned dst = smem_u32(s_rec) + (s_dst[i] + gl) * (8 * KW);
            for (unsigned x = gl; x < len; x += glanes, src += glanes * KW, dst += glanes * 8 * KW) cp_async<8 * KW>(dst, src);
          }
        } else for (unsigned i = gi; i < nt; i += gn) {
          const unsigned a = s_off[i * (kSplitBuckets + 1) + j], len = s_off[i * (kSplitBuckets + 1) + j + 1] - a;
          const unsigned d = s_dst[i];
          if (d >= w0 + n || d + len <= w0) continue;
          const unsigned x0 = d < w0 ? w0 - d : 0u, x1 = d + len > w0 + n ? w0 + n - d : len;
          const u64* src = T.recs + ((u64)(t0 + i) * kPartTile + a) * KW;
          for (unsigned x = x0 + gl; x < x1; x += glanes)
            cp_async<8 * KW>(smem_u32(s_rec + (size_t)(d + x - w0) * KW), src + (u64)x * KW);
        }
        cp_async_wait_all();
        __syncthreads();
        unsigned pr[kSplitItems];
#pragma unroll
        for (int y = 0; y < kSplitItems; ++y) {
          const unsigned x = y * kSplitThreads + tid;
          pr[y] = 0xFFFFFFFFu;
          if (x < n) {
            const unsigned p = sub_of(s_rec[x * KW], G.log_b, n_sub);
            pr[y] = (p << 13) | atomicAdd(&s_bin[p], 1u);
          }
        }
        __syncthreads();
        unsigned c[kSplitMaxPer];
        u64 at[kSplitMaxPer];
        unsigned lc = 0, tot2;
#pragma unroll
        for (unsigned x = 0; x < kSplitMaxPer; ++x) {  // places taken; in flight during the scan
          if (x >= per_sub) break;
          const unsigned p = x * kSplitThreads + tid;
          c[x] = p < n_sub ? s_bin[p] : 0u;
          at[x] = c[x] ? atomicAdd(&S.fill[sub0 + p], (u64)c[x]) : 0;
          lc += c[x];
        }
        unsigned ro = block_scan<kSplitThreads>(lc, s_wsum, tot2);
#pragma unroll
        for (unsigned x = 0; x < kSplitMaxPer; ++x) {
          if (x >= per_sub) break;
          const unsigned p = x * kSplitThreads + tid;
          if (p < n_sub) {
            s_bin[p] = ro;
            ro += c[x];
          }
        }
        __syncthreads();
#pragma unroll
        for (int y = 0; y < kSplitItems; ++y) {
          if (pr[y] == 0xFFFFFFFFu) continue;
          s_ord[s_bin[pr[y] >> 13] + (pr[y] & 8191u)] = (unsigned short)(y * kSplitThreads + tid);
        }
        unsigned over = 0;  // the places, taken by now
#pragma unroll
        for (unsigned x = 0; x < kSplitMaxPer; ++x) {
          if (x >= per_sub) break;
          const unsigned p = x * kSplitThreads + tid;
          if (p < n_sub) {
            const unsigned room = at[x] < G.cap ? G.cap - (unsigned)at[x] : 0u, fits = c[x] < room ? c[x] : room;
            const unsigned o = s_bin[p];
            s_to[p] = p * G.cap + (unsigned)at[x] - o;
            s_lim[p] = (unsigned short)(o + fits);
            c[x] -= fits;
            over += c[x];
          }
        }
        const int any_over = __syncthreads_or(over != 0);
        if (any_over) {  // the block's records that found no room: numbered, and a segment for them
          unsigned n_over;
          unsigned o = block_scan<kSplitThreads>(over, s_wsum, n_over);
#pragma unroll
          for (unsigned x = 0; x < kSplitMaxPer; ++x) {
            if (x >= per_sub) break;
            const unsigned p = x * kSplitThreads + tid;
            if (p < n_sub) {
              s_bin[p] = o - s_lim[p];  // overflow number minus sorted position
              o += c[x];
            }
          }
          if (tid == 0) {
            const u64 pos = atomicAdd(S.over_n, (u64)n_over);
            const unsigned b = bb + j - S.b0;
            PartSegment sg;
            sg.pos = pos;
            sg.n = n_over;
            sg.pad = 0;
            S.segs[S.seg_base[b] + atomicAdd(&S.n_segs[b], 1u)] = sg;
            s_over = pos;
          }
          __syncthreads();
        }
        if (!any_over) {
#pragma unroll
          for (int y = 0; y < kSplitItems; ++y) {
            const unsigned i = y * kSplitThreads + tid;
            if (i >= n) break;
            u64 v0, v1 = 0;
            if (KW == 1) {
              v0 = s_rec[s_ord[i]];
            } else {
              const ulonglong2 v = reinterpret_cast<const ulonglong2*>(s_rec)[s_ord[i]];
              v0 = v.x;
              v1 = v.y;
            }
            u64* to = out + (u64)(s_to[sub_of(v0, G.log_b, n_sub)] + i) * KW;
            if (KW == 1) *to = v0;
            else *reinterpret_cast<ulonglong2*>(to) = make_ulonglong2(v0, v1);
          }
        } else {
          for (unsigned i = tid; i < n; i += kSplitThreads) {
            u64 v0, v1 = 0;
            if (KW == 1) {
              v0 = s_rec[s_ord[i]];
            } else {
              const ulonglong2 v = reinterpret_cast<const ulonglong2*>(s_rec)[s_ord[i]];
              v0 = v.x;
              v1 = v.y;
            }
            const unsigned p = sub_of(v0, G.log_b, n_sub);
            u64* to = i < s_lim[p] ? out + (u64)(s_to[p] + i) * KW : S.over + (s_over + (s_bin[p] + i)) * KW;
            if (KW == 1) *to = v0;
            else *reinterpret_cast<ulonglong2*>(to) = make_ulonglong2(v0, v1);
          }
        }
        __syncthreads();  // s_bin, s_rec and s_wsum are rewritten
      }
      if (total == 0) __syncthreads();  // s_wsum
    }
  }
}

// ------------------------------------------------------------------ count
//
// One work item = one sub-bucket, brought into shared memory by bulk copies while the previous
// one is counted (two buffers, two CTAs per SM). Then
//  1. every record writes its number at the entry its hash picks, the last one wins;
//  2. it compares its key with the winner's: equal keys share the winner as their representative,
//     without an atomic or a loop. The others (fewer than one in ten) find theirs in a second table
//     by compare-and-swap and probing, compacted into full warps first;
//  3. representatives that another record joined take a block of ten 16-bit counters (a staged
//     sub-bucket has fewer than 2^16 records);
//  4. every record of such a key adds its two outcomes;
//  5. these keys with their counters (all keys without the singleton filter) are appended to a
//     list for part_build_kernel: inserted here, a few keys per sub-bucket would leave most threads
//     waiting for the table's round trips (34 ms -> 47 ms for 2.4 G windows).
// Sub-buckets that overflowed (very frequent k-mers) and those with more keys than the second
// table holds are listed for part_large_kernel.
//
// Bound by the barriers between the steps and by shared memory (207 instructions a record, 56 % of
// the issue slots used). 166 M records of 16 bytes: 1.65 ms; 2.4 G of them: 23.0 ms. Rejected: a
// table with the keys and counters themselves that records are added to from registers (a probe of
// a 16-byte key behind a 64-bit compare-and-swap takes 70 instructions for 32 records, 12 in all
// per record and warp instead of 6).

constexpr int kCountThreads = 640;  // 512 and 768: 1 % and 6 % slower
constexpr int kCountCtas = 2;                // per SM
constexpr unsigned kEntries = 8192;          // first entries, 16 bits (4096: 4 % slower, more records for the second table)
constexpr unsigned kEntries2 = 1024;         // second table, 32 bits
constexpr unsigned kNoEntry = 0xFFFFFFFFu;   // empty entry
constexpr unsigned kOnce = 0xFFFFu;          // counter block of a representative nobody joined, and of no representative
constexpr unsigned kJoined = 0xFFFEu;        // joined, block not taken yet
constexpr unsigned kLone = 0x8000u;          // without the singleton filter: number among the keys seen once
constexpr unsigned kRangeBits = 20;          // hash bits 21..40: part_large_kernel takes a range of them at a time

// Counters of a key in 16-bit halves of six words: left A C G T none, (a half not used), right
// A C G T none, (not used). The outcome bits of a record lie in the top byte of its first word:
// v = outcome bits << 2. Byte offset of the counter's word, and 1 in the counter's half of it:
__device__ __forceinline__ unsigned left_word(unsigned v) { return (v >> 1) & 12u; }
__device__ __forceinline__ unsigned left_one(unsigned v) { return 1u << ((v << 2) & 16u); }
__device__ __forceinline__ unsigned right_word(unsigned v) { return 12u + ((v >> 4) & 12u); }
__device__ __forceinline__ unsigned right_one(unsigned v) { return 1u << ((v >> 1) & 16u); }
constexpr unsigned kCtrWords = 6;

// An entry of the list of counted keys: the six counter words (the half not used of the third
// one is undefined), then h and hi.
template <int KW>
constexpr unsigned kKeyWords = kCtrWords + 2 * KW;

template <int KW>
struct CountShape {
  static constexpr unsigned kCap = KW == 1 ? kCountCap1 : kCountCap2;
  static constexpr size_t kRec = (size_t)kCap * KW * 8;
  static constexpr size_t kIdx = ((size_t)kCap * 2 + 15) & ~(size_t)15;  // representative; counter block
  static constexpr size_t kTab = (size_t)kEntries * 2 + kEntries2 * 4 + kIdx;  // entries, second table, list of step 2
  static constexpr size_t kCtr = ((size_t)(kCap / 2) * kCtrWords * 4 + 15) & ~(size_t)15;
  static constexpr size_t kSmem = 2 * kRec + 2 * kIdx + (kTab > kCtr ? kTab : kCtr);  // steps 1 and 2 share the counters' room
  static_assert(kCap < kLone && kCap % 2 == 0, "record numbers are 16 bits, bulk copies of 16 bytes");
};

// Slot-to-be of one key in the table: the key's words and where its probes begin.
struct Place {
  Slot* sub;
  u64 lo, hi, idx;
};
__device__ __forceinline__ Place place_of(const PartGeom& G, u64 h, u64 hi) {
  Place p;
  p.lo = key_lo(h, hi);
  p.hi = hi;
  p.sub = G.table + (u64)part_of(h, G.P) * G.Sp;
  p.idx = table_index(h, G.Sp, G.P);
  return p;
}

// A slot of 64 bytes: key, counters without a neighbour, counters.
__device__ __forceinline__ void write_slot(Slot* s, const unsigned (&ctr)[10]) {
  *reinterpret_cast<uint4*>(&s->none[0]) = make_uint4(ctr[4], ctr[9], 0u, 0u);
  *reinterpret_cast<uint4*>(&s->ext[0]) = make_uint4(ctr[0], ctr[1], ctr[2], ctr[3]);
  *reinterpret_cast<uint4*>(&s->ext[4]) = make_uint4(ctr[5], ctr[6], ctr[7], ctr[8]);
}

// Puts a key with its ten counters (left A C G T none, right A C G T none) into the table, whose
// slots below S.end have been written. The key is in no slot yet and no other thread inserts it, so
// the first empty slot takes it. If that lies in the next group's part of the table the key is
// carried over to it (no more than kMaxProbe can be: every one of them takes one of the next
// kMaxProbe slots, or the table is full).
__device__ __forceinline__ bool insert_key(const PartGeom& G, const PartSplit& S, u64 h, u64 hi, const unsigned (&ctr)[10]) {
  Place p = place_of(G, h, hi);
  const u64 limit = G.Sp < kMaxProbe ? G.Sp : kMaxProbe;
  for (u64 n = 0; n < limit; ++n) {
    if (p.sub + p.idx == G.table + S.end) {
      const u64 at = atomicAdd(S.n_carry_out, 1ull);
      if (at >= kMaxProbe) break;
      unsigned* c = S.carry_out + at * kCarryWords;
#pragma unroll
      for (int x = 0; x < 10; ++x) c[x] = ctr[x];
      c[10] = (unsigned)h;
      c[11] = (unsigned)(h >> 32);
      c[12] = (unsigned)hi;
      c[13] = (unsigned)(hi >> 32);
      return false;
    }
    u64 olo, ohi;
    cas128(p.sub + p.idx, kEmpty, kEmpty, p.lo, p.hi, olo, ohi);
    if (olo == kEmpty && ohi == kEmpty) {
      write_slot(p.sub + p.idx, ctr);
      return true;
    }
    p.idx = (p.idx + 1 == G.Sp) ? 0 : p.idx + 1;
  }
  atomicOr(&G.status->flags, kFlagFull);
  return false;
}

// Count of a key (its left outcomes; 0xFFFFFFFF and a flag above 32 bits), and its record at place
// `at` of the output. Returns whether both sides are unique.
__device__ __forceinline__ unsigned key_count(const PartGeom& G, const unsigned (&ctr)[10]) {
  return slot_count(ctr[4], make_uint4(ctr[0], ctr[1], ctr[2], ctr[3]), G.status);
}
__device__ __forceinline__ bool write_record(const PartGeom& G, const PartOut& O, u64 at, u64 lo, u64 hi, unsigned count,
                                             const unsigned (&ctr)[10]) {
  const unsigned l = side_code(ctr, O.min_ext), r = side_code(ctr + 5, O.min_ext);
  if (at < O.cap) {
    reinterpret_cast<ulonglong2*>(O.keys)[at] = make_ulonglong2(lo, hi);
    O.counts[at] = count;
    reinterpret_cast<uint4*>(O.ext)[2 * at] = make_uint4(ctr[0], ctr[1], ctr[2], ctr[3]);
    reinterpret_cast<uint4*>(O.ext)[2 * at + 1] = make_uint4(ctr[5], ctr[6], ctr[7], ctr[8]);
    reinterpret_cast<uchar2*>(O.codes)[at] = make_uchar2((unsigned char)l, (unsigned char)r);
  } else {
    atomicOr(&G.status->flags, kFlagOutput);
  }
  return l < 4 && r < 4;
}

constexpr u64 kFree = ~0ull;                 // part_large_kernel: first key word of an empty slot
constexpr u64 kLock = 1ull << 63;            // slot taken, second key word not written yet
constexpr unsigned kProbes = 128;

// One probe of part_large_kernel's table at `pos` for key (h, hi): kSame (the slot holds the key, taken
// for it now if it was empty), kOther, or (two-word keys) kAgain: a new key of two words is
// written behind a lock bit, within this call, so a lane that meets the locked slot of its own
// hash only has to come back.
enum : unsigned { kOther = 0, kSame = 1, kAgain = 2 };
template <int KW>
__device__ __forceinline__ unsigned probe_slot(u64* k0, u64* k1, unsigned pos, u64 h, u64 hi) {
  u64 e = *reinterpret_cast<volatile u64*>(&k0[pos]);
  if (e == kFree) {
    e = atomicCAS(&k0[pos], kFree, KW == 1 ? h : h | kLock);
    if (e == kFree) {
      if (KW == 2) {
        *reinterpret_cast<volatile u64*>(&k1[pos]) = hi;
        __threadfence_block();
        *reinterpret_cast<volatile u64*>(&k0[pos]) = h;
      }
      return kSame;
    }
  }
  if (KW == 1) return e == h ? kSame : kOther;
  if (e == h) return *reinterpret_cast<volatile u64*>(&k1[pos]) == hi ? kSame : kOther;
  return e == (h | kLock) ? kAgain : kOther;
}

// A sub-bucket of any size: its records (`n_in` in place, the rest among the bucket's overflow
// segments) are streamed from HBM through a shared-memory table with 32-bit counters, as often as
// its distinct keys need: one range of the hash at a time, halved when a probe of kProbes slots
// finds no place. Lanes with equal outcomes of equal keys act as one (frequent k-mers are
// accumulated in the warp first, Section 5.1). The keys go straight to the HBM table.
//
// Bound by the latency of the segments' records: a moderately frequent key has a few in every
// segment (a lane per segment), a hot one thousands (four rows of them in flight). A kernel of
// its own, whose CTAs take the next sub-bucket when they are done: as a function of the count
// kernel it held that to 64 registers (now 40) and left most CTAs waiting for those with a hot
// key. 343 M windows, 30 % of them a satellite's: 10.6 ms -> 5.4 ms with the counting.
constexpr int kLargeThreads = 512;
constexpr unsigned kLargeSlots = 2048;  // keys counted at a time

__host__ __device__ constexpr size_t large_smem(int kw) { return (size_t)kLargeSlots * (kw * 8 + 2 * 5 * 4); }

template <int KW>
__global__ void __launch_bounds__(kLargeThreads, 2) part_large_kernel(const __grid_constant__ PartGeom G,
                                                                      const __grid_constant__ PartSplit S,
                                                                      const __grid_constant__ PartOut O) {
  extern __shared__ __align__(128) unsigned char s_raw[];
  constexpr unsigned kSlots = kLargeSlots;
  __shared__ unsigned s_bad, s_item;
  u64* k0 = reinterpret_cast<u64*>(s_raw);                            // [slots] first key words
  u64* k1 = k0 + kSlots * (KW - 1);                                   // [slots] second ones
  unsigned* left = reinterpret_cast<unsigned*>(k0 + kSlots * KW);     // [slots * 5]
  unsigned* right = left + kSlots * 5;                                // [slots * 5]
  const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned n_sub = sub_buckets(G), n_items = (unsigned)__ldcg(S.n_large);
  unsigned acc_ins = 0, acc_first = 0;
  for (;;) {
    __syncthreads();
    if (tid == 0) s_item = atomicAdd(reinterpret_cast<unsigned*>(S.next_large), 1u);
    __syncthreads();
    if (s_item >= n_items) break;
    const unsigned item = S.large[s_item], b = S.b0 + item / n_sub, s = item % n_sub;
    const u64 fill = S.fill[item];
    const unsigned n_in = fill < G.cap ? (unsigned)fill : G.cap;
    const u64 htop = (u64)(b >> (G.log_b - kInfoBits)) << (64 - kInfoBits);
    const unsigned n_segs = fill > G.cap ? S.n_segs[b - S.b0] : 0u, order = sub_order(s, n_sub);
    const PartSegment* segs = S.segs + S.seg_base[b - S.b0];
    u64 lo = 0, width = 1ull << kRangeBits;
    while (lo < (1ull << kRangeBits)) {
      __syncthreads();
      for (unsigned i = tid; i < kSlots; i += kLargeThreads) k0[i] = kFree;
      for (unsigned i = tid; i < kSlots * 5; i += kLargeThreads) left[i] = right[i] = 0;
      if (tid == 0) s_bad = 0;
      __syncthreads();
      // one row of 32 records: lane's record (if `in`)
      auto row = [&](bool in, u64 r, u64 hi) {
        const u64 h = r & kHashMask, x = (h >> 21) & ((1u << kRangeBits) - 1);
        bool act = in && x >= lo && x < lo + width;
        if (*reinterpret_cast<volatile unsigned*>(&s_bad)) act = false;  // this range is counted again
        if (!__any_sync(0xffffffffu, act)) return;
        unsigned pos = (unsigned)h & (kSlots - 1), got = kOther;
        const unsigned jump = (unsigned)(h >> 11) | 1u;
        const bool mine = act;
        for (unsigned step = 0; step < kProbes; ++step) {
          if (act) {
            got = probe_slot<KW>(k0, k1, pos, h, hi);
            act = got != kSame;
            if (got == kOther) pos = (pos + jump) & (kSlots - 1);
          }
          if (!__any_sync(0xffffffffu, act)) break;
        }
        const bool hit = mine && got == kSame;
        if (mine && !hit) s_bad = 1;
        const unsigned l = left_outcome(r), o = right_outcome(r);
        const unsigned ml = __match_any_sync(0xffffffffu, hit ? pos * 8 + l : ~0u);
        const unsigned mo = __match_any_sync(0xffffffffu, hit ? pos * 8 + o : ~0u);
        if (hit) {
          bool wrap = false;
          if (lane == __ffs(ml) - 1) wrap |= atomicAdd(&left[pos * 5 + l], __popc(ml)) > 0xFFFFFFFFu - __popc(ml);
          if (lane == __ffs(mo) - 1) wrap |= atomicAdd(&right[pos * 5 + o], __popc(mo)) > 0xFFFFFFFFu - __popc(mo);
          if (wrap) atomicOr(&G.status->flags, kFlagOverflow);
        }
      };
      auto load = [&](const u64* p, u64& r, u64& hi) {
        if (KW == 1) {
          r = __ldg(p);
        } else {
          const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
          r = v.x;
          hi = v.y;
        }
      };
      const u64* in = S.recs + ((u64)(b - S.b0) * n_sub + s) * G.cap * KW;
      for (unsigned x0 = warp * 32; x0 < n_in; x0 += kLargeThreads) {
        u64 r = 0, hi = 0;
        if (x0 + lane < n_in) load(in + (u64)(x0 + lane) * KW, r, hi);
        row(x0 + lane < n_in, r, hi);
      }
      // the sub-bucket's records in the segments: each lane searches one segment, which is ordered by
      // sub-bucket, for the first of them. Neighbouring segments go to different warps: a bucket of a
      // small sample has a few of them, which one warp alone took one after another (4 Mbases,
      // 30 % of them a satellite's: 203 us -> 54 us)
      for (unsigned g0 = 0; g0 < n_segs; g0 += kLargeThreads) {
        const unsigned g = g0 + lane * (kLargeThreads / 32) + warp;
        PartSegment sg = {0, 0, 0};
        unsigned from = 0;
        if (g < n_segs) {
          sg = segs[g];
          unsigned end = sg.n;
          while (from < end) {
            const unsigned mid = (from + end) / 2;
            if (sub_order(sub_of(__ldg(S.over + (sg.pos + mid) * KW), G.log_b, n_sub), n_sub) < order) from = mid + 1;
            else end = mid;
          }
        }
        // the first few of every segment, a lane each
        constexpr int kFew = 4;
        u64 r[kFew], hi[kFew];
#pragma unroll
        for (int y = 0; y < kFew; ++y) {
          r[y] = hi[y] = 0;
          if (from + y < sg.n) load(S.over + (sg.pos + from + y) * KW, r[y], hi[y]);
        }
        bool more = true;
#pragma unroll
        for (int y = 0; y < kFew; ++y) {
          more = more && from + y < sg.n && sub_of(r[y], G.log_b, n_sub) == s;
          if (__any_sync(0xffffffffu, more)) row(more, r[y], hi[y]);
        }
        // the rest of the long ones (a hot key's), the warp together
        unsigned todo = __ballot_sync(0xffffffffu, more);
        for (; todo; todo &= todo - 1) {
          const int src = __ffs(todo) - 1;
          const u64 pos = __shfl_sync(0xffffffffu, sg.pos, src);
          const unsigned n = __shfl_sync(0xffffffffu, sg.n, src);
          for (unsigned x0 = __shfl_sync(0xffffffffu, from, src) + kFew; x0 < n; x0 += kFew * 32) {
#pragma unroll
            for (int y = 0; y < kFew; ++y) {
              const unsigned x = x0 + y * 32 + lane;
              if (x < n) load(S.over + (pos + x) * KW, r[y], hi[y]);
            }
            unsigned m = 0;
#pragma unroll
            for (int y = 0; y < kFew; ++y) {
              const bool mine = x0 + y * 32 + lane < n && sub_of(r[y], G.log_b, n_sub) == s;
              m = __ballot_sync(0xffffffffu, mine);
              if (m) row(mine, r[y], hi[y]);
            }
            if (m != 0xffffffffu) break;  // the last of them
          }
        }
      }
      __syncthreads();
      if (s_bad) {  // uniform
        if (width > 1) {
          width >>= 1;
          continue;
        }
        if (tid == 0) atomicOr(&G.status->flags, kFlagFull);  // cannot be: the hash has more bits than the range
      }
      for (unsigned i = tid; i < kSlots; i += kLargeThreads) {
        const u64 h = k0[i];
        if (h == kFree) continue;
        ++acc_first;
        unsigned v[10];
        u64 n = 0;
#pragma unroll
        for (int x = 0; x < 5; ++x) {
          v[x] = left[i * 5 + x];
          v[5 + x] = right[i * 5 + x];
          n += v[x];
        }
        if (n < G.min_count) continue;
        const u64 hi = KW == 2 ? k1[i] : 0;
        acc_ins += insert_key(G, S, h | htop, hi, v);
        const unsigned count = key_count(G, v);
        if (count >= O.min_depth && write_record(G, O, atomicAdd(&G.status->n_out, 1ull), key_lo(h | htop, hi), hi, count, v))
          atomicAdd(&G.status->n_uu, 1ull);
      }
      lo += width;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    acc_ins += __shfl_down_sync(0xffffffffu, acc_ins, o);
    acc_first += __shfl_down_sync(0xffffffffu, acc_first, o);
  }
  if (lane == 0) {
    if (acc_ins) atomicAdd(&G.status->table_keys, (u64)acc_ins);
    if (acc_first && G.min_count > 1) atomicAdd(&G.status->first_sightings, (u64)acc_first);
  }
}

template <int KW>
__global__ void __launch_bounds__(kCountThreads, kCountCtas) part_count_kernel(const __grid_constant__ PartGeom G,
                                                                               const __grid_constant__ PartSplit S) {
  using C = CountShape<KW>;
  extern __shared__ __align__(128) unsigned char s_raw[];
  __shared__ __align__(8) unsigned long long s_bar[2];
  __shared__ u64 s_fill[2], s_ahead, s_base;  // s_ahead: records of the item after the one whose copy is under way
  __shared__ unsigned s_nctr, s_nlone, s_nlist, s_state;
  const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned short* s_rep = reinterpret_cast<unsigned short*>(s_raw + 2 * C::kRec);           // [cap] representative
  unsigned short* s_q = reinterpret_cast<unsigned short*>(s_raw + 2 * C::kRec + C::kIdx);   // [cap] its counter block
  unsigned* s_ent2 = reinterpret_cast<unsigned*>(s_raw + 2 * C::kRec + 2 * C::kIdx);        // [entries2]
  unsigned short* s_ent = reinterpret_cast<unsigned short*>(s_ent2 + kEntries2);            // [entries]
  unsigned short* s_list = s_ent + kEntries;                                                // [cap] not settled yet (step 2)
  unsigned char* s_ctr = s_raw + 2 * C::kRec + 2 * C::kIdx;                                 // [cap / 2][kCtrWords * 4]
  const unsigned n_sub = sub_buckets(G);
  const unsigned n_items = (S.b1 - S.b0) * n_sub;  // at most 2^22
  unsigned acc_first = 0;  // per thread: below 2^32
  // thread 0: copy a sub-bucket's records into buffer `buf`
  auto issue = [&](unsigned buf, unsigned item, u64 fill) {
    s_fill[buf] = fill;
    const unsigned n = fill < G.cap ? (unsigned)fill : G.cap;
    const unsigned bytes = (n * (8 * KW) + 15u) & ~15u, bar = smem_u32(&s_bar[buf]);
    fence_proxy_async_smem();
    mbar_expect_tx(bar, bytes);
    const unsigned char* src = reinterpret_cast<const unsigned char*>(S.recs + (u64)item * G.cap * KW);
    const unsigned dst = smem_u32(s_raw) + buf * (unsigned)C::kRec;
    for (unsigned o = 0; o < bytes; o += 16384u) tma_load_1d(dst + o, src + o, bytes - o < 16384u ? bytes - o : 16384u, bar);
  };
  if (tid == 0) {
    mbar_init(smem_u32(&s_bar[0]), 1);
    mbar_init(smem_u32(&s_bar[1]), 1);
    s_state = s_nlist = 0;
    if (blockIdx.x < n_items) issue(0, blockIdx.x, __ldcg(&S.fill[blockIdx.x]));
    if (blockIdx.x + gridDim.x < n_items) s_ahead = __ldcg(&S.fill[blockIdx.x + gridDim.x]);
  }
  __syncthreads();
  unsigned phases = 0, buf = 0;  // bit b: parity to wait for on buffer b
  for (unsigned item = blockIdx.x; item < n_items; item += gridDim.x, buf ^= 1) {
    // bit 0 of s_state: a wait gave up; bit 1: the second table is full
    if (!mbar_wait_bounded(smem_u32(&s_bar[buf]), (phases >> buf) & 1u, kWaitPolls)) atomicOr(&s_state, 1u);
    __syncthreads();  // everyone is done with the previous sub-bucket
    const u64 fill = s_fill[buf];
    const unsigned n = fill < G.cap ? (unsigned)fill : G.cap;
    u64* s_rec = reinterpret_cast<u64*>(s_raw + buf * C::kRec);  // [cap * KW]
    // 1: numbers to the first entries
#pragma unroll 2
    for (unsigned x = tid; x < n; x += kCountThreads) {
      s_ent[(unsigned)s_rec[(size_t)x * KW] & (kEntries - 1)] = (unsigned short)x;
      s_q[x] = (unsigned short)kOnce;
    }
    if (tid < kEntries2 / 4) reinterpret_cast<uint4*>(s_ent2)[tid] = make_uint4(kNoEntry, kNoEntry, kNoEntry, kNoEntry);
    __syncthreads();
    if (s_state) {  // uniform: a copy did not land. Report; those in flight land now (bounded)
      if (tid == 0) {
        atomicOr(&G.status->flags, kFlagTimeout);
        mbar_drain(smem_u32(&s_bar[buf]), (phases >> buf) & 1u, kWaitPolls);
      }
      break;
    }
    phases ^= 1u << buf;
    if (tid == 0) {
      const unsigned next = item + gridDim.x;
      if (next < n_items) issue(buf ^ 1, next, s_ahead);
      if (next + gridDim.x < n_items) s_ahead = __ldcg(&S.fill[next + gridDim.x]);
      s_nctr = s_nlone = 0;
    }
    if (fill > G.cap) {  // uniform: left to part_large_kernel
      if (tid == 0) S.large[atomicAdd(S.n_large, 1ull)] = item;
      continue;
    }
    // 2: a representative for every record. The key of record z is (a0, a1)?
    auto same_key = [&](unsigned z, u64 a0, u64 a1) -> bool {
      if (KW == 1) return ((s_rec[z] ^ a0) & kHashMask) == 0;
      const ulonglong2 v = reinterpret_cast<const ulonglong2*>(s_rec)[z];
      return (((v.x ^ a0) & kHashMask) | (v.y ^ a1)) == 0;
    };
    unsigned firsts = 0;
#pragma unroll 2
    for (unsigned x0 = tid - lane; x0 < n; x0 += kCountThreads) {
      const unsigned x = x0 + lane;
      bool left = false;
      if (x < n) {
        u64 a0, a1 = 0;
        if (KW == 1) {
          a0 = s_rec[x];
        } else {
          const ulonglong2 v = reinterpret_cast<const ulonglong2*>(s_rec)[x];
          a0 = v.x;
          a1 = v.y;
        }
        const unsigned z = s_ent[(unsigned)a0 & (kEntries - 1)];
        const bool same = same_key(z, a0, a1);
        left = !same;
        firsts += z == x;
        if (same) s_rep[x] = (unsigned short)z;
        if (same && z != x) s_q[z] = (unsigned short)kJoined;
      }
      const unsigned lm = __ballot_sync(0xffffffffu, left);
      if (lm) {
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(&s_nlist, __popc(lm));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(lm & ((1u << lane) - 1u));
        if (left) s_list[at] = (unsigned short)x;
      }
    }
    __syncthreads();
    for (unsigned i = tid; i < s_nlist; i += kCountThreads) {
      const unsigned x = s_list[i];
      u64 a0, a1 = 0;
      if (KW == 1) {
        a0 = s_rec[x];
      } else {
        const ulonglong2 v = reinterpret_cast<const ulonglong2*>(s_rec)[x];
        a0 = v.x;
        a1 = v.y;
      }
      unsigned pos = (unsigned)(a0 >> 13) & (kEntries2 - 1), z = x, step = 0;
      const unsigned jump = (unsigned)(a0 >> 22) | 1u;  // odd: comes by every entry
      for (; step < kEntries2; ++step) {
        z = *reinterpret_cast<volatile unsigned*>(&s_ent2[pos]);
        if (z == kNoEntry) {
          z = atomicCAS(&s_ent2[pos], kNoEntry, x);
          if (z == kNoEntry) {
            z = x;
            ++firsts;
            break;
          }
        }
        if (same_key(z, a0, a1)) {
          s_q[z] = (unsigned short)kJoined;
          break;
        }
        pos = (pos + jump) & (kEntries2 - 1);
      }
      if (step == kEntries2) atomicOr(&s_state, 2u);  // more keys than the second table holds
      s_rep[x] = (unsigned short)z;
    }
    __syncthreads();
    if (s_state) {  // uniform
      __syncthreads();
      if (tid == 0) {
        s_state = s_nlist = 0;
        S.large[atomicAdd(S.n_large, 1ull)] = item;
      }
      continue;
    }
    acc_first += firsts;
    // 3: counter blocks
    for (unsigned x0 = warp * 32; x0 < n; x0 += kCountThreads) {
      const unsigned x = x0 + lane;
      const unsigned q0 = x < n ? s_q[x] : kOnce;
      const unsigned mm = __ballot_sync(0xffffffffu, q0 == kJoined);
      if (mm) {
        unsigned q = 0;
        if (lane == 0) q = atomicAdd(&s_nctr, __popc(mm));
        q = __shfl_sync(0xffffffffu, q, 0) + __popc(mm & ((1u << lane) - 1u));
        if (q0 == kJoined) {
          s_q[x] = (unsigned short)q;
          uint2* c = reinterpret_cast<uint2*>(s_ctr + q * (kCtrWords * 4));
          c[0] = make_uint2(0, 0);
          c[1] = make_uint2(x << 16, 0);  // the representative's number, in the half not used
          c[2] = make_uint2(0, 0);
        }
      }
      if (G.min_count <= 1) {
        const bool lone = x < n && q0 == kOnce && s_rep[x] == x;
        const unsigned lm = __ballot_sync(0xffffffffu, lone);
        unsigned q = 0;
        if (lane == 0 && lm) q = atomicAdd(&s_nlone, __popc(lm));
        q = __shfl_sync(0xffffffffu, q, 0) + __popc(lm & ((1u << lane) - 1u));
        if (lone) s_q[x] = (unsigned short)(kLone | q);
      }
    }
    __syncthreads();
    // 4: outcomes
    if (tid == 0) s_nlist = 0;
    if (tid == 0) {
      unsigned nk = s_nctr + s_nlone;
      s_base = nk ? atomicAdd(S.n_keys, (u64)nk) : 0;
      if (s_base + nk > S.keys_cap) {  // more keys than slots
        atomicOr(&G.status->flags, kFlagFull);
        nk = s_nctr = s_nlone = 0;
      }
      S.key_base[item] = s_base;
      S.key_n[item] = nk;
    }
#pragma unroll 2
    for (unsigned x = tid; x < n; x += kCountThreads) {
      const unsigned q = s_q[s_rep[x]];
      if (q < kLone) {
        const unsigned v = reinterpret_cast<const unsigned char*>(s_rec)[(size_t)x * (8 * KW) + 7];
        unsigned char* c = s_ctr + q * (kCtrWords * 4);
        atomicAdd(reinterpret_cast<unsigned*>(c + left_word(v)), left_one(v));
        atomicAdd(reinterpret_cast<unsigned*>(c + right_word(v)), right_one(v));
      }
    }
    __syncthreads();
    // 5: to the list
    const unsigned nq = s_nctr;
    const u64 htop = (u64)((S.b0 + item / n_sub) >> (G.log_b - kInfoBits)) << (64 - kInfoBits);
    unsigned* out = S.keys + s_base * kKeyWords<KW>;
    for (unsigned e = tid; e < nq * kKeyWords<KW>; e += kCountThreads) {
      const unsigned q = e / kKeyWords<KW>, w = e - q * kKeyWords<KW>;
      const unsigned* c = reinterpret_cast<const unsigned*>(s_ctr) + q * kCtrWords;
      unsigned v;
      if (w < kCtrWords) {
        v = c[w];
      } else {
        v = reinterpret_cast<const unsigned*>(s_rec + (size_t)(c[2] >> 16) * KW)[w - kCtrWords];
        if (w == kCtrWords + 1) v = (v & (unsigned)(kHashMask >> 32)) | (unsigned)(htop >> 32);
      }
      out[e] = v;
    }
    if (s_nlone) {
      for (unsigned x = tid; x < n; x += kCountThreads) {
        const unsigned q = s_q[x];
        if (q < kLone || q >= kJoined) continue;
        const u64 r = s_rec[(size_t)x * KW];
        const unsigned v = (unsigned)(r >> 56);
        unsigned* c = out + (size_t)(nq + (q & ~kLone)) * kKeyWords<KW>;
#pragma unroll
        for (unsigned w = 0; w < kCtrWords; ++w)
          c[w] = (left_word(v) == 4 * w ? left_one(v) : 0u) + (right_word(v) == 4 * w ? right_one(v) : 0u);
        const u64 kh = (r & kHashMask) | htop;
        c[kCtrWords] = (unsigned)kh;
        c[kCtrWords + 1] = (unsigned)(kh >> 32);
        if (KW == 2) {
          const u64 khi = s_rec[(size_t)x * KW + KW - 1];
          c[kKeyWords<KW> - 2] = (unsigned)khi;
          c[kKeyWords<KW> - 1] = (unsigned)(khi >> 32);
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc_first += __shfl_down_sync(0xffffffffu, acc_first, o);
  if (lane == 0 && acc_first && G.min_count > 1) atomicAdd(&G.status->first_sightings, (u64)acc_first);
}

// ------------------------------------------------------------------ table
//
// The table's slots follow the hash, so the keys of neighbouring sub-buckets go to a range of
// slots of their own: one CTA makes that range in shared memory, empty slots and all, and writes
// it with bulk copies (kBuildSlots at a time: as many sub-buckets as fill them, or a part of one).
// Nothing is cleared before and no slot is claimed in HBM. A key that finds no empty slot in its
// range (or whose first slot lies behind it) is marked; part_insert_kernel puts it into the table
// when all ranges of the group have been written.
//
// Bound by the latency of an item's few loads behind one another and by the table's write; one
// sub-bucket at a time was twice as slow. With the records (part_insert_kernel) 7.4 ms for 115 M
// keys in 317 M slots; clearing the table and claiming every slot with a compare-and-swap took
// 10.5 ms. 512 slots and 6 CTAs, 1024 and 3, 256 and 12: 7.5, 8.1, 7.4 ms.

constexpr int kBuildThreads = 256;
constexpr int kBuildCtas = 4;               // per SM
constexpr unsigned kBuildSlots = 768;
constexpr unsigned kBuildSubs = 16;         // sub-buckets at a time, at most
constexpr size_t kBuildSmem = (size_t)kBuildSlots * (sizeof(Slot) + 4);

// Slot of a hash in the whole table (never decreases with it), and the first one of sub-bucket s of
// n of bucket b.
__device__ __forceinline__ u64 slot_of(const PartGeom& G, u64 h) {
  return (u64)part_of(h, G.P) * G.Sp + table_index(h, G.Sp, G.P);
}
__device__ __forceinline__ u64 first_slot(const PartGeom& G, unsigned b, unsigned s, unsigned n) {
  if (b >> G.log_b) return (u64)G.P * G.Sp;
  const u64 x = (((u64)s << 32) + n - 1) / n;  // the smallest that sub_of takes to s
  return slot_of(G, ((u64)b << (64 - G.log_b)) | (x << (32 - G.log_b)));
}

template <int KW>
__global__ void __launch_bounds__(kBuildThreads, kBuildCtas) part_build_kernel(const __grid_constant__ PartGeom G,
                                                                      const __grid_constant__ PartSplit S) {
  extern __shared__ __align__(128) unsigned char s_raw[];
  uint4* s_slot = reinterpret_cast<uint4*>(s_raw);                                       // [slots][4]
  unsigned* s_taken = reinterpret_cast<unsigned*>(s_raw + kBuildSlots * sizeof(Slot));   // [slots]
  __shared__ u64 s_first[2][kBuildSubs];                 // first list entry of each sub-bucket, less the keys before it
  __shared__ unsigned s_upto[2][kBuildSubs];             // keys up to and with it
  const unsigned tid = threadIdx.x, n_sub = sub_buckets(G), n_subs = (S.b1 - S.b0) * n_sub;
  // as many neighbouring sub-buckets as fill the slots in shared memory
  const double ranges = (double)n_sub * (double)(1u << G.log_b), slots = (double)G.P * (double)G.Sp;
  const double fit = 0.95 * kBuildSlots * ranges / slots;
  const unsigned m = fit >= kBuildSubs ? kBuildSubs : fit < 2.0 ? 1u : (unsigned)fit;
  const unsigned n_items = (n_subs + m - 1) / m;
  unsigned acc_ins = 0, buf = 0;
  // the first warp: lists of an item's sub-buckets (loaded an item ahead)
  auto lists = [&](unsigned item, unsigned to) {
    if (tid >= 32) return;
    const unsigned sub = item * m + tid;
    const bool in = tid < m && item < n_items && sub < n_subs;
    const unsigned n = in ? S.key_n[sub] : 0u;
    const u64 base = n ? S.key_base[sub] : 0ull;
    unsigned upto = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned x = __shfl_up_sync(0xffffffffu, upto, o);
      if (tid >= (unsigned)o) upto += x;
    }
    if (tid < m) {
      s_upto[to][tid] = upto;
      s_first[to][tid] = base - (upto - n);
    }
  };
  lists(blockIdx.x, 0);
  for (unsigned item = blockIdx.x; item < n_items; item += gridDim.x, buf ^= 1) {
    const unsigned sub0 = item * m, sub1 = sub0 + m < n_subs ? sub0 + m : n_subs;
    const u64 begin = first_slot(G, S.b0 + sub0 / n_sub, sub0 % n_sub, n_sub);
    const u64 end = first_slot(G, S.b0 + sub1 / n_sub, sub1 % n_sub, n_sub);
    for (u64 c0 = begin; c0 < end || c0 == begin; c0 += kBuildSlots) {
      const unsigned ns = end - c0 < kBuildSlots ? (unsigned)(end - c0) : kBuildSlots;
      if (tid == 0) tma_store_wait_read();  // the previous slots have left shared memory
      __syncthreads();
      for (unsigned i = tid; i < ns * 4; i += kBuildThreads) {
        const unsigned v = i & 3 ? 0u : 0xFFFFFFFFu;
        s_slot[i] = make_uint4(v, v, v, v);
      }
      for (unsigned i = tid; i < ns; i += kBuildThreads) s_taken[i] = 0;
      __syncthreads();
      if (c0 == begin) lists(item + gridDim.x, buf ^ 1);  // read after the next barriers
      const unsigned nk = s_upto[buf][m - 1];
      for (unsigned i = tid; i < nk; i += kBuildThreads) {
        unsigned at = 0;
        while (i >= s_upto[buf][at]) ++at;
        unsigned* e = S.keys + (s_first[buf][at] + i) * kKeyWords<KW>;
        const uint2 hw = *reinterpret_cast<const uint2*>(e + kCtrWords);
        const u64 h = ((u64)hw.y << 32) | hw.x, g = slot_of(G, h);
        if (g >= end ? c0 + ns < end : g - c0 >= ns) continue;  // not of these slots (g >= begin)
        // probes go round at the end of the partition, which may lie inside the range
        const u64 round = ((u64)part_of(h, G.P) + 1) * G.Sp - c0;
        const unsigned last = round < ns ? (unsigned)round : ns;
        unsigned x = g < end ? (unsigned)(g - c0) : ns;
        while (x < last && atomicExch(&s_taken[x], 1u)) ++x;
        const uint2* w = reinterpret_cast<const uint2*>(e);
        const uint2 w2 = w[2];
        if (x >= last) {
          e[5] = w2.y | 0x10000u;  // marked, in the half not used
          continue;
        }
        const uint2 w0 = w[0], w1 = w[1];
        const u64 hi = KW == 2 ? *reinterpret_cast<const u64*>(e + kKeyWords<KW> - 2) : 0ull, lo = key_lo(h, hi);
        s_slot[4 * x] = make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
        s_slot[4 * x + 1] = make_uint4(w1.x & 0xFFFFu, w2.y & 0xFFFFu, 0u, 0u);
        s_slot[4 * x + 2] = make_uint4(w0.x & 0xFFFFu, w0.x >> 16, w0.y & 0xFFFFu, w0.y >> 16);
        s_slot[4 * x + 3] = make_uint4(w1.y & 0xFFFFu, w1.y >> 16, w2.x & 0xFFFFu, w2.x >> 16);
        ++acc_ins;
      }
      fence_proxy_async_smem();
      __syncthreads();
      if (tid == 0 && ns) {
        unsigned char* dst = reinterpret_cast<unsigned char*>(G.table + c0);
        const unsigned bytes = ns * (unsigned)sizeof(Slot);
        for (unsigned o = 0; o < bytes; o += 16384u)
          tma_store_1d(dst + o, smem_u32(s_raw) + o, bytes - o < 16384u ? bytes - o : 16384u);
        tma_store_commit();
      }
    }
  }
  if (tid == 0) tma_store_wait();  // complete before the CTA may leave
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc_ins += __shfl_down_sync(0xffffffffu, acc_ins, o);
  if ((tid & 31) == 0 && acc_ins) atomicAdd(&G.status->table_keys, (u64)acc_ins);
}

// ------------------------------------------------------------------ insert
//
// The output records of the listed keys that are frequent enough (Section 5.1's depth filter, the
// side codes of Sections 2 and 4.1), and the marked keys into the table: a few at the end of each
// range, by compare-and-swap behind those that are there. A tile's output places are reserved
// together: the atomics on that one counter take 6 ns each. Writing the records here saves the
// scan of the whole table (64 bytes per slot, half of them empty).

constexpr int kInsertThreads = 256;
constexpr int kInsertKeys = 2;
constexpr unsigned kInsertTile = kInsertThreads * kInsertKeys;

template <int KW>
__global__ void __launch_bounds__(kInsertThreads) part_insert_kernel(const __grid_constant__ PartGeom G,
                                                                     const __grid_constant__ PartSplit S,
                                                                     const __grid_constant__ PartOut O) {
  __shared__ unsigned s_wsum[32];
  __shared__ u64 s_base;
  const u64 listed = __ldcg(S.n_keys), n = listed < S.keys_cap ? listed : S.keys_cap;  // more: the table is full
  const unsigned* keys = S.keys;
  unsigned acc_ins = 0, acc_uu = 0;
  // the keys carried over from the groups before
  u64 carried = __ldcg(S.n_carry_in);
  if (carried > kMaxProbe) carried = kMaxProbe;
  for (u64 i = (u64)blockIdx.x * kInsertThreads + threadIdx.x; i < carried; i += (u64)gridDim.x * kInsertThreads) {
    const unsigned* c = S.carry_in + i * kCarryWords;
    unsigned v[10];
#pragma unroll
    for (int x = 0; x < 10; ++x) v[x] = c[x];
    acc_ins += insert_key(G, S, ((u64)c[11] << 32) | c[10], ((u64)c[13] << 32) | c[12], v);
  }
  // key i into the table if it is marked; its record at `at` if it has the depth
  auto put = [&](u64 i, u64 at) {
    const uint2* c = reinterpret_cast<const uint2*>(keys + i * kKeyWords<KW>);
    uint2 w[kKeyWords<KW> / 2];
#pragma unroll
    for (unsigned x = 0; x < kKeyWords<KW> / 2; ++x) w[x] = __ldg(c + x);
    const u64 h = ((u64)w[3].y << 32) | w[3].x;
    const u64 hi = KW == 2 ? ((u64)w[kKeyWords<KW> / 2 - 1].y << 32) | w[kKeyWords<KW> / 2 - 1].x : 0ull;
    const unsigned v[10] = {w[0].x & 0xFFFFu, w[0].x >> 16, w[0].y & 0xFFFFu, w[0].y >> 16, w[1].x & 0xFFFFu,
                            w[1].y & 0xFFFFu, w[1].y >> 16, w[2].x & 0xFFFFu, w[2].x >> 16, w[2].y & 0xFFFFu};
    if (w[2].y >> 16) acc_ins += insert_key(G, S, h, hi, v);
    const unsigned count = key_count(G, v);
    if (count < O.min_depth) return false;
    acc_uu += write_record(G, O, at, key_lo(h, hi), hi, count, v);
    return true;
  };
  if (O.min_depth <= G.min_count) {
    // every key of the list has the depth: records in list order, nothing to number
    const u64 base = __ldcg(&G.status->n_out), stride = (u64)gridDim.x * kInsertThreads;
    for (u64 i = (u64)blockIdx.x * kInsertThreads + threadIdx.x; i < n; i += stride) put(i, base + i);
    __syncthreads();  // all of the block have read base
    if (threadIdx.x == 0) {
      __threadfence();
      const bool last = atomicAdd(reinterpret_cast<unsigned*>(S.inserted), 1u) == gridDim.x - 1;  // everyone has read it
      if (last && n) atomicAdd(&G.status->n_out, n);
    }
  } else {
    for (u64 t = blockIdx.x; t * kInsertTile < n; t += gridDim.x) {
      // the records this thread's keys make
      unsigned keep = 0;
#pragma unroll
      for (int y = 0; y < kInsertKeys; ++y) {
        const u64 i = t * kInsertTile + y * kInsertThreads + threadIdx.x;
        if (i < n) {
          const uint2* c = reinterpret_cast<const uint2*>(keys + i * kKeyWords<KW>);
          const uint2 a = __ldg(c);
          const unsigned none = __ldg(&c[1].x) & 0xFFFFu;
          keep += (a.x & 0xFFFFu) + (a.x >> 16) + (a.y & 0xFFFFu) + (a.y >> 16) + none >= O.min_depth;
        }
      }
      unsigned total;
      const unsigned before = block_scan<kInsertThreads>(keep, s_wsum, total);
      if (threadIdx.x == 0) s_base = total ? atomicAdd(&G.status->n_out, (u64)total) : 0;
      __syncthreads();
      u64 at = s_base + before;
#pragma unroll 1
      for (int y = 0; y < kInsertKeys; ++y) {
        const u64 i = t * kInsertTile + y * kInsertThreads + threadIdx.x;
        if (i >= n) break;
        at += put(i, at);
      }
      __syncthreads();  // s_wsum and s_base are rewritten
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    acc_ins += __shfl_down_sync(0xffffffffu, acc_ins, o);
    acc_uu += __shfl_down_sync(0xffffffffu, acc_uu, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (acc_ins) atomicAdd(&G.status->table_keys, (u64)acc_ins);
    if (acc_uu) atomicAdd(&G.status->n_uu, (u64)acc_uu);
  }
}

// ------------------------------------------------------------------ launchers

cudaError_t allow_dynamic_smem(const void* fn, size_t need) {
  static std::mutex mu;
  static std::vector<std::pair<std::pair<const void*, int>, int>> done;  // (kernel, device) -> limit
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  int limit = -1;
  for (const auto& d : done)
    if (d.first.first == fn && d.first.second == dev) limit = d.second;
  if (limit < 0) {
    int optin = 0;
    cudaFuncAttributes fa;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess ||
        (e = cudaFuncGetAttributes(&fa, fn)) != cudaSuccess)
      return e;
    limit = optin - (int)fa.sharedSizeBytes;
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, limit)) != cudaSuccess) return e;
    done.push_back({{fn, dev}, limit});
  }
  return need <= (size_t)limit ? cudaSuccess : cudaErrorInvalidValue;
}

static u64 grid_for(const void* fn, int threads, size_t smem, int num_sms, u64 items) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    per_sm = 1;
  }
  const u64 g = (u64)num_sms * (per_sm > 0 ? per_sm : 1);
  return items < g ? items : g;
}

cudaError_t launch_part_scatter(const PartGeom& g, const PartWindows& w, const PartTiles& t, cudaStream_t stream,
                                int num_sms) {
  if (w.q1 <= w.q0) return cudaSuccess;
  const int kw = g.k > 32 ? 2 : 1;
  const size_t smem = scatter_smem(g.log_b, kw);
  const void* fn = kw == 2 ? (const void*)part_scatter_kernel<2> : (const void*)part_scatter_kernel<1>;
  cudaError_t e = allow_dynamic_smem(fn, smem);
  if (e != cudaSuccess) return e;
  const unsigned grid =
      (unsigned)grid_for(fn, kScatterThreads, smem, num_sms, (w.q1 - w.q0 + kScatterTile - 1) / kScatterTile);
  if (kw == 2) part_scatter_kernel<2><<<grid, kScatterThreads, smem, stream>>>(g, w, t);
  else part_scatter_kernel<1><<<grid, kScatterThreads, smem, stream>>>(g, w, t);
  return cudaGetLastError();
}

cudaError_t launch_part_base(const unsigned long long* totals, const PartSplit& s, cudaStream_t stream) {
  part_base_kernel<<<1, kBaseThreads, 0, stream>>>(totals, s.b0, s.b1, s.n_chunks, s.seg_base);
  return cudaGetLastError();
}

cudaError_t launch_part_split(const PartGeom& g, const PartTiles& t, const PartSplit& s, cudaStream_t stream,
                              int num_sms) {
  if (t.n_tiles == 0 || s.b1 <= s.b0) return cudaSuccess;
  if (s.chunk_tiles == 0 || s.chunk_tiles > kMaxChunkTiles || s.b0 % kSplitBuckets || t.stride % 8) return cudaErrorInvalidValue;
  const int kw = g.k > 32 ? 2 : 1;
  const size_t smem = split_smem(s.chunk_tiles, g.sub_max, kw);
  const void* fn = kw == 2 ? (const void*)part_split_kernel<2> : (const void*)part_split_kernel<1>;
  cudaError_t e = allow_dynamic_smem(fn, smem);
  if (e != cudaSuccess) return e;
  const u64 items = (u64)((t.n_tiles + s.chunk_tiles - 1) / s.chunk_tiles) *
                    ((s.b1 - s.b0 + kSplitBuckets - 1) / kSplitBuckets);
  const unsigned grid = (unsigned)grid_for(fn, kSplitThreads, smem, num_sms, items);
  if (kw == 2) part_split_kernel<2><<<grid, kSplitThreads, smem, stream>>>(g, t, s);
  else part_split_kernel<1><<<grid, kSplitThreads, smem, stream>>>(g, t, s);
  return cudaGetLastError();
}

cudaError_t launch_part_count(const PartGeom& g, const PartSplit& s, cudaStream_t stream, int num_sms) {
  if (s.b1 <= s.b0) return cudaSuccess;
  const int kw = g.k > 32 ? 2 : 1;
  const size_t smem = kw == 2 ? CountShape<2>::kSmem : CountShape<1>::kSmem;
  const void* fn = kw == 2 ? (const void*)part_count_kernel<2> : (const void*)part_count_kernel<1>;
  cudaError_t e = allow_dynamic_smem(fn, smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)grid_for(fn, kCountThreads, smem, num_sms, (u64)(s.b1 - s.b0) * g.sub_max);
  if (kw == 2) part_count_kernel<2><<<grid, kCountThreads, smem, stream>>>(g, s);
  else part_count_kernel<1><<<grid, kCountThreads, smem, stream>>>(g, s);
  return cudaGetLastError();
}

cudaError_t launch_part_large(const PartGeom& g, const PartSplit& s, const PartOut& o, cudaStream_t stream, int num_sms) {
  if (s.b1 <= s.b0) return cudaSuccess;
  const int kw = g.k > 32 ? 2 : 1;
  const void* fn = kw == 2 ? (const void*)part_large_kernel<2> : (const void*)part_large_kernel<1>;
  cudaError_t e = allow_dynamic_smem(fn, large_smem(kw));
  if (e != cudaSuccess) return e;
  // their number is known on the device only
  const unsigned grid = (unsigned)grid_for(fn, kLargeThreads, large_smem(kw), num_sms, (u64)(s.b1 - s.b0) * g.sub_max);
  if (kw == 2) part_large_kernel<2><<<grid, kLargeThreads, large_smem(2), stream>>>(g, s, o);
  else part_large_kernel<1><<<grid, kLargeThreads, large_smem(1), stream>>>(g, s, o);
  return cudaGetLastError();
}

cudaError_t launch_part_build(const PartGeom& g, const PartSplit& s, cudaStream_t stream, int num_sms) {
  if (s.b1 <= s.b0) return cudaSuccess;
  const void* fn = g.k > 32 ? (const void*)part_build_kernel<2> : (const void*)part_build_kernel<1>;
  cudaError_t e = allow_dynamic_smem(fn, kBuildSmem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)grid_for(fn, kBuildThreads, kBuildSmem, num_sms, (u64)(s.b1 - s.b0) * g.sub_max);
  if (g.k > 32) part_build_kernel<2><<<grid, kBuildThreads, kBuildSmem, stream>>>(g, s);
  else part_build_kernel<1><<<grid, kBuildThreads, kBuildSmem, stream>>>(g, s);
  return cudaGetLastError();
}

cudaError_t launch_part_insert(const PartGeom& g, const PartSplit& s, const PartOut& o, cudaStream_t stream, int num_sms) {
  // the number of keys is known on the device only: as many CTAs as run at a time
  const void* fn = g.k > 32 ? (const void*)part_insert_kernel<2> : (const void*)part_insert_kernel<1>;
  const unsigned grid = (unsigned)grid_for(fn, kInsertThreads, 0, num_sms, ~0ull);
  if (g.k > 32) part_insert_kernel<2><<<grid, kInsertThreads, 0, stream>>>(g, s, o);
  else part_insert_kernel<1><<<grid, kInsertThreads, 0, stream>>>(g, s, o);
  return cudaGetLastError();
}

}  // namespace kma
