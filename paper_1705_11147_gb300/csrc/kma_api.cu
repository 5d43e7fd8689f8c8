// Host side of the C ABI declared in include/kmer_analysis.h: parameter checks, sizing
// (Bloom filter, table, arena), device memory, staging of host inputs, launch sequencing
// and status reporting. Every computation on reads and k-mers runs in kma_kernels.cu.
#include <cuda_runtime.h>
#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "../../include/kmer_analysis.h"
#include "kma_internal.cuh"

using namespace kma;
typedef unsigned long long u64;

namespace {

thread_local std::string g_last_cuda_error;

int cuda_fail(cudaError_t e, const char* what) {
  g_last_cuda_error = std::string(what) + ": " + cudaGetErrorString(e);
  return KMA_ECUDA;
}

#define KMA_CUDA(call)                                        \
  do {                                                        \
    cudaError_t e_ = (call);                                  \
    if (e_ != cudaSuccess) return cuda_fail(e_, #call);       \
  } while (0)

constexpr u64 kArenaSlack = 64ull * 4096;  // padding positions for per-batch 64-alignment
constexpr u64 kBatchSlack = 256;            // invalid positions kept behind the last batch
constexpr u64 kDefaultStaging = 256ull << 20;
// Host reads are copied and worked on in pieces of an eighth of the call, so that most of the
// work overlaps the copies, but not less than this (below it the launches take longer than the
// copy, 40 us).
constexpr u64 kHostPiece = 8ull << 20;

// ------------------------------------------------------------------ Bloom sizing
//
// Section 5.1 sizes the filter from the number of distinct k-mers m, the filter size n and
// h hash functions with Pr(e) = (1 - e^{-h m / n})^h, optimal h = ln 2 * n / m (the printed
// version swaps m and n in the exponent and in h; this is the standard form). Here all h
// bits of a k-mer lie in one 64-bit word (so one atomicOr is a linearisable test-and-set),
// which raises the rate: a word receives j other k-mers with j ~ Poisson(m / W) for W words,
// and given j the probability that one bit is set is 1 - (63/64)^{h j}. The estimate is the
// Poisson mixture of (1 - (63/64)^{h j})^h.
double blocked_fpr(double m, double words, unsigned h) {
  if (words <= 0) return 1.0;
  const double lam = m / words;
  const double q = std::log(63.0 / 64.0);
  // sum the Poisson(lam) pmf over lam +- 12 sd (+40); the mass outside counts as certain
  // false positives, which only makes the estimate conservative
  const double sd = std::sqrt(lam);
  const long j0 = (long)std::max(0.0, std::floor(lam - 12.0 * sd - 40.0));
  const long j1 = (long)std::ceil(lam + 12.0 * sd + 40.0);
  double fpr = 0.0, mass = 0.0;
  for (long j = j0; j <= j1; ++j) {
    const double pmf = lam > 0 ? std::exp(-lam + (double)j * std::log(lam) - std::lgamma((double)j + 1.0))
                               : (j == 0 ? 1.0 : 0.0);
    mass += pmf;
    fpr += pmf * std::pow(1.0 - std::exp(q * h * (double)j), (double)h);
  }
  return std::min(1.0, fpr + std::max(0.0, 1.0 - mass));
}

void size_bloom(double m, double target, uint64_t& words, uint32_t& hbits, double& est) {
  words = 0;
  hbits = 0;
  est = 1.0;
  if (m < 1) m = 1;
  for (unsigned h = 1; h <= 10; ++h) {
    // smallest W with blocked_fpr <= target (monotone in W)
    double lo = 1, hi = std::max(1.0, m / 64.0);  // start at one bit per key
    while (blocked_fpr(m, hi, h) > target && hi < 1e15) hi *= 2;
    if (blocked_fpr(m, hi, h) > target) continue;
    lo = std::max(1.0, hi / 2);
    while (hi - lo > std::max(1.0, hi * 1e-4)) {
      const double mid = std::floor((lo + hi) / 2);
      if (blocked_fpr(m, mid, h) <= target) hi = mid; else lo = mid;
    }
    const uint64_t w = (uint64_t)std::ceil(hi);
    if (words == 0 || w < words) {
      words = w;
      hbits = h;
      est = blocked_fpr(m, (double)w, h);
    }
  }
}

struct Derived {
  kma_plan plan;
  u64 codes_words, bit_words, mark_words;
  u64 staging;
  unsigned P;      // on-chip partitions (1: one table)
  u64 Sp;          // table slots per partition
  u64 rec_bytes;   // bytes per record in partitioned mode
  unsigned log_b, sub_max, avg;  // partitioned mode: buckets, sub-buckets per bucket, records per sub-bucket
};

// Partitioned mode sorts records into buckets, then sub-buckets of about this part of what the
// count kernel stages, and does both sorts with about as many bins. The rest is for the spread of
// their sizes: at 30x coverage one in a thousand overflows.
constexpr double kSubBucketFill = 0.72;
// The sorted copy of the records made by the split: as large as all of them below this size, one
// launch; above it the buckets are split and counted in groups that share a smaller copy. Smaller
// groups leave the GPU idle at each one's end (2 GiB, 1 GiB, 256 MiB: 250 Mbases, k = 51 5.41,
// 5.47, 5.98 ms; 430 Mbases, 30 % of them a satellite's, 10.9, 11.7, 17.3 ms; 12 and 24 groups of 3
// Gbases 78.0 and 78.9 ms), so they are taken only where there is no memory for more. A handle is
// planned with the second pair.
constexpr u64 kSplitAtOnce = 2ull << 30;
constexpr u64 kSplitGroups = 12;
constexpr u64 kSplitPlanned = 256ull << 20;
constexpr u64 kSplitGroupsPlanned = 48;
constexpr u64 kSplitLeast = 16ull << 20;

// Partitioned above these: filter + table bytes, and bases the kernels have to count; a table so
// large that clearing and scanning it (one table) costs more than the seven kernels of the sorts
// always. One table against partitions, us from reads to answers, 30x of 150 bases:
//   with the singleton filter, 64 MB, k = 25: 0.6 Mbases 144 / 161, 1.2 174 / 172, 2.5 233 / 194, 10 655 / 341
//     (k = 51: 142 / 173, 167 / 180, 218 / 205, 618 / 346)
//   every k-mer: 1.2 Mbases, 64 MB 166 / 187, 2.5 Mbases, 128 MB 209 / 234 (with hot k-mers 206 / 301);
//     10 Mbases, 512 MB 840 / 501 (787 / 550)
//   512 MB: 0.3 Mbases 272 / 294, 0.6 292 / 236; every k-mer 268 / 334, 290 / 289, 1.2 316 / 266
constexpr u64 kAutoPartitionAbove = 32ull << 20;
constexpr u64 kAutoPartitionBases = 1200000;
constexpr u64 kAutoPartitionBasesAll = 4000000;  // every k-mer goes into the table
constexpr u64 kAutoPartitionAlways = 512ull << 20;
constexpr u64 kPartitionTarget = 64ull << 20;      // filter + table bytes per partition

int check_params(const kma_params* p) {
  if (!p) return KMA_EINVAL;
  if (p->k < 1 || p->k > 63) return KMA_EINVAL;
  if (p->canonical && (p->k % 2 == 0)) return KMA_EINVAL;
  if (p->min_depth < 1) return KMA_EINVAL;
  if (p->use_bloom && p->min_depth < 2) return KMA_EINVAL;
  if (p->bloom_fpr < 0 || p->bloom_fpr >= 1) return KMA_EINVAL;
  if (p->load_factor < 0 || p->load_factor > 0.95) return KMA_EINVAL;
  if (p->max_bases == 0) return KMA_EINVAL;
  if (p->block_threads && (p->block_threads < 64 || p->block_threads > 256 || p->block_threads % 32))
    return KMA_EINVAL;
  if (p->windows_per_thread && p->windows_per_thread != 1 && p->windows_per_thread != 2 &&
      p->windows_per_thread != 4 && p->windows_per_thread != 8)
    return KMA_EINVAL;
  if (p->slot_prefetch > 2) return KMA_EINVAL;
  if (p->fault_inject > 1) return KMA_EINVAL;
  if (p->heavy_hitters > 1) return KMA_EINVAL;
  if (p->partitions > (p->k > 32 ? kMaxPartitionsWide : kMaxPartitions)) return KMA_EINVAL;
  if (p->n_parts > 1 && p->part >= p->n_parts) return KMA_EINVAL;
  return KMA_OK;
}

int derive(const kma_params* p, Derived& d) {
  int rc = check_params(p);
  if (rc) return rc;
  std::memset(&d, 0, sizeof(d));
  const u64 windows_bound = p->max_bases;
  const double distinct = p->expected_distinct ? (double)p->expected_distinct : (double)windows_bound;
  if (p->use_bloom) {
    const double target = p->bloom_fpr > 0 ? p->bloom_fpr : 0.01;
    size_bloom(distinct, target, d.plan.bloom_words, d.plan.bloom_hashes, d.plan.bloom_fpr_est);
    if (d.plan.bloom_words == 0) return KMA_EINVAL;
  }
  if (p->table_capacity) {
    d.plan.table_slots = p->table_capacity;
  } else {
    const double keys = p->expected_keys ? (double)p->expected_keys : distinct;
    const double lf = p->load_factor > 0 ? p->load_factor : 0.5;
    d.plan.table_slots = (u64)std::ceil(keys / lf) + 64;
  }
  // on-chip partitions of the table
  {
    const u64 W = d.plan.bloom_words, S = d.plan.table_slots;
    const u64 bytes = W * 8 + S * sizeof(Slot);
    u64 P = p->partitions;
    if (P == 0) {
      const bool large = p->max_bases >= (p->use_bloom ? kAutoPartitionBases : kAutoPartitionBasesAll);
      const bool split = bytes > kAutoPartitionAbove && (large || bytes >= kAutoPartitionAlways);
      P = split ? std::max<u64>(2, (bytes + kPartitionTarget - 1) / kPartitionTarget) : 1;
    }
    const u64 max_parts = p->k > 32 ? kMaxPartitionsWide : kMaxPartitions;
    if (P > max_parts) P = max_parts;
    if (P < 1) P = 1;
    d.P = (unsigned)P;
    d.Sp = (S + P - 1) / P;
    if (P > 1) {
      if (d.Sp < 64) d.Sp = 64;
      d.plan.bloom_words = W ? (W + P - 1) / P * P : 0;
      d.plan.table_slots = d.Sp * P;
    } else {
      d.Sp = S;
    }
    d.plan.partitions = d.P;
    d.rec_bytes = p->k > 32 ? 16 : 8;
    const double parts = p->n_parts > 1 ? p->n_parts : 1;
    d.avg = (unsigned)((p->k > 32 ? kCountCap2 : kCountCap1) * kSubBucketFill);
    const double subs = (double)p->max_bases / parts / d.avg;
    const long lb = std::lround(0.5 * std::log2(std::max(subs, 1.0)));
    d.log_b = (unsigned)std::min<long>(std::max<long>(lb, kMinLogBuckets), kMaxLogBuckets);
    d.sub_max = (unsigned)std::min<double>(std::ceil(subs / (double)(1u << d.log_b)) + 1.0, kMaxSubBuckets);
  }
  // bit slices of the key hash address at most 2^32 Bloom words and 2^32 slots per partition
  if (d.plan.bloom_words >= (1ull << 32) || d.Sp >= (1ull << 32)) return KMA_EINVAL;
  const u64 reads = p->max_reads ? p->max_reads : p->max_bases / 32 + 1;
  // every piece of host reads starts at a multiple of 64 positions; two in a row exceed kHostPiece
  const u64 pieces = 2 * (p->max_bases / kHostPiece + 1);
  const u64 pos = ((p->max_bases + reads + kArenaSlack + 63) / 64 + pieces) * 64;
  d.plan.arena_positions = pos;
  d.codes_words = pos / 32 + 4;
  d.bit_words = pos / 64 + 4;
  d.mark_words = pos / 32 + 4;
  d.staging = p->staging_bytes ? p->staging_bytes : kDefaultStaging;
  d.plan.device_bytes = 2 * d.codes_words * 8 + 2 * d.bit_words * 8 + d.mark_words * 4 +
                        (d.P > 1 ? 0 : d.plan.bloom_words * 8) + d.plan.table_slots * sizeof(Slot) +
                        sizeof(DevStatus) + 2 * (2 * d.staging + (d.staging / 16 + 2) * 8);
  if (d.P > 1) {  // scatter tiles with their offset rows, and count_records' temporaries
    const u64 tiles = pos / kPartTile + 1;
    d.plan.device_bytes += tiles * (kPartTile * d.rec_bytes + (((u64)1 << d.log_b) + 8) * 2);
    const double windows = (double)p->max_bases, all = windows * d.rec_bytes;  // any of them may be counted
    const double group = all <= (double)kSplitPlanned ? 1.0 : std::max((double)kSplitPlanned / all, 1.0 / kSplitGroupsPlanned);
    const double most = group * windows, subs = (most / d.avg + (1 << d.log_b)) * 1.05;
    const double slots = group * (double)d.plan.table_slots + 2 * kMaxProbe;
    d.plan.device_bytes += (u64)(subs * ((double)(p->k > 32 ? kCountCap2 : kCountCap1) * d.rec_bytes + 24) + most * d.rec_bytes +
                                 std::min(most / (p->use_bloom ? 2 : 1), slots) * (d.rec_bytes == 8 ? 32 : 40) +
                                 2 * kMaxProbe * kCarryWords * 4);
  }
  return KMA_OK;
}

// Library-private stream-ordered pool per device: handles of a serving loop come and go,
// and freed blocks are reused instead of going back to the driver.
std::mutex g_pool_mu;
cudaMemPool_t g_pools[64];
bool g_pool_init[64];

int get_pool(int dev, cudaMemPool_t* out) {
  std::lock_guard<std::mutex> lk(g_pool_mu);
  if (dev < 0 || dev >= 64) return KMA_EINVAL;
  if (!g_pool_init[dev]) {
    cudaMemPoolProps props;
    std::memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    KMA_CUDA(cudaMemPoolCreate(&g_pools[dev], &props));
    u64 thr = ~0ull;
    KMA_CUDA(cudaMemPoolSetAttribute(g_pools[dev], cudaMemPoolAttrReleaseThreshold, &thr));
    g_pool_init[dev] = true;
  }
  *out = g_pools[dev];
  return KMA_OK;
}

// Small pinned host blocks (a handle's status word and group counts), kept in a free list
// for the life of the process: cudaFreeHost synchronises the whole device, so a handle
// destroyed in one thread would otherwise stall the GPU work other threads have queued.
constexpr size_t kPinnedBlock = 256;
std::mutex g_pinned_mu;
std::vector<void*> g_pinned_free;

void* pinned_take() {
  std::lock_guard<std::mutex> lk(g_pinned_mu);
  if (g_pinned_free.empty()) {
    char* page = nullptr;
    constexpr size_t kPerPage = 64;
    if (cudaMallocHost((void**)&page, kPinnedBlock * kPerPage) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    for (size_t i = 0; i < kPerPage; ++i) g_pinned_free.push_back(page + i * kPinnedBlock);
  }
  void* b = g_pinned_free.back();
  g_pinned_free.pop_back();
  return b;
}

void pinned_give(void* b) {
  if (!b) return;
  std::lock_guard<std::mutex> lk(g_pinned_mu);
  g_pinned_free.push_back(b);
}

}  // namespace

// finalize_to_host splits the counting and classification into this many groups of
// partitions (of table slots with one table), so that each group's records are copied to the
// host while the next group is still being counted.
constexpr unsigned kFinalizeGroups = 8;

struct kma_handle {
  kma_params p;
  Derived d;
  cudaStream_t stream = nullptr;
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t copied[2] = {nullptr, nullptr};
  cudaEvent_t consumed[2] = {nullptr, nullptr};
  int device = 0;
  int num_sms = 0;
  cudaMemPool_t pool = nullptr;
  LaunchShape shape{256, 4, 0};
  bool agg = false;
  unsigned prefetch = 1;

  u64* codes = nullptr;
  u64* rcodes = nullptr;
  u64* inv = nullptr;
  u64* hq = nullptr;
  unsigned* marks = nullptr;
  u64* bloom = nullptr;      // one-table mode
  Slot* table = nullptr;
  DevStatus* status = nullptr;
  DevStatus* host_status = nullptr;  // pinned
  unsigned char* stage_seq[2] = {nullptr, nullptr};
  unsigned char* stage_qual[2] = {nullptr, nullptr};
  u64* stage_offs[2] = {nullptr, nullptr};
  u64 stage_offs_cap = 0;
  int stage_next = 0;

  u64 q_used = 0, reads_used = 0, bases_used = 0;
  // One table: windows counted since the last reset, an upper bound on the occurrences of any
  // one key. Below 2^32 no counter can wrap and the passes count with plain reductions.
  u64 count_bound = 0;
  bool finalized = false;
  bool failed = false;
  bool pack_only = false;  // estimation handles: count() packs the reads, no counting pass

  // partitioned mode: the scatter tiles of the count() calls, in slabs kept until finalize has
  // counted them, and the records per bucket
  struct Slab { u64* recs; unsigned short* offs; u64 cap, used; double windows, positions, bases; };
  std::vector<Slab> slabs;
  u64* totals = nullptr;

  // contigs of the finalized result (kmer_analysis_contigs), freed by reset / destroy
  char* contig_seq = nullptr;
  u64* contig_offsets = nullptr;
  u64 contig_n = 0, contig_bases = 0, contig_vertices = 0, contig_cycles = 0;
  u64* out_keys = nullptr;
  unsigned* out_counts = nullptr;
  unsigned* out_ext = nullptr;
  unsigned char* out_codes = nullptr;
  u64 out_cap = 0;
  kma_result res;
  // finalize_to_host: per-group record counts (pinned) and the events that publish them
  u64* host_groups = nullptr;
  cudaEvent_t group_ev[kFinalizeGroups] = {};

  // tracing
  bool profiling = false;
  struct ProfRec { int kind; cudaEvent_t a, b; };
  std::vector<ProfRec> prof;
  std::vector<cudaEvent_t> event_pool;
  double ms[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  u64 launches[8] = {0, 0, 0, 0, 0, 0, 0, 0};
};

namespace {

template <typename T>
int dalloc(kma_handle* h, T** ptr, u64 count) {
  *ptr = nullptr;
  if (count == 0) return KMA_OK;
  cudaError_t e = cudaMallocFromPoolAsync((void**)ptr, count * sizeof(T), h->pool, h->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *ptr = nullptr;
    return e == cudaErrorMemoryAllocation ? KMA_ENOMEM : cuda_fail(e, "cudaMallocFromPoolAsync");
  }
  return KMA_OK;
}

template <typename T>
void dfree(kma_handle* h, T*& ptr) {
  if (ptr) cudaFreeAsync(ptr, h->stream);
  ptr = nullptr;
}

cudaEvent_t take_event(kma_handle* h) {
  if (!h->event_pool.empty()) {
    cudaEvent_t e = h->event_pool.back();
    h->event_pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

// Launch one library kernel on `stream`, counting it and (when profiling) bracketing it
// with a pair of CUDA events on that stream.
template <typename F>
int timed_launch(kma_handle* h, int kind, cudaStream_t stream, bool has_work, F&& launch) {
  if (!has_work) return KMA_OK;
  cudaEvent_t a = nullptr, b = nullptr;
  if (h->profiling) {
    a = take_event(h);
    b = take_event(h);
    if (a) cudaEventRecord(a, stream);
  }
  cudaError_t e = launch();
  if (e != cudaSuccess) return cuda_fail(e, "kernel launch");
  h->launches[kind]++;
  if (h->profiling && a && b) {
    cudaEventRecord(b, stream);
    h->prof.push_back({kind, a, b});
  }
  return KMA_OK;
}

void free_records(kma_handle* h) {
  for (auto& b : h->slabs) {
    if (b.recs) cudaFreeAsync(b.recs, h->stream);
    if (b.offs) cudaFreeAsync(b.offs, h->stream);
  }
  h->slabs.clear();
}

void free_contigs(kma_handle* h) {
  if (h->contig_seq) cudaFreeAsync(h->contig_seq, h->stream);
  if (h->contig_offsets) cudaFreeAsync(h->contig_offsets, h->stream);
  h->contig_seq = nullptr;
  h->contig_offsets = nullptr;
  h->contig_n = h->contig_bases = h->contig_vertices = h->contig_cycles = 0;
}

void free_all(kma_handle* h) {
  free_records(h);
  dfree(h, h->codes); dfree(h, h->rcodes); dfree(h, h->inv); dfree(h, h->hq); dfree(h, h->marks);
  dfree(h, h->bloom); dfree(h, h->totals); dfree(h, h->table); dfree(h, h->status);
  for (int i = 0; i < 2; ++i) { dfree(h, h->stage_seq[i]); dfree(h, h->stage_qual[i]); dfree(h, h->stage_offs[i]); }
  dfree(h, h->out_keys); dfree(h, h->out_counts); dfree(h, h->out_ext); dfree(h, h->out_codes);
  free_contigs(h);
  if (h->stream) cudaStreamSynchronize(h->stream);
  pinned_give(h->host_status);
  h->host_status = nullptr;
  pinned_give(h->host_groups);
  h->host_groups = nullptr;
  for (auto& e : h->group_ev) {
    if (e) cudaEventDestroy(e);
    e = nullptr;
  }
  for (int i = 0; i < 2; ++i) {
    if (h->copied[i]) cudaEventDestroy(h->copied[i]);
    if (h->consumed[i]) cudaEventDestroy(h->consumed[i]);
    h->copied[i] = h->consumed[i] = nullptr;
  }
  if (h->copy_stream) cudaStreamDestroy(h->copy_stream);
  h->copy_stream = nullptr;
  for (auto& r : h->prof) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
  h->prof.clear();
  for (auto e : h->event_pool) cudaEventDestroy(e);
  h->event_pool.clear();
}

// Back to the empty state: status, Bloom filter, bucket totals and table cleared on the handle's
// stream. The arena is not cleared: every count() rewrites the words of its batch and sets the
// slack words behind it invalid (reserve_batch).
int clear_state(kma_handle* h) {
  free_records(h);
  free_contigs(h);
  KMA_CUDA(cudaMemsetAsync(h->status, 0, sizeof(DevStatus), h->stream));
  if (h->bloom) KMA_CUDA(cudaMemsetAsync(h->bloom, 0, h->d.plan.bloom_words * 8, h->stream));
  if (h->totals) KMA_CUDA(cudaMemsetAsync(h->totals, 0, sizeof(u64) << h->d.log_b, h->stream));
  // (partitioned mode: the table is written as a whole when its keys are known)
  int rc = timed_launch(h, KMA_KERNEL_INIT, h->stream, h->d.P <= 1 && h->d.plan.table_slots > 0,
                        [&] { return launch_table_init(h->table, h->d.plan.table_slots, h->stream); });
  if (rc) return rc;
  h->q_used = h->reads_used = h->bases_used = 0;
  h->count_bound = 0;
  h->finalized = false;
  h->failed = false;
  std::memset(&h->res, 0, sizeof(h->res));
  return KMA_OK;
}

void choose_shape(kma_handle* h) {
  h->shape.block_threads = h->p.block_threads ? (int)h->p.block_threads : 256;
  h->shape.windows_per_thread = h->p.windows_per_thread ? (int)h->p.windows_per_thread : 2;
  h->agg = h->p.warp_aggregate != 0;
  h->prefetch = h->p.slot_prefetch == 1 ? 1u : 0u;
  int per_sm = h->p.ctas_per_sm ? (int)h->p.ctas_per_sm
                                : pass_max_ctas_per_sm(h->shape.block_threads, h->shape.windows_per_thread, h->agg);
  if (per_sm < 1) per_sm = 1;
  h->shape.grid = h->num_sms * per_sm;
}

int flags_to_code(unsigned flags) {
  if (flags & kFlagTimeout) return KMA_ETIMEOUT;
  if (flags & kFlagBadOffsets) return KMA_EINVAL;
  if (flags & (kFlagFull | kFlagOutput)) return KMA_EFULL;
  if (flags & kFlagOverflow) return KMA_EOVERFLOW;
  return KMA_OK;
}

int read_status(kma_handle* h) {
  KMA_CUDA(cudaMemcpyAsync(h->host_status, h->status, sizeof(DevStatus), cudaMemcpyDeviceToHost, h->stream));
  KMA_CUDA(cudaStreamSynchronize(h->stream));
  return KMA_OK;
}

PassDesc pass_desc(kma_handle* h, unsigned mode, u64 q0, u64 q1) {
  PassDesc d;
  std::memset(&d, 0, sizeof(d));
  d.codes = h->codes; d.rcodes = h->rcodes; d.inv = h->inv; d.hq = h->hq; d.marks = h->marks;
  d.bloom = h->bloom; d.table = h->table; d.status = h->status;
  d.bloom_words = h->d.plan.bloom_words; d.slots = h->d.plan.table_slots;
  d.q0 = q0; d.q1 = q1;
  d.k = h->p.k; d.bloom_h = h->d.plan.bloom_hashes; d.canonical = h->p.canonical;
  d.mode = mode;
  d.n_parts = h->p.n_parts > 1 ? h->p.n_parts : 1;
  d.part = h->p.n_parts > 1 ? h->p.part : 0;
  d.no_overflow = h->count_bound < (1ull << 32) ? 1u : 0u;
  return d;
}

// Staging-copy wait policy of the pack kernel: a generous poll limit, or (fault injection
// for tests) copies that are never issued and a short limit, which must end in KMA_ETIMEOUT.
void set_pack_waits(kma_handle* h, PackBatch& pb) {
  pb.skip_copy = h->p.fault_inject == 1 ? 1u : 0u;
  pb.wait_limit = h->p.fault_inject == 1 ? kWaitPollsInjected : kWaitPolls;
}

// Arena positions of a batch: its bases and a separator behind every read.
u64 batch_positions(u64 n_reads, u64 n_bases) { return std::max<u64>(1, (n_bases + n_reads + 63) / 64) * 64; }

// Reserve arena positions for a batch of n_reads reads (n_bases bases), packed on stream `st`,
// and describe it for the pack kernel. The windows of the batch read up to 192 positions past
// its end; the 256 positions behind it are set invalid here (ordered before the packing on
// `st`), and the next batch's packing overwrites them.
int reserve_batch(kma_handle* h, u64 n_reads, u64 n_bases, PackDesc& pd, u64& q0, u64& n_pos, cudaStream_t st) {
  n_pos = batch_positions(n_reads, n_bases);
  if (h->q_used + n_pos + kBatchSlack > h->d.plan.arena_positions) return KMA_EFULL;
  if (h->bases_used + n_bases > h->p.max_bases) return KMA_EFULL;
  q0 = h->q_used;
  {
    const u64 e = q0 + n_pos;  // a multiple of 64
    KMA_CUDA(cudaMemsetAsync(h->inv + e / 64, 0xFF, kBatchSlack / 64 * 8, st));
    KMA_CUDA(cudaMemsetAsync(h->hq + e / 64, 0, kBatchSlack / 64 * 8, st));
    KMA_CUDA(cudaMemsetAsync(h->codes + e / 32, 0, kBatchSlack / 32 * 8, st));
    KMA_CUDA(cudaMemsetAsync(h->rcodes + e / 32, 0xFF, kBatchSlack / 32 * 8, st));
  }
  std::memset(&pd, 0, sizeof(pd));
  pd.n_reads = n_reads; pd.n_bases = n_bases; pd.q0 = q0; pd.n_pos = n_pos;
  pd.codes = h->codes; pd.rcodes = h->rcodes; pd.inv = h->inv; pd.hq = h->hq; pd.status = h->status;
  pd.qual_min = (unsigned)h->p.qual_offset + (unsigned)h->p.qual_threshold;
  h->q_used += n_pos;
  h->reads_used += n_reads;
  h->bases_used += n_bases;
  return KMA_OK;
}

PartGeom part_geom(kma_handle* h) {
  PartGeom g;
  std::memset(&g, 0, sizeof(g));
  g.table = h->table;
  g.status = h->status;
  g.Sp = h->d.Sp;
  g.P = h->d.P;
  g.k = h->p.k;
  g.canonical = h->p.canonical;
  g.n_parts = h->p.n_parts > 1 ? h->p.n_parts : 1;
  g.part = h->p.n_parts > 1 ? h->p.part : 0;
  g.log_b = h->d.log_b;
  g.sub_max = h->d.sub_max;
  g.avg = h->d.avg;
  g.cap = h->p.k > 32 ? kCountCap2 : kCountCap1;
  g.min_count = h->p.use_bloom ? 2 : 1;
  return g;
}

// Scatter tiles of slab `sl` (tile0: where the next scatter launch writes).
PartTiles tiles_of(kma_handle* h, const kma_handle::Slab& sl, u64 tile0) {
  PartTiles t;
  t.recs = sl.recs;
  t.offs = sl.offs;
  t.totals = h->totals;
  t.tile0 = tile0;
  t.n_tiles = (unsigned)sl.used;
  t.stride = (1u << h->d.log_b) + 8;
  return t;
}

u64 tiles_for(u64 n_pos) { return (n_pos + kPartTile - 1) / kPartTile; }

// Partitioned mode: room for `tiles` more scatter tiles in the handle's last slab, or a new slab
// that also has room for later calls (up to what max_bases allows, 2048 tiles at most), so that
// many small count() calls fill common chunks.
int prepare_tiles(kma_handle* h, u64 tiles, cudaStream_t st) {
  if (!h->slabs.empty() && h->slabs.back().used + tiles <= h->slabs.back().cap) return KMA_OK;
  const u64 left = tiles_for(h->d.plan.arena_positions - std::min<u64>(h->q_used, h->d.plan.arena_positions)) + 1;
  const u64 cap = std::max<u64>(tiles, std::min<u64>(left, 2048));
  if (cap >= (1ull << 31)) return KMA_EINVAL;  // tile numbers are 32-bit
  kma_handle::Slab sl{nullptr, nullptr, cap, 0, 0.0, 0.0, 0.0};
  cudaError_t e = cudaMallocFromPoolAsync((void**)&sl.recs, (size_t)cap * kPartTile * h->d.rec_bytes, h->pool, st);
  if (e == cudaSuccess)
    e = cudaMallocFromPoolAsync((void**)&sl.offs, (size_t)cap * (((u64)1 << h->d.log_b) + 8) * 2, h->pool, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    if (sl.recs) cudaFreeAsync(sl.recs, st);
    return e == cudaErrorMemoryAllocation ? KMA_ENOMEM : cuda_fail(e, "scatter tiles");
  }
  h->slabs.push_back(sl);
  return KMA_OK;
}

// Partitioned mode: the windows [q0, q0 + n_pos) (n_reads reads, n_bases bases) into the last
// slab, which has room for them.
int scatter_windows(kma_handle* h, u64 q0, u64 n_pos, u64 n_reads, u64 n_bases, cudaStream_t st) {
  const PartGeom g = part_geom(h);
  PartWindows w;
  w.codes = h->codes; w.rcodes = h->rcodes; w.inv = h->inv; w.hq = h->hq;
  w.q0 = q0; w.q1 = q0 + n_pos;
  kma_handle::Slab& sl = h->slabs.back();
  const PartTiles t = tiles_of(h, sl, sl.used);
  sl.used += tiles_for(n_pos);
  sl.positions += (double)n_pos;
  sl.bases += (double)n_bases;
  const u64 k1 = h->p.k - 1;
  sl.windows += (n_bases > k1 * n_reads ? (double)(n_bases - k1 * n_reads) : 0.0) / std::max(1u, h->p.n_parts);
  return timed_launch(h, KMA_KERNEL_SCATTER, st, n_pos > 0,
                      [&] { return launch_part_scatter(g, w, t, st, h->num_sms); });
}

void drop_output(kma_handle* h) {
  dfree(h, h->out_keys); dfree(h, h->out_counts); dfree(h, h->out_ext); dfree(h, h->out_codes);
  h->out_cap = 0;
}

// Room for `need` output records; all of it or, on an error, none.
int ensure_output(kma_handle* h, u64 need) {
  if (need <= h->out_cap && h->out_keys) return KMA_OK;
  drop_output(h);
  u64 cap = std::max<u64>(need + need / 8, 1024);
  int rc;
  if ((rc = dalloc(h, &h->out_keys, 2 * cap)) || (rc = dalloc(h, &h->out_counts, cap)) ||
      (rc = dalloc(h, &h->out_ext, 8 * cap)) || (rc = dalloc(h, &h->out_codes, 2 * cap))) {
    drop_output(h);
    return rc;
  }
  h->out_cap = cap;
  return KMA_OK;
}

ClassDesc class_desc(kma_handle* h) {
  ClassDesc c;
  std::memset(&c, 0, sizeof(c));
  c.table = h->table; c.status = h->status; c.slots = h->d.plan.table_slots;
  c.out_keys = h->out_keys; c.out_counts = h->out_counts; c.out_ext = h->out_ext;
  c.out_codes = h->out_codes; c.out_cap = h->out_cap;
  c.min_depth = h->p.min_depth;
  c.min_ext = h->p.min_ext_count ? h->p.min_ext_count : 1;
  return c;
}

PartOut part_out(kma_handle* h) {
  PartOut o;
  std::memset(&o, 0, sizeof(o));
  o.keys = h->out_keys;
  o.counts = h->out_counts;
  o.ext = h->out_ext;
  o.codes = h->out_codes;
  o.cap = h->out_keys ? h->out_cap : 0;
  o.min_depth = h->p.min_depth;
  o.min_ext = h->p.min_ext_count ? h->p.min_ext_count : 1;
  return o;
}

// Partitioned mode: output room before anything is in the table, for as many keys as it was
// sized for, if there is memory for them (more records than fit are classified again afterwards).
int guess_output(kma_handle* h) {
  const double load = h->p.load_factor > 0 ? h->p.load_factor : 0.5;
  const int rc = ensure_output(h, (u64)((double)h->d.plan.table_slots * load));
  return rc == KMA_ENOMEM ? KMA_OK : rc;
}

// Lanes (log2) that copy one run of `len` records on average.
unsigned lanes_for(double len) {
  const double l = std::floor(std::log2(std::max(len, 1.0)) + 0.3);
  return (unsigned)std::min(5.0, l);
}

// Partitioned mode: counts the handle's records into its table and output records on stream `st`,
// the buckets in order, `parts` groups of them or more, and calls after(end) when the buckets
// below `end` have been enqueued. The groups share the sorted copy of the split: all records at once when
// they are few, otherwise from the bucket totals, a twelfth of the records or the largest bucket;
// smaller ones when there is no memory for that. When the call may not wait for the GPU (may_sync
// = false, capture) the groups are of equal numbers of buckets, as many as there are 2 GiB of
// records (twelve at most), and only the room for records without a place in their sub-bucket is
// for all (any bucket may hold them): a graph of 64 samples of up to 1.3 Gbases takes 281 ms (299
// with twelve groups for each sample above 2 GiB, 276 in one with twice the memory).
template <typename F>
int count_records(kma_handle* h, kma_handle* timed, cudaStream_t st, bool may_sync, unsigned parts, F&& after) {
  const unsigned B = 1u << h->d.log_b;
  u64 bound = 0, n_chunks = 0;
  double windows = 0, positions = 0, bases = 0;
  std::vector<unsigned> chunk_tiles;
  for (auto& sl : h->slabs) {
    const double least = 0.5 / std::max(1u, h->p.n_parts);  // against many reads shorter than k
    const double occ = std::min(1.0, std::max(least, sl.positions > 0 ? sl.windows / sl.positions : 1.0));
    // a bucket's records from one chunk fill 85 % of a sub-tile
    const double c = 0.85 * kPartSubTile * B / (kPartTile * occ);
    chunk_tiles.push_back((unsigned)std::min<double>(std::max(1.0, std::floor(c)), kMaxChunkTiles));
    n_chunks += (sl.used + chunk_tiles.back() - 1) / chunk_tiles.back();
    bound += std::min<u64>(sl.used * kPartTile, (u64)sl.bases);
    windows += sl.windows;
    positions += sl.positions;
    bases += sl.bases;
  }
  if (n_chunks == 0) {
    const int rc = timed_launch(timed, KMA_KERNEL_INIT, st, true,
                                [&] { return launch_table_init(h->table, h->d.plan.table_slots, st); });
    return rc ? rc : after(B);
  }
  constexpr unsigned kStep = kSplitBuckets;  // groups are whole work items of the split
  if (!may_sync) parts = std::max(parts, (unsigned)std::min<u64>(kSplitGroups, bound * h->d.rec_bytes / kSplitAtOnce + 1));
  parts = std::min(parts, B / kStep);
  double counted = bases / std::max(1u, h->p.n_parts);  // windows there may be
  PartSplit s;
  std::memset(&s, 0, sizeof(s));
  PartGeom g = part_geom(h);
  PartOut o = part_out(h);
  // first slot of the hashes of bucket b (part_of, table_index)
  auto first_slot = [&](unsigned b) -> u64 {
    const u64 top = (u64)b << (32 - h->d.log_b);
    return b < B ? (top * g.P >> 32) * g.Sp + ((top * g.P & 0xFFFFFFFFull) * g.Sp >> 32) : (u64)g.P * g.Sp;
  };
  // Temporaries, in one allocation. While the stream is busy an allocation from the pool takes the
  // host 1 us, and 3.5 us more for every other stream that the pool's free memory was used on
  // (ten of them, after eight batch graphs on streams of their own: 0.72 -> 0.90 ms for 12 Mbases).
  std::vector<u64> totals;     // records per bucket
  std::vector<unsigned> ends;  // of the groups
  unsigned most_buckets = 0;   // of a group
  u64 n_subs = 0, n_zero = 0, n_keys = 0, block_bytes = 0;
  u64 at_recs, at_over, at_keys, at_zero, at_large, at_base, at_n_carry, at_carry, at_segs, at_seg_base;
  unsigned char* block = nullptr;
  for (u64 at_once = kSplitAtOnce, at_most = kSplitGroups;; at_once /= 2, at_most *= 2) {
    u64 most = bound, most_slots = 0;  // records and table slots of a group
    ends.clear();
    if (!may_sync || bound * h->d.rec_bytes <= at_once) {
      for (unsigned i = 0; i < parts; ++i) ends.push_back((unsigned)((u64)(B / kStep) * (i + 1) / parts) * kStep);
    } else {
      if (totals.empty()) {
        totals.resize(B);
        KMA_CUDA(cudaMemcpyAsync(totals.data(), h->totals, B * sizeof(u64), cudaMemcpyDeviceToHost, st));
        KMA_CUDA(cudaStreamSynchronize(st));
      }
      u64 all = 0;
      for (u64 t : totals) all += t;
      counted = (double)all;
      const u64 aim = std::max(at_once / h->d.rec_bytes, all / at_most);
      std::vector<u64> step(B / kStep, 0);  // records per step of buckets
      for (unsigned b = 0; b < B; ++b) step[b / kStep] += totals[b];
      const unsigned widest = (B / kStep + parts - 1) / parts;
      most = 0;
      for (unsigned b = 0; b < B / kStep;) {
        unsigned e = b;
        u64 sum = 0;
        do sum += step[e++];
        while (e < B / kStep && e - b < widest && sum + step[e] <= aim);
        ends.push_back(e * kStep);
        most = std::max(most, sum);
        b = e;
      }
    }
    most_buckets = 0;
    for (size_t i = 0; i < ends.size(); ++i) {
      const unsigned b0 = i ? ends[i - 1] : 0;
      most_buckets = std::max(most_buckets, ends[i] - b0);
      most_slots = std::max(most_slots, first_slot(ends[i]) - first_slot(b0));
    }
    // Room for the sub-buckets of the windows there may be (sub_buckets makes as many as there are
    // windows for). Not of n_bases - (k - 1) * n_reads windows: reads shorter than k take from the
    // others' there, and with too few sub-buckets all of them overflow (1 Mbp, 30x of 35 to 75 bases,
    // k = 63: 3.80 ms instead of 0.48, 3.43 of them in part_large_kernel).
    g.sub_max = (unsigned)std::min<double>(h->d.sub_max, std::ceil(1.05 * counted / ((double)g.avg * B)) + 1.0);
    n_subs = (u64)most_buckets * g.sub_max;
    const u64 n_segs = most / kPartSubTile + (u64)most_buckets * n_chunks + 1;
    if (n_chunks >= (1ull << 31) || n_segs >= (1ull << 32)) return KMA_EINVAL;
    // [sub-buckets], overflow records, list entries, large sub-buckets, those taken, CTAs done,
    // then segments per bucket and keys per sub-bucket (32 bits)
    n_zero = n_subs + 5 + (most_buckets + n_subs + 1) / 2;
    const unsigned key_words = kMaxKeyWords - (h->d.rec_bytes == 8 ? 2 : 0);
    // The keys of a group go to its slots, or kMaxProbe further on, or (round the end of a partition
    // that began before it) to the first kMaxProbe of that: with more of them the table is full.
    n_keys = std::min<u64>(most / (h->p.use_bloom ? 2 : 1), most_slots + 2 * kMaxProbe) + 1;
    block_bytes = 0;
    auto room = [&](u64 bytes) -> u64 {
      const u64 at = block_bytes;
      block_bytes += (bytes + 255) & ~255ull;
      return at;
    };
    at_recs = room(n_subs * g.cap * h->d.rec_bytes), at_over = room(most * h->d.rec_bytes);
    at_keys = room(n_keys * key_words * 4), at_zero = room(n_zero * 8), at_large = room(n_subs * sizeof(unsigned));
    at_base = room(n_subs * 8), at_n_carry = room(2 * 8);
    at_carry = room(2 * (u64)kMaxProbe * kCarryWords * 4);  // two lists, taken in turn
    at_segs = room(n_segs * sizeof(PartSegment)), at_seg_base = room(most_buckets * sizeof(unsigned));
    const cudaError_t e = cudaMallocFromPoolAsync((void**)&block, block_bytes, h->pool, st);
    if (e == cudaSuccess) break;
    cudaGetLastError();
    if (e != cudaErrorMemoryAllocation) return cuda_fail(e, "split output");
    if (!may_sync) return KMA_ENOMEM;
    if (at_once <= kSplitLeast) {  // then without output room: the records are classified when their number is known
      if (!h->out_keys) return KMA_ENOMEM;
      const cudaStream_t own = h->stream;
      h->stream = st;
      drop_output(h);
      h->stream = own;
      o = part_out(h);
      at_once = 2 * kSplitAtOnce, at_most = kSplitGroups / 2;
    }
    KMA_CUDA(cudaStreamSynchronize(st));  // what has been freed on it is there for the next attempt
  }
  auto run = [&]() -> int {
    int rc;
    u64* zero = (u64*)(block + at_zero);
    u64* n_carry = (u64*)(block + at_n_carry);
    unsigned* carry = (unsigned*)(block + at_carry);
    s.recs = (u64*)(block + at_recs);
    s.over = (u64*)(block + at_over);
    s.keys = (unsigned*)(block + at_keys);
    s.large = (unsigned*)(block + at_large);
    s.key_base = (u64*)(block + at_base);
    s.segs = (PartSegment*)(block + at_segs);
    s.seg_base = (unsigned*)(block + at_seg_base);
    s.fill = zero;
    s.over_n = zero + n_subs;
    s.n_keys = zero + n_subs + 1;
    s.n_large = zero + n_subs + 2;
    s.next_large = zero + n_subs + 3;
    s.inserted = zero + n_subs + 4;
    s.n_segs = reinterpret_cast<unsigned*>(zero + n_subs + 5);
    s.key_n = s.n_segs + most_buckets;
    s.keys_cap = n_keys;
    s.n_chunks = (unsigned)n_chunks;
    KMA_CUDA(cudaMemsetAsync(n_carry, 0, 2 * 8, st));
    const double occ = std::min(1.0, std::max(0.3, positions > 0 ? windows / positions : 1.0));
    s.log_lanes = lanes_for(kPartTile * occ / B);
    for (size_t i = 0; i < ends.size(); ++i) {
      s.b0 = i ? ends[i - 1] : 0;
      s.b1 = ends[i];
      KMA_CUDA(cudaMemsetAsync(zero, 0, n_zero * 8, st));
      s.end = first_slot(s.b1);  // the group's slots end there
      s.carry_in = carry + (i & 1) * (u64)kMaxProbe * kCarryWords;
      s.carry_out = carry + ((i + 1) & 1) * (u64)kMaxProbe * kCarryWords;
      s.n_carry_in = n_carry + (i & 1);
      s.n_carry_out = n_carry + ((i + 1) & 1);
      KMA_CUDA(cudaMemsetAsync(s.n_carry_out, 0, 8, st));
      if ((rc = timed_launch(timed, KMA_KERNEL_SCATTER, st, true,
                             [&] { return launch_part_base(h->totals, s, st); })))
        return rc;
      for (size_t j = 0; j < h->slabs.size(); ++j) {
        const PartTiles t = tiles_of(h, h->slabs[j], 0);
        s.chunk_tiles = chunk_tiles[j];
        if ((rc = timed_launch(timed, KMA_KERNEL_SCATTER, st, t.n_tiles > 0,
                               [&] { return launch_part_split(g, t, s, st, h->num_sms); })))
          return rc;
      }
      if ((rc = timed_launch(timed, KMA_KERNEL_PASS, st, true,
                             [&] { return launch_part_count(g, s, st, h->num_sms); })) ||
          (rc = timed_launch(timed, KMA_KERNEL_RECOUNT, st, true,
                             [&] { return launch_part_build(g, s, st, h->num_sms); })) ||
          (rc = timed_launch(timed, KMA_KERNEL_PASS, st, true,
                             [&] { return launch_part_large(g, s, o, st, h->num_sms); })) ||
          (rc = timed_launch(timed, KMA_KERNEL_RECOUNT, st, true,
                             [&] { return launch_part_insert(g, s, o, st, h->num_sms); })))
        return rc;
      if ((rc = after(s.b1))) return rc;
    }
    return KMA_OK;
  };
  const int rc = run();
  cudaFreeAsync(block, st);
  return rc;
}

// Partitioned mode: the figures that count_records adds to start at zero (again, if an earlier
// finalize ran out of memory for another handle of its batch).
int reset_counted(kma_handle* h, cudaStream_t st) {
  static_assert(offsetof(DevStatus, first_sightings) - offsetof(DevStatus, table_keys) == 3 * sizeof(u64), "they are in a row");
  KMA_CUDA(cudaMemsetAsync(&h->status->table_keys, 0, 4 * sizeof(u64), st));
  return KMA_OK;
}

// First pass over the windows [q0, q0 + n_pos) of one packed batch (n_reads reads, n_bases
// bases) on stream `st`. One table: Bloom test-and-set (or counting) in place. Partitions:
// scatter into tiles, which finalize counts. Nothing here waits for the GPU.
int first_pass(kma_handle* h, u64 q0, u64 n_pos, u64 n_reads, u64 n_bases, cudaStream_t st) {
  const unsigned mode = h->p.use_bloom ? kModeBloom : kModeCount;
  if (h->d.P <= 1) {
    h->count_bound += n_pos;
    PassBatch b;
    std::memset(&b, 0, offsetof(PassBatch, d) + sizeof(PassDesc));
    b.n = 1;
    b.prefetch = h->prefetch;
    b.d[0] = pass_desc(h, mode, q0, q0 + n_pos);
    const u64 tile = (u64)h->shape.block_threads * h->shape.windows_per_thread;
    b.d[0].tile_begin = 0;
    b.total_tiles = (n_pos + tile - 1) / tile;
    return timed_launch(h, KMA_KERNEL_PASS, st, b.total_tiles > 0,
                        [&] { return launch_pass(b, h->shape, h->agg, st); });
  }
  int rc = prepare_tiles(h, tiles_for(n_pos), st);
  return rc ? rc : scatter_windows(h, q0, n_pos, n_reads, n_bases, st);
}

int run_pack_and_pass(kma_handle* h, const PackDesc& pd) {
  PackBatch pb;
  std::memset(&pb, 0, offsetof(PackBatch, d) + sizeof(PackDesc));
  pb.n = 1;
  set_pack_waits(h, pb);
  pb.d[0] = pd;
  pb.d[0].chunk_begin = 0;
  pb.total_chunks = (pd.n_pos / 64 + kPackChunkWords - 1) / kPackChunkWords;
  int rc = timed_launch(h, KMA_KERNEL_PACK, h->stream, pb.total_chunks > 0,
                        [&] { return launch_pack(pb, h->stream, h->num_sms); });
  if (rc) return rc;
  if (h->pack_only) return KMA_OK;
  return first_pass(h, pd.q0, pd.n_pos, pd.n_reads, pd.n_bases, h->stream);
}

constexpr u64 kClassTile = 256 * 4;  // slots per classify block tile (kernel constants)

void fill_result(kma_handle* h) {
  kma_result& r = h->res;
  r.n = h->host_status->n_out;
  r.n_uu = h->host_status->n_uu;
  r.valid_windows = h->host_status->valid_windows;
  r.table_keys = h->host_status->table_keys;
  r.keys = (const uint64_t*)h->out_keys;
  r.counts = h->out_counts;
  r.ext = h->out_ext;
  r.codes = h->out_codes;
}

// HyperLogLog estimate of 2^p registers (Flajolet, Fusy, Gandouet, Meunier 2007): the raw
// estimate alpha_m m^2 / sum 2^-M[j], replaced by linear counting m ln(m / V) in the small
// range (raw <= 5m/2 with V > 0 empty registers). 64-bit hashes need no large-range
// correction.
double hll_estimate(const uint8_t* regs, unsigned p) {
  const double m = (double)(1u << p);
  double sum = 0.0;
  u64 zeros = 0;
  for (u64 j = 0; j < (1ull << p); ++j) {
    sum += std::ldexp(1.0, -(int)regs[j]);
    zeros += regs[j] == 0;
  }
  const double alpha = p == 4 ? 0.673 : p == 5 ? 0.697 : p == 6 ? 0.709 : 0.7213 / (1.0 + 1.079 / m);
  const double raw = alpha * m * m / sum;
  if (raw <= 2.5 * m && zeros > 0) return m * std::log(m / (double)zeros);
  return raw;
}

// Answers into pageable host arrays. A copy to pages that are not there yet waits for their faults:
// 152 MB take 6.4 ms, 8 MB 0.48 ms, to pages in place 0.83 and 0.05 ms. So a few threads bring such
// pages in while the lookups run (with the copy 2.2 and 0.31 ms); they call nothing of CUDA's, and
// the copies stay the caller's, on its stream. A page is brought in by a store of 0, which is what
// a page never written holds, and only where the kernel says that it is missing. (Reading the byte
// first maps the page twice, 20 us more; an atomic does too; MADV_POPULATE_WRITE is slower in
// eight threads than in one.)
// Arrays whose pages are there (malloc hands blocks below 32 MB out again as they are) and pinned
// ones are copied at once: looking through them takes 10 us for 152 MB. A thread takes 50 us to
// start: one for every 4 MB (16 MB: 0.40 ms with four, 0.73 with one, 0.85 without). Up to
// 1 MB the faults take less than the look.
constexpr u64 kTouchFrom = 1ull << 20;
constexpr u64 kTouchPerThread = 4ull << 20;
constexpr unsigned kTouchThreads = 8;

struct HostArray {
  char* at;
  u64 bytes;
};

// Calls missing(first byte of [at, end) on it) for every page that is not there, looking at kLook
// pages at a time. Stops where it cannot be told.
template <typename F>
void missing_pages(char* at, char* end, u64 page, F&& missing) {
  constexpr u64 kLook = 256;
  unsigned char there[kLook];
  for (u64 p = (u64)at / page * page; p < (u64)end; p += kLook * page) {
    const u64 n = std::min(kLook, ((u64)end - p + page - 1) / page);
    if (mincore((void*)p, n * page, there) != 0) return;
    for (u64 i = 0; i < n; ++i)
      if (!(there[i] & 1)) missing(std::max(at, (char*)(p + i * page)));
  }
}

void bring_pages_in(std::initializer_list<HostArray> arrays) {
  const long ps = sysconf(_SC_PAGESIZE);
  if (ps <= 0) return;
  const u64 page = (u64)ps, piece = std::max<u64>(1ull << 20, page);
  HostArray todo[4];
  unsigned n = 0;
  u64 total = 0, missing = 0;
  for (const HostArray& a : arrays) total += a.bytes;
  if (total < kTouchFrom) return;
  for (const HostArray& a : arrays) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, a.at) != cudaSuccess) cudaGetLastError(), at.type = cudaMemoryTypeUnregistered;
    if (n == 4 || at.type != cudaMemoryTypeUnregistered) continue;
    const u64 before = missing;
    missing_pages(a.at, a.at + a.bytes, page, [&](char*) { missing += page; });
    if (missing != before) todo[n++] = a;
  }
  if (!missing) return;
  std::atomic<u64> next{0};
  auto work = [&] {
    for (;;) {
      u64 i = next.fetch_add(1);  // piece i of the arrays together
      unsigned j = 0;
      for (; j < n && i >= (todo[j].bytes + piece - 1) / piece; ++j) i -= (todo[j].bytes + piece - 1) / piece;
      if (j == n) return;
      missing_pages(todo[j].at + i * piece, todo[j].at + std::min(todo[j].bytes, (i + 1) * piece), page,
                    [](char* p) { *(volatile char*)p = 0; });
    }
  };
  std::thread th[kTouchThreads - 1];
  const u64 T = std::min<u64>({missing / kTouchPerThread, kTouchThreads, std::max(1u, std::thread::hardware_concurrency())});
  try {
    for (u64 t = 1; t < T; ++t) th[t - 1] = std::thread(work);
  } catch (...) {  // no more threads: those there are do it all
  }
  work();
  for (auto& x : th)
    if (x.joinable()) x.join();
}

}  // namespace

extern "C" {

int kmer_analysis_plan(const kma_params* params, kma_plan* out) {
  if (!out) return KMA_EINVAL;
  Derived d;
  int rc = derive(params, d);
  if (rc) return rc;
  *out = d.plan;
  return KMA_OK;
}

int kmer_analysis_create(const kma_params* params, void* cuda_stream, kma_handle** out) {
  if (!out) return KMA_EINVAL;
  *out = nullptr;
  Derived d;
  int rc = derive(params, d);
  if (rc) return rc;
  kma_handle* h = new kma_handle();
  h->p = *params;
  h->d = d;
  h->stream = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaGetDevice(&h->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
  if (e != cudaSuccess) { delete h; return cuda_fail(e, "cudaGetDevice"); }
  if ((rc = get_pool(h->device, &h->pool))) { delete h; return rc; }
  choose_shape(h);
  h->stage_offs_cap = d.staging / 16 + 2;
  if ((rc = dalloc(h, &h->codes, d.codes_words)) || (rc = dalloc(h, &h->rcodes, d.codes_words)) ||
      (rc = dalloc(h, &h->inv, d.bit_words)) ||
      (rc = dalloc(h, &h->hq, d.bit_words)) || (rc = dalloc(h, &h->marks, d.mark_words)) ||
      (rc = dalloc(h, &h->bloom, d.P > 1 ? 0 : d.plan.bloom_words)) ||
      (rc = dalloc(h, &h->totals, d.P > 1 ? 1ull << d.log_b : 0)) ||
      (rc = dalloc(h, &h->table, d.plan.table_slots)) || (rc = dalloc(h, &h->status, 1))) {
    free_all(h);
    delete h;
    return rc;
  }
  static_assert(sizeof(DevStatus) <= kPinnedBlock && kFinalizeGroups * sizeof(u64) <= kPinnedBlock,
                "pinned blocks hold a status word and the group counts");
  h->host_status = static_cast<DevStatus*>(pinned_take());
  if (!h->host_status) { free_all(h); delete h; return KMA_ENOMEM; }

  std::memset(h->host_status, 0, sizeof(DevStatus));
  if ((rc = clear_state(h))) { free_all(h); delete h; return rc; }
  *out = h;
  return KMA_OK;
}

// offsets[0..n] non-decreasing? Large read sets are checked by several host threads (the
// check is a stream over 8 bytes per read, done before any input is copied).
static bool offsets_nondecreasing(const uint64_t* offsets, u64 n) {
  auto check = [offsets](u64 a, u64 b) {
    unsigned bad = 0;
    for (u64 r = a; r < b; ++r) bad |= offsets[r + 1] < offsets[r];
    return bad == 0;
  };
  const unsigned hw = std::thread::hardware_concurrency();
  const unsigned T = n < (1u << 20) ? 1u : std::max(1u, std::min(8u, hw));
  if (T == 1) return check(0, n);
  std::vector<char> ok(T, 0);
  std::vector<std::thread> th;
  for (unsigned t = 0; t < T; ++t)
    th.emplace_back([&, t] { ok[t] = check(n * t / T, n * (t + 1) / T); });
  for (auto& x : th) x.join();
  return std::all_of(ok.begin(), ok.end(), [](char v) { return v != 0; });
}

static int setup_staging(kma_handle* h) {
  if (h->stage_seq[0]) return KMA_OK;
  int rc;
  for (int i = 0; i < 2; ++i) {
    if ((rc = dalloc(h, &h->stage_seq[i], h->d.staging)) || (rc = dalloc(h, &h->stage_qual[i], h->d.staging)) ||
        (rc = dalloc(h, &h->stage_offs[i], h->stage_offs_cap)))
      return rc;
    KMA_CUDA(cudaEventCreateWithFlags(&h->copied[i], cudaEventDisableTiming));
    KMA_CUDA(cudaEventCreateWithFlags(&h->consumed[i], cudaEventDisableTiming));
  }
  KMA_CUDA(cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking));
  // the staging buffers were allocated on h->stream: make the copy stream wait for that
  KMA_CUDA(cudaEventRecord(h->consumed[0], h->stream));
  KMA_CUDA(cudaEventRecord(h->consumed[1], h->stream));
  return KMA_OK;
}

int kmer_analysis_count(kma_handle* h, const char* seq, const char* qual, const uint64_t* offsets,
                        uint64_t n_reads, int on_device) {
  if (!h) return KMA_EINVAL;
  if (h->finalized || h->failed) return KMA_ESTATE;
  if (!offsets) return KMA_EINVAL;
  if (n_reads == 0) return KMA_OK;
  if (!seq || !qual) return KMA_EINVAL;
  int rc;
  if (on_device) {
    u64 ends[2];
    KMA_CUDA(cudaMemcpyAsync(&ends[0], offsets, 8, cudaMemcpyDeviceToHost, h->stream));
    KMA_CUDA(cudaMemcpyAsync(&ends[1], offsets + n_reads, 8, cudaMemcpyDeviceToHost, h->stream));
    KMA_CUDA(cudaStreamSynchronize(h->stream));
    if (ends[1] < ends[0]) return KMA_EINVAL;
    PackDesc pd;
    u64 q0, n_pos;
    if ((rc = reserve_batch(h, n_reads, ends[1] - ends[0], pd, q0, n_pos, h->stream))) return rc;
    pd.seq = (const unsigned char*)seq;
    pd.qual = (const unsigned char*)qual;
    pd.offsets = (const unsigned long long*)offsets;
    pd.delta = 0;
    return run_pack_and_pass(h, pd);
  }
  // Host input: validate offsets, then stream chunks through two staging buffers; the copy
  // of chunk i+1 overlaps the packing and first pass of chunk i.
  if (!offsets_nondecreasing(offsets, n_reads)) return KMA_EINVAL;
  const u64 nb_all = offsets[n_reads] - offsets[0];
  if (nb_all + h->bases_used > h->p.max_bases) return KMA_EFULL;
  const u64 piece = std::min(h->d.staging, std::max(kHostPiece, nb_all / 8));
  // one past the last read of the piece that starts at read r0: the reads that end inside it
  // (offsets do not decrease), at least one
  auto piece_end = [&](u64 r0) -> u64 {
    const u64 r_max = std::min<u64>(n_reads, r0 + h->stage_offs_cap - 1);
    const u64 r1 = (u64)(std::upper_bound(offsets + r0 + 1, offsets + r_max + 1, offsets[r0] + piece) - offsets) - 1;
    return std::max(r1, r0 + 1);
  };
  // all of the call or, on an error, none of it
  u64 q = h->q_used;
  for (u64 r0 = 0, r1; r0 < n_reads; r0 = r1) {
    r1 = piece_end(r0);
    if (offsets[r1] - offsets[r0] > h->d.staging) return KMA_EINVAL;  // a single read longer than the staging buffer
    q += batch_positions(r1 - r0, offsets[r1] - offsets[r0]);
    if (q + kBatchSlack > h->d.plan.arena_positions) return KMA_EFULL;
  }
  if ((rc = setup_staging(h))) return rc;
  // With partitions, every staged chunk is packed and scattered, so the copy of the next chunk
  // overlaps both.
  const bool parts = h->d.P > 1 && !h->pack_only;
  if (parts) {
    // tiles of the whole call: every chunk starts a tile, and a chunk ends only when the next
    // read would overflow the piece or the staged read offsets
    const u64 chunks = 2 * (nb_all / piece + n_reads / (h->stage_offs_cap - 1) + 1);
    if ((rc = prepare_tiles(h, tiles_for(nb_all + n_reads + 64 * chunks) + chunks, h->stream))) return rc;
  }
  u64 r0 = 0;
  while (r0 < n_reads) {
    const u64 r1 = piece_end(r0);
    const u64 nb = offsets[r1] - offsets[r0];
    PackDesc pd;
    u64 q0, n_pos;
    if ((rc = reserve_batch(h, r1 - r0, nb, pd, q0, n_pos, h->stream))) return rc;
    const int b = h->stage_next;
    h->stage_next ^= 1;
    KMA_CUDA(cudaStreamWaitEvent(h->copy_stream, h->consumed[b], 0));
    KMA_CUDA(cudaMemcpyAsync(h->stage_seq[b], seq + offsets[r0], nb, cudaMemcpyHostToDevice, h->copy_stream));
    KMA_CUDA(cudaMemcpyAsync(h->stage_qual[b], qual + offsets[r0], nb, cudaMemcpyHostToDevice, h->copy_stream));
    KMA_CUDA(cudaMemcpyAsync(h->stage_offs[b], offsets + r0, (r1 - r0 + 1) * 8, cudaMemcpyHostToDevice, h->copy_stream));
    KMA_CUDA(cudaEventRecord(h->copied[b], h->copy_stream));
    KMA_CUDA(cudaStreamWaitEvent(h->stream, h->copied[b], 0));
    pd.seq = h->stage_seq[b];
    pd.qual = h->stage_qual[b];
    pd.offsets = h->stage_offs[b];
    pd.delta = (long long)offsets[r0];
    PackBatch pb;
    std::memset(&pb, 0, offsetof(PackBatch, d) + sizeof(PackDesc));
    pb.n = 1;
    set_pack_waits(h, pb);
    pb.d[0] = pd;
    pb.total_chunks = (n_pos / 64 + kPackChunkWords - 1) / kPackChunkWords;
    if ((rc = timed_launch(h, KMA_KERNEL_PACK, h->stream, true,
                           [&] { return launch_pack(pb, h->stream, h->num_sms); })))
      return rc;
    KMA_CUDA(cudaEventRecord(h->consumed[b], h->stream));
    if (parts) {
      if ((rc = scatter_windows(h, q0, n_pos, r1 - r0, nb, h->stream))) return rc;
    } else if (!h->pack_only && (rc = first_pass(h, q0, n_pos, r1 - r0, nb, h->stream))) {
      return rc;
    }
    r0 = r1;
  }
  // Host buffers may be reused once the call returns: wait for the copies.
  KMA_CUDA(cudaStreamSynchronize(h->copy_stream));
  return KMA_OK;
}

// What is left of the counting: one launch of the recount (first sightings) for all one-table
// Bloom handles, and the records of the partitioned ones. Enqueued on h0's stream; may_sync:
// see count_records.
static int enqueue_recount(kma_handle* const* hs, uint32_t n, bool may_sync) {
  kma_handle* h0 = hs[0];
  PassBatch pb;
  std::memset(&pb, 0, sizeof(pb));
  pb.prefetch = h0->prefetch;
  const u64 tile = (u64)h0->shape.block_threads * h0->shape.windows_per_thread;
  u64 tiles = 0;
  for (uint32_t i = 0; i < n; ++i) {
    kma_handle* h = hs[i];
    if (!h->p.use_bloom || h->q_used == 0 || h->d.P > 1) continue;
    PassDesc d = pass_desc(h, kModeRecount, 0, h->q_used);
    d.tile_begin = tiles;
    tiles += (h->q_used + tile - 1) / tile;
    pb.d[pb.n++] = d;
  }
  pb.total_tiles = tiles;
  int rc = timed_launch(h0, KMA_KERNEL_RECOUNT, h0->stream, pb.n > 0 && tiles > 0,
                        [&] { return launch_pass(pb, h0->shape, h0->agg, h0->stream); });
  if (rc) return rc;
  for (uint32_t i = 0; i < n; ++i) {
    kma_handle* h = hs[i];
    if (h->d.P <= 1) continue;
    auto nothing = [](unsigned) { return (int)KMA_OK; };
    if ((rc = reset_counted(h, h0->stream)) || (rc = count_records(h, h0, h0->stream, may_sync, 1, nothing))) return rc;
  }
  return KMA_OK;
}

// Classification + compaction of the handles with ok[i] into their current output buffers,
// one launch; then their records are released. Enqueued on h0's stream.
static int enqueue_classify(kma_handle* const* hs, uint32_t n, const std::vector<int>& ok) {
  kma_handle* h0 = hs[0];
  for (uint32_t i = 0; i < n; ++i)
    if (ok[i]) KMA_CUDA(cudaMemsetAsync(&hs[i]->status->n_out, 0, 2 * sizeof(u64), h0->stream));
  ClassBatch cb;
  std::memset(&cb, 0, sizeof(cb));
  cb.write = 1;
  u64 blocks = 0;
  for (uint32_t i = 0; i < n; ++i) {
    if (!ok[i]) continue;
    ClassDesc c = class_desc(hs[i]);
    c.block_begin = blocks;
    blocks += (c.slots + kClassTile - 1) / kClassTile;
    cb.d[cb.n++] = c;
  }
  cb.total_blocks = blocks;
  int rc = timed_launch(h0, KMA_KERNEL_CLASSIFY, h0->stream, cb.n > 0 && blocks > 0,
                        [&] { return launch_classify(cb, h0->stream, h0->num_sms); });
  if (rc) return rc;
  for (uint32_t i = 0; i < n; ++i) {  // the records are not needed any more
    cudaStream_t saved = hs[i]->stream;
    hs[i]->stream = h0->stream;
    free_records(hs[i]);
    hs[i]->stream = saved;
  }
  return KMA_OK;
}

static int check_batch(kma_handle* const* hs, uint32_t n) {
  if (!hs || n == 0 || n > KMA_MAX_BATCH) return KMA_EINVAL;
  for (uint32_t i = 0; i < n; ++i) {
    if (!hs[i]) return KMA_EINVAL;
    if (hs[i]->finalized || hs[i]->failed) return KMA_ESTATE;
    for (uint32_t j = 0; j < i; ++j)
      if (hs[j] == hs[i]) return KMA_EINVAL;
  }
  return KMA_OK;
}

static int finalize_many(kma_handle* const* hs, uint32_t n, kma_result* out) {
  int rc = check_batch(hs, n);
  if (rc) return rc;
  kma_handle* h0 = hs[0];
  // make every handle's stream work visible to h0's stream
  for (uint32_t i = 1; i < n; ++i) {
    if (hs[i]->stream != h0->stream) {
      cudaEvent_t ev;
      KMA_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
      cudaError_t e = cudaEventRecord(ev, hs[i]->stream);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(h0->stream, ev, 0);
      cudaEventDestroy(ev);
      if (e != cudaSuccess) return cuda_fail(e, "stream ordering");
    }
  }
  for (uint32_t i = 0; i < n; ++i) {
    if (hs[i]->d.P <= 1) continue;
    cudaStream_t saved = hs[i]->stream;
    hs[i]->stream = h0->stream;
    rc = guess_output(hs[i]);
    hs[i]->stream = saved;
    if (rc) return rc;
  }
  if ((rc = enqueue_recount(hs, n, true))) return rc;
  // statuses -> output capacities (table_keys bounds the records). The partitioned handles have
  // their records already, unless there was not enough room.
  for (uint32_t i = 0; i < n; ++i)
    KMA_CUDA(cudaMemcpyAsync(hs[i]->host_status, hs[i]->status, sizeof(DevStatus), cudaMemcpyDeviceToHost, h0->stream));
  KMA_CUDA(cudaStreamSynchronize(h0->stream));
  int first_err = KMA_OK;
  std::vector<int> ok(n, 0), todo(n, 0);  // done without an error; to be classified
  for (uint32_t i = 0; i < n; ++i) {
    kma_handle* h = hs[i];
    int e = flags_to_code(h->host_status->flags & ~(h->d.P > 1 ? kFlagOutput : 0u));
    if (e) { h->failed = true; if (!first_err) first_err = e; continue; }
    ok[i] = 1;
    if (h->d.P > 1 && !(h->host_status->flags & kFlagOutput)) continue;
    cudaStream_t saved = h->stream;
    h->stream = h0->stream;
    e = ensure_output(h, h->d.P > 1 ? h->host_status->n_out : h->host_status->table_keys);
    h->stream = saved;
    if (e) { h->failed = true; ok[i] = 0; if (!first_err) first_err = e; continue; }
    if (h->d.P > 1) KMA_CUDA(cudaMemsetAsync(&h->status->flags, 0, sizeof(h->status->flags), h0->stream));
    todo[i] = 1;
  }
  if ((rc = enqueue_classify(hs, n, todo))) return rc;
  for (uint32_t i = 0; i < n; ++i)
    if (todo[i]) KMA_CUDA(cudaMemcpyAsync(hs[i]->host_status, hs[i]->status, sizeof(DevStatus), cudaMemcpyDeviceToHost, h0->stream));
  if (std::any_of(todo.begin(), todo.end(), [](int v) { return v != 0; })) KMA_CUDA(cudaStreamSynchronize(h0->stream));
  for (uint32_t i = 0; i < n; ++i) {
    kma_handle* h = hs[i];
    if (!ok[i]) { if (out) std::memset(&out[i], 0, sizeof(kma_result)); continue; }
    int e = flags_to_code(h->host_status->flags);
    if (e) { h->failed = true; if (!first_err) first_err = e; if (out) std::memset(&out[i], 0, sizeof(kma_result)); continue; }
    fill_result(h);
    h->finalized = true;
    if (out) out[i] = h->res;
  }
  return first_err;
}

int kmer_analysis_finalize(kma_handle* h, kma_result* out) {
  if (!h) return KMA_EINVAL;
  kma_handle* hs[1] = {h};
  return finalize_many(hs, 1, out);
}

int kmer_analysis_finalize_batch(kma_handle* const* hs, uint32_t n, kma_result* out) {
  return finalize_many(hs, n, out);
}

int kmer_analysis_reserve_output(kma_handle* h, uint64_t n_records) {
  if (!h) return KMA_EINVAL;
  return ensure_output(h, n_records);
}

int kmer_analysis_finalize_batch_async(kma_handle* const* hs, uint32_t n) {
  int rc = check_batch(hs, n);
  if (rc) return rc;
  for (uint32_t i = 0; i < n; ++i)
    if (!hs[i]->out_keys) return KMA_ESTATE;  // kmer_analysis_reserve_output first
  if ((rc = enqueue_recount(hs, n, false))) return rc;
  std::vector<int> todo(n, 0);  // the partitioned handles have their records already
  for (uint32_t i = 0; i < n; ++i) todo[i] = hs[i]->d.P <= 1;
  if ((rc = enqueue_classify(hs, n, todo))) return rc;
  for (uint32_t i = 0; i < n; ++i) hs[i]->finalized = true;
  return KMA_OK;
}

int kmer_analysis_fetch_result(kma_handle* h, kma_result* out) {
  if (!h) return KMA_EINVAL;
  if (!h->finalized) return KMA_ESTATE;
  int rc = read_status(h);
  if (rc) return rc;
  fill_result(h);
  if (out) *out = h->res;
  rc = flags_to_code(h->host_status->flags);
  if (!rc && h->host_status->n_out > h->out_cap) rc = KMA_EFULL;
  return rc;
}

int kmer_analysis_count_batch(kma_handle* const* hs, const kma_reads* reads, uint32_t n) {
  if (!hs || !reads || n == 0 || n > KMA_MAX_BATCH) return KMA_EINVAL;
  kma_handle* h0 = hs[0];
  for (uint32_t i = 0; i < n; ++i) {
    if (!hs[i]) return KMA_EINVAL;
    if (hs[i]->finalized || hs[i]->failed) return KMA_ESTATE;
    if (hs[i]->device != h0->device) return KMA_EINVAL;
    for (uint32_t j = 0; j < i; ++j)
      if (hs[j] == hs[i]) return KMA_EINVAL;
    if (reads[i].n_reads && (!reads[i].seq || !reads[i].qual || !reads[i].offsets)) return KMA_EINVAL;
  }
  PackBatch pk;
  std::memset(&pk, 0, sizeof(pk));
  set_pack_waits(h0, pk);
  struct Later { kma_handle* h; u64 q0, n_pos, n_reads, n_bases; };
  std::vector<Later> part_later;
  PassBatch ps;
  std::memset(&ps, 0, sizeof(ps));
  ps.prefetch = h0->prefetch;
  const u64 tile = (u64)h0->shape.block_threads * h0->shape.windows_per_thread;
  u64 words = 0, tiles = 0;
  for (uint32_t i = 0; i < n; ++i) {
    kma_handle* h = hs[i];
    if (reads[i].n_reads == 0) continue;
    PackDesc pd;
    u64 q0, n_pos;
    int rc = reserve_batch(h, reads[i].n_reads, reads[i].n_bases, pd, q0, n_pos, h0->stream);
    if (rc) return rc;
    pd.seq = (const unsigned char*)reads[i].seq;
    pd.qual = (const unsigned char*)reads[i].qual;
    pd.offsets = (const unsigned long long*)reads[i].offsets;
    pd.delta = 0;
    pd.chunk_begin = words;
    words += (n_pos / 64 + kPackChunkWords - 1) / kPackChunkWords;
    pk.d[pk.n++] = pd;
    if (h->d.P > 1) {  // partitioned: its own scatter after the packing
      part_later.push_back({h, q0, n_pos, reads[i].n_reads, reads[i].n_bases});
      continue;
    }
    h->count_bound += n_pos;
    PassDesc d = pass_desc(h, h->p.use_bloom ? kModeBloom : kModeCount, q0, q0 + n_pos);
    d.tile_begin = tiles;
    tiles += (n_pos + tile - 1) / tile;
    ps.d[ps.n++] = d;
  }
  pk.total_chunks = words;
  ps.total_tiles = tiles;
  int rc = timed_launch(h0, KMA_KERNEL_PACK, h0->stream, pk.n > 0 && words > 0,
                        [&] { return launch_pack(pk, h0->stream, h0->num_sms); });
  if (rc) return rc;
  rc = timed_launch(h0, KMA_KERNEL_PASS, h0->stream, ps.n > 0 && tiles > 0,
                    [&] { return launch_pass(ps, h0->shape, h0->agg, h0->stream); });
  if (rc) return rc;
  for (auto& l : part_later)
    if ((rc = first_pass(l.h, l.q0, l.n_pos, l.n_reads, l.n_bases, h0->stream))) return rc;
  return KMA_OK;
}

int kmer_analysis_copy_result(kma_handle* h, uint64_t* keys, uint32_t* counts, uint32_t* ext,
                              uint8_t* codes, uint64_t capacity, int on_device) {
  if (!h) return KMA_EINVAL;
  if (!h->finalized) return KMA_ESTATE;
  const u64 n = h->res.n;
  if (capacity < n) return KMA_EINVAL;
  const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  if (n) {
    if (keys) KMA_CUDA(cudaMemcpyAsync(keys, h->out_keys, n * 16, kind, h->stream));
    if (counts) KMA_CUDA(cudaMemcpyAsync(counts, h->out_counts, n * 4, kind, h->stream));
    if (ext) KMA_CUDA(cudaMemcpyAsync(ext, h->out_ext, n * 32, kind, h->stream));
    if (codes) KMA_CUDA(cudaMemcpyAsync(codes, h->out_codes, n * 2, kind, h->stream));
  }
  KMA_CUDA(cudaStreamSynchronize(h->stream));
  return KMA_OK;
}

int kmer_analysis_finalize_to_host(kma_handle* h, uint64_t* keys, uint32_t* counts, uint32_t* ext,
                                   uint8_t* codes, uint64_t capacity, kma_result* out) {
  if (!h) return KMA_EINVAL;
  if (h->finalized || h->failed) return KMA_ESTATE;
  if (!h->host_groups) {
    h->host_groups = static_cast<u64*>(pinned_take());
    if (!h->host_groups) return KMA_ENOMEM;
    for (auto& e : h->group_ev) KMA_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  }
  if (!h->copy_stream) KMA_CUDA(cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking));
  const bool parts = h->d.P > 1;
  const u64 S = h->d.plan.table_slots;
  // One table: the keys counted so far bound the records. Partitions: nothing is in the table
  // yet; room for as many records as the caller has room for, if there is memory for them (more:
  // classified again below).
  int rc = read_status(h);
  if (rc) return rc;
  if ((rc = flags_to_code(h->host_status->flags))) { h->failed = true; return rc; }
  rc = ensure_output(h, parts ? std::min<u64>(capacity, S) : h->host_status->table_keys);
  if (rc && !(parts && rc == KMA_ENOMEM)) { h->failed = true; return rc; }
  if (parts) {
    if ((rc = reset_counted(h, h->stream))) return rc;
  } else {
    KMA_CUDA(cudaMemsetAsync(&h->status->n_out, 0, 2 * sizeof(u64), h->stream));
  }
  const unsigned G = (unsigned)std::max<u64>(1, std::min<u64>(kFinalizeGroups, parts ? h->d.P : S / kClassTile));
  unsigned published = 0;  // groups whose records have been appended to the output
  // Publish the record count so far.
  auto announce = [&]() -> int {
    KMA_CUDA(cudaMemcpyAsync(&h->host_groups[published], &h->status->n_out, sizeof(u64), cudaMemcpyDeviceToHost, h->stream));
    KMA_CUDA(cudaEventRecord(h->group_ev[published], h->stream));
    ++published;
    return KMA_OK;
  };
  // Classify the table slots [s0, s1), then the same.
  auto publish = [&](u64 s0, u64 s1) -> int {
    ClassBatch cb;
    std::memset(&cb, 0, sizeof(cb));
    cb.write = 1;
    cb.n = 1;
    cb.d[0] = class_desc(h);
    cb.d[0].table = h->table + s0;
    cb.d[0].slots = s1 - s0;
    cb.total_blocks = (s1 - s0 + kClassTile - 1) / kClassTile;
    int rc2 = timed_launch(h, KMA_KERNEL_CLASSIFY, h->stream, cb.total_blocks > 0,
                           [&] { return launch_classify(cb, h->stream, h->num_sms); });
    return rc2 ? rc2 : announce();
  };
  if (!parts) {
    // the recount is a pass over the windows: the groups only split the classification
    if (h->p.use_bloom) {
      kma_handle* hs[1] = {h};
      if ((rc = enqueue_recount(hs, 1, true))) return rc;
    }
    for (unsigned i = 0; i < G; ++i)
      if ((rc = publish(S * i / G, S * (i + 1) / G))) return rc;
  } else {
    // the records are appended to the output as each group of buckets is counted
    const unsigned B = 1u << h->d.log_b;
    rc = count_records(h, h, h->stream, true, G, [&](unsigned end) -> int {
      if (end != B && (u64)end * G / B <= published) return KMA_OK;
      return announce();
    });
    if (rc) return rc;
  }
  KMA_CUDA(cudaMemcpyAsync(h->host_status, h->status, sizeof(DevStatus), cudaMemcpyDeviceToHost, h->stream));
  // As each group completes, its records go to the host on the copy stream while the GPU
  // counts the next group.
  const u64 cap = std::min<u64>(capacity, h->out_cap);
  u64 done = 0;
  for (unsigned i = 0; i < published; ++i) {
    KMA_CUDA(cudaEventSynchronize(h->group_ev[i]));
    const u64 upto = std::min<u64>(h->host_groups[i], cap);
    if (upto <= done) continue;
    const u64 n = upto - done;
    KMA_CUDA(cudaStreamWaitEvent(h->copy_stream, h->group_ev[i], 0));
    if (keys) KMA_CUDA(cudaMemcpyAsync(keys + 2 * done, h->out_keys + 2 * done, n * 16, cudaMemcpyDeviceToHost, h->copy_stream));
    if (counts) KMA_CUDA(cudaMemcpyAsync(counts + done, h->out_counts + done, n * 4, cudaMemcpyDeviceToHost, h->copy_stream));
    if (ext) KMA_CUDA(cudaMemcpyAsync(ext + 8 * done, h->out_ext + 8 * done, n * 32, cudaMemcpyDeviceToHost, h->copy_stream));
    if (codes) KMA_CUDA(cudaMemcpyAsync(codes + 2 * done, h->out_codes + 2 * done, n * 2, cudaMemcpyDeviceToHost, h->copy_stream));
    done = upto;
  }
  free_records(h);
  KMA_CUDA(cudaStreamSynchronize(h->stream));
  KMA_CUDA(cudaStreamSynchronize(h->copy_stream));
  if (h->host_status->n_out > h->out_cap && !(h->host_status->flags & ~kFlagOutput)) {
    // more records than the caller (and so the device output) has room for: all of them into a
    // larger device output; the host has the first `capacity` of the same set. Or there was no memory
    // for that output before the counting: then the host gets them now
    if ((rc = ensure_output(h, h->host_status->n_out))) { h->failed = true; return rc; }
    KMA_CUDA(cudaMemsetAsync(&h->status->flags, 0, sizeof(h->status->flags), h->stream));
    KMA_CUDA(cudaMemsetAsync(&h->status->n_out, 0, 2 * sizeof(u64), h->stream));
    published = 0;
    if ((rc = publish(0, S)) || (rc = read_status(h))) { h->failed = true; return rc; }
    const u64 n = std::min<u64>(capacity, h->host_status->n_out);
    if (done < n) {
      if (keys) KMA_CUDA(cudaMemcpyAsync(keys, h->out_keys, n * 16, cudaMemcpyDeviceToHost, h->stream));
      if (counts) KMA_CUDA(cudaMemcpyAsync(counts, h->out_counts, n * 4, cudaMemcpyDeviceToHost, h->stream));
      if (ext) KMA_CUDA(cudaMemcpyAsync(ext, h->out_ext, n * 32, cudaMemcpyDeviceToHost, h->stream));
      if (codes) KMA_CUDA(cudaMemcpyAsync(codes, h->out_codes, n * 2, cudaMemcpyDeviceToHost, h->stream));
      KMA_CUDA(cudaStreamSynchronize(h->stream));
    }
  }
  if ((rc = flags_to_code(h->host_status->flags))) {
    h->failed = true;
    if (out) std::memset(out, 0, sizeof(kma_result));
    return rc;
  }
  fill_result(h);
  h->finalized = true;
  if (out) *out = h->res;
  return h->res.n > capacity ? KMA_EFULL : KMA_OK;
}

int kmer_analysis_query(kma_handle* h, const uint64_t* keys, uint64_t n, uint32_t* counts,
                        uint32_t* ext, uint8_t* codes, int on_device) {
  if (!h) return KMA_EINVAL;
  if (!h->finalized) return KMA_ESTATE;
  if (n == 0) return KMA_OK;
  if (!keys || !counts || !ext || !codes) return KMA_EINVAL;
  const unsigned min_ext = h->p.min_ext_count ? h->p.min_ext_count : 1;
  if (on_device) {
    return timed_launch(h, KMA_KERNEL_QUERY, h->stream, true, [&] {
      return launch_query(h->table, h->d.Sp, h->d.P, h->p.k, h->p.canonical, h->p.min_depth,
                          min_ext, (const u64*)keys, n, counts, ext, codes, h->status, h->stream);
    });
  }
  u64* dk = nullptr;
  unsigned *dc = nullptr, *de = nullptr;
  unsigned char* dcode = nullptr;
  int rc;
  if ((rc = dalloc(h, &dk, 2 * n)) || (rc = dalloc(h, &dc, n)) || (rc = dalloc(h, &de, 8 * n)) ||
      (rc = dalloc(h, &dcode, 2 * n))) {
    dfree(h, dk); dfree(h, dc); dfree(h, de); dfree(h, dcode);
    return rc;
  }
  cudaError_t e = cudaMemcpyAsync(dk, keys, n * 16, cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess) {
    rc = timed_launch(h, KMA_KERNEL_QUERY, h->stream, true, [&] {
      return launch_query(h->table, h->d.Sp, h->d.P, h->p.k, h->p.canonical, h->p.min_depth,
                          min_ext, dk, n, dc, de, dcode, h->status, h->stream);
    });
    if (rc) { dfree(h, dk); dfree(h, dc); dfree(h, de); dfree(h, dcode); return rc; }
  }
  if (e == cudaSuccess) {
    bring_pages_in({{(char*)counts, n * 4}, {(char*)ext, n * 32}, {(char*)codes, n * 2}});
    e = cudaMemcpyAsync(counts, dc, n * 4, cudaMemcpyDeviceToHost, h->stream);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(ext, de, n * 32, cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(codes, dcode, n * 2, cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  dfree(h, dk); dfree(h, dc); dfree(h, de); dfree(h, dcode);
  if (e != cudaSuccess) return cuda_fail(e, "query");
  return KMA_OK;
}

int kmer_analysis_reset(kma_handle* h) {
  if (!h) return KMA_EINVAL;
  return clear_state(h);
}

int kmer_analysis_set_stream(kma_handle* h, void* cuda_stream) {
  if (!h) return KMA_EINVAL;
  h->stream = (cudaStream_t)cuda_stream;
  return KMA_OK;
}

int kmer_analysis_status(kma_handle* h) {
  if (!h) return KMA_EINVAL;
  int rc = read_status(h);
  if (rc) return rc;
  return flags_to_code(h->host_status->flags);
}

uint64_t kmer_analysis_device_bytes(const kma_handle* h) {
  if (!h) return 0;
  return h->d.plan.device_bytes + h->out_cap * (16 + 4 + 32 + 2);
}

int kmer_analysis_set_profiling(kma_handle* h, int enable) {
  if (!h) return KMA_EINVAL;
  h->profiling = enable != 0;
  return KMA_OK;
}

int kmer_analysis_timings(kma_handle* h, kma_timings* out, int reset) {
  if (!h || !out) return KMA_EINVAL;
  KMA_CUDA(cudaStreamSynchronize(h->stream));
  for (auto& r : h->prof) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, r.a, r.b) == cudaSuccess && r.kind >= 0 && r.kind < 8) h->ms[r.kind] += ms;
    h->event_pool.push_back(r.a);
    h->event_pool.push_back(r.b);
  }
  h->prof.clear();
  cudaGetLastError();
  std::memset(out, 0, sizeof(*out));
  for (int i = 0; i < 8; ++i) {
    out->ms[i] = h->ms[i];
    out->launches[i] = h->launches[i];
    out->total_launches += h->launches[i];
  }
  int rc = read_status(h);
  if (rc) return rc;
  out->first_sightings = h->host_status->first_sightings;
  if (reset) {
    for (int i = 0; i < 8; ++i) { h->ms[i] = 0; h->launches[i] = 0; }
  }
  return KMA_OK;
}

int kmer_analysis_contigs(kma_handle* h, kma_contigs* out) {
  if (!h || !out) return KMA_EINVAL;
  if (!h->finalized) return KMA_ESTATE;
  free_contigs(h);
  cudaError_t err = cudaSuccess;
  const int rc = contig_pass(h->out_keys, h->out_codes, h->res.n, h->p.k, h->p.canonical, h->pool, h->stream,
                             &h->contig_seq, &h->contig_offsets, &h->contig_n, &h->contig_bases,
                             &h->contig_vertices, &h->contig_cycles, &h->status->flags, &err);
  if (rc == KMA_ECUDA) return cuda_fail(err, "contig generation");
  if (rc) return rc;
  int st = read_status(h);
  if (st) return st;
  if (h->host_status->flags & (kFlagFull | kFlagOutput)) return KMA_EFULL;
  out->n_contigs = h->contig_n;
  out->n_bases = h->contig_bases;
  out->n_vertices = h->contig_vertices;
  out->n_cycles = h->contig_cycles;
  out->seq = h->contig_seq;
  out->offsets = (const uint64_t*)h->contig_offsets;
  return KMA_OK;
}

int kmer_analysis_copy_contigs(kma_handle* h, char* seq, uint64_t* offsets, int on_device) {
  if (!h) return KMA_EINVAL;
  if (!h->contig_offsets) return KMA_ESTATE;
  const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  if (seq && h->contig_bases) KMA_CUDA(cudaMemcpyAsync(seq, h->contig_seq, h->contig_bases, kind, h->stream));
  if (offsets) KMA_CUDA(cudaMemcpyAsync(offsets, h->contig_offsets, (h->contig_n + 1) * 8, kind, h->stream));
  KMA_CUDA(cudaStreamSynchronize(h->stream));
  return KMA_OK;
}

int kmer_analysis_hll_estimate(const uint8_t* registers, uint32_t precision, double* distinct) {
  if (!registers || !distinct || precision < KMA_HLL_MIN_PRECISION || precision > KMA_HLL_MAX_PRECISION)
    return KMA_EINVAL;
  *distinct = hll_estimate(registers, precision);
  return KMA_OK;
}

int kmer_analysis_estimate(const kma_params* params, const char* seq, const char* qual,
                           const uint64_t* offsets, uint64_t n_reads, int on_device, void* cuda_stream,
                           kma_estimate* est, uint8_t* registers) {
  if (!params || !est || !offsets) return KMA_EINVAL;
  const unsigned p = est->precision ? est->precision : 14;
  if (p < KMA_HLL_MIN_PRECISION || p > KMA_HLL_MAX_PRECISION) return KMA_EINVAL;
  if (n_reads && (!seq || !qual)) return KMA_EINVAL;
  int rc = check_params(params);
  if (rc) return rc;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  // bases of the read set (device offsets: read back the two ends)
  u64 ends[2] = {0, 0};
  if (n_reads) {
    if (on_device) {
      KMA_CUDA(cudaMemcpyAsync(&ends[0], offsets, 8, cudaMemcpyDeviceToHost, stream));
      KMA_CUDA(cudaMemcpyAsync(&ends[1], offsets + n_reads, 8, cudaMemcpyDeviceToHost, stream));
      KMA_CUDA(cudaStreamSynchronize(stream));
    } else {
      ends[0] = offsets[0];
      ends[1] = offsets[n_reads];
    }
    if (ends[1] < ends[0]) return KMA_EINVAL;
  }
  // a handle that only packs: the read arena, no Bloom filter, a token table
  kma_params q = *params;
  q.use_bloom = 0;
  q.table_capacity = 64;
  q.expected_keys = 0;
  q.expected_distinct = 0;
  q.partitions = 1;
  q.fault_inject = 0;
  q.max_bases = std::max<u64>(q.max_bases, std::max<u64>(ends[1] - ends[0], 1));
  q.max_reads = std::max<u64>(q.max_reads, std::max<u64>(n_reads, 1));
  kma_handle* h = nullptr;
  if ((rc = kmer_analysis_create(&q, cuda_stream, &h))) return rc;
  h->pack_only = true;
  const u64 m = 1ull << p;
  std::vector<unsigned> regs32(m, 0);
  if (registers)
    for (u64 j = 0; j < m; ++j) regs32[j] = registers[j];
  // device temporaries: sketch registers, the CTAs' heavy-hitter summaries, and (host input)
  // the reads, copied whole so that they are packed as one batch (the sampled stream is
  // defined on the positions of one packed batch)
  const unsigned grid = hll_grid(p, params->k, h->num_sms);
  const u64 mg_n = (u64)grid * kMgBuckets * kMgCounters;
  std::vector<void*> temps;
  auto finish = [&](int code) {
    for (void* t : temps) cudaFreeAsync(t, h->stream);
    kmer_analysis_destroy(h);
    return code;
  };
  auto temp = [&](void** ptr, u64 bytes) -> int {
    cudaError_t e = cudaMallocFromPoolAsync(ptr, std::max<u64>(bytes, 16), h->pool, h->stream);
    if (e != cudaSuccess) {
      cudaGetLastError();
      *ptr = nullptr;
      return e == cudaErrorMemoryAllocation ? KMA_ENOMEM : cuda_fail(e, "estimate temporaries");
    }
    temps.push_back(*ptr);
    return KMA_OK;
  };
  unsigned* d_regs = nullptr;
  MgOut mg{};
  // one zeroed block: items, totals, merge tables, merged counts; merged entries and the items
  // come back together
  const u64 slots = mg_table_slots(grid);
  const u64 zeroed = kMgBuckets * 8 + mg_n * 8 + kMgBuckets * slots * 4 + kMgBuckets * 4;
  char* zero = nullptr;
  if ((rc = temp((void**)&d_regs, m * 4)) || (rc = temp((void**)&mg.lo, mg_n * 8)) ||
      (rc = temp((void**)&mg.hi, mg_n * 8)) || (rc = temp((void**)&mg.count, mg_n * 4)) ||
      (rc = temp((void**)&mg.merged, kMgBuckets * kMgCounters * sizeof(MgEntry))) ||
      (rc = temp((void**)&zero, zeroed)))
    return finish(rc);
  mg.items = (unsigned long long*)zero;
  mg.total = mg.items + kMgBuckets;
  mg.table = (unsigned*)(mg.total + mg_n);
  mg.n_merged = mg.table + kMgBuckets * slots;
  cudaError_t e;
  if ((e = cudaMemsetAsync(zero, 0, zeroed, h->stream)) != cudaSuccess) return finish(cuda_fail(e, "summaries"));
  if ((e = cudaMemcpyAsync(d_regs, regs32.data(), m * 4, cudaMemcpyHostToDevice, h->stream)) != cudaSuccess)
    return finish(cuda_fail(e, "sketch registers in"));
  if (n_reads) {
    const char *s_in = seq, *q_in = qual;
    const uint64_t* o_in = offsets;
    if (!on_device) {
      const u64 nb = ends[1] - ends[0];
      void *ds = nullptr, *dq = nullptr, *dof = nullptr;
      if ((rc = temp(&ds, nb)) || (rc = temp(&dq, nb)) || (rc = temp(&dof, (n_reads + 1) * 8))) return finish(rc);
      if ((e = cudaMemcpyAsync(ds, seq + ends[0], nb, cudaMemcpyHostToDevice, h->stream)) != cudaSuccess ||
          (e = cudaMemcpyAsync(dq, qual + ends[0], nb, cudaMemcpyHostToDevice, h->stream)) != cudaSuccess ||
          (e = cudaMemcpyAsync(dof, offsets, (n_reads + 1) * 8, cudaMemcpyHostToDevice, h->stream)) != cudaSuccess)
        return finish(cuda_fail(e, "estimate reads in"));
      // the device copy of the bases starts at offsets[0]
      s_in = (const char*)ds - ends[0];
      q_in = (const char*)dq - ends[0];
      o_in = (const uint64_t*)dof;
    }
    if ((rc = kmer_analysis_count(h, s_in, q_in, o_in, n_reads, 1))) return finish(rc);
  }
  PartWindows w;
  w.codes = h->codes; w.rcodes = h->rcodes; w.inv = h->inv; w.hq = h->hq;
  w.q0 = 0; w.q1 = h->q_used;
  const unsigned n_parts = params->n_parts > 1 ? params->n_parts : 1;
  const unsigned part = params->n_parts > 1 ? params->part : 0;
  if ((e = launch_hll(w, params->k, params->canonical, n_parts, part, p, d_regs, h->status, mg, grid,
                      h->stream)) != cudaSuccess)
    return finish(cuda_fail(e, "hll_kernel"));
  if ((e = launch_mg_merge(mg, grid, h->stream)) != cudaSuccess) return finish(cuda_fail(e, "mg_merge"));
  unsigned n_merged[kMgBuckets];
  u64 bucket_n[kMgBuckets];
  std::vector<MgEntry> summary(kMgBuckets * kMgCounters);
  if ((e = cudaMemcpyAsync(regs32.data(), d_regs, m * 4, cudaMemcpyDeviceToHost, h->stream)) != cudaSuccess ||
      (e = cudaMemcpyAsync(summary.data(), mg.merged, summary.size() * sizeof(MgEntry), cudaMemcpyDeviceToHost,
                           h->stream)) != cudaSuccess ||
      (e = cudaMemcpyAsync(n_merged, mg.n_merged, sizeof n_merged, cudaMemcpyDeviceToHost, h->stream)) !=
          cudaSuccess ||
      (e = cudaMemcpyAsync(bucket_n, mg.items, sizeof bucket_n, cudaMemcpyDeviceToHost, h->stream)) != cudaSuccess)
    return finish(cuda_fail(e, "estimate results out"));
  if ((rc = read_status(h))) return finish(rc);
  if ((rc = flags_to_code(h->host_status->flags))) return finish(rc);
  std::vector<uint8_t> regs8(m);
  for (u64 j = 0; j < m; ++j) regs8[j] = (uint8_t)regs32[j];
  if (registers) std::memcpy(registers, regs8.data(), m);
  est->precision = p;
  est->distinct = hll_estimate(regs8.data(), p);
  est->rel_std_error = 1.04 / std::sqrt((double)m);
  est->valid_windows = h->host_status->valid_windows;
  // heavy hitters: the keys of all buckets by count
  struct Heavy {
    MgEntry e;
    unsigned bucket;
  };
  std::vector<Heavy> merged;
  for (unsigned b = 0; b < kMgBuckets; ++b)
    for (unsigned i = 0; i < std::min(n_merged[b], kMgCounters); ++i) merged.push_back({summary[b * kMgCounters + i], b});
  std::sort(merged.begin(), merged.end(), [](const Heavy& x, const Heavy& y) {
    if (x.e.count != y.e.count) return x.e.count > y.e.count;
    return x.e.hi != y.e.hi ? x.e.hi < y.e.hi : x.e.lo < y.e.lo;
  });
  u64 sampled = 0;
  for (u64 x : bucket_n) sampled += x;
  est->sampled_windows = sampled;
  est->heavy_threshold = std::max<u64>(1, sampled / 2048);
  est->heavy_hitters = !merged.empty() && merged[0].e.count >= est->heavy_threshold ? 1u : 0u;
  est->n_summary = merged.size();
  const u64 rows = std::min<u64>(est->summary_capacity, merged.size());
  for (u64 i = 0; i < rows; ++i) {
    if (est->summary_keys) { est->summary_keys[2 * i] = merged[i].e.lo; est->summary_keys[2 * i + 1] = merged[i].e.hi; }
    if (est->summary_counts) est->summary_counts[i] = merged[i].e.count;
    if (est->summary_bucket) est->summary_bucket[i] = merged[i].bucket;
  }
  if (est->bucket_windows)
    for (unsigned b = 0; b < kMgBuckets; ++b) est->bucket_windows[b] = bucket_n[b];
  return finish(KMA_OK);
}

int kmer_analysis_parse_fastq(const char* text, uint64_t n_bytes, int on_device, char* seq, char* qual,
                              uint64_t* offsets, uint64_t cap_bases, uint64_t cap_reads, uint64_t* n_reads,
                              uint64_t* n_bases, void* cuda_stream) {
  if (!n_reads || !n_bases || !offsets || (n_bytes && !text)) return KMA_EINVAL;
  *n_reads = *n_bases = 0;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int dev = 0, rc;
  KMA_CUDA(cudaGetDevice(&dev));
  cudaMemPool_t pool;
  if ((rc = get_pool(dev, &pool))) return rc;
  std::vector<void*> temps;
  auto alloc = [&](void** p, u64 bytes) -> int {
    cudaError_t e = cudaMallocFromPoolAsync(p, std::max<u64>(bytes, 8), pool, st);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return e == cudaErrorMemoryAllocation ? KMA_ENOMEM : cuda_fail(e, "fastq temporaries");
    }
    temps.push_back(*p);
    return KMA_OK;
  };
  auto done = [&](int code) {
    for (void* p : temps) cudaFreeAsync(p, st);
    cudaStreamSynchronize(st);
    return code;
  };
#define FQ_CUDA(call)                                              \
  do {                                                             \
    cudaError_t e_ = (call);                                       \
    if (e_ != cudaSuccess) return done(cuda_fail(e_, #call));      \
  } while (0)
  if (n_bytes == 0) {
    FQ_CUDA(cudaMemsetAsync(offsets, 0, 8, st));
    return done(KMA_OK);
  }
  const unsigned char* d_text = (const unsigned char*)text;
  if (!on_device) {
    void* t = nullptr;
    if ((rc = alloc(&t, n_bytes))) return done(rc);
    FQ_CUDA(cudaMemcpyAsync(t, text, n_bytes, cudaMemcpyHostToDevice, st));
    d_text = (const unsigned char*)t;
  }
  // 1-2: newlines per chunk, scanned (one extra element receives the total)
  const u64 chunks = fastq_chunks(n_bytes);
  u64 *cc = nullptr, *tmp = nullptr;
  if ((rc = alloc((void**)&cc, (chunks + 1) * 8)) ||
      (rc = alloc((void**)&tmp, scan_scratch_items(std::max<u64>(chunks + 1, 1)) * 8)))
    return done(rc);
  unsigned short* masks = nullptr;
  if ((rc = alloc((void**)&masks, fastq_masks(n_bytes) * 2))) return done(rc);
  FQ_CUDA(launch_fastq_count(d_text, n_bytes, masks, cc, st));
  FQ_CUDA(cudaMemsetAsync(cc + chunks, 0, 8, st));
  FQ_CUDA(scan_exclusive(cc, chunks + 1, tmp, st));
  u64 n_lines = 0;
  FQ_CUDA(cudaMemcpyAsync(&n_lines, cc + chunks, 8, cudaMemcpyDeviceToHost, st));
  FQ_CUDA(cudaStreamSynchronize(st));
  // 3: line ends
  u64* line_end = nullptr;
  if ((rc = alloc((void**)&line_end, n_lines * 8))) return done(rc);
  FQ_CUDA(launch_fastq_lines(d_text, n_bytes, masks, cc, line_end, st));
  // lines after the last complete record must be empty
  const u64 extra = n_lines % 4;
  if (extra) {
    const u64 first = n_lines - extra;  // first extra line
    u64 ends[4] = {0, 0, 0, 0};
    const u64 from = first ? first - 1 : 0, cnt = first ? extra + 1 : extra;
    FQ_CUDA(cudaMemcpyAsync(ends, line_end + from, cnt * 8, cudaMemcpyDeviceToHost, st));
    FQ_CUDA(cudaStreamSynchronize(st));
    u64 prev_end = first ? ends[0] : (u64)-1;  // (u64)-1 + 1 == 0: the text's first byte
    for (u64 i = 0; i < extra; ++i) {
      const u64 e = ends[first ? i + 1 : i];
      const u64 len = e - (prev_end + 1);
      if (len > 1) return done(KMA_EINVAL);
      if (len == 1) {  // a lone '\r' is an empty line too
        char c = 0;
        FQ_CUDA(cudaMemcpyAsync(&c, d_text + prev_end + 1, 1, cudaMemcpyDeviceToHost, st));
        FQ_CUDA(cudaStreamSynchronize(st));
        if (c != '\r') return done(KMA_EINVAL);
      }
      prev_end = e;
    }
  }
  const u64 nr = (n_lines - extra) / 4;
  *n_reads = nr;
  if (nr > cap_reads) return done(KMA_EFULL);
  // 4-5: record checks, bases per record, scanned into the offsets
  unsigned long long* bad = nullptr;
  if ((rc = alloc((void**)&bad, 8))) return done(rc);
  u64* scan_tmp = nullptr;
  if ((rc = alloc((void**)&scan_tmp, scan_scratch_items(nr + 1) * 8))) return done(rc);
  FQ_CUDA(cudaMemsetAsync(bad, 0xFF, 8, st));
  FQ_CUDA(launch_fastq_records(d_text, line_end, nr, (u64*)offsets, bad, st));
  FQ_CUDA(cudaMemsetAsync(offsets + nr, 0, 8, st));
  FQ_CUDA(scan_exclusive((u64*)offsets, nr + 1, scan_tmp, st));
  u64 back[2] = {0, 0};
  FQ_CUDA(cudaMemcpyAsync(&back[0], offsets + nr, 8, cudaMemcpyDeviceToHost, st));
  FQ_CUDA(cudaMemcpyAsync(&back[1], bad, 8, cudaMemcpyDeviceToHost, st));
  FQ_CUDA(cudaStreamSynchronize(st));
  if (back[1] != ~0ull) return done(KMA_EINVAL);
  *n_bases = back[0];
  if (back[0] > cap_bases) return done(KMA_EFULL);
  if (nr && (!seq || !qual)) return done(KMA_EINVAL);
  // 6: bases and qualities
  FQ_CUDA(launch_fastq_copy(d_text, line_end, nr, (const u64*)offsets, (unsigned char*)seq,
                            (unsigned char*)qual, st));
  return done(KMA_OK);
#undef FQ_CUDA
}

void kmer_analysis_destroy(kma_handle* h) {
  if (!h) return;
  free_all(h);
  delete h;
}

const char* kmer_analysis_strerror(int code) {
  switch (code) {
    case KMA_OK: return "ok";
    case KMA_EINVAL: return "invalid argument";
    case KMA_ENOMEM: return "out of device memory";
    case KMA_EFULL: return "capacity exceeded (hash table or read arena)";
    case KMA_ESTATE: return "call not allowed in this state";
    case KMA_ETIMEOUT: return "device wait timed out";
    case KMA_EOVERFLOW: return "k-mer counter overflow";
    case KMA_ECUDA: return g_last_cuda_error.empty() ? "CUDA error" : g_last_cuda_error.c_str();
    case KMA_ETOOLARGE: return "input exceeds a fixed limit (allocation-free scratch, or 2^31 contig vertices)";
    default: return "unknown error";
  }
}

}  // extern "C"
