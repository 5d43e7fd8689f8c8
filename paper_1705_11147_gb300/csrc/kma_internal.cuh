// Internal layout shared by the library's CUDA translation units (not part of the C ABI).
//
// Device data of one handle ("sample"):
//   packed-read arena  positions q = 0 .. arena_positions-1. Each count() batch starts at a
//                      multiple of 64; read r of a batch occupies [ps_r, ps_r + len_r) and is
//                      followed by one separator position (invalid), so no window can span
//                      two reads and the bases before/after a read are never usable.
//     codes  u64[arena/32]  2 bits per position, first position in the two most significant
//                           bits (A0 C1 G2 T3; 0 for invalid positions)
//     rcodes u64[arena/32]  complemented codes (3 - code), first position in the two LEAST
//                           significant bits: bits [2i, 2i+2k) of consecutive words read as
//                           one number are the reverse complement of the window at i
//     inv    u64[arena/64]  1 = position is not A/C/G/T (separator, N, padding), MSB first
//     hq     u64[arena/64]  1 = A/C/G/T with Phred >= qual_threshold, MSB first
//     marks  u32[arena/32]  Bloom pass: 1 = this window was the first sighting of its k-mer
//   bloom    u64[bloom_words]  blocked Bloom filter: all bits of a k-mer in one word
//   table    Slot[slots]       open addressing, linear probing, 64-byte slots
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace kma {

constexpr uint64_t kEmpty = ~0ull;          // both key words of an empty slot
constexpr uint32_t kMaxProbe = 1u << 14;    // probe limit before reporting a full table
constexpr int kMaxBatch = 64;

// Bounded device waits (bulk-copy staging): polls of an mbarrier before giving up, each poll
// suspending the thread for at most kWaitHintNs (about 1.3 s in all), and the short limit of
// the fault-injection test.
constexpr unsigned kWaitHintNs = 10000;
constexpr unsigned kWaitPolls = 1u << 17;
constexpr unsigned kWaitPollsInjected = 1u << 6;

// Status flags raised on the device.
constexpr uint32_t kFlagFull = 1u;
constexpr uint32_t kFlagOverflow = 2u;
constexpr uint32_t kFlagBadOffsets = 4u;
constexpr uint32_t kFlagTimeout = 8u;     // a bounded device wait gave up
constexpr uint32_t kFlagOutput = 16u;     // more records than the output arrays hold

// One hash-table slot. Every occurrence has exactly one left outcome (a usable base A/C/G/T
// or none) and one right outcome, so the slot keeps five counters per side and no separate
// count: count = none[0] + ext[0..3] = none[1] + ext[4..7]. An occurrence costs two
// counter updates. The key and the two "none" counters share the first 32-byte sector, the
// eight extension counters fill the second.
struct __align__(64) Slot {
  unsigned long long lo, hi;
  unsigned int none[2];  // occurrences without a usable left / right extension base
  unsigned int pad[2];
  unsigned int ext[8];   // left A C G T, right A C G T
};
static_assert(sizeof(Slot) == 64, "slot must be 64 bytes");

struct DevStatus {
  unsigned int flags;
  unsigned int pad;
  unsigned long long valid_windows;
  unsigned long long table_keys;
  unsigned long long n_out;
  unsigned long long n_uu;
  unsigned long long first_sightings;  // Bloom pass: windows marked as first sightings
  unsigned long long reserved[2];
};

// Per-sample view the pass kernels need. Passed by value inside kernel parameters.
struct PassDesc {
  const unsigned long long* codes;
  const unsigned long long* rcodes;
  const unsigned long long* inv;
  const unsigned long long* hq;
  unsigned int* marks;
  unsigned long long* bloom;
  Slot* table;
  DevStatus* status;
  unsigned long long bloom_words;
  unsigned long long slots;
  unsigned long long q0;          // first window start of this launch (multiple of 64)
  unsigned long long q1;          // one past the last window start
  unsigned long long tile_begin;  // first global tile index of this sample
  unsigned int k;
  unsigned int bloom_h;
  unsigned int canonical;
  unsigned int mode;              // kModeBloom / kModeCount / kModeRecount
  unsigned int n_parts;           // owner-computes partition: count only keys owned by `part`
  unsigned int part;
  unsigned int no_overflow;       // 1: no count can reach 2^32 (host bound), counts use red.add
  unsigned int pad;
};

struct PassBatch {
  unsigned int n;
  unsigned int prefetch;          // 1: L2-prefetch each window's first table slot in the Bloom pass
  unsigned long long total_tiles;
  PassDesc d[kMaxBatch];
};

constexpr unsigned int kModeBloom = 0;    // Bloom test-and-set; "seen" -> insert + count; else mark
constexpr unsigned int kModeCount = 1;    // no Bloom: insert + count every window
constexpr unsigned int kModeRecount = 2;  // marked windows: count if the key is in the table

// Pack kernel per-sample input.
struct PackDesc {
  const unsigned char* seq;
  const unsigned char* qual;
  const unsigned long long* offsets;  // n_reads + 1 entries
  long long delta;                    // seq/qual index of base b is offsets-relative b - delta
  unsigned long long n_reads;
  unsigned long long n_bases;         // offsets[n_reads] - offsets[0] as the host believes
  unsigned long long q0;              // arena start (multiple of 64)
  unsigned long long n_pos;           // n_bases + n_reads, rounded up to a multiple of 64
  unsigned long long chunk_begin;     // prefix of 256-word pack chunks over the batch
  unsigned long long* codes;
  unsigned long long* rcodes;
  unsigned long long* inv;
  unsigned long long* hq;
  DevStatus* status;
  unsigned int qual_min;              // qual byte >= qual_min <=> Phred >= threshold
  unsigned int pad;
};

constexpr unsigned long long kPackChunkWords = 256;  // 64-position words per pack CTA chunk

struct PackBatch {
  unsigned int n;
  unsigned int skip_copy;             // testing: wait for staging copies that were never issued
  unsigned int wait_limit;            // polls of the staging barrier before giving up
  unsigned int pad;
  unsigned long long total_chunks;
  PackDesc d[kMaxBatch];
};

struct ClassDesc {
  const Slot* table;
  DevStatus* status;
  unsigned long long slots;
  unsigned long long* out_keys;
  unsigned int* out_counts;
  unsigned int* out_ext;
  unsigned char* out_codes;
  unsigned long long out_cap;
  unsigned long long block_begin;
  unsigned int min_depth;
  unsigned int min_ext;
};

struct ClassBatch {
  unsigned int n;
  unsigned int write;   // 0: count survivors only; 1: compact into out_*
  unsigned long long total_blocks;
  ClassDesc d[kMaxBatch];
};

// ---- Partitioned mode ("owner-computes on chip", Section 5.1's k-mer -> owner map) -------
// The k-mer space is split by the key hash twice: 2^log_b buckets (its top bits), then up to
// sub_max sub-buckets of each, small enough to be counted in one SM's shared memory
// (kma_partition.cu). The table is laid out in P partitions by the same hash: partition p owns
// slots [p*Sp, (p+1)*Sp), so the keys of one bucket go to one or two partitions.
constexpr unsigned kMaxPartitions = 4096;      // k <= 32 (one-word keys)
constexpr unsigned kMaxPartitionsWide = 2048;  // k > 32

constexpr unsigned kMinLogBuckets = 6;         // the record's outcome bits take the place of 6 hash bits
constexpr unsigned kMaxLogBuckets = 11;
constexpr unsigned kMaxSubBuckets = 2048;
constexpr unsigned kPartTile = 8192;           // window starts (and records, at most) per scatter tile
constexpr unsigned kPartSubTile = 4096;        // records per sub-tile of the split
constexpr unsigned kMaxChunkTiles = 1024;      // scatter tiles gathered together by the split
constexpr unsigned kSplitBuckets = 8;          // adjacent buckets per work item of the split
constexpr unsigned kCountCap1 = 3072;          // records of a sub-bucket counted in one go (k <= 32)
constexpr unsigned kCountCap2 = 2304;          // (k > 32)

struct PartGeom {
  Slot* table;
  DevStatus* status;
  unsigned long long Sp;        // table slots per partition
  unsigned int P;
  unsigned int k;
  unsigned int canonical;
  unsigned int n_parts;         // multi-GPU owner filter (as PassDesc)
  unsigned int part;
  unsigned int log_b;           // log2 of the buckets
  unsigned int sub_max;         // most sub-buckets per bucket
  unsigned int avg;             // records per sub-bucket aimed at
  unsigned int cap;             // records a sub-bucket has room for
  unsigned int min_count;       // a key reaches the table with at least this many occurrences (1 or 2)
};

struct PartWindows {
  const unsigned long long* codes;
  const unsigned long long* rcodes;
  const unsigned long long* inv;
  const unsigned long long* hq;
  unsigned long long q0, q1;    // window starts of one count() batch (multiples of 64)
};

// Scatter tiles: tile i holds its records, sorted by bucket, from recs + i * kPartTile records on;
// row i of offs (stride entries) holds the buckets' first records and, at [2^log_b], their number.
struct PartTiles {
  unsigned long long* recs;     // one word per record (k <= 32) or two
  unsigned short* offs;
  unsigned long long* totals;   // [2^log_b] records per bucket (added to by the scatter)
  unsigned long long tile0;     // scatter: first tile of this launch
  unsigned int n_tiles;         // split: tiles to gather from
  unsigned int stride;
};

// Split output for the buckets [b0, b1): sub-bucket s of bucket b has the G.cap places from
// recs[((b - b0) * n_sub + s) * cap] on, and fill[(b - b0) * n_sub + s] records; those beyond cap
// lie in the bucket's overflow segments, over[pos .. pos + n) each.
struct PartSegment {
  unsigned long long pos;
  unsigned int n, pad;
};
constexpr unsigned kCarryWords = 14;  // an entry of carry_in and carry_out: ten counters, h, hi

struct PartSplit {
  unsigned long long* recs;
  unsigned long long* fill;     // starts at 0
  unsigned long long* over;     // room for all records of the buckets
  unsigned long long* over_n;   // records in it; starts at 0
  PartSegment* segs;            // the buckets' segments, bucket b's from seg_base[b - b0] on
  unsigned int* seg_base;       // [b1 - b0]
  unsigned int* n_segs;         // [b1 - b0], starts at 0
  unsigned int b0, b1;
  unsigned int n_chunks;        // chunks of all record slabs
  unsigned int chunk_tiles;     // tiles per chunk
  unsigned int log_lanes;       // lanes per gathered run (log2)
  unsigned int pad;
  unsigned int* keys;           // count: the counted keys for the table (kma_partition.cu)
  unsigned long long* n_keys;   // their number; starts at 0
  unsigned long long keys_cap;  // most that the table can take; the list has room for them
  unsigned int* large;          // [sub-buckets] count: those left to part_large_kernel
  unsigned long long* n_large;  // their number, and how many have been taken; start at 0
  unsigned long long* next_large;
  unsigned long long* key_base; // [sub-buckets] count: the sub-bucket's first key in the list
  unsigned int* key_n;          // [sub-buckets] and their number; starts at 0
  unsigned long long end;       // first table slot behind the group's (all slots: the last group's)
  unsigned int* carry_in;       // keys that go to a slot behind their group's, from the groups before
  unsigned int* carry_out;      // and for the next one (kMaxProbe entries)
  unsigned long long* n_carry_in;
  unsigned long long* n_carry_out;  // starts at 0
  unsigned long long* inserted; // CTAs of part_insert_kernel that are done; starts at 0
};

// Output records of the keys inserted (as ClassDesc).
struct PartOut {
  unsigned long long* keys;
  unsigned int* counts;
  unsigned int* ext;
  unsigned char* codes;
  unsigned long long cap;
  unsigned int min_depth;
  unsigned int min_ext;
};

cudaError_t launch_part_scatter(const PartGeom& g, const PartWindows& w, const PartTiles& t, cudaStream_t stream,
                                int num_sms);
cudaError_t launch_part_base(const unsigned long long* totals, const PartSplit& s, cudaStream_t stream);
cudaError_t launch_part_split(const PartGeom& g, const PartTiles& t, const PartSplit& s, cudaStream_t stream,
                              int num_sms);
cudaError_t launch_part_count(const PartGeom& g, const PartSplit& s, cudaStream_t stream, int num_sms);
cudaError_t launch_part_large(const PartGeom& g, const PartSplit& s, const PartOut& o, cudaStream_t stream, int num_sms);
cudaError_t launch_part_build(const PartGeom& g, const PartSplit& s, cudaStream_t stream, int num_sms);
cudaError_t launch_part_insert(const PartGeom& g, const PartSplit& s, const PartOut& o, cudaStream_t stream, int num_sms);
constexpr unsigned kMaxKeyWords = 10;          // words of one counted key in the list

// FASTQ parsing (kma_fastq.cu) and the device-wide exclusive scan it uses.
unsigned long long scan_scratch_items(unsigned long long n);
cudaError_t scan_exclusive(unsigned long long* data, unsigned long long n, unsigned long long* tmp,
                           cudaStream_t stream);
unsigned long long fastq_chunks(unsigned long long n_bytes);
unsigned long long fastq_masks(unsigned long long n_bytes);  // newline masks, one per 16 bytes
cudaError_t launch_fastq_count(const unsigned char* text, unsigned long long n, unsigned short* masks,
                               unsigned long long* chunk_counts,
                               cudaStream_t stream);
cudaError_t launch_fastq_lines(const unsigned char* text, unsigned long long n, const unsigned short* masks,
                               const unsigned long long* chunk_offsets, unsigned long long* line_end,
                               cudaStream_t stream);
cudaError_t launch_fastq_records(const unsigned char* text, const unsigned long long* line_end,
                                 unsigned long long n_reads, unsigned long long* seq_len,
                                 unsigned long long* bad, cudaStream_t stream);
cudaError_t launch_fastq_copy(const unsigned char* text, const unsigned long long* line_end,
                              unsigned long long n_reads, const unsigned long long* offsets, unsigned char* seq,
                              unsigned char* qual, cudaStream_t stream);

// Contig generation over finalized records (kma_contig.cu). Returns 0, a negative KMA_E*
// code (-7 = CUDA error in *err), and on success pool allocations in *seq_out / *offsets_out.
int contig_pass(const unsigned long long* keys, const unsigned char* codes, unsigned long long n, unsigned k,
                unsigned canonical, cudaMemPool_t pool, cudaStream_t st, char** seq_out,
                unsigned long long** offsets_out, unsigned long long* n_contigs, unsigned long long* n_bases,
                unsigned long long* n_vertices, unsigned long long* n_cycles, unsigned* dev_flags, cudaError_t* err);

// Heavy-hitter summaries of the cardinality pass (kma_hll.cu): the windows at every
// 2^kMgSampleShift-th arena position, split by the top kMgBucketBits bits of the key hash into
// kMgBuckets sub-streams, one Misra-Gries summary of kMgCounters counters per sub-stream and CTA.
constexpr unsigned kMgSampleShift = 6;
constexpr unsigned kMgBucketBits = 5;
constexpr unsigned kMgBuckets = 1u << kMgBucketBits;
constexpr unsigned kMgCounters = 32;

struct MgEntry {
  unsigned long long lo, hi, count;
};

// Where the CTAs leave their summaries: entry [cta][bucket][counter] (lo, hi, count; count 0
// = unused), items[bucket] = sampled windows of that bucket; and the merged summaries, at most
// kMgCounters entries a bucket. items, table, total and n_merged start at zero. lo == nullptr:
// no summaries.
struct MgOut {
  unsigned long long* lo;
  unsigned long long* hi;
  unsigned* count;
  unsigned long long* items;  // [kMgBuckets]
  unsigned* table;            // [kMgBuckets][mg_table_slots(grid)]
  unsigned long long* total;  // one per entry: the key's count over all CTAs, at its first entry
  MgEntry* merged;            // [kMgBuckets][kMgCounters]
  unsigned* n_merged;         // [kMgBuckets]
};

// Lets `fn` launch with up to the device's opt-in shared memory per block (less its static
// shared memory) and checks that `need` dynamic bytes fit. The limit is a property of the
// kernel, shared by every host thread: handles counting on several threads launch the same
// kernel with different sizes, and a limit set to one launch's own size could be lowered by
// another thread between that thread's set and its launch. So it is only ever set to the
// maximum (once per kernel and device).
cudaError_t allow_dynamic_smem(const void* fn, size_t need);

// HyperLogLog registers (2^p, 32-bit each) of the windows [w.q0, w.q1), and the heavy-hitter
// summaries of `grid` CTAs (kma_hll.cu); hll_grid gives the number of resident CTAs.
unsigned hll_grid(unsigned p, unsigned k, int num_sms);
cudaError_t launch_hll(const PartWindows& w, unsigned k, unsigned canonical, unsigned n_parts, unsigned part,
                       unsigned p, unsigned* regs, DevStatus* st, const MgOut& mg, unsigned grid,
                       cudaStream_t stream);
unsigned mg_table_slots(unsigned grid);
cudaError_t launch_mg_merge(const MgOut& mg, unsigned grid, cudaStream_t stream);

struct LaunchShape {
  int block_threads;
  int windows_per_thread;
  int grid;
};

// Launchers (kma_kernels.cu). All enqueue on `stream`.
cudaError_t launch_pack(const PackBatch& b, cudaStream_t stream, int num_sms);
cudaError_t launch_pass(const PassBatch& b, const LaunchShape& shape, bool warp_aggregate,
                        cudaStream_t stream);
cudaError_t launch_classify(const ClassBatch& b, cudaStream_t stream, int num_sms);
cudaError_t launch_table_init(Slot* table, unsigned long long slots, cudaStream_t stream);
cudaError_t launch_query(const Slot* table, unsigned long long slots, unsigned int parts,
                         unsigned int k,
                         unsigned int canonical, unsigned int min_depth, unsigned int min_ext,
                         const unsigned long long* keys, unsigned long long n,
                         unsigned int* counts, unsigned int* ext, unsigned char* codes,
                         DevStatus* status, cudaStream_t stream);
int pass_max_ctas_per_sm(int block_threads, int windows_per_thread, bool warp_aggregate);

}  // namespace kma
