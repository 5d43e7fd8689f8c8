// FASTQ text -> reads (the input side of the k-mer analysis stage, Section 2 item 1: the
// stage reads sequencing reads with per-base qualities). A FASTQ record is four lines:
// "@name", the bases, "+" (optionally followed by the name again) and the qualities, one
// character per base. Quality lines may begin with '@' or '+', so records are found by line
// number (line 4r starts record r), never by scanning for markers.
//
// Device steps (all on the caller's stream):
//   1. newlines per 64 KiB chunk of text, masks      fastq_count_kernel
//   2. exclusive scan of the chunk counts           scan kernels (device-wide, u64)
//   3. newline positions, in order                  fastq_lines_kernel
//   4. per record: check the '@' and '+' lines, base and quality line lengths equal
//                                                   fastq_record_kernel
//   5. exclusive scan of the base counts -> offsets scan kernels
//   6. bases and qualities copied out, 8 lanes a line
//                                                   fastq_copy_kernel
// A line may end in "\r\n"; the '\r' is not part of it. A final line without '\n' counts.
#include "kma_device.cuh"

namespace kma {

constexpr int kFqThreads = 1024;
constexpr int kFqBytesPerThread = 16;
constexpr int kFqPieces = 4;  // 16-byte pieces per thread; with one the two passes took 69 and 75 instead of 50 and 26 us
constexpr u64 kFqChunk = (u64)kFqThreads * kFqBytesPerThread * kFqPieces;  // 64 KiB of text per CTA

// ------------------------------------------------------------------ device-wide scan (u64)

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr u64 kScanBlock = (u64)kScanThreads * kScanItems;

// Exclusive scan of one block's kScanBlock items in place; the block's total to sums[blk].
__global__ void __launch_bounds__(kScanThreads) scan_block_kernel(u64* data, u64 n, u64* sums) {
  __shared__ u64 warp_tot[kScanThreads / 32];
  const u64 base = (u64)blockIdx.x * kScanBlock + (u64)threadIdx.x * kScanItems;
  u64 v[kScanItems];
  u64 local = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    v[j] = base + j < n ? data[base + j] : 0;
    local += v[j];
  }
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u64 incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (unsigned)o) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const u64 w = lane < kScanThreads / 32 ? warp_tot[lane] : 0;
    u64 wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= (unsigned)o) wi += t;
    }
    if (lane < kScanThreads / 32) warp_tot[lane] = wi - w;  // exclusive warp offsets
    if (lane == kScanThreads / 32 - 1 && sums) sums[blockIdx.x] = wi;
  }
  __syncthreads();
  u64 run = warp_tot[warp] + incl - local;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    if (base + j < n) data[base + j] = run;
    run += v[j];
  }
}

__global__ void scan_add_kernel(u64* data, u64 n, const u64* block_offsets) {
  const u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) data[i] += block_offsets[i / kScanBlock];
}

// Exclusive scan of data[0, n) in place; `tmp` holds scan_scratch_items(n) u64.
u64 scan_scratch_items(u64 n) {
  u64 total = 0;
  while (n > kScanBlock) {
    n = (n + kScanBlock - 1) / kScanBlock;
    total += n;
  }
  return total + 1;
}

cudaError_t scan_exclusive(u64* data, u64 n, u64* tmp, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const u64 blocks = (n + kScanBlock - 1) / kScanBlock;
  if (blocks == 1) {
    scan_block_kernel<<<1, kScanThreads, 0, stream>>>(data, n, nullptr);
    return cudaGetLastError();
  }
  u64* sums = tmp;
  scan_block_kernel<<<(unsigned)blocks, kScanThreads, 0, stream>>>(data, n, sums);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if ((e = scan_exclusive(sums, blocks, tmp + blocks, stream)) != cudaSuccess) return e;
  scan_add_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(data, n, sums);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ FASTQ kernels

// The 16 text bytes from position i on (i a multiple of 16 from the text's first aligned address:
// `head` bytes before it belong to the same 16 bytes), with a bit per byte: bit j of the result is
// set if byte i + j is a newline, or the text's last byte and none (the end of an unterminated
// line). Bytes outside [0, n) count as none. Bound by the text's one read; a byte load per
// thread and byte took 13 times as many requests.
__device__ __forceinline__ unsigned newline_mask(const unsigned char* text, u64 n, long long i) {
  if (i >= (long long)n) return 0;
  uint4 v;
  if (i >= 0 && i + 16 <= (long long)n) {
    v = __ldg(reinterpret_cast<const uint4*>(text + i));
  } else {  // the first or the last piece: byte by byte
    unsigned w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (i + j >= 0 && i + j < (long long)n) w[j >> 2] |= (unsigned)text[i + j] << (8 * (j & 3));
    v = make_uint4(w[0], w[1], w[2], w[3]);
  }
  // one bit per byte: compare, keep bit 0 of each byte, gather the four of a word
  const unsigned nl = 0x0A0A0A0Au;
  const unsigned m0 = ((__vcmpeq4(v.x, nl) & 0x01010101u) * 0x01020408u) >> 24;
  const unsigned m1 = ((__vcmpeq4(v.y, nl) & 0x01010101u) * 0x01020408u) >> 24;
  const unsigned m2 = ((__vcmpeq4(v.z, nl) & 0x01010101u) * 0x01020408u) >> 24;
  const unsigned m3 = ((__vcmpeq4(v.w, nl) & 0x01010101u) * 0x01020408u) >> 24;
  unsigned m = (m0 & 15u) | ((m1 & 15u) << 4) | ((m2 & 15u) << 8) | ((m3 & 15u) << 12);
  const long long last = (long long)n - 1 - i;
  if (last < 16) m |= 1u << last;  // the last byte ends a line either way
  return m;
}

// Newlines in each chunk (plus one for a final line that does not end in '\n'), and their
// masks, an eighth of the text, for the next pass (reading the text again took it 104 us for 100
// Mbases).
__global__ void __launch_bounds__(kFqThreads) fastq_count_kernel(const unsigned char* text, u64 n, unsigned head,
                                                                 unsigned short* masks, u64* chunk_counts) {
  __shared__ unsigned warp_cnt[kFqThreads / 32];
  const u64 c = blockIdx.x;
  unsigned cnt = 0, m[kFqPieces];
#pragma unroll
  for (int j = 0; j < kFqPieces; ++j)
    m[j] = newline_mask(text, n, (long long)(c * kFqChunk + (u64)(j * kFqThreads + threadIdx.x) * kFqBytesPerThread) - head);
#pragma unroll
  for (int j = 0; j < kFqPieces; ++j) {
    masks[(c * kFqPieces + j) * kFqThreads + threadIdx.x] = (unsigned short)m[j];
    cnt += __popc(m[j]);
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if ((threadIdx.x & 31) == 0) warp_cnt[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x < 32) {
    const unsigned t = __reduce_add_sync(0xffffffffu, warp_cnt[threadIdx.x]);
    if (threadIdx.x == 0) chunk_counts[c] = t;
  }
}

// Line ends (position of each '\n', or n for an unterminated last line), in text order.
__global__ void __launch_bounds__(kFqThreads) fastq_lines_kernel(const unsigned char* text, u64 n, unsigned head,
                                                                 const unsigned short* masks, const u64* chunk_offsets,
                                                                 u64* line_end) {
  __shared__ unsigned warp_off[kFqThreads / 32];
  const u64 c = blockIdx.x;
  // four pieces in a row
  static_assert(kFqPieces == 4 && kFqBytesPerThread == 16, "a thread's masks are one 64-bit word");
  const long long i = (long long)(c * kFqChunk + (u64)threadIdx.x * (kFqBytesPerThread * kFqPieces)) - head;
  u64 m = reinterpret_cast<const u64*>(masks)[c * kFqThreads + threadIdx.x];
  const unsigned cnt = __popcll(m);
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (unsigned)o) incl += t;
  }
  if (lane == 31) warp_off[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const unsigned t = warp_off[lane];
    unsigned run = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned x = __shfl_up_sync(0xffffffffu, run, o);
      if (lane >= (unsigned)o) run += x;
    }
    warp_off[lane] = run - t;
  }
  __syncthreads();
  u64 out = chunk_offsets[c] + warp_off[warp] + incl - cnt;
  for (; m; m &= m - 1) {
    const u64 at = (u64)(i + __ffsll((long long)m) - 1);
    line_end[out++] = at == n - 1 && text[at] != '\n' ? n : at;  // unterminated last line
  }
}

// Line l occupies [start, end) with the '\r' of a "\r\n" ending removed.
__device__ __forceinline__ void line_span(const unsigned char* text, const u64* line_end, u64 l, u64& s, u64& e) {
  s = l ? line_end[l - 1] + 1 : 0;
  e = line_end[l];
  if (e > s && text[e - 1] == '\r') --e;
}

// Record r: '@' line, bases, '+' line, qualities; bases per record to seq_len[r]. The first
// malformed record's index goes to *bad (atomicMin).
__global__ void fastq_record_kernel(const unsigned char* text, const u64* line_end, u64 n_reads, u64* seq_len,
                                    unsigned long long* bad) {
  const u64 r = (u64)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_reads) return;
  u64 s0, e0, s1, e1, s2, e2, s3, e3;
  line_span(text, line_end, 4 * r, s0, e0);
  line_span(text, line_end, 4 * r + 1, s1, e1);
  line_span(text, line_end, 4 * r + 2, s2, e2);
  line_span(text, line_end, 4 * r + 3, s3, e3);
  const bool ok = e0 > s0 && text[s0] == '@' && e2 > s2 && text[s2] == '+' && e1 - s1 == e3 - s3;
  seq_len[r] = ok ? e1 - s1 : 0;
  if (!ok) atomicMin(bad, (unsigned long long)r);
}

// Eight text bytes starting at any address, from the one or two aligned words that hold them.
__device__ __forceinline__ u64 load8(const unsigned char* p) {
  const u64 a = reinterpret_cast<u64>(p);
  const u64* w = reinterpret_cast<const u64*>(a & ~7ull);
  const unsigned s = (unsigned)(a & 7) * 8;
  u64 v = __ldg(w) >> s;
  if (s) v |= __ldg(w + 1) << (64 - s);
  return v;
}

// `len` bytes from src to dst by kLineLanes lanes: bytes up to an 8-byte boundary of dst,
// then a word per lane, then the bytes left. Reads and writes nothing outside the ranges but the
// rest of the aligned words that hold source bytes.
constexpr unsigned kLineLanes = 8;
__device__ __forceinline__ void copy_line(const unsigned char* src, unsigned char* dst, u64 len, unsigned lane) {
  u64 head = (8 - (reinterpret_cast<u64>(dst) & 7)) & 7;
  if (head > len) head = len;
  if (lane < head) dst[lane] = src[lane];
  const u64 words = (len - head) / 8;
  for (u64 w = lane; w < words; w += kLineLanes) *reinterpret_cast<u64*>(dst + head + 8 * w) = load8(src + head + 8 * w);
  const u64 done = head + 8 * words;
  if (lane < len - done) dst[done + lane] = src[done + lane];
}

// A quarter of a warp per line, bases or qualities, to its place in the output, eight bytes a lane:
// a byte per lane took eight times the requests on both sides, and with half a warp per line 41 %
// of the lanes had nothing to do for lines of 150 bytes.
__global__ void fastq_copy_kernel(const unsigned char* text, const u64* line_end, u64 n_reads, const u64* offsets,
                                  unsigned char* seq, unsigned char* qual) {
  const u64 line = ((u64)blockIdx.x * blockDim.x + threadIdx.x) / kLineLanes, r = line / 2;
  const unsigned lane = threadIdx.x % kLineLanes, which = (unsigned)line & 1;
  if (r >= n_reads) return;
  const u64 o = offsets[r], len = offsets[r + 1] - o;
  const u64 l = 4 * r + 1 + 2 * which;  // the bases' line, or the qualities'
  copy_line(text + line_end[l - 1] + 1, (which ? qual : seq) + o, len, lane);
}

// ------------------------------------------------------------------ launchers

// Chunks begin at a 16-byte boundary: `head` bytes before the text belong to the first one.
static unsigned fastq_head(const unsigned char* text) { return (unsigned)(reinterpret_cast<uintptr_t>(text) & 15); }

u64 fastq_masks(u64 n_bytes) { return fastq_chunks(n_bytes) * (kFqThreads * kFqPieces); }

u64 fastq_chunks(u64 n_bytes) { return n_bytes ? (n_bytes + 15 + kFqChunk - 1) / kFqChunk : 0; }

cudaError_t launch_fastq_count(const unsigned char* text, u64 n, unsigned short* masks, u64* chunk_counts,
                               cudaStream_t stream) {
  const u64 chunks = fastq_chunks(n);
  if (!chunks) return cudaSuccess;
  fastq_count_kernel<<<(unsigned)chunks, kFqThreads, 0, stream>>>(text, n, fastq_head(text), masks, chunk_counts);
  return cudaGetLastError();
}

cudaError_t launch_fastq_lines(const unsigned char* text, u64 n, const unsigned short* masks, const u64* chunk_offsets,
                               u64* line_end, cudaStream_t stream) {
  const u64 chunks = fastq_chunks(n);
  if (!chunks) return cudaSuccess;
  fastq_lines_kernel<<<(unsigned)chunks, kFqThreads, 0, stream>>>(text, n, fastq_head(text), masks, chunk_offsets, line_end);
  return cudaGetLastError();
}

cudaError_t launch_fastq_records(const unsigned char* text, const u64* line_end, u64 n_reads, u64* seq_len,
                                 unsigned long long* bad, cudaStream_t stream) {
  if (!n_reads) return cudaSuccess;
  fastq_record_kernel<<<(unsigned)((n_reads + 255) / 256), 256, 0, stream>>>(text, line_end, n_reads, seq_len, bad);
  return cudaGetLastError();
}

cudaError_t launch_fastq_copy(const unsigned char* text, const u64* line_end, u64 n_reads, const u64* offsets,
                              unsigned char* seq, unsigned char* qual, cudaStream_t stream) {
  if (!n_reads) return cudaSuccess;
  const u64 threads = n_reads * 2 * kLineLanes;
  fastq_copy_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, stream>>>(text, line_end, n_reads, offsets, seq,
                                                                          qual);
  return cudaGetLastError();
}

}  // namespace kma
