// Device helpers shared by the library's kernels (not part of the C ABI): hashing, 2-bit
// k-mer words, window extraction from the packed-read arena, and the hash-table operations.
#pragma once
#include "kma_internal.cuh"

namespace kma {

typedef unsigned long long u64;
typedef unsigned __int128 u128;

// ------------------------------------------------------------------ hashing

// 64-bit finaliser of MurmurHash3 (Appleby).
__device__ __forceinline__ u64 fmix64(u64 x) {
  x ^= x >> 33;
  x *= 0xff51afd7ed558ccdull;
  x ^= x >> 33;
  x *= 0xc4ceb9fe1a85ec53ull;
  x ^= x >> 33;
  return x;
}

// 64-bit hash of a 128-bit key: the high word is spread by an odd multiplier (plus a
// constant), folded into the low word, and the result mixed by one finaliser.
__device__ __forceinline__ u64 key_hash(u64 lo, u64 hi) {
  return fmix64(lo ^ (hi * 0x9e3779b97f4a7c15ull + 0x632be59bd9b4e019ull));
}

// Everything derived from the 64-bit key hash h uses cheap 32-bit slices of h and of two
// more products, instead of further 64-bit mixes:
//   on-chip partition   high 32 bits of h                  (part_of)
//   Bloom word          low 32 bits of h                   (bloom_index; < 2^32 words)
//   table slot          high 32 bits of h, the part behind the partition (table_index; < 2^32 slots per part)
//   Bloom bit positions 6-bit fields from the top of (h ^ h >> 32) * c   (bloom_mask)
// The bit positions must not depend on the low bits of h alone: those also pick the word, and
// keys sharing a word would then share most of their bits (a much higher false-positive rate).
// Slot of a key in its partition (of `parts`): in the order of the hash, so that the keys of one
// sub-bucket (partitioned mode counts in hash order) go to neighbouring slots and every line of
// the table is brought in and written back once.
__device__ __forceinline__ u64 table_index(u64 h, u64 slots, unsigned parts = 1) {
  return __umulhi((unsigned)(h >> 32) * parts, (unsigned)slots);
}
__device__ __forceinline__ u64 bloom_index(u64 h, u64 words) {
  return __umulhi((unsigned)h, (unsigned)words);
}
// Owner GPU of a k-mer (multi-GPU owner-computes), independent of the bits above.
__device__ __forceinline__ unsigned owner_of(u64 h, unsigned n_parts) {
  return __umulhi((unsigned)(fmix64(h ^ 0x9fb21c651e98df25ull) >> 32), n_parts);
}

// On-chip partition (partitioned mode) of a k-mer with hash h, 0 .. P-1.
__device__ __forceinline__ unsigned part_of(u64 h, unsigned P) {
  return __umulhi((unsigned)(h >> 32), P);
}

// Mask with bit x set for each 6-bit field x taken from the top of g (field i at bits
// 58 - 6i .. 63 - 6i, i < nbits <= kMaxHashBits), built in 32-bit halves. The loop is unrolled
// so that every field is extracted with constant shifts.
constexpr unsigned kMaxHashBits = 10;
__device__ __forceinline__ u64 mask_from_fields(u64 g, unsigned nbits) {
  const unsigned gh = (unsigned)(g >> 32), gl = (unsigned)g;
  unsigned lo = 0, hi = 0;
#pragma unroll
  for (int i = 0; i < (int)kMaxHashBits; ++i) {
    if (i < (int)nbits) {
      const int off = 58 - 6 * i;
      const unsigned x = off >= 32 ? (gh >> (off - 32)) & 63u
                                   : (off + 6 <= 32 ? (gl >> off) & 63u : __funnelshift_r(gl, gh, off) & 63u);
      const unsigned bit = 1u << (x & 31u);
      if (x & 32u) hi |= bit; else lo |= bit;
    }
  }
  return ((u64)hi << 32) | lo;
}

__device__ __forceinline__ u64 bloom_mask(u64 h, unsigned nbits) {
  return mask_from_fields((h ^ (h >> 32)) * 0xd6e8feb86659fd93ull, nbits);
}

// ------------------------------------------------------------------ bulk copies (TMA)

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// 1-D TMA bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16),
// completion signalled on the mbarrier as transaction bytes.
__device__ __forceinline__ void tma_load_1d(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Orders this thread's earlier generic-proxy accesses to shared memory before later bulk
// copies into it (a buffer read by the CTA, then refilled by a copy).
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Test for the phase; while it is incomplete the thread may be suspended, and it resumes when
// the phase completes or after at most kWaitHintNs nanoseconds. A waiting warp therefore
// sleeps instead of spinning (no issue slots spent on polling).
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned phase) {
  unsigned done;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(done) : "r"(bar), "r"(phase), "n"(kWaitHintNs) : "memory");
  return done != 0;
}

// Bounded wait for the mbarrier phase: returns false (and the caller raises a status flag)
// if the copies have not completed after `limit` polls (at most limit * kWaitHintNs ns).
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned phase, unsigned limit) {
  for (unsigned it = 0; it < limit; ++it)
    if (mbar_try_wait(bar, phase)) return true;
  return false;
}

// After a wait that gave up: before the CTA may exit, the bulk copies already issued into its
// shared memory must land. Waits up to 8 times the first limit (still bounded; copies that
// have not landed by then are reported by the flag the caller already raised).
__device__ __forceinline__ bool mbar_drain(unsigned bar, unsigned phase, unsigned limit) {
  for (unsigned r = 0; r < 8; ++r)
    if (mbar_wait_bounded(bar, phase, limit)) return true;
  return false;
}

// ------------------------------------------------------------------ 2-bit words

// Reverse the order of the 32 two-bit groups of x.
__device__ __forceinline__ u64 rev2(u64 x) {
  x = __brevll(x);
  return ((x >> 1) & 0x5555555555555555ull) | ((x & 0x5555555555555555ull) << 1);
}

// Reverse complement of a k-mer held in the low 2k bits of (hi:lo).
__device__ __forceinline__ void revcomp(u64 lo, u64 hi, unsigned k, u64& rlo, u64& rhi) {
  u128 r = ((u128)rev2(lo) << 64) | (u128)rev2(hi);
  r = ~r;
  r >>= (128 - 2 * k);
  rlo = (u64)r;
  rhi = (u64)(r >> 64);
}

__device__ __forceinline__ unsigned code_at(const u64* codes, u64 p) {
  return (unsigned)(codes[p >> 5] >> (62 - 2 * (p & 31))) & 3u;
}

__device__ __forceinline__ unsigned bit_at(const u64* bits, u64 p) {
  return (unsigned)(bits[p >> 6] >> (63 - (p & 63))) & 1u;
}

struct Window {
  u64 lo, hi;        // canonical key
  unsigned lb, rb;   // extension bases in the key's orientation
  bool lu, ru;       // usable (exists, A/C/G/T, Phred >= threshold)
};

// (a:b) << s, top 64 bits, for 0 <= s < 64.
__device__ __forceinline__ u64 fshl(u64 a, u64 b, unsigned s) { return s ? (a << s) | (b >> (64 - s)) : a; }
// (b:a) >> s, low 64 bits, for 0 <= s < 64.
__device__ __forceinline__ u64 fshr(u64 a, u64 b, unsigned s) { return s ? (a >> s) | (b << (64 - s)) : a; }

// Window starting at arena position q: returns false if any of its k positions is invalid.
// The forward k-mer is read MSB-first from `codes`, its reverse complement LSB-first from
// `rcodes` (both one funnel shift per 64-bit word), the canonical key is the smaller.
__device__ __forceinline__ bool load_window(const u64* codes, const u64* rcodes, const u64* inv,
                                            const u64* hq, unsigned k, unsigned canonical, u64 q,
                                            Window& w) {
  const u64 v = q >> 6;
  const unsigned t = (unsigned)(q & 63);
  if (fshl(inv[v], inv[v + 1], t) >> (64 - k)) return false;

  const u64 wi = q >> 5;
  const unsigned s = 2 * (unsigned)(q & 31);
  const u64 a = codes[wi], b = codes[wi + 1];
  const u64 top = fshl(a, b, s);  // first 32 bases of the window, MSB-first
  u64 flo, fhi, rlo, rhi;
  const u64 r0 = rcodes[wi], r1 = rcodes[wi + 1];
  const u64 bot = fshr(r0, r1, s);  // reverse complement, low 64 bits
  if (k > 32) {
    const u64 c = codes[wi + 2];
    const u64 mid = fshl(b, c, s);
    const unsigned sh = 128 - 2 * k;  // 2 .. 62
    flo = (mid >> sh) | (top << (64 - sh));
    fhi = top >> sh;
    const u64 r2 = rcodes[wi + 2];
    rlo = bot;
    rhi = fshr(r1, r2, s) & ((1ull << (2 * k - 64)) - 1);
  } else {
    flo = top >> (64 - 2 * k);
    fhi = 0;
    rlo = k == 32 ? bot : bot & ((1ull << (2 * k)) - 1);
    rhi = 0;
  }

  // Extension bases: position q-1 (before) and q+k (after).
  const bool bu = q > 0 && bit_at(hq, q - 1);
  const bool au = bit_at(hq, q + k) != 0;
  const unsigned bb = q > 0 ? code_at(codes, q - 1) : 0u;
  const unsigned ab = code_at(codes, q + k);

  const bool forward = !canonical || (fhi < rhi) || (fhi == rhi && flo <= rlo);
  if (forward) {
    w.lo = flo; w.hi = fhi;
    w.lb = bb; w.lu = bu;
    w.rb = ab; w.ru = au;
  } else {
    w.lo = rlo; w.hi = rhi;
    w.lb = 3u - ab; w.lu = au;
    w.rb = 3u - bb; w.ru = bu;
  }
  return true;
}

__device__ __forceinline__ bool load_window(const PassDesc& D, u64 q, Window& w) {
  return load_window(D.codes, D.rcodes, D.inv, D.hq, D.k, D.canonical, q, w);
}

// Eight consecutive windows starting at q (a multiple of 8), in 32-bit words. The base streams
// are aligned once per run (one funnel shift per word): fw holds the forward stream so that
// window 0 ends with fw[2 KW - 1] and the following bases are in fw[2 KW], rv the reverse
// complement stream from window 0 on. Window j is then 2 KW funnel shifts by the constant 2 j of
// each, right-aligned as it is needed (rolling the two 128-bit numbers base by base took about
// twice the instructions). Valid windows are a range of j: invalid positions before the first
// window's eighth one cut it from below, those behind the first window's end from above.
// Extension outcomes of all eight windows are put together in bytes beforehand, for either
// orientation.
template <int KW>
struct WindowRun {
  unsigned fw[2 * KW + 1], rv[2 * KW + 1];
  unsigned m_top, m_next;     // masks of the words that hold bits 2k and above
  unsigned valid;             // bit j: window j has no invalid position
  unsigned ext[2][2];         // [forward?][j & 1]: byte j / 2 = outcome bits << 2 (left, right << 3)

  __device__ __forceinline__ static unsigned spread2(unsigned x) {  // 8 pairs -> 8 nibbles
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    return (x | (x << 2)) & 0x33333333u;
  }
  __device__ __forceinline__ static unsigned spread1(unsigned x) {  // 8 bits -> 8 nibbles
    x = (x | (x << 12)) & 0x000F000Fu;
    x = (x | (x << 6)) & 0x03030303u;
    return (x | (x << 3)) & 0x11111111u;
  }
  // Outcome nibbles (0-3 base, 4 none) of eight positions: codes in the top 16 bits of c and
  // high-quality flags in the top 8 bits of u, first position first; comp: of the complements.
  __device__ __forceinline__ static unsigned outcomes(unsigned c, unsigned u, unsigned& comp) {
    c = __brev(c) & 0xFFFFu;  // first position in the low pair, its bits swapped
    c = ((c >> 1) & 0x5555u) | ((c & 0x5555u) << 1);
    const unsigned on = spread1(__brev(u) & 0xFFu), on3 = on * 3u;
    const unsigned n = (spread2(c) & on3) | ((on ^ 0x11111111u) << 2);
    comp = n ^ on3;
    return n;
  }

  // q counts from the first position of the words given (the arena's or a staged part of it),
  // `first`: window q starts the arena. With outcomes = false only the keys are wanted.
  __device__ __forceinline__ void init(const u64* codes, const u64* rcodes, const u64* inv, const u64* hq, unsigned k,
                                       u64 q, bool first, bool with_outcomes) {
    const unsigned* c32 = reinterpret_cast<const unsigned*>(codes);   // word w of 16 positions: c32[w ^ 1]
    const unsigned* r32 = reinterpret_cast<const unsigned*>(rcodes);  // word w of 16 positions: r32[w]
    const unsigned* h32 = reinterpret_cast<const unsigned*>(hq);      // word w of 32 positions: h32[w ^ 1]
    // forward: the 16 * 2 KW positions that end where window 0 ends, and the 16 behind them
    // (positions before the arena are masked off below)
    const u64 e = q + k;
    const long long ie = (long long)(e >> 4);
    const unsigned se = 2 * (unsigned)(e & 15);
    unsigned prev = 0;
#pragma unroll
    for (int m = 0; m <= 2 * KW + 1; ++m) {
      const long long w = ie - 2 * KW + m;
      const unsigned x = c32[(u64)(w > 0 ? w : 0) ^ 1];
      if (m > 0) fw[m - 1] = __funnelshift_l(x, prev, se);
      prev = x;
    }
    const u64 iq = q >> 4;
    const unsigned sq = 2 * (unsigned)(q & 15);
    prev = r32[iq];
#pragma unroll
    for (int m = 0; m <= 2 * KW; ++m) {
      const unsigned x = r32[iq + m + 1];
      rv[m] = __funnelshift_r(prev, x, sq);
      prev = x;
    }
    const unsigned over = 64u * KW - 2u * k;  // bits above the key: 0 .. 62
    m_top = over >= 32 ? 0u : 0xFFFFFFFFu >> over;
    m_next = over >= 32 ? 0xFFFFFFFFu >> (over - 32) : 0xFFFFFFFFu;
    // validity
    const u64 v = q >> 6;
    const unsigned t = (unsigned)(q & 63);
    const u64 i0 = inv[v], i1 = inv[v + 1], i2 = inv[v + 2];
    const u64 b0 = fshl(i0, i1, t), b1 = fshl(i1, i2, t);  // invalid bits from q, first in the top bit
    if (k >= 8) {
      const unsigned low = (unsigned)(b0 >> 57);                             // positions 0 .. 6
      const unsigned high = (unsigned)(((b0 << k) | (b1 >> (64 - k))) >> 57);  // positions k .. k + 6
      const unsigned from = low ? 8u - (unsigned)__ffs(low) : 0u;            // behind the last of the former
      const unsigned upto = high ? (unsigned)__clz(high) - 25u : 7u;         // the first of the latter ends it
      const bool all_bad = k > 7 && ((b0 << 7) >> (71 - k)) != 0;            // positions 7 .. k - 1
      valid = all_bad ? 0u : (0xFFu << from) & (0xFFu >> (7 - upto));
    } else {
      valid = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) valid |= (((b0 << j) >> (64 - k)) == 0 ? 1u : 0u) << j;
    }
    if (with_outcomes) {
      // left: positions q - 1 .. q + 6 (none before the arena), right: e .. e + 7
      unsigned lc = 0, lu = 0;
      if (!first) {
        const u64 p = q - 1;
        lc = __funnelshift_l(c32[((p >> 4) + 1) ^ 1], c32[(p >> 4) ^ 1], 2 * (unsigned)(p & 15));
        lu = __funnelshift_l(h32[((p >> 5) + 1) ^ 1], h32[(p >> 5) ^ 1], (unsigned)(p & 31));
      } else {
        lc = c32[1] >> 2;
        lu = h32[1] >> 1;
      }
      const unsigned ru = __funnelshift_l(h32[((e >> 5) + 1) ^ 1], h32[(e >> 5) ^ 1], (unsigned)(e & 31));
      unsigned lcomp, rcomp;
      const unsigned l = outcomes(lc, lu, lcomp), r = outcomes(fw[2 * KW], ru, rcomp);
      constexpr unsigned kEven = 0x07070707u;
      ext[1][0] = ((l & kEven) << 2) | ((r & kEven) << 5);
      ext[1][1] = (((l >> 4) & kEven) << 2) | (((r >> 4) & kEven) << 5);
      ext[0][0] = ((rcomp & kEven) << 2) | ((lcomp & kEven) << 5);
      ext[0][1] = (((rcomp >> 4) & kEven) << 2) | (((lcomp >> 4) & kEven) << 5);
    }
  }

  // Canonical key of window j (a constant when unrolled); returns whether it is read forward.
  __device__ __forceinline__ bool key(int j, unsigned canonical, u64& lo, u64& hi) const {
    unsigned f[2 * KW], r[2 * KW];  // least significant word first
#pragma unroll
    for (int m = 0; m < 2 * KW; ++m) {
      f[2 * KW - 1 - m] = __funnelshift_l(fw[m + 1], fw[m], 2 * j);
      r[m] = __funnelshift_r(rv[m], rv[m + 1], 2 * j);
    }
    f[2 * KW - 1] &= m_top;
    r[2 * KW - 1] &= m_top;
    f[2 * KW - 2] &= m_next;
    r[2 * KW - 2] &= m_next;
    const u64 f0 = ((u64)f[1] << 32) | f[0], r0 = ((u64)r[1] << 32) | r[0];
    if (KW == 1) {
      const bool forward = !canonical || f0 <= r0;
      lo = forward ? f0 : r0;
      hi = 0;
      return forward;
    }
    const u64 f1 = ((u64)f[2 * KW - 1] << 32) | f[2 * KW - 2], r1 = ((u64)r[2 * KW - 1] << 32) | r[2 * KW - 2];
    const bool forward = !canonical || f1 < r1 || (f1 == r1 && f0 <= r0);
    lo = forward ? f0 : r0;
    hi = forward ? f1 : r1;
    return forward;
  }

  // Outcome bits of window j in the top byte (<< 26), read forward or not.
  __device__ __forceinline__ unsigned info(int j, bool forward) const {
    const unsigned w = forward ? ext[1][j & 1] : ext[0][j & 1];
    return __byte_perm(w, 0u, 0x0444u | ((unsigned)(j >> 1) << 12));
  }
};

// ------------------------------------------------------------------ table

__device__ __forceinline__ void cas128(Slot* s, u64 cmp_lo, u64 cmp_hi, u64 new_lo, u64 new_hi,
                                       u64& old_lo, u64& old_hi) {
  asm volatile(
      "{\n\t"
      ".reg .b128 d, c, n;\n\t"
      "mov.b128 c, {%2, %3};\n\t"
      "mov.b128 n, {%4, %5};\n\t"
      "atom.global.cas.b128 d, [%6], c, n;\n\t"
      "mov.b128 {%0, %1}, d;\n\t"
      "}"
      : "=l"(old_lo), "=l"(old_hi)
      : "l"(cmp_lo), "l"(cmp_hi), "l"(new_lo), "l"(new_hi), "l"(s)
      : "memory");
}

// Lookup in a table no thread is modifying. nullptr if absent; sets `full` if the probe
// limit was reached without finding an empty slot.
__device__ __forceinline__ const Slot* find(const Slot* table, u64 slots, unsigned parts, u64 lo, u64 hi, u64 h,
                                            bool& full) {
  u64 idx = table_index(h, slots, parts);
  const u64 limit = slots < kMaxProbe ? slots : kMaxProbe;
  full = false;
  for (u64 n = 0; n < limit; ++n) {
    const Slot* s = table + idx;
    const ulonglong2 kv = __ldcg(reinterpret_cast<const ulonglong2*>(s));
    if (kv.x == lo && kv.y == hi) return s;
    if (kv.y == kEmpty) return nullptr;
    idx = (idx + 1 == slots) ? 0 : idx + 1;
  }
  full = true;
  return nullptr;
}

// Counter of the occurrence's left / right outcome.
__device__ __forceinline__ unsigned* left_counter(Slot* s, const Window& w) {
  return w.lu ? &s->ext[w.lb] : &s->none[0];
}
__device__ __forceinline__ unsigned* right_counter(Slot* s, const Window& w) {
  return w.ru ? &s->ext[4 + w.rb] : &s->none[1];
}

// One occurrence (inc of them) of the slot's key, with wrap detection: every counter is at
// most the key's count, so a wrap of either updated counter is the only way one can be lost
// (a total count above 2^32 is caught when the counters are summed).
__device__ __forceinline__ void add_occurrence(Slot* s, const Window& w, unsigned inc,
                                               DevStatus* st) {
  const unsigned a = atomicAdd(left_counter(s, w), inc);
  const unsigned b = atomicAdd(right_counter(s, w), inc);
  if (a > 0xFFFFFFFFu - inc || b > 0xFFFFFFFFu - inc) atomicOr(&st->flags, kFlagOverflow);
}

// Count update when no counter can reach 2^32 (the host bounds the occurrences a key can
// have before the next reset): reductions without a returned value, nothing to wait for.
__device__ __forceinline__ void red_add(unsigned* a, unsigned v) {
  asm volatile("red.global.add.u32 [%0], %1;" ::"l"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void add_occurrence_red(Slot* s, const Window& w) {
  red_add(left_counter(s, w), 1u);
  red_add(right_counter(s, w), 1u);
}

// Warp-aggregated variant: lanes in `act` adding to the same counter merge their updates.
__device__ __forceinline__ void add_occurrence_agg(unsigned act, Slot* s, const Window& w,
                                                   DevStatus* st) {
  const int lane = threadIdx.x & 31;
  unsigned* l = left_counter(s, w);
  unsigned* r = right_counter(s, w);
  const unsigned ml = __match_any_sync(act, reinterpret_cast<u64>(l));
  const unsigned mr = __match_any_sync(act, reinterpret_cast<u64>(r));
  bool wrap = false;
  if (lane == __ffs(ml) - 1) {
    const unsigned inc = __popc(ml);
    wrap |= atomicAdd(l, inc) > 0xFFFFFFFFu - inc;
  }
  if (lane == __ffs(mr) - 1) {
    const unsigned inc = __popc(mr);
    wrap |= atomicAdd(r, inc) > 0xFFFFFFFFu - inc;
  }
  if (wrap) atomicOr(&st->flags, kFlagOverflow);
}

// Count of a slot (sum of its left outcomes), flagged if it does not fit 32 bits.
__device__ __forceinline__ unsigned slot_count(unsigned none_l, uint4 el, DevStatus* st) {
  const u64 c = (u64)none_l + el.x + el.y + el.z + el.w;
  if (c > 0xFFFFFFFFull) {
    atomicOr(&st->flags, kFlagOverflow);
    return 0xFFFFFFFFu;
  }
  return (unsigned)c;
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Insert-if-absent continuing from a first probe whose slot (index idx) is already loaded.
__device__ __forceinline__ Slot* resolve_insert(Slot* table, u64 slots, u64 idx, ulonglong2 kv,
                                                u64 lo, u64 hi, bool& inserted) {
  const u64 limit = slots < kMaxProbe ? slots : kMaxProbe;
  inserted = false;
  for (u64 n = 0; n < limit; ++n) {
    Slot* s = table + idx;
    if (n) kv = __ldcg(reinterpret_cast<const ulonglong2*>(s));
    if (kv.x == lo && kv.y == hi) return s;
    if (kv.y == kEmpty || kv.x == kEmpty) {
      u64 olo, ohi;
      cas128(s, kEmpty, kEmpty, lo, hi, olo, ohi);
      if (olo == kEmpty && ohi == kEmpty) { inserted = true; return s; }
      if (olo == lo && ohi == hi) return s;
    }
    idx = (idx + 1 == slots) ? 0 : idx + 1;
  }
  return nullptr;
}

// Lookup (table not being modified) continuing from a loaded first probe.
__device__ __forceinline__ Slot* resolve_find(Slot* table, u64 slots, u64 idx, ulonglong2 kv,
                                              u64 lo, u64 hi, bool& full) {
  const u64 limit = slots < kMaxProbe ? slots : kMaxProbe;
  full = false;
  for (u64 n = 0; n < limit; ++n) {
    Slot* s = table + idx;
    if (n) kv = __ldcg(reinterpret_cast<const ulonglong2*>(s));
    if (kv.x == lo && kv.y == hi) return s;
    if (kv.y == kEmpty) return nullptr;
    idx = (idx + 1 == slots) ? 0 : idx + 1;
  }
  full = true;
  return nullptr;
}

__device__ __forceinline__ unsigned side_code(const unsigned* e, unsigned min_ext) {
  unsigned n = 0, b = 0;
#pragma unroll
  for (unsigned j = 0; j < 4; ++j)
    if (e[j] >= min_ext) { ++n; b = j; }
  return n == 0 ? 4u : (n >= 2 ? 5u : b);
}

}  // namespace kma
