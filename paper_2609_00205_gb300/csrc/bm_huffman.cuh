// Huffman stage (the lossless stage of the pipeline, Sec. III-B: outlier
// handling, histogram, codebook, encoding, concatenation of chunk codes).
//
// Codebook: code lengths of the two-queue Huffman construction (leaves sorted
// by (frequency, symbol); on equal weight a leaf goes before an internal
// node; internal nodes in creation order), canonical codes by (length,
// symbol), lengths above 32 bits avoided by re-running on max(1, f >> t).
// The GPU builds exactly that tree in parallel rounds: with X the sum of the
// two lightest remaining nodes, every remaining node of weight <= X is
// consumed, in merged order, before any node created from now on (new nodes
// weigh >= X and lose ties), so all those pairs are formed at once.
#pragma once

#include <stddef.h>

#include <cooperative_groups.h>

#include "bm_common.cuh"

namespace bm {

constexpr int kCbThreads = 1024;
constexpr int kLutBits = 14;
// Entries of the code table window the encoder keeps in shared memory (a
// window of the dictionary, 4 bytes an entry): kEncWinSmall in CTAs of eight
// warps, four per SM, when every present symbol lies within so many consecutive
// symbols; kEncWin in one CTA of kEncWarps warps per SM, beside the warps'
// staging words, when they lie within that.
constexpr int kEncWin = 49152;
constexpr int kEncWinSmall = 8192;
constexpr int kEncWarps = 32;
// The window's entry of a symbol: its code, left-justified, and its length in
// the low five bits.  Codes longer than kPackLen bits do not fit: a codebook
// with one (fields beyond about 10^8 symbols) takes the split table.
constexpr unsigned kPackLen = 27;
__host__ __device__ constexpr unsigned enc_entry(unsigned code, unsigned len) {
  return len >= 1 && len <= kPackLen ? (code << (32 - len)) | len : 0u;
}
// Every chunk is split into eight equal runs; the stream stores the bit
// offsets of runs 1..7 so that eight decoders can work on one chunk.
constexpr int kSplits = 8;

// Canonical-code tables shared by encoder and decoder.
struct CanonTables {
  unsigned first_code[kMaxLen + 2];
  unsigned first_pos[kMaxLen + 2];
  unsigned count[kMaxLen + 2];
  unsigned long long limit[kMaxLen + 2];  // (first_code + count) << (32 - L), left-justified
  unsigned n;                             // present symbols
  unsigned max_len;
};

struct DecodeTables {
  CanonTables ct;
  alignas(16) uint16_t canon[kMaxDict];  // symbols in canonical order
};

// ---------------------------------------------------------------------------
// Block-wide helpers (blockDim.x == kCbThreads)
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned block_excl_scan(unsigned v, unsigned* warp_tot, unsigned* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[wid] = x;
  __syncthreads();
  if (wid == 0) {
    unsigned t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    warp_tot[lane] = t;  // inclusive
  }
  __syncthreads();
  const unsigned before = (wid ? warp_tot[wid - 1] : 0u) + x - v;
  if (total && threadIdx.x == 0) *total = warp_tot[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before;
}

// Exclusive scan over the warps of a block of one count per warp (every lane
// of a warp passes the same value); returns the sum of the warps before this
// one to every lane, and the total in *total.  scan_tmp: 32 u32.
__device__ __forceinline__ unsigned warp_excl_scan_block(unsigned v, unsigned* scan_tmp, unsigned* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) scan_tmp[wid] = v;
  __syncthreads();
  if (wid == 0) {
    const unsigned c = lane < nw ? scan_tmp[lane] : 0u;
    unsigned x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane < nw) scan_tmp[lane] = x - c;
    if (lane == 31 && total) *total = x;
  }
  __syncthreads();
  const unsigned r = scan_tmp[wid];
  __syncthreads();
  return r;
}

// Per-warp running counts of a counting pass, stored by (digit, warp) with
// the warp index swizzled by the digit so that the lanes of a warp reading
// counts of different digits hit different banks.
__device__ __forceinline__ int wc_idx(unsigned d, int w) { return (int)(d * 32u + ((unsigned)w ^ (d & 31u))); }

// Stable LSD radix sort (8-bit digits) of n <= kMaxDict (key, payload) pairs
// by key, one block of kCbThreads threads.  Warp w owns the contiguous rows
// w*rows .. w*rows+rows-1 of 32 pairs, so (warp, row, lane) is index order.
// Each pass: a counting walk (every warp ranks its rows by digit with
// __match_any_sync, keeping a running count per (digit, warp)), one block
// scan over (digit, warp) for every group's start, and a scatter walk over
// the same rows in the same order that recomputes each pair's rank (so no
// per-row state is kept in registers and n is not limited by them).  As many
// passes as maxkey has bytes.  Input in (ka, sa); returns 0 when the sorted
// pairs are in (ka, sa), 1 when in (kb, sb).  wcnt: 256 * 32 u32 of scratch.
__device__ int radix_sort_pairs(unsigned* ka, uint16_t* sa, unsigned* kb, uint16_t* sb, unsigned* wcnt, int n,
                                unsigned maxkey, unsigned* scan_tmp) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int rows = (n + kCbThreads - 1) / kCbThreads;
  const int seg = rows * 32;
  int passes = 1;
  while (passes < 4 && (maxkey >> (8 * passes)) != 0u) ++passes;
  int cur = 0;
  for (int p = 0; p < passes; ++p) {
    const int shift = 8 * p;
    const unsigned* kin = cur ? kb : ka;
    const uint16_t* sin = cur ? sb : sa;
    unsigned* kout = cur ? ka : kb;
    uint16_t* sout = cur ? sa : sb;
    for (int i = threadIdx.x; i < 256 * 32; i += blockDim.x) wcnt[i] = 0u;
    __syncthreads();
    for (int r0 = 0; r0 < rows; r0 += 8) {  // counting walk, eight rows' keys loaded ahead
      unsigned kk[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int i = wid * seg + (r0 + t) * 32 + lane;
        kk[t] = (r0 + t < rows && i < n) ? kin[i] : 0u;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        if (r0 + t >= rows) break;
        const int i = wid * seg + (r0 + t) * 32 + lane;
        const bool ok = i < n;
        const unsigned d = (kk[t] >> shift) & 255u;
        const unsigned m = __match_any_sync(0xffffffffu, ok ? d : 256u + (unsigned)lane);
        if (ok && (m & ((1u << lane) - 1u)) == 0u) wcnt[wc_idx(d, wid)] += (unsigned)__popc(m);
        __syncwarp();
      }
    }
    __syncthreads();
    // exclusive scan in (digit, warp) order: thread t owns entries 8t .. 8t+7
    unsigned v[8], sum = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = threadIdx.x * 8 + j;
      v[j] = wcnt[wc_idx((unsigned)k >> 5, k & 31)];
      sum += v[j];
    }
    unsigned pre = block_excl_scan(sum, scan_tmp, nullptr);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = threadIdx.x * 8 + j;
      wcnt[wc_idx((unsigned)k >> 5, k & 31)] = pre;
      pre += v[j];
    }
    __syncthreads();
    for (int r0 = 0; r0 < rows; r0 += 8) {  // scatter walk, eight rows loaded ahead
      unsigned kk[8];
      uint16_t pp[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int i = wid * seg + (r0 + t) * 32 + lane;
        const bool ok = r0 + t < rows && i < n;
        kk[t] = ok ? kin[i] : 0u;
        pp[t] = ok ? sin[i] : (uint16_t)0;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        if (r0 + t >= rows) break;
        const int i = wid * seg + (r0 + t) * 32 + lane;
        const bool ok = i < n;
        const unsigned d = (kk[t] >> shift) & 255u;
        const unsigned m = __match_any_sync(0xffffffffu, ok ? d : 256u + (unsigned)lane);
        const unsigned lt = m & ((1u << lane) - 1u);
        const unsigned base = ok ? wcnt[wc_idx(d, wid)] : 0u;
        if (ok) {
          const unsigned dst = base + (unsigned)__popc(lt);
          kout[dst] = kk[t];
          sout[dst] = pp[t];
        }
        __syncwarp();
        if (ok && lt == 0u) wcnt[wc_idx(d, wid)] = base + (unsigned)__popc(m);
        __syncwarp();
      }
    }
    __syncthreads();
    cur ^= 1;
  }
  return cur;
}
// The same sort of at most 8 kCbThreads pairs, whose keys, payloads and ranks
// within (digit, warp) stay in registers between the counting and the scatter:
// one walk instead of two.
__device__ int radix_sort_pairs_small(unsigned* ka, uint16_t* sa, unsigned* kb, uint16_t* sb, unsigned* wcnt, int n,
                                      unsigned maxkey, unsigned* scan_tmp) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int rows = (n + kCbThreads - 1) / kCbThreads;  // at most 8
  const int base_i = wid * rows * 32 + lane;
  int passes = 1;
  while (passes < 4 && (maxkey >> (8 * passes)) != 0u) ++passes;
  int cur = 0;
  for (int p = 0; p < passes; ++p) {
    const int shift = 8 * p;
    const unsigned* kin = cur ? kb : ka;
    const uint16_t* sin = cur ? sb : sa;
    unsigned* kout = cur ? ka : kb;
    uint16_t* sout = cur ? sa : sb;
    unsigned kk[8], rk[8];
    uint16_t pp[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = base_i + 32 * t;
      const bool ok = t < rows && i < n;
      kk[t] = ok ? kin[i] : 0u;
      pp[t] = ok ? sin[i] : (uint16_t)0;
    }
    for (int i = threadIdx.x; i < 256 * 32; i += blockDim.x) wcnt[i] = 0u;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (t < rows) {
        const bool ok = base_i + 32 * t < n;
        const unsigned d = (kk[t] >> shift) & 255u;
        const unsigned m = __match_any_sync(0xffffffffu, ok ? d : 256u);
        const unsigned lt = m & ((1u << lane) - 1u);
        const unsigned before = ok ? wcnt[wc_idx(d, wid)] : 0u;
        __syncwarp();
        if (ok && lt == 0u) wcnt[wc_idx(d, wid)] = before + (unsigned)__popc(m);
        rk[t] = before + (unsigned)__popc(lt);
        __syncwarp();
      }
    }
    __syncthreads();
    // exclusive scan in (digit, warp) order: thread t owns entries 8t .. 8t+7
    unsigned v[8], sum = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = threadIdx.x * 8 + j;
      v[j] = wcnt[wc_idx((unsigned)k >> 5, k & 31)];
      sum += v[j];
    }
    unsigned pre = block_excl_scan(sum, scan_tmp, nullptr);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = threadIdx.x * 8 + j;
      wcnt[wc_idx((unsigned)k >> 5, k & 31)] = pre;
      pre += v[j];
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (t < rows && base_i + 32 * t < n) {
        const unsigned dst = wcnt[wc_idx((kk[t] >> shift) & 255u, wid)] + rk[t];
        kout[dst] = kk[t];
        sout[dst] = pp[t];
      }
    }
    __syncthreads();
    cur ^= 1;
  }
  return cur;
}

// upper_bound by the 32 lanes of a warp (all lanes call it with the same
// arguments and get the same result): each step probes the last element of 32
// equal segments and keeps the first segment whose last element exceeds v.
__device__ __forceinline__ int warp_upper_bound_u32(const unsigned* a, int lo, int hi, unsigned v) {
  const int lane = threadIdx.x & 31;
  while (hi - lo > 32) {
    const int step = (hi - lo + 31) >> 5;
    const int p = min(lo + (lane + 1) * step, hi) - 1;
    const unsigned m = __ballot_sync(0xffffffffu, a[p] > v);
    if (m == 0u) return hi;
    const int f = __ffs(m) - 1;
    const int nlo = lo + f * step;
    hi = min(nlo + step, hi);
    lo = nlo;
  }
  const unsigned m = __ballot_sync(0xffffffffu, lane < hi - lo && a[lo + lane] > v);
  return m ? lo + __ffs(m) - 1 : hi;
}
// upper_bound over the sorted a[lo, hi) by the 32 lanes of a warp, with
// samples smp[k] = a[64 k + 63] in shared memory for the blocks k < nfull (a
// last block shorter than 64 elements, if any, follows them unsampled): a
// 32-ary search of the samples finds the block that holds the bound, then one
// coalesced read of that block (the search's only global round trip).
__device__ __forceinline__ int warp_upper_bound_sampled(const unsigned* a, const unsigned* smp, int lo, int hi,
                                                        int nfull, unsigned v) {
  const int lane = threadIdx.x & 31;
  if (lo >= hi) return hi;
  int klo = lo >> 6, khi = nfull;  // the first block in [klo, khi) whose sample exceeds v, else khi
  while (khi - klo > 32) {
    const int step = (khi - klo + 31) / 32;
    const int p = min(klo + (lane + 1) * step, khi) - 1;
    const unsigned m = __ballot_sync(0xffffffffu, smp[p] > v);
    if (m == 0u) {
      klo = khi;
      break;
    }
    const int f = __ffs(m) - 1;
    const int nlo = klo + f * step;
    khi = min(nlo + step, khi);
    klo = nlo;
  }
  if (klo < khi) {
    const unsigned m = __ballot_sync(0xffffffffu, lane < khi - klo && smp[klo + lane] > v);
    klo = m ? klo + __ffs(m) - 1 : khi;
  }
  const int b0 = max(lo, klo << 6), b1 = min(hi, (klo << 6) + 64);
  if (b0 >= b1) return hi;
  const int i0 = b0 + lane, i1 = b0 + 32 + lane;
  const unsigned x0 = i0 < b1 ? a[i0] : 0u, x1 = i1 < b1 ? a[i1] : 0u;
  const unsigned m0 = __ballot_sync(0xffffffffu, i0 < b1 && x0 > v);
  if (m0) return b0 + __ffs(m0) - 1;
  const unsigned m1 = __ballot_sync(0xffffffffu, i1 < b1 && x1 > v);
  return m1 ? b0 + 32 + __ffs(m1) - 1 : hi;
}
// Merge path split by the 32 lanes of a warp: the number of A elements among
// the first d of merge(A[0..na), B[0..nb)) when A's element goes first on
// equal weight, i.e. the first i in [max(0, d - nb), min(d, na)] with
// A[i] > B[d - 1 - i] (a 32-ary search: each step probes 32 equal segments).
__device__ __forceinline__ int warp_merge_split(const unsigned* A, int na, const unsigned* B, int nb, int d) {
  const int lane = threadIdx.x & 31;
  int lo = max(0, d - nb), hi = min(d, na);
  auto after = [&](int i) { return A[i] > B[d - 1 - i]; };  // A[i] is not among the first d
  while (hi - lo > 32) {
    const int step = (hi - lo + 31) / 32;
    const int p = min(lo + (lane + 1) * step, hi) - 1;
    const unsigned m = __ballot_sync(0xffffffffu, after(p));
    if (m == 0u) return hi;
    const int f = __ffs(m) - 1;
    const int nlo = lo + f * step;
    hi = min(nlo + step, hi);
    lo = nlo;
  }
  const unsigned m = __ballot_sync(0xffffffffu, lane < hi - lo && after(lo + lane));
  return m ? lo + __ffs(m) - 1 : hi;
}

// First codes, first positions, left-justified limits, the symbol count and
// the longest length of canonical codes from the count of codes of each
// length (ct->count[1..kMaxLen], count[kMaxLen + 1] = 0); one thread.
__device__ inline void canon_from_counts(CanonTables* ct) {
  unsigned code = 0, p = 0, maxl = 0;
  ct->count[0] = 0;
  for (int L = 1; L <= kMaxLen + 1; ++L) {
    code = (code + (L > 1 ? ct->count[L - 1] : 0u)) << 1;
    if (L == 1) code = 0;
    ct->first_code[L] = code;
    ct->first_pos[L] = p;
    p += ct->count[L];
    if (ct->count[L]) maxl = L;
  }
  for (int L = 1; L <= kMaxLen; ++L) ct->limit[L] = ((unsigned long long)ct->first_code[L] + ct->count[L]) << (32 - L);
  ct->limit[kMaxLen + 1] = 1ull << 32;
  ct->n = p;
  ct->max_len = maxl;
}

// Canonical-code tables from the code lengths of the n present symbols held
// in symbol order (len[i]: length of the i-th present symbol): canon[] gets
// the indices i in (length, symbol) order, by one stable counting pass over
// the lengths (at most kMaxLen): warps rank their rows of 32 as in
// radix_sort_pairs (counting walk, scan, ranking walk), warp L-1 scans length
// L's counts over the warps, and each index lands at first_pos[len] + (indices
// of its length before it).  wcnt is scratch of at least (kMaxLen + 1) * 32 u32.
// `add` is added to the indices in canon[].
__device__ void build_canonical(const uint8_t* len, int n, unsigned* wcnt, uint16_t* canon, CanonTables* ct,
                                unsigned add = 0u) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x < kMaxLen + 2) ct->count[threadIdx.x] = 0;
  for (int i = threadIdx.x; i < (kMaxLen + 1) * 32; i += blockDim.x) wcnt[i] = 0u;
  __syncthreads();
  const int rows = (n + kCbThreads - 1) / kCbThreads;
  const int seg = rows * 32;
  for (int r0 = 0; r0 < rows; r0 += 8) {
    unsigned ll[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = wid * seg + (r0 + t) * 32 + lane;
      ll[t] = (r0 + t < rows && i < n) ? len[i] : 0u;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (r0 + t >= rows) break;
      const unsigned L = ll[t];
      const bool ok = L != 0u && L <= (unsigned)kMaxLen;
      if (!__any_sync(0xffffffffu, ok)) continue;
      const unsigned m = __match_any_sync(0xffffffffu, ok ? L : 64u);  // few distinct values: match takes a step each
      if (ok && (m & ((1u << lane) - 1u)) == 0u) wcnt[wc_idx(L, wid)] += (unsigned)__popc(m);
      __syncwarp();
    }
  }
  __syncthreads();
  if (wid < kMaxLen) {  // length L = wid + 1: exclusive scan of its counts over the warps
    const unsigned L = (unsigned)wid + 1u;
    const unsigned c = wcnt[wc_idx(L, lane)];
    unsigned x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    wcnt[wc_idx(L, lane)] = x - c;
    if (lane == 31) ct->count[L] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) canon_from_counts(ct);
  __syncthreads();
  for (int r0 = 0; r0 < rows; r0 += 8) {
    unsigned ll[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = wid * seg + (r0 + t) * 32 + lane;
      ll[t] = (r0 + t < rows && i < n) ? len[i] : 0u;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (r0 + t >= rows) break;
      const int i = wid * seg + (r0 + t) * 32 + lane;
      const unsigned L = ll[t];
      const bool ok = L != 0u && L <= (unsigned)kMaxLen;
      if (!__any_sync(0xffffffffu, ok)) continue;
      const unsigned m = __match_any_sync(0xffffffffu, ok ? L : 64u);
      const unsigned lt = m & ((1u << lane) - 1u);
      const unsigned base = ok ? wcnt[wc_idx(L, wid)] : 0u;
      if (ok) canon[ct->first_pos[L] + base + (unsigned)__popc(lt)] = (uint16_t)(add + (unsigned)i);
      __syncwarp();
      if (ok && lt == 0u) wcnt[wc_idx(L, wid)] = base + (unsigned)__popc(m);
      __syncwarp();
    }
  }
  __syncthreads();
}

struct CodebookArgs {
  const unsigned* hist;  // [dict]
  int dict;
  uint8_t* lens;         // [dict] out
  unsigned* codes;       // [dict] out
  uint8_t* out;          // stream base (codebook runs written at out + off), may be null
  unsigned long long off;
  unsigned long long capacity;
  Scalars* sc;
  int esc_mode;                  // symbol 0 is the escape of an outlier code
  unsigned long long nch;        // chunks
  unsigned long long raw_total;  // size of the raw stream (~0: no raw fallback)
  unsigned char* big;            // global scratch for more than kCbSmemSyms present symbols (cb_big_bytes())
  unsigned* packed;              // [dict] out: the encoder's entries, enc_entry(code, len)
  unsigned* first_code;          // [kMaxLen + 1] out: first code of each length
  int presorted;                 // cb_presort_kernel ran: tables cleared, symbols compacted into the
                                 // global arrays and, above kCbSmemSyms of them, sorted
};

// Present symbols the codebook keeps in shared memory; more use global
// scratch (L2-resident) with the same code.
constexpr int kCbSmemSyms = 8192;

// Arrays of the codebook construction over the n present symbols, indexed by
// their rank in symbol order ("compact index"); node ids of the Huffman tree
// are leaves 0..n-1 (sorted order) and internal nodes n.. (creation order).
struct CbArrays {
  uint16_t* csym;      // [n] symbol of compact index
  uint8_t* clen;       // [n] code length of compact index
  unsigned* ka;        // [n] sort keys -> sorted leaf weights (lw)
  uint16_t* sa;        // [n] compact indices -> sorted leaf order (ls)
  unsigned* kb;        // [n] sort buffer (aliases iw in shared memory)
  uint16_t* sb;        // [n] sort buffer (aliases parent in shared memory)
  unsigned* iw;        // [n] internal weights
  uint16_t* parent;    // [2n]; more symbols than shared memory holds: [n], the leaves' (internal node by creation)
  uint8_t* depth;      // [2n] (in shared memory only, as round_end)
  unsigned* wcnt;      // [256*32] sort counts (aliases round_end in shared memory)
  uint16_t* round_end; // [n] internal nodes created up to the end of each round
  uint16_t* canon;     // [n] compact indices in canonical order (aliases iw)
  unsigned* run_start; // [n] compact index of each run's first symbol (aliases ka)
  unsigned* run_end;   // [n] one past its last (aliases iw, after the canonical codes are out)
  unsigned* run_off;   // [n] byte offset of the run in the codebook section (aliases wcnt)
};

// Shared-memory layout for at most kCbSmemSyms present symbols (16-bit ids).
struct CbSmem {
  unsigned scan_tmp[64];
  CanonTables ct;
  unsigned ka[kCbSmemSyms];                 // 32 KB
  unsigned iw[kCbSmemSyms];                 // 32 KB (sort: kb; later canon)
  unsigned wcnt[256 * 32];                  // 32 KB (rounds: round_end u16[N])
  uint16_t parent[2 * kCbSmemSyms];         // 32 KB (sort: sb)
  uint8_t depth[2 * kCbSmemSyms];           // 16 KB
  uint16_t sa[kCbSmemSyms];                 // 16 KB
  uint16_t csym[kCbSmemSyms];               // 16 KB
  uint8_t clen[kCbSmemSyms];                //  8 KB
};
static_assert(sizeof(CbSmem) <= 227 * 1024, "codebook shared memory");
static_assert(256 * 32 >= kCbSmemSyms, "run offsets over the sort counts");

// Shared memory of the global-scratch variant's tree: a tile of merged ranks
// (the weights of its leaves, then of its internal nodes), samples of the two
// queues, and the parent of every internal node.
// After the rounds the tile holds a depth byte per internal node, and at the
// end the parents' place the leaves' lengths, gathered there before an
// in-order copy out.
constexpr int kCbTile = 20480;  // ranks of a tile (even)
struct CbBigSmem {
  unsigned scan_tmp[64];
  CanonTables ct;
  alignas(16) unsigned wcnt[256 * 32];  // the sort's counts, before the rounds (then part of the tile)
  unsigned tile_rest[kCbTile - 256 * 32];
  unsigned samp[2 * (kMaxDict / 64)];
  uint16_t par[kMaxDict];
  __device__ __forceinline__ unsigned* tile() { return wcnt; }
};
static_assert(sizeof(CbBigSmem) <= 227 * 1024, "codebook shared memory");
static_assert(kCbTile * sizeof(unsigned) >= kMaxDict, "a depth byte per internal node");
constexpr size_t kCbSmemBytes = sizeof(CbSmem) > sizeof(CbBigSmem) ? sizeof(CbSmem) : sizeof(CbBigSmem);

// Global scratch of the large variant: n <= kMaxDict present symbols, 32-bit ids.
constexpr int kPreCtas = 64;  // CTAs of cb_presort_kernel
// Counts of the multi-CTA presort, after the arrays in the global scratch.
struct CbPre {
  unsigned n, maxk, passes, pad;
  unsigned cnt[kPreCtas];          // present symbols of each CTA's dictionary segment
  unsigned dcnt[kPreCtas * 256];   // per (CTA, digit) keys of the current pass; then per (CTA, length) codes
  unsigned rcnt[kPreCtas];         // run starts of each CTA's segment of compact indices
  unsigned bsum[kPreCtas];         // codebook-section bytes of each CTA's runs
  unsigned long long bits;         // sum of f len
};
__host__ __device__ constexpr size_t cb_big_bytes() {
  return (size_t)kMaxDict * (2 + 1 + 4 + 2 + 4 + 2 + 4 + 2 + 2) + 3 * 4 * (size_t)kMaxDict + 16 * 256 +
         sizeof(CbPre) + 256;
}

__device__ __forceinline__ CbArrays cb_small(CbSmem& S) {
  CbArrays v;
  v.csym = S.csym; v.clen = S.clen; v.ka = S.ka; v.sa = S.sa;
  v.kb = S.iw; v.sb = S.parent; v.iw = S.iw; v.parent = S.parent; v.depth = S.depth;
  v.wcnt = S.wcnt;
  v.round_end = reinterpret_cast<uint16_t*>(S.wcnt);
  v.canon = reinterpret_cast<uint16_t*>(S.iw);
  v.run_start = S.ka;
  v.run_end = S.iw;
  v.run_off = S.wcnt;
  return v;
}

__device__ __forceinline__ CbArrays cb_big(unsigned char* g, unsigned* smem_wcnt) {
  auto take = [&](size_t bytes) {
    unsigned char* p = g;
    g += (bytes + 255) & ~size_t(255);
    return p;
  };
  const size_t N = kMaxDict;
  CbArrays v;
  v.csym = reinterpret_cast<uint16_t*>(take(2 * N));
  v.clen = take(N);
  v.ka = reinterpret_cast<unsigned*>(take(4 * N));
  v.sa = reinterpret_cast<uint16_t*>(take(2 * N));
  v.kb = reinterpret_cast<unsigned*>(take(4 * N));
  v.sb = reinterpret_cast<uint16_t*>(take(2 * N));
  v.iw = reinterpret_cast<unsigned*>(take(4 * N));
  v.parent = reinterpret_cast<uint16_t*>(take(2 * N));
  v.depth = nullptr;
  v.round_end = nullptr;
  v.canon = reinterpret_cast<uint16_t*>(take(2 * N));
  v.run_start = reinterpret_cast<unsigned*>(take(4 * N));
  v.run_end = reinterpret_cast<unsigned*>(take(4 * N));
  v.run_off = reinterpret_cast<unsigned*>(take(4 * N));
  v.wcnt = smem_wcnt;  // the counting passes stay in shared memory
  return v;
}
// The presort's counts: after the arrays of cb_big.
__device__ __forceinline__ CbPre* cb_pre(unsigned char* g) {
  const size_t N = kMaxDict;
  size_t off = 0;
  const size_t parts[] = {2 * N, N, 4 * N, 2 * N, 4 * N, 2 * N, 4 * N, 2 * N, 2 * N, 4 * N, 4 * N, 4 * N};
  for (size_t b : parts) off += (b + 255) & ~size_t(255);
  return reinterpret_cast<CbPre*>(g + off);
}

// Pairs of the ranks [d0, d1) of merge(A[0..na), B[0..nb)) (A first on equal
// weight), d0 even, whose first i0 = split(d0) ranks came from A: appends
// the pairs' weights to iw at qe + d/2 and sets the parents.  Ids: A[i] is
// node aid0 + i, B[j] is node bid0 + j.
__device__ __forceinline__ unsigned merge_pairs(const unsigned* A, int na, const unsigned* B, int nb, int d0, int d1,
                                                int i, int aid0, int bid0, int qe, unsigned* iw, uint16_t* parent,
                                                int n) {
  unsigned leaves = 0;
  int j = d0 - i;
  for (int d = d0; d < d1; d += 2) {
    // both queues' next two read together (~0u past a queue's end: a weight is
    // below 2^31, and a pair's two nodes exist)
    const unsigned a0 = i < na ? A[i] : ~0u, a1 = i + 1 < na ? A[i + 1] : ~0u;
    const unsigned b0 = j < nb ? B[j] : ~0u, b1 = j + 1 < nb ? B[j + 1] : ~0u;
    const bool f = a0 <= b0;                    // the first is a leaf
    const bool s = f ? a1 <= b0 : a0 <= b1;     // the second is a leaf
    const int i2 = i + (f ? 1 : 0), j2 = j + (f ? 0 : 1);
    const int id0 = f ? aid0 + i : bid0 + j, id1 = s ? aid0 + i2 : bid0 + j2;
    const unsigned w = (f ? a0 : b0) + (s ? (f ? a1 : a0) : (f ? b0 : b1));
    i = i2 + (s ? 1 : 0);
    j = j2 + (s ? 0 : 1);
    leaves += (f ? 1u : 0u) + (s ? 1u : 0u);
    const int k = d >> 1;
    iw[qe + k] = w;
    parent[id0] = (uint16_t)(n + qe + k);
    parent[id1] = (uint16_t)(n + qe + k);
  }
  return leaves;
}
// The sum of the two smallest remaining weights of both queues: the first two
// of each, read together (a weight is below 2^31, so ~0u marks an empty slot).
__device__ __forceinline__ unsigned two_smallest(const unsigned* lw, unsigned lp, unsigned n, const unsigned* iw,
                                                 unsigned qp, unsigned qe) {
  const unsigned c0 = lp < n ? lw[lp] : ~0u, c1 = lp + 1 < n ? lw[lp + 1] : ~0u;
  const unsigned d0 = qp < qe ? iw[qp] : ~0u, d1 = qp + 1 < qe ? iw[qp + 1] : ~0u;
  return c0 <= d0 ? c0 + min(c1, d0) : d0 + min(c0, d1);
}

// Leaves by ascending weight (ties in symbol order) into (V.ka, V.sa), for
// the weights max(1, f >> shift): the whole block.
__device__ void codebook_sort(const CodebookArgs& a, const CbArrays& V, int n, unsigned* scan_tmp, int shift) {
  __shared__ unsigned s_maxk;
  if (threadIdx.x == 0) s_maxk = 0;
  __syncthreads();
  unsigned mk = 0;
  for (int i0 = threadIdx.x; i0 < n; i0 += 8 * blockDim.x) {  // eight loads in flight
    unsigned sy[8], f[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = i0 + t * (int)blockDim.x;
      sy[t] = i < n ? (unsigned)V.csym[i] : 0u;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) f[t] = i0 + t * (int)blockDim.x < n ? a.hist[sy[t]] : 0u;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = i0 + t * (int)blockDim.x;
      if (i < n) {
        const unsigned fs = shift ? max(1u, f[t] >> shift) : f[t];
        V.ka[i] = fs;
        V.sa[i] = (uint16_t)i;
        V.clen[i] = 0;
        mk = max(mk, fs);
      }
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) mk = max(mk, __shfl_xor_sync(0xffffffffu, mk, o));
  if ((threadIdx.x & 31) == 0 && mk) atomicMax(&s_maxk, mk);
  __syncthreads();
  const int which = n <= 8 * kCbThreads ? radix_sort_pairs_small(V.ka, V.sa, V.kb, V.sb, V.wcnt, n, s_maxk, scan_tmp)
                                        : radix_sort_pairs(V.ka, V.sa, V.kb, V.sb, V.wcnt, n, s_maxk, scan_tmp);
  if (which) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      V.ka[i] = V.kb[i];
      V.sa[i] = V.sb[i];
    }
  }
  __syncthreads();
}

// The codebook over the compact arrays V (n present symbols, already in
// V.csym): Huffman lengths into V.clen.  The lengths are those of the
// sequential two-queue construction; lengths above kMaxLen are avoided by
// re-running on max(1, f >> t), t = 1, 2, ...
// At most kCbSmemSyms present symbols: every array in shared memory.
__device__ void codebook_lengths(const CodebookArgs& a, CbArrays V, int n, unsigned* scan_tmp) {
  __shared__ unsigned s_p[2], s_leaves, s_maxd;
  if (n <= 1) {
    if (n == 1 && threadIdx.x == 0) V.clen[0] = 1;
    __syncthreads();
    return;
  }
  for (int shift = 0;; ++shift) {
    // 1. (freq', compact index) pairs sorted
    codebook_sort(a, V, n, scan_tmp, shift);
    const unsigned* lw = V.ka;
    const uint16_t* ls = V.sa;
    // 2. parallel rounds of the two-queue construction: a round pairs all nodes
    // of weight <= X (X = the two smallest weights summed), found by warp-wide
    // searches of both sorted queues.  Every thread keeps the queues' state; the
    // leaves a round takes come from the thread that owns the round's last rank.
    // Bound by the latency of a round's steps (about 1,900 cycles, 18 rounds for
    // 1,749 symbols).  With the leaves counted by atomics and folded into a
    // shared state behind a third barrier, and the sort in two walks, the whole
    // codebook of 65^3 at 1e-3 took 63 us against 57 (1535x2049, 3,660 symbols:
    // 75 against 67); every warp making the searches for itself, one barrier a
    // round, was no faster than that (the tree 25 us against 22).
    unsigned lp = 0, qp = 0, qe = 0;
    int rounds = 0;
    while (qe < (unsigned)(n - 1)) {
      if (threadIdx.x < 64) {  // warps 0 and 1: the leaves and the internal nodes that weigh at most X
        const unsigned X = two_smallest(lw, lp, (unsigned)n, V.iw, qp, qe);
        const bool first = threadIdx.x < 32;
        const int from = (int)(first ? lp : qp);
        const int cnt = warp_upper_bound_u32(first ? lw : V.iw, from, first ? n : (int)qe, X) - from;
        if ((threadIdx.x & 31) == 0) s_p[first ? 0 : 1] = (unsigned)cnt;
      }
      __syncthreads();
      const int pl = (int)s_p[0], pq = (int)s_p[1];
      const int npairs = (pl + pq) >> 1;
      // the first 2*npairs nodes of the merged order (leaf first on equal
      // weight) pair up in order.  Merge path: thread t takes the ranks
      // [d0, d1) (d0 even), finds how many of the first d0 are leaves by one
      // binary search, then walks its ranks sequentially and forms its pairs.
      const unsigned* A = lw + lp;
      const unsigned* Bq = V.iw + qp;
      const int T = 2 * npairs;
      const int seg = 2 * ((npairs + (int)blockDim.x - 1) / (int)blockDim.x);
      const int d0 = min(T, (int)threadIdx.x * seg), d1 = min(T, d0 + seg);
      if (d0 < d1) {
        int lo = max(0, d0 - pq), hi = min(d0, pl);
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (A[mid] <= Bq[d0 - 1 - mid]) lo = mid + 1; else hi = mid;
        }
        const unsigned leaves = merge_pairs(A, pl, Bq, pq, d0, d1, lo, (int)lp, n + (int)qp, (int)qe, V.iw, V.parent, n);
        if (d1 == T) s_leaves = (unsigned)lo + leaves;
      }
      if (threadIdx.x == 0) V.round_end[rounds] = (uint16_t)(qe + npairs);
      __syncthreads();
      const unsigned taken = s_leaves;  // written again after the next barrier
      lp += taken;
      qp += (unsigned)T - taken;
      qe += (unsigned)npairs;
      ++rounds;
    }
    // 3. depths, rounds in reverse (a parent is always created in a later
    // round)
    const int root = 2 * n - 2;
    if (threadIdx.x == 0) {
      V.depth[root] = 0;
      s_maxd = 0;
    }
    __syncthreads();
    for (int r = rounds - 1; r >= 0; --r) {
      const int jb = r ? (int)V.round_end[r - 1] : 0, je = (int)V.round_end[r];
      for (int j = jb + threadIdx.x; j < je; j += blockDim.x) {
        const int v = n + j;
        if (v != root) V.depth[v] = V.depth[V.parent[v]] + 1;
      }
      __syncthreads();
    }
    unsigned md = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const unsigned dd = (unsigned)V.depth[V.parent[i]] + 1u;
      V.clen[ls[i]] = (uint8_t)min(dd, 255u);
      md = max(md, dd);
    }
    if (md) atomicMax(&s_maxd, md);
    __syncthreads();
    if (s_maxd <= (unsigned)kMaxLen) break;
    __syncthreads();
  }
}

// More present symbols: the queues in global scratch, a round's nodes staged
// in tiles of merged ranks, one pass over a tile: the leaves' parents and the
// new weights go straight to global memory, the internal nodes' parents stay
// in shared memory, where the depths follow them.  Bound by the latency of a
// round's steps (19 to 28 rounds) and one SM's issue rate.  With the results
// staged per queue and every parent in global memory the tree of 65,468
// symbols (100x500x500 at 1e-4) took 0.195 ms against 0.153; ranks found by
// a binary search per node instead of the merge path took 0.211.
__device__ void codebook_lengths_big(const CodebookArgs& a, CbArrays V, int n, CbBigSmem& S,
                                     int pre_passes) {
  __shared__ unsigned s_lp, s_qp, s_qe, s_pl, s_pq, s_rounds, s_maxd;
  __shared__ int s_split;
  // a round's X is at least 1.5 times the one before (a node left over by an
  // odd count weighs at least X / 2): at most 54 rounds
  __shared__ unsigned s_rend[64];
  unsigned* const lsamp = S.samp;
  unsigned* const isamp = S.samp + kMaxDict / 64;
  unsigned* const tw = S.tile();  // a tile's weights: leaves, then internal nodes
  uint16_t* const lpar = V.parent;  // of the leaves
  for (int shift = 0;; ++shift) {
    if (shift == 0 && pre_passes > 0) {  // pairs sorted by cb_presort_kernel
      if (pre_passes & 1) {  // into (kb, sb)
        unsigned* tk = V.ka;
        V.ka = V.kb;
        V.kb = tk;
        uint16_t* ts = V.sa;
        V.sa = V.sb;
        V.sb = ts;
      }
    } else {
      codebook_sort(a, V, n, S.scan_tmp, shift);
    }
    const unsigned* lw = V.ka;
    const uint16_t* ls = V.sa;
    // the leaves' samples (the last block's is the last leaf)
    for (int k = threadIdx.x; k < (n + 63) >> 6; k += blockDim.x) lsamp[k] = lw[min(64 * k + 63, n - 1)];
    if (threadIdx.x == 0) { s_lp = 0; s_qp = 0; s_qe = 0; s_rounds = 0; }
    __syncthreads();
    while (true) {
      if (threadIdx.x < 64) {
        const unsigned lp = s_lp, qp = s_qp, qe = s_qe;
        if (qe < (unsigned)(n - 1)) {
          const unsigned X = two_smallest(lw, lp, (unsigned)n, V.iw, qp, qe);
          if (threadIdx.x < 32) {
            const int pl = warp_upper_bound_sampled(lw, lsamp, (int)lp, n, (n + 63) >> 6, X) - (int)lp;
            if (threadIdx.x == 0) s_pl = (unsigned)pl;
          } else {
            const int pq = warp_upper_bound_sampled(V.iw, isamp, (int)qp, (int)qe, (int)(qe >> 6), X) - (int)qp;
            if (threadIdx.x == 32) s_pq = (unsigned)pq;
          }
        }
      }
      __syncthreads();
      if (s_qe >= (unsigned)(n - 1)) break;
      const int lp = s_lp, qp = s_qp, qe = s_qe, pl = s_pl, pq = s_pq;
      const int npairs = (pl + pq) >> 1;
      const unsigned* A = lw + lp;
      const unsigned* Bq = V.iw + qp;
      const int T = 2 * npairs;
      int ia = 0;
      for (int tb = 0; tb < T; tb += kCbTile) {
        const int te = min(T, tb + kCbTile);
        int ib;
        if (te == pl + pq) {  // every node of both queues
          ib = pl;
        } else {
          if (te == T) {  // all but the last of the merged order (A first on equal weight)
            if (threadIdx.x == 0) s_split = pq == 0 ? pl - 1 : pl == 0 ? 0 : A[pl - 1] <= Bq[pq - 1] ? pl : pl - 1;
          } else if (threadIdx.x < 32) {
            const int sp = warp_merge_split(A, pl, Bq, pq, te);
            if (threadIdx.x == 0) s_split = sp;
          }
          __syncthreads();
          ib = s_split;
        }
        const int ja = tb - ia, na = ib - ia, tl = te - tb, nb = tl - na;
        for (int k0 = threadIdx.x; k0 < tl; k0 += 10 * blockDim.x) {  // ten loads in flight
          unsigned x[10];
#pragma unroll
          for (int t = 0; t < 10; ++t) {
            const int k = k0 + t * (int)blockDim.x;
            x[t] = k < na ? A[ia + k] : k < tl ? Bq[ja + k - na] : 0u;
          }
#pragma unroll
          for (int t = 0; t < 10; ++t)
            if (k0 + t * (int)blockDim.x < tl) tw[k0 + t * blockDim.x] = x[t];
        }
        __syncthreads();
        // merge path: thread t takes the tile's ranks [d0, d1) (d0 even), finds
        // how many of the first d0 are leaves by one binary search, then walks
        // its ranks, one look-up each (~0u past a queue's end)
        const int kb0 = qe + (tb >> 1);
        const int seg = 2 * ((tl / 2 + (int)blockDim.x - 1) / (int)blockDim.x);
        const int d0 = min(tl, (int)threadIdx.x * seg), d1 = min(tl, d0 + seg);
        if (d0 < d1) {
          const unsigned* sB = tw + na;
          int lo = max(0, d0 - nb), hi = min(d0, na);
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (tw[mid] <= sB[d0 - 1 - mid]) lo = mid + 1; else hi = mid;
          }
          int i = lo, j = na + d0 - lo;  // next leaf, next internal node (indices into tw)
          unsigned x = i < na ? tw[i] : ~0u, y = j < tl ? tw[j] : ~0u;
          for (int d = d0; d < d1; d += 2) {
            unsigned w = 0;
            const uint16_t parent = (uint16_t)(kb0 + (d >> 1));
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const bool leaf = x <= y;
              w += leaf ? x : y;
              if (leaf) lpar[lp + ia + i] = parent;
              else S.par[qp + ja + j - na] = parent;
              const int nx = leaf ? ++i : ++j;
              const unsigned v = nx < (leaf ? na : tl) ? tw[nx] : ~0u;
              x = leaf ? v : x;
              y = leaf ? y : v;
            }
            V.iw[parent] = w;
            if ((parent & 63) == 63) isamp[parent >> 6] = w;
          }
        }
        ia = ib;
        if (te < T) __syncthreads();
      }
      if (threadIdx.x == 0) {
        s_lp = lp + ia;
        s_qp = qp + T - ia;
        s_qe = qe + npairs;
        s_rend[s_rounds++] = (unsigned)(qe + npairs);
      }
      __syncthreads();
    }
    // depths, rounds in reverse (a parent is always created in a later round),
    // one byte each in the tile's place (a depth stays below 64 for counts
    // below 2^32), indexed by creation order
    uint8_t* const dsh = reinterpret_cast<uint8_t*>(S.tile());
    if (threadIdx.x == 0) {
      dsh[n - 2] = 0;
      s_maxd = 0;
    }
    __syncthreads();
    for (int r = (int)s_rounds - 1; r >= 0; --r) {
      const int jb = r ? (int)s_rend[r - 1] : 0, je = (int)s_rend[r];
      for (int j = jb + threadIdx.x; j < je; j += blockDim.x)
        if (j != n - 2) dsh[j] = (uint8_t)(dsh[S.par[j]] + 1);
      __syncthreads();
    }
    // the leaves' lengths, gathered over the parents (scattered byte stores),
    // then copied out in compact-index order
    uint8_t* const lens = reinterpret_cast<uint8_t*>(S.par);
    unsigned md = 0;
    for (int i0 = threadIdx.x; i0 < n; i0 += 8 * blockDim.x) {  // sixteen loads in flight
      unsigned pa[8], li[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int i = i0 + t * (int)blockDim.x;
        pa[t] = i < n ? (unsigned)lpar[i] : 0u;
        li[t] = i < n ? (unsigned)ls[i] : 0u;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (i0 + t * (int)blockDim.x < n) {
          const unsigned dd = (unsigned)dsh[pa[t]] + 1u;
          lens[li[t]] = (uint8_t)min(dd, 255u);
          md = max(md, dd);
        }
    }
    if (md) atomicMax(&s_maxd, md);
    __syncthreads();
    for (int i = threadIdx.x; i < n / 4; i += blockDim.x)
      reinterpret_cast<unsigned*>(V.clen)[i] = reinterpret_cast<const unsigned*>(lens)[i];
    if (threadIdx.x < (unsigned)(n & 3)) V.clen[(n & ~3) + threadIdx.x] = lens[(n & ~3) + threadIdx.x];
    __syncthreads();
    if (s_maxd <= (unsigned)kMaxLen) break;
    __syncthreads();
  }
}

// The codebook's decisions (one thread): section sizes and offsets, the
// encoder's table and window, the lower bound on the stream size and the
// raw-copy decision.  smin / smax: the smallest and largest present symbol;
// bits: sum of f_s len_s.
__device__ inline void codebook_decide(const CodebookArgs& a, unsigned smin, unsigned smax, unsigned long long total,
                                       int nruns, unsigned max_len, unsigned long long bits, bool fits) {
  {
    Scalars* sc = a.sc;
    sc->codebook_bytes = total;
    sc->n_runs = (unsigned long long)nruns;
    sc->max_len = max_len;
    // the encoder's table: a shared-memory window of enc_entry words when every
    // present symbol lies in kEncWinSmall or in kEncWin consecutive symbols and
    // no code is too long for an entry, else the split table of the whole
    // dictionary (three shared-memory look-ups per code instead of one: 0.284
    // ms for the window at 1e-3 against 0.397 for the split table at 1e-4, 513^3)
    unsigned wn = kEncWin;
    sc->enc_lo = 0;
    sc->enc_mode = 2;
    if (max_len <= kPackLen && smax - smin < (unsigned)kEncWinSmall) {
      sc->enc_lo = a.dict <= kEncWinSmall ? 0u : min(smin, (unsigned)(a.dict - kEncWinSmall));
      sc->enc_mode = 0;
      wn = kEncWinSmall;
    } else if (max_len <= kPackLen && smax - smin < (unsigned)kEncWin) {
      sc->enc_lo = a.dict <= kEncWin ? 0u : min(smin, (unsigned)(a.dict - kEncWin));
      sc->enc_mode = 3;
    }
    // the window's entries above the largest present symbol are never read
    sc->enc_n = smax >= sc->enc_lo ? min(wn, smax + 1u - sc->enc_lo) : 0u;
    if (a.out && !fits) atomicOr(&sc->status, ST_CAPACITY | ST_RAW);
    const unsigned long long nout = a.esc_mode ? (unsigned long long)a.hist[0] : 0ull;
    const unsigned long long off_ce = a.off + pad8(total);
    const unsigned long long off_out = off_ce + (nout ? pad8(4ull * a.nch) : 0ull);
    const unsigned long long off_bits = off_out + pad8(4ull * nout);
    const unsigned long long min_total = off_bits + pad8(4ull * ((bits + 31ull) / 32ull));
    sc->n_outliers = nout;
    sc->off_chunk_esc = off_ce;
    sc->off_outliers = off_out;
    sc->off_bits = off_bits;
    // a quantisation overflow, a size bound at or above the raw copy, or sections
    // that do not fit all make the stream a raw copy: skip the encoder
    if ((sc->status & ST_OVERFLOW) || min_total >= a.raw_total || off_bits > a.capacity) atomicOr(&sc->status, ST_RAW);
    sc->skip = (sc->status & ST_RAW) ? 1u : 0u;
  }
}

// Canonical codes, the lookup tables of the encoder, the codebook section of
// the stream and the offsets of the sections after it, from the lengths.
__device__ void codebook_emit(const CodebookArgs& a, CbArrays V, int n, unsigned* scan_tmp, CanonTables* ct) {
  __shared__ unsigned s_total, s_nruns;
  __shared__ unsigned long long s_bits;
  if (threadIdx.x == 0) s_bits = 0;
  // 4. canonical codes (the counting pass in the sort counts' shared memory)
  build_canonical(V.clen, n, V.wcnt, V.canon, ct);
  const int nc = (int)ct->n;
  if (threadIdx.x <= kMaxLen) a.first_code[threadIdx.x] = ct->first_code[threadIdx.x];
  for (int i0 = threadIdx.x; i0 < nc; i0 += 8 * blockDim.x) {  // eight loads in flight
    unsigned ci[8], L[8], sy[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = i0 + t * (int)blockDim.x;
      ci[t] = i < nc ? (unsigned)V.canon[i] : 0u;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const bool ok = i0 + t * (int)blockDim.x < nc;
      L[t] = ok ? (unsigned)V.clen[ci[t]] : 0u;
      sy[t] = ok ? (unsigned)V.csym[ci[t]] : 0u;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = i0 + t * (int)blockDim.x;
      if (i < nc) {
        const unsigned c = ct->first_code[L[t]] + (unsigned)(i - (int)ct->first_pos[L[t]]);
        a.codes[sy[t]] = c;
        a.packed[sy[t]] = enc_entry(c, L[t]);
        a.lens[sy[t]] = (uint8_t)L[t];
      }
    }
  }
  // 5. codebook runs {u32 first, u32 count, u8 len[count], pad to 4}: a run
  // starts at every present symbol whose predecessor is absent.  Warp w walks
  // its contiguous rows of 32 compact indices (coalesced loads): run starts
  // by ballot, one scan over the warps, then each start's run index.
  unsigned* run_start = V.run_start;
  unsigned* run_end = V.run_end;
  unsigned* run_off = V.run_off;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int rows = (n + 31) / 32, rpw = (rows + nwarps - 1) / nwarps;
  const int r0 = wid * rpw, r1 = min(rows, r0 + rpw);
  // run-start masks of eight rows at once (sixteen loads in flight)
  auto start_masks = [&](int r, unsigned (&m)[8]) {
    unsigned c[8], p[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = (r + t) * 32 + lane;
      const bool ok = r + t < r1 && i < n;
      c[t] = ok ? (unsigned)V.csym[i] : 0u;
      p[t] = ok && i > 0 ? (unsigned)V.csym[i - 1] : 0u;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = (r + t) * 32 + lane;
      m[t] = __ballot_sync(0xffffffffu, r + t < r1 && i < n && (i == 0 || c[t] != p[t] + 1u));
    }
  };
  unsigned nst = 0;
  for (int r = r0; r < r1; r += 8) {
    unsigned m[8];
    start_masks(r, m);
#pragma unroll
    for (int t = 0; t < 8; ++t) nst += (unsigned)__popc(m[t]);
  }
  const unsigned rbase = warp_excl_scan_block(nst, scan_tmp, &s_nruns);
  {
    unsigned q = rbase;
    for (int r = r0; r < r1; r += 8) {
      unsigned m[8];
      start_masks(r, m);
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        if ((m[t] >> lane) & 1u)
          run_start[q + (unsigned)__popc(m[t] & ((1u << lane) - 1u))] = (unsigned)((r + t) * 32 + lane);
        q += (unsigned)__popc(m[t]);
      }
    }
  }
  __syncthreads();
  const int nruns = (int)s_nruns;
  for (int q = threadIdx.x; q < nruns; q += blockDim.x) run_end[q] = q + 1 < nruns ? run_start[q + 1] : (unsigned)n;
  __syncthreads();
  unsigned my_bytes = 0;
  const int rper = (nruns + blockDim.x - 1) / blockDim.x;
  const int q0 = threadIdx.x * rper;
  for (int q = q0; q < q0 + rper && q < nruns; ++q) my_bytes += 8u + (((run_end[q] - run_start[q]) + 3u) & ~3u);
  unsigned off = block_excl_scan(my_bytes, scan_tmp, &s_total);
  for (int q = q0; q < q0 + rper && q < nruns; ++q) {
    run_off[q] = off;
    off += 8u + (((run_end[q] - run_start[q]) + 3u) & ~3u);
  }
  __syncthreads();
  const unsigned long long total = s_total;
  const bool fits = a.out && a.off + pad8(total) <= a.capacity;
  if (fits) {
    for (int q = threadIdx.x; q < nruns; q += blockDim.x) {
      const unsigned first = run_start[q], cntq = run_end[q] - first;
      uint8_t* p = a.out + a.off + run_off[q];
      *reinterpret_cast<unsigned*>(p) = (unsigned)V.csym[first];
      *reinterpret_cast<unsigned*>(p + 4) = cntq;
      for (unsigned t = cntq; t < ((cntq + 3u) & ~3u); ++t) p[8 + t] = 0;
    }
    // length bytes: compact index i of run q goes to run_off[q] + 8 + (i -
    // run_start[q]), q = (run starts up to i) - 1, from the same row walk
    unsigned q = rbase;
    for (int r = r0; r < r1; r += 8) {
      unsigned m[8], qi[8], ro[8], rs[8], cl[8];
      start_masks(r, m);
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        qi[t] = q + (unsigned)__popc(m[t] & ((2u << lane) - 1u)) - 1u;
        q += (unsigned)__popc(m[t]);
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int i = (r + t) * 32 + lane;
        const bool ok = r + t < r1 && i < n;
        ro[t] = ok ? run_off[qi[t]] : 0u;
        rs[t] = ok ? run_start[qi[t]] : 0u;
        cl[t] = ok ? (unsigned)V.clen[i] : 0u;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int i = (r + t) * 32 + lane;
        if (r + t < r1 && i < n) a.out[a.off + ro[t] + 8 + (i - rs[t])] = (uint8_t)cl[t];
      }
    }
    if (threadIdx.x == 0)
      for (unsigned long long t = total; t < pad8(total); ++t) a.out[a.off + t] = 0;
  }
  // 6. layout of the rest of the stream (escape counts, outlier codes, then
  // the bitstream) and a lower bound on its size: the bitstream holds exactly
  // sum_s f_s len_s bits plus the padding of each chunk to whole words
  unsigned long long my_bits = 0;
  for (int i0 = threadIdx.x; i0 < n; i0 += 8 * blockDim.x) {  // eight loads in flight
    unsigned sy[8], cl[8], f[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = i0 + t * (int)blockDim.x;
      sy[t] = i < n ? (unsigned)V.csym[i] : 0u;
      cl[t] = i < n ? (unsigned)V.clen[i] : 0u;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) f[t] = i0 + t * (int)blockDim.x < n ? a.hist[sy[t]] : 0u;
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (i0 + t * (int)blockDim.x < n) my_bits += (unsigned long long)f[t] * cl[t];
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) my_bits += __shfl_xor_sync(0xffffffffu, my_bits, o);
  if ((threadIdx.x & 31) == 0 && my_bits) atomicAdd(&s_bits, my_bits);
  __syncthreads();
  if (threadIdx.x == 0)
    codebook_decide(a, n ? V.csym[0] : 0u, n ? V.csym[n - 1] : 0u, total, nruns, ct->max_len, s_bits, fits);
}

// Multi-CTA start of the codebook for wide code distributions: one
// cooperative launch of kPreCtas CTAs with grid-wide barriers between the
// phases.  It clears the code tables, compacts the present symbols (symbol
// order) into the global arrays with their frequencies as keys, the compact
// index as payload and zero lengths, and, when more than kCbSmemSyms symbols
// are present, sorts the pairs by key, stably, with 8-bit LSD passes: each
// CTA owns a contiguous segment of the pairs; in a pass its warps rank their
// rows by digit, and after the barrier every pair goes to the digit's global
// offset (all keys of smaller digits, then those of digit d in the CTAs and
// the warps before) plus its rank, so equal keys keep their order.  One
// thread per digit walking the segment instead took 26 us a pass (65,468
// pairs: the launch 91 us against 31).  The sorted pairs are in
// (ka, sa) after an even number of passes and in (kb, sb) after an odd one
// (CbPre::passes; 0 when the codebook kernel sorts in shared memory itself).
constexpr int kPreThreads = 256;
constexpr int kPreSeg = kMaxDict / kPreCtas;  // pairs per CTA at most
constexpr int kPreWarps = kPreThreads / 32, kPreRows = kPreSeg / kPreThreads;  // rows of 32 pairs per warp
__global__ void __launch_bounds__(kPreThreads) cb_presort_kernel(CodebookArgs a) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  CbPre* pre = cb_pre(a.big);
  const CbArrays V = cb_big(a.big, nullptr);
  const int dict = a.dict, c = blockIdx.x, G = gridDim.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __shared__ unsigned s_red[kPreThreads / 32];
  __shared__ unsigned s_scan[32], s_tot;
  __shared__ unsigned s_wc[kPreWarps * 256];
  __shared__ unsigned s_base, s_n, s_maxk;
  auto block_sum = [&](unsigned v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) s_red[wid] = v;
    __syncthreads();
    unsigned t = 0;
    for (int w = 0; w < kPreThreads / 32; ++w) t += s_red[w];
    return t;
  };
  auto block_excl = [&](unsigned v, unsigned* total) { return block_excl_scan(v, s_scan, total); };
  // 0. tables cleared; present symbols of this CTA's dictionary segment counted
  for (int s = c * kPreThreads + threadIdx.x; s < dict; s += G * kPreThreads) {
    a.lens[s] = 0;
    a.codes[s] = 0;
    a.packed[s] = 0;
  }
  const int dseg = (dict + G - 1) / G, d0 = min(dict, c * dseg), d1 = min(dict, d0 + dseg);
  unsigned my = 0;
  for (int s = d0 + threadIdx.x; s < d1; s += kPreThreads) my += a.hist[s] != 0u;
  const unsigned cnt = block_sum(my);
  if (threadIdx.x == 0) {
    pre->cnt[c] = cnt;
    if (c == 0) {
      pre->maxk = 0;
      pre->bits = 0;
    }
  }
  grid.sync();
  // 1. compaction in symbol order: (frequency, compact index) pairs
  if (threadIdx.x == 0) {
    unsigned b = 0, t = 0;
    for (int k = 0; k < G; ++k) {
      const unsigned v = pre->cnt[k];
      if (k < c) b += v;
      t += v;
    }
    s_base = b;
    s_n = t;
  }
  __syncthreads();
  unsigned pos = s_base, mk = 0;
  for (int s0 = d0; s0 < d1; s0 += kPreThreads) {
    const int s = s0 + threadIdx.x;
    const unsigned f = s < d1 ? a.hist[s] : 0u;
    const unsigned r = block_excl(f != 0u ? 1u : 0u, &s_tot);
    if (f) {
      const unsigned i = pos + r;
      V.csym[i] = (uint16_t)s;
      V.clen[i] = 0;
      V.ka[i] = f;
      V.sa[i] = (uint16_t)i;
      mk = max(mk, f);
    }
    pos += s_tot;
    __syncthreads();
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) mk = max(mk, __shfl_xor_sync(0xffffffffu, mk, o));
  if (lane == 0 && mk) atomicMax(&pre->maxk, mk);
  if (c == 0 && threadIdx.x == 0) pre->n = s_n;
  grid.sync();
  const int n = (int)s_n;
  if (threadIdx.x == 0) s_maxk = pre->maxk;
  __syncthreads();
  int passes = 0;
  if (n > kCbSmemSyms) {
    passes = 1;
    while (passes < 4 && (s_maxk >> (8 * passes)) != 0u) ++passes;
  }
  if (c == 0 && threadIdx.x == 0) pre->passes = (unsigned)passes;
  const int pseg = (n + G - 1) / G, p0 = min(n, c * pseg), p1 = min(n, p0 + pseg);
  for (int p = 0; p < passes; ++p) {
    const int shift = 8 * p;
    const unsigned* kin = (p & 1) ? V.kb : V.ka;
    const uint16_t* sin = (p & 1) ? V.sb : V.sa;
    unsigned* kout = (p & 1) ? V.ka : V.kb;
    uint16_t* sout = (p & 1) ? V.sa : V.sb;
    // every warp ranks its four rows of 32 pairs by digit (match), with a
    // running count per (warp, digit): the pair's rank among the warp's
    for (int i = threadIdx.x; i < kPreWarps * 256; i += kPreThreads) s_wc[i] = 0u;
    __syncthreads();
    unsigned key[kPreRows], rank[kPreRows];
    uint16_t val[kPreRows];
#pragma unroll
    for (int t = 0; t < kPreRows; ++t) {
      const int i = p0 + (wid * kPreRows + t) * 32 + lane;
      key[t] = i < p1 ? kin[i] : 0u;
      val[t] = i < p1 ? sin[i] : (uint16_t)0;
    }
#pragma unroll
    for (int t = 0; t < kPreRows; ++t) {
      const bool ok = p0 + (wid * kPreRows + t) * 32 + lane < p1;
      const unsigned d = (key[t] >> shift) & 255u;
      const unsigned m = __match_any_sync(0xffffffffu, ok ? d : 256u);
      const unsigned lt = m & ((1u << lane) - 1u), seen = ok ? s_wc[wid * 256 + d] : 0u;
      rank[t] = seen + (unsigned)__popc(lt);
      __syncwarp();
      if (ok && lt == 0u) s_wc[wid * 256 + d] = seen + (unsigned)__popc(m);
      __syncwarp();
    }
    __syncthreads();
    {  // thread d: the digit's count over the warps, and each warp's offset in it
      unsigned t = 0;
#pragma unroll
      for (int w = 0; w < kPreWarps; ++w) {
        const unsigned v = s_wc[w * 256 + threadIdx.x];
        s_wc[w * 256 + threadIdx.x] = t;
        t += v;
      }
      pre->dcnt[c * 256 + threadIdx.x] = t;
    }
    grid.sync();
    // offsets of digit d (thread d): keys of smaller digits, then of digit d
    // in the CTAs before this one
    const unsigned d = threadIdx.x;
    unsigned col = 0, part = 0;
#pragma unroll 16
    for (int k = 0; k < G; ++k) {
      const unsigned v = pre->dcnt[k * 256 + d];
      if (k < c) part += v;
      col += v;
    }
    const unsigned off = block_excl(col, nullptr) + part;
#pragma unroll
    for (int w = 0; w < kPreWarps; ++w) s_wc[w * 256 + d] += off;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kPreRows; ++t)
      if (p0 + (wid * kPreRows + t) * 32 + lane < p1) {
        const unsigned o = s_wc[wid * 256 + ((key[t] >> shift) & 255u)] + rank[t];
        kout[o] = key[t];
        sout[o] = val[t];
      }
    grid.sync();
  }
}

// Multi-CTA end of the codebook for wide code distributions (after the one-CTA
// tree, above kCbSmemSyms present symbols; cooperative launch of kPreCtas
// CTAs, grid-wide barriers between the phases): what codebook_emit does, each
// CTA over its segment of compact indices.  Codes: per-(CTA, length) counts
// and the warps' ranks by length (symbol order within a length), as in the
// presort (one thread per length walking the segment: the launch 45 us
// against 29).  Runs of consecutive
// present symbols: per-CTA start counts give each start's run index; the
// runs' section bytes are summed per CTA for their offsets.  The sums of the
// size bound and of the encoder's window go to global atomics; CTA 0 makes
// the decisions.
__global__ void __launch_bounds__(kPreThreads) cb_emit_kernel(CodebookArgs a) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  CbPre* pre = cb_pre(a.big);
  const CbArrays V = cb_big(a.big, nullptr);
  const int n = (int)pre->n;
  if (n <= kCbSmemSyms) return;  // the one-CTA kernel emitted everything (the same for every CTA)
  const int c = blockIdx.x, G = gridDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  __shared__ uint8_t s_len[kPreSeg];
  __shared__ uint16_t s_sym[kPreSeg];
  __shared__ unsigned s_wl[kPreWarps * 64];  // per (warp, length): codes, then offsets
  __shared__ unsigned s_scan[32], s_tot;
  __shared__ unsigned s_red[kPreThreads / 32];
  __shared__ unsigned long long s_r64[kPreThreads / 32];
  __shared__ CanonTables s_ct;
  __shared__ unsigned s_prev, s_rbase, s_nruns, s_boff, s_total;
  auto block_excl = [&](unsigned v, unsigned* total) { return block_excl_scan(v, s_scan, total); };
  const int pseg = (n + G - 1) / G, e0 = min(n, c * pseg), e1 = min(n, e0 + pseg), m = e1 - e0;
  // E0: the segment staged; its length counts, run starts and size sums
  for (int i = tid; i < kPreWarps * 64; i += kPreThreads) s_wl[i] = 0u;
  if (tid == 0) s_prev = e0 > 0 ? (unsigned)V.csym[e0 - 1] : 0u;
  __syncthreads();
  unsigned long long my_bits = 0;
  for (int i = tid; i < m; i += kPreThreads) {
    const unsigned L = V.clen[e0 + i], sy = V.csym[e0 + i];
    s_len[i] = (uint8_t)L;
    s_sym[i] = (uint16_t)sy;
    my_bits += (unsigned long long)a.hist[sy] * L;
  }
  __syncthreads();
  auto is_start = [&](int i) {  // i: index within the segment
    return e0 + i == 0 || (unsigned)s_sym[i] != (i ? (unsigned)s_sym[i - 1] : s_prev) + 1u;
  };
  unsigned my_st = 0;
  for (int i = tid; i < m; i += kPreThreads) my_st += is_start(i);
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    my_bits += __shfl_xor_sync(0xffffffffu, my_bits, o);
    my_st += __shfl_xor_sync(0xffffffffu, my_st, o);
  }
  if (lane == 0) {
    s_r64[wid] = my_bits;
    s_red[wid] = my_st;
  }
  __syncthreads();
  if (tid == 0) {
    unsigned long long b = 0;
    unsigned st = 0;
    for (int k = 0; k < kPreThreads / 32; ++k) {
      b += s_r64[k];
      st += s_red[k];
    }
    atomicAdd(&pre->bits, b);
    pre->rcnt[c] = st;
  }
  // ranks by length: every warp's rows in order, as in the presort
  unsigned rank[kPreRows];
#pragma unroll
  for (int t = 0; t < kPreRows; ++t) {
    const int i = (wid * kPreRows + t) * 32 + lane;
    const bool ok = i < m && s_len[i] >= 1 && s_len[i] <= kMaxLen;
    const unsigned L = ok ? (unsigned)s_len[i] : 0u;
    const unsigned mm = __match_any_sync(0xffffffffu, L);
    const unsigned lt = mm & ((1u << lane) - 1u), seen = s_wl[wid * 64 + L];
    rank[t] = seen + (unsigned)__popc(lt);
    __syncwarp();
    if (lt == 0u) s_wl[wid * 64 + L] = seen + (unsigned)__popc(mm);
    __syncwarp();
  }
  __syncthreads();
  if (tid <= kMaxLen) {
    unsigned t = 0;
    for (int w = 0; w < kPreWarps; ++w) {
      const unsigned v = s_wl[w * 64 + tid];
      s_wl[w * 64 + tid] = t;
      t += v;
    }
    pre->dcnt[c * 256 + tid] = tid ? t : 0u;
  }
  grid.sync();
  // E1: canonical tables (every CTA, the same), this segment's canonical
  // positions; run bases
  unsigned part = 0;
  if (tid <= kMaxLen + 1) {
    unsigned tot = 0;
#pragma unroll 16
    for (int k = 0; k < G; ++k) {
      const unsigned v = tid <= kMaxLen ? pre->dcnt[k * 256 + tid] : 0u;
      if (k < c) part += v;
      tot += v;
    }
    s_ct.count[tid] = tid == 0 || tid == kMaxLen + 1 ? 0u : tot;
  }
  if (tid == 0) {
    unsigned rb = 0, rt = 0;
    for (int k = 0; k < G; ++k) {
      const unsigned v = pre->rcnt[k];
      if (k < c) rb += v;
      rt += v;
    }
    s_rbase = rb;
    s_nruns = rt;
  }
  __syncthreads();
  if (tid == 0) canon_from_counts(&s_ct);
  __syncthreads();
  if (tid <= kMaxLen)
    for (int w = 0; w < kPreWarps; ++w) s_wl[w * 64 + tid] += part;
  if (c == 0 && tid <= kMaxLen) a.first_code[tid] = s_ct.first_code[tid];
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kPreRows; ++t) {  // a symbol's code: its length's first one plus its rank
    const int i = (wid * kPreRows + t) * 32 + lane;
    const unsigned L = i < m ? (unsigned)s_len[i] : 0u;
    if (L >= 1u && L <= (unsigned)kMaxLen) {
      const unsigned cd = s_ct.first_code[L] + s_wl[wid * 64 + L] + rank[t], sy = s_sym[i];
      a.codes[sy] = cd;
      a.packed[sy] = enc_entry(cd, L);
      a.lens[sy] = (uint8_t)L;
    }
  }
  const int nruns = (int)s_nruns;
  {  // run starts of the segment at their run indices
    unsigned q = s_rbase;
    for (int i0 = 0; i0 < m; i0 += kPreThreads) {
      const int i = i0 + tid;
      const bool st = i < m && is_start(i);
      const unsigned r = block_excl(st ? 1u : 0u, &s_tot);
      if (st) V.run_start[q + r] = (unsigned)(e0 + i);
      q += s_tot;
      __syncthreads();
    }
  }
  grid.sync();
  // E2: section bytes of this CTA's runs
  const int rq = (nruns + G - 1) / G, q0 = min(nruns, c * rq), q1 = min(nruns, q0 + rq);
  unsigned my_b = 0;
  for (int q = q0 + tid; q < q1; q += kPreThreads) {
    const unsigned st = V.run_start[q], en = q + 1 < nruns ? V.run_start[q + 1] : (unsigned)n;
    V.run_end[q] = en;
    my_b += 8u + (((en - st) + 3u) & ~3u);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) my_b += __shfl_xor_sync(0xffffffffu, my_b, o);
  if (lane == 0) s_red[wid] = my_b;
  __syncthreads();
  if (tid == 0) {
    unsigned t = 0;
    for (int k = 0; k < kPreThreads / 32; ++k) t += s_red[k];
    pre->bsum[c] = t;
  }
  grid.sync();
  // E3: run offsets and headers
  if (tid == 0) {
    unsigned b = 0, t = 0;
    for (int k = 0; k < G; ++k) {
      const unsigned v = pre->bsum[k];
      if (k < c) b += v;
      t += v;
    }
    s_boff = b;
    s_total = t;
  }
  __syncthreads();
  const unsigned long long total = s_total;
  const bool fits = a.out && a.off + pad8(total) <= a.capacity;
  {
    unsigned off = s_boff;
    for (int qb = q0; qb < q1; qb += kPreThreads) {
      const int q = qb + tid;
      const unsigned st = q < q1 ? V.run_start[q] : 0u, en = q < q1 ? V.run_end[q] : 0u;
      const unsigned bq = q < q1 ? 8u + (((en - st) + 3u) & ~3u) : 0u;
      const unsigned r = block_excl(bq, &s_tot);
      if (q < q1) {
        V.run_off[q] = off + r;
        if (fits) {
          uint8_t* p = a.out + a.off + off + r;
          *reinterpret_cast<unsigned*>(p) = (unsigned)V.csym[st];
          *reinterpret_cast<unsigned*>(p + 4) = en - st;
          for (unsigned t = en - st; t < (((en - st) + 3u) & ~3u); ++t) p[8 + t] = 0;
        }
      }
      off += s_tot;
      __syncthreads();
    }
  }
  grid.sync();
  // E4: the length bytes, each at its run's offset; CTA 0's decisions
  if (fits) {
    unsigned q = s_rbase;  // run index of the next start
    for (int i0 = 0; i0 < m; i0 += kPreThreads) {
      const int i = i0 + tid;
      const bool st = i < m && is_start(i);
      const unsigned r = block_excl(st ? 1u : 0u, &s_tot);
      if (i < m) {
        const unsigned qi = q + r + (st ? 1u : 0u) - 1u;  // starts up to and including i, minus one
        a.out[a.off + V.run_off[qi] + 8 + ((unsigned)(e0 + i) - V.run_start[qi])] = s_len[i];
      }
      q += s_tot;
      __syncthreads();
    }
    if (c == 0 && tid == 0)
      for (unsigned long long t = total; t < pad8(total); ++t) a.out[a.off + t] = 0;
  }
  if (c == 0 && tid == 0)
    codebook_decide(a, V.csym[0], V.csym[n - 1], total, nruns, s_ct.max_len, pre->bits, fits);
}

// The codebook of one compress call, built by one CTA (the whole block).
__device__ void codebook_block(const CodebookArgs& a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CbSmem& S = *reinterpret_cast<CbSmem*>(smem_raw);
  __shared__ unsigned s_n;
  const int dict = a.dict;
  if (a.presorted) {  // cb_presort_kernel cleared the tables and compacted the symbols
    const CbPre* pre = cb_pre(a.big);
    const int n = (int)pre->n;
    const int passes = (int)pre->passes;
    if (n <= kCbSmemSyms) {
      const uint16_t* gsym = cb_big(a.big, S.wcnt).csym;
      for (int i = threadIdx.x; i < n; i += blockDim.x) S.csym[i] = gsym[i];
      __syncthreads();
      const CbArrays V = cb_small(S);
      codebook_lengths(a, V, n, S.scan_tmp);
      codebook_emit(a, V, n, S.scan_tmp, &S.ct);
    } else {  // the tree here; cb_emit_kernel emits the codes on many CTAs afterwards
      CbBigSmem& L = *reinterpret_cast<CbBigSmem*>(smem_raw);
      codebook_lengths_big(a, cb_big(a.big, L.wcnt), n, L, passes);
    }
    return;
  }
  // 0. every dictionary entry starts without a code
  for (int s = threadIdx.x; s < dict; s += blockDim.x) {
    a.lens[s] = 0;
    a.codes[s] = 0;
    a.packed[s] = 0;
  }
  // present symbols, in symbol order, compacted: warp w walks its contiguous
  // rows of 32 symbols (coalesced loads, eight rows in flight), counting by
  // ballot; one scan over the warps; a second walk writes each present
  // symbol at its warp's offset plus its rank in the row
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int rows = (dict + 31) / 32, rpw = (rows + nwarps - 1) / nwarps;
  const int r0 = wid * rpw, r1 = min(rows, r0 + rpw);
  unsigned cnt = 0;
  for (int r = r0; r < r1; r += 8) {
    unsigned f[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int s = (r + k) * 32 + lane;
      f[k] = (r + k < r1 && s < dict) ? a.hist[s] : 0u;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) cnt += (unsigned)__popc(__ballot_sync(0xffffffffu, f[k] != 0u));
  }
  if (lane == 0) S.scan_tmp[32 + wid] = cnt;
  __syncthreads();
  if (wid == 0) {
    const unsigned c = lane < nwarps ? S.scan_tmp[32 + lane] : 0u;
    unsigned x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane < nwarps) S.scan_tmp[lane] = x - c;
    if (lane == 31) s_n = x;
  }
  __syncthreads();
  const int n = (int)s_n;
  const bool small = n <= kCbSmemSyms;
  uint16_t* csym = small ? S.csym : cb_big(a.big, S.wcnt).csym;
  unsigned pos = S.scan_tmp[wid];
  for (int r = r0; r < r1; r += 8) {
    unsigned f[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int s = (r + k) * 32 + lane;
      f[k] = (r + k < r1 && s < dict) ? a.hist[s] : 0u;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const unsigned m = __ballot_sync(0xffffffffu, f[k] != 0u);
      if (f[k]) csym[pos + (unsigned)__popc(m & ((1u << lane) - 1u))] = (uint16_t)((r + k) * 32 + lane);
      pos += (unsigned)__popc(m);
    }
  }
  __syncthreads();
  if (small) {
    const CbArrays V = cb_small(S);
    codebook_lengths(a, V, n, S.scan_tmp);
    codebook_emit(a, V, n, S.scan_tmp, &S.ct);
  } else {
    CbBigSmem& L = *reinterpret_cast<CbBigSmem*>(smem_raw);
    const CbArrays V = cb_big(a.big, L.wcnt);
    codebook_lengths_big(a, V, n, L, -1);
    codebook_emit(a, V, n, L.scan_tmp, &L.ct);
  }
}

__global__ void __launch_bounds__(kCbThreads) codebook_kernel(CodebookArgs a) { codebook_block(a); }

// The codebooks of several compress calls (a batch), one CTA each.
__global__ void __launch_bounds__(kCbThreads) codebook_batch_kernel(const CodebookArgs* __restrict__ args) {
  const CodebookArgs a = args[blockIdx.x];
  codebook_block(a);
}

// Histogram of a symbol array (stand-alone Huffman entry point): a shared
// window of kHistWin bins around the dictionary's middle, global atomics
// outside it; symbols not below dict are flagged.
__global__ void __launch_bounds__(256) hist_kernel(const uint16_t* __restrict__ sym, unsigned long long n, int dict,
                                                   unsigned* hist, Scalars* sc) {
  __shared__ unsigned hs[kHistWin];
  const int lo = max(0, min(dict / 2 - kHistWin / 2, dict - kHistWin));
  const int w = min(dict, kHistWin);
  for (int i = threadIdx.x; i < w; i += blockDim.x) hs[i] = 0;
  __syncthreads();
  bool bad = false;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned s = sym[i];
    const unsigned k = s - (unsigned)lo;
    if (k < (unsigned)w) atomicAdd(hs + k, 1u);
    else if (s < (unsigned)dict) atomicAdd(hist + s, 1u);
    else bad = true;
  }
  if (bad) atomicOr(&sc->status, ST_CORRUPT);
  __syncthreads();
  for (int i = threadIdx.x; i < w; i += blockDim.x)
    if (hs[i]) atomicAdd(hist + lo + i, hs[i]);
}

// Histogram of a symbol range [s0, s1) with 16-byte loads.  Build-time choice
// BM_HIST_METHOD: 1 = the centre symbol (code 0) counted in a register, the
// rest with shared atomics; 7 = the seven symbols around the centre in
// registers; 0 = equal symbols of a warp instruction merged first
// (__match_any_sync), one shared atomic per distinct symbol.  Shared bins
// cover kHistWin symbols around the centre; the rest go to global atomics.
#ifndef BM_HIST_METHOD
#define BM_HIST_METHOD 1
#endif
#ifndef BM_HIST_INFLIGHT
#define BM_HIST_INFLIGHT 8
#endif
__global__ void __launch_bounds__(256) hist_range_kernel(const uint16_t* __restrict__ sym, unsigned long long s0,
                                                         unsigned long long s1, int dict, unsigned centre_sym,
                                                         unsigned* hist) {
  __shared__ unsigned hs[kHistWin];
  const unsigned wlo = (unsigned)max(0, min((int)centre_sym - kHistWin / 2, dict - kHistWin));
  const unsigned wn = (unsigned)min(dict, kHistWin);
  for (int i = threadIdx.x; i < (int)wn; i += blockDim.x) hs[i] = 0;
  __syncthreads();
  constexpr int NC = BM_HIST_METHOD == 7 ? 7 : 1;
  unsigned cnt[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) cnt[j] = 0;
  unsigned n_esc = 0;  // the escape symbol 0: outside the window for large dictionaries, and frequent
  const unsigned lo = centre_sym - (NC / 2);
  auto bin = [&](unsigned s, unsigned c) {
    const unsigned k = s - wlo;
    if (k < wn) atomicAdd(hs + k, c);
    else if (s < (unsigned)dict) atomicAdd(hist + s, c);
  };
  auto count = [&](unsigned s) {
    if (BM_HIST_METHOD == 0) {
      const unsigned m = __match_any_sync(__activemask(), s);
      if ((unsigned)(threadIdx.x & 31) == (unsigned)(__ffs(m) - 1)) bin(s, __popc(m));
      return;
    }
    const unsigned d = s - lo;
#pragma unroll
    for (int j = 0; j < NC; ++j) cnt[j] += d == (unsigned)j;
    n_esc += s == 0u;
    if (d >= (unsigned)NC && s != 0u) bin(s, 1u);
  };
  const unsigned long long a0 = min(s1, (s0 + 7) & ~7ull);  // 16-byte aligned start
  const unsigned long long tid = blockIdx.x * 256ull + threadIdx.x, nth = gridDim.x * 256ull;
  for (unsigned long long i = s0 + tid; i < a0; i += nth) count(sym[i]);
  const unsigned long long nv = (s1 - a0) / 8;
  const uint4* pv = reinterpret_cast<const uint4*>(sym + a0);
  // BM_HIST_INFLIGHT 16-byte loads per thread are issued before any is counted
  constexpr int NF = BM_HIST_INFLIGHT;
  for (unsigned long long v = tid; v < nv; v += NF * nth) {
    uint4 q[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const unsigned long long vf = v + f * nth;
      q[f] = vf < nv ? __ldg(pv + vf) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      if (v + f * nth >= nv) break;
      const unsigned w4[4] = {q[f].x, q[f].y, q[f].z, q[f].w};
#pragma unroll
      for (int h = 0; h < 4; ++h) { count(w4[h] & 0xFFFFu); count(w4[h] >> 16); }
    }
  }
  for (unsigned long long i = a0 + nv * 8 + tid; i < s1; i += nth) count(sym[i]);
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    unsigned c = cnt[j];
#pragma unroll
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (BM_HIST_METHOD != 0 && (threadIdx.x & 31) == 0 && c) bin(lo + j, c);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) n_esc += __shfl_xor_sync(0xffffffffu, n_esc, o);
  if ((threadIdx.x & 31) == 0 && n_esc) bin(0u, n_esc);
  __syncthreads();
  for (int i = threadIdx.x; i < (int)wn; i += blockDim.x)
    if (hs[i]) atomicAdd(hist + wlo + i, hs[i]);
}

// Histogram of a symbol range [s0, s1) for dictionaries larger than the
// small window: one CTA of kHistWideThreads threads per SM keeps a private
// window of hist_wide_bins(dict) bins centred on the centre symbol (as much
// of the dictionary as fits in shared memory: at most kHistWideMax bins) and
// counts with shared atomics; symbols outside it (thin tails of very wide
// code distributions) go to global atomics; the centre and the escape symbol
// 0 are counted in registers.  Symbols not below dict are flagged (sc, when
// given).  Measured on GB300 faster than spreading the whole dictionary over
// a thread-block cluster in distributed shared memory (remote reductions on
// the frequent bins serialise at their owner).
constexpr int kHistWideThreads = 1024;
constexpr int kHistWideMax = 49152;
__host__ __device__ constexpr int hist_wide_bins(int dict) { return dict < kHistWideMax ? dict : kHistWideMax; }

__global__ void __launch_bounds__(kHistWideThreads)
    hist_wide_kernel(const uint16_t* __restrict__ sym, unsigned long long s0, unsigned long long s1, int dict,
                     unsigned centre_sym, unsigned* hist, Scalars* sc) {
  extern __shared__ __align__(16) unsigned hw[];
  const int W = hist_wide_bins(dict);
  const unsigned wlo = (unsigned)max(0, min((int)centre_sym - W / 2, dict - W));
  for (int i = threadIdx.x; i < W; i += blockDim.x) hw[i] = 0;
  __syncthreads();
  unsigned n_centre = 0, n_esc = 0;
  bool bad = false;
  auto count = [&](unsigned s) {
    n_centre += s == centre_sym;
    n_esc += s == 0u;
    if (s == centre_sym || s == 0u) return;
    const unsigned k = s - wlo;
    if (k < (unsigned)W) atomicAdd(hw + k, 1u);
    else if (s < (unsigned)dict) atomicAdd(hist + s, 1u);
    else bad = true;
  };
  // the 16-byte aligned start (a caller's symbols may begin at any address)
  const unsigned head = (unsigned)((16u - (reinterpret_cast<uintptr_t>(sym + s0) & 15u)) & 15u) / 2u;
  const unsigned long long a0 = min(s1, s0 + head);
  const unsigned long long tid = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  const unsigned long long nth = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = s0 + tid; i < a0; i += nth) count(sym[i]);
  const unsigned long long nv = (s1 - a0) / 8;
  const uint4* pv = reinterpret_cast<const uint4*>(sym + a0);
  constexpr int NF = 4;
  for (unsigned long long v = tid; v < nv; v += NF * nth) {
    uint4 q[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const unsigned long long vf = v + f * nth;
      q[f] = vf < nv ? __ldg(pv + vf) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      if (v + f * nth >= nv) break;
      const unsigned w4[4] = {q[f].x, q[f].y, q[f].z, q[f].w};
#pragma unroll
      for (int h = 0; h < 4; ++h) { count(w4[h] & 0xFFFFu); count(w4[h] >> 16); }
    }
  }
  for (unsigned long long i = a0 + nv * 8 + tid; i < s1; i += nth) count(sym[i]);
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    n_centre += __shfl_xor_sync(0xffffffffu, n_centre, o);
    n_esc += __shfl_xor_sync(0xffffffffu, n_esc, o);
  }
  if ((threadIdx.x & 31) == 0) {  // the window always holds the centre (it is centred on it, or holds all)
    if (n_centre) atomicAdd(hw + (centre_sym - wlo), n_centre);
    if (n_esc) atomicAdd(hist, n_esc);
  }
  if (bad && sc) atomicOr(&sc->status, ST_CORRUPT);
  __syncthreads();
  for (int i = threadIdx.x; i < W; i += blockDim.x) {
    const unsigned v = hw[i];
    if (v) atomicAdd(hist + wlo + i, v);
  }
}

// ---------------------------------------------------------------------------
// Single-pass encoder (decoupled look-back, Merrill & Garland 2016)
// ---------------------------------------------------------------------------
// Status word of a chunk for the look-back: [flag:2][words:31][escapes:31],
// so one load sees a consistent pair (inputs hold fewer than 2^31 symbols).
constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagIncl = 2ull << 62;
constexpr unsigned long long kM31 = (1ull << 31) - 1;
constexpr long kSpinLimit = 1l << 24;
__device__ __forceinline__ unsigned long long pack_status(unsigned long long flag, unsigned long long w,
                                                          unsigned long long e) {
  return flag | ((w & kM31) << 31) | (e & kM31);
}

struct FusedEncodeArgs {
  const uint16_t* sym;
  const int32_t* esc;            // codes of escaped symbols (stream mode) or null
  unsigned long long n;
  int chunk;                     // multiple of 32
  const uint8_t* lens;
  const unsigned* codes;
  const unsigned* packed;        // [dict] enc_entry(code, len) per symbol (written by the codebook)
  const unsigned* first_code;    // [kMaxLen + 1] first code of each length (written by the codebook)
  int dict;
  unsigned long long nch;
  unsigned* ticket;              // zeroed before launch
  unsigned long long* st;        // [nch] look-back status words (zeroed)
  unsigned* chunk_words;         // stream chunk table
  uint16_t* splits;              // stream split offsets [nch][7]
  uint8_t* out;                  // stream base; the codebook kernel put the section offsets in sc
  unsigned long long capacity;
  Scalars* sc;
  int win;                       // entries of the shared-memory window (MODE 0, 3)
};

__device__ __forceinline__ unsigned long long ld_volatile_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}

constexpr int kEncSteps = 8;  // 256-symbol steps of the longest chunk (2048 symbols)
// Warps (and consecutive chunks) of a tile, by the CTA's warps: with one
// look-back per chunk and 32 warps per SM a warp walked back over thousands
// of unfinished predecessors (half of the kernel's instructions); larger
// tiles wait longer at their barriers.  At 513^3, 1e-2 / 1e-3 / 1e-4 / 1e-5
// (the small window, the large one, the split table twice), tiles of one
// chunk took 0.309 / 0.316 / 0.417 / 0.529 ms, of four 0.271 / 0.284 / 0.397
// / 0.502, of eight 0.260 / 0.294 / 0.427 / 0.558.
constexpr int enc_group(int warps) { return warps > 8 ? 4 : 8; }

// Tables of the encoder in shared memory, by the kernel's MODE:
//   0, 3  a window of the dictionary, one enc_entry per symbol (`lo` its first
//         symbol): every symbol met lies in it and no code is longer than
//         kPackLen bits;
//   2     the whole dictionary split into the symbol's rank among the codes of
//         its length (u16, `low`) and the length (u8, `len`): any code is
//         first_code[len] + rank, with the left-justified first codes in `fc`.
// and, left in global memory (encode_small_kernel):
//   4     the whole dictionary, one enc_entry per symbol, as in 0 and 3;
//   5     its lengths and codes, split as in 2 at the look-up.
constexpr bool enc_split(int mode) { return mode == 2 || mode == 5; }
template <int MODE, bool CLAMP>
struct EncTab {
  const unsigned* ent;
  const uint16_t* low;
  const uint8_t* len;
  const unsigned* fc;  // [kMaxLen + 1] first codes, left-justified
  const unsigned* codes;       // mode 5
  const unsigned* first_code;
  unsigned lo;
  // What a symbol's look-up keeps in a register: the window's entry, or
  // rank | len << 16.
  __device__ __forceinline__ unsigned entry(unsigned s) const {
    if (MODE == 2) return (unsigned)low[s] | ((unsigned)len[s] << 16);
    if (MODE == 5) {
      const unsigned L = len[s];
      return ((codes[s] - first_code[L]) & 0xFFFFu) | (L << 16);
    }
    return ent[s - lo];
  }
  __device__ __forceinline__ unsigned length(unsigned s) const {
    return enc_split(MODE) ? (unsigned)len[s] : ent[s - lo] & 31u;
  }
  // Symbol i of a lane's eight.
  __device__ __forceinline__ static unsigned symbol(const unsigned (&w)[4], int i, unsigned dmax) {
    const unsigned s = (i & 1) ? w[i >> 1] >> 16 : w[i >> 1] & 0xFFFFu;
    return CLAMP ? min(s, dmax) : s;
  }
  __device__ __forceinline__ static unsigned bits(unsigned e) { return enc_split(MODE) ? e >> 16 : e & 31u; }
  // The code left-justified in 32 bits.
  __device__ __forceinline__ unsigned code(unsigned e, unsigned L) const {
    if (enc_split(MODE)) return fc[L] + ((e & 0xFFFFu) << (32u - L));
    return e & ~31u;
  }
};
// Shared memory of the encoder: the table, then a step's packed words for
// each warp (256 symbols of at most 32 bits from any bit of the first word on).
constexpr int kEncStage = 260;
template <int MODE>
__host__ __device__ constexpr size_t enc_table_bytes(int win, int dict) {
  return MODE == 2 ? (size_t)(dict + 7) / 8 * 8 * 3 + 4 * (kMaxLen + 4)
         : MODE == 5 ? 4 * (kMaxLen + 4)
         : MODE == 4 ? 0
                     : 4 * (size_t)win;
}
template <int MODE>
__host__ __device__ constexpr size_t enc_smem(int warps, int win, int dict) {
  return enc_table_bytes<MODE>(win, dict) + (size_t)warps * kEncStage * 4;
}
static_assert(enc_smem<3>(kEncWarps, kEncWin, 0) <= 227 * 1024 && enc_smem<2>(kEncWarps, 0, kMaxDict) <= 227 * 1024,
              "encoder shared memory");

// Publishes tile c's (words, escapes) aggregate and walks back over its
// predecessors (a window of 32 per step, one per lane of the calling warp)
// until one has published an inclusive prefix, then publishes its own.  Every
// lane gets the words and escapes before the tile; false when the bounded
// wait ran out.
__device__ __forceinline__ bool enc_lookback(unsigned long long* st, unsigned long long c, unsigned W, unsigned esc,
                                             unsigned long long& pw_out, unsigned long long& pe_out) {
  const int lane = threadIdx.x & 31;
  unsigned long long pw = 0, pe = 0;
  int timed_out = 0;
  if (c == 0) {
    if (lane == 0) atomicExch(st + 0, pack_status(kFlagIncl, W, esc));
  } else {
    if (lane == 0) atomicExch(st + c, pack_status(kFlagAgg, W, esc));
    long long top = (long long)c - 1;  // highest predecessor not yet summed
    long spins = 0;
    while (top >= 0) {
      const long long pidx = top - lane;
      const unsigned long long sv = pidx >= 0 ? ld_volatile_u64(st + pidx) : kFlagIncl;  // before chunk 0: prefix 0
      const unsigned flag = (unsigned)(sv >> 62);
      // only the lanes up to the first unpublished one can be used
      const unsigned unpub = __ballot_sync(0xffffffffu, flag == 0);
      const unsigned incl = __ballot_sync(0xffffffffu, flag == 2);
      const int first_incl = incl ? __ffs(incl) - 1 : 32;
      const int first_unpub = unpub ? __ffs(unpub) - 1 : 32;
      if (first_unpub <= first_incl && first_unpub < 32) {
        if (first_unpub == 0) {  // nearest predecessor not published yet: wait
          if (++spins > kSpinLimit) { timed_out = 1; break; }
          __nanosleep(32);
          continue;
        }
      }
      const int take = min(first_incl + 1, first_unpub);  // lanes [0, take) are summed
      unsigned long long w = 0, e = 0;
      if (lane < take && pidx >= 0) { w = (sv >> 31) & kM31; e = sv & kM31; }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        w += __shfl_xor_sync(0xffffffffu, w, o);
        e += __shfl_xor_sync(0xffffffffu, e, o);
      }
      pw += w;
      pe += e;
      if (first_incl < take) break;  // reached an inclusive prefix (or the start)
      top -= take;
    }
    timed_out = __shfl_sync(0xffffffffu, timed_out, 0);
    if (!timed_out && lane == 0) {
      __threadfence();
      atomicExch(st + c, pack_status(kFlagIncl, pw + W, pe + esc));
    }
  }
  pw_out = pw;  // every lane holds the same sums
  pe_out = pe;
  return !timed_out;
}

// A shared-memory store where `pred` holds, and an OR into shared memory
// (predicated instructions: lanes that fill a word at different symbols do
// not diverge).
__device__ __forceinline__ void st_shared_if(unsigned addr, unsigned v, bool pred) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.shared.u32 [%0], %1;\n}\n" ::"r"(addr), "r"(v),
               "r"((unsigned)pred)
               : "memory");
}
__device__ __forceinline__ void red_shared_or(unsigned addr, unsigned v) {
  asm volatile("red.shared.or.b32 [%0], %1;\n" ::"r"(addr), "r"(v) : "memory");
}

// Which of a lane's eight symbols are escapes (symbol 0).
__device__ __forceinline__ unsigned escape_mask(const unsigned (&w)[4]) {
  unsigned m = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m |= (w[i] & 0xFFFFu) == 0u ? 1u << (2 * i) : 0u;
    m |= (w[i] >> 16) == 0u ? 2u << (2 * i) : 0u;
  }
  return m;
}

// The outlier codes of a step's escapes (m8: this lane's eight symbols), at
// stream order positions from ep on; s: the step's first symbol; rank: the
// escapes of the lanes before, total: of the warp.  Many escapes are copied
// 32 consecutive symbols at a time (coalesced), few by the lanes that hold
// them.
__device__ __forceinline__ void enc_outliers(const int32_t* __restrict__ esc, int32_t* __restrict__ ocode,
                                             unsigned long long n_out, unsigned m8, unsigned long long s,
                                             unsigned long long ep, unsigned rank, unsigned total) {
  const int lane = threadIdx.x & 31;
  if (total >= 32u) {
    unsigned x = m8 << (8 * (lane & 3));
    x |= __shfl_xor_sync(0xffffffffu, x, 1);
    x |= __shfl_xor_sync(0xffffffffu, x, 2);
    int32_t v[8];
    unsigned m[8];
#pragma unroll
    for (int g = 0; g < 8; ++g) {  // eight loads in flight
      m[g] = __shfl_sync(0xffffffffu, x, 4 * g);
      v[g] = ((m[g] >> lane) & 1u) ? __ldg(esc + s + 32 * g + lane) : 0;
    }
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const unsigned long long p = ep + __popc(m[g] & ((1u << lane) - 1u));
      if (((m[g] >> lane) & 1u) && p < n_out) ocode[p] = v[g];
      ep += __popc(m[g]);
    }
  } else {
    ep += rank;
    while (m8) {
      const int i = __ffs(m8) - 1;
      m8 &= m8 - 1u;
      if (ep < n_out) ocode[ep] = __ldg(esc + s + 8 * lane + i);
      ++ep;
    }
  }
}

// The codebook's choice of table (sc->enc_mode, the kernel's MODE): 0 when
// every symbol met lies in a window of kEncWinSmall entries, 3 when they all
// lie in one of kEncWin entries, and no code is longer than kPackLen bits;
// 2 (the split table of the whole dictionary) otherwise.  For the
// compressor's own symbols (CLAMP = false) all three are launched, the ones
// that do not match returning at once; caller-supplied symbols (clamped to
// the dictionary) take 0 or 2 by the dictionary's size and the longest code.
//
// Groups of warps take tiles of consecutive chunks in ticket order, one chunk
// per warp, with one look-back per tile.  Chunks of whole 256-symbol steps: in
// step k lane l holds symbols 256 k + 8 l .. + 7 (one coalesced 16-byte load),
// so the warp's lanes code one contiguous run of the stream at a time.  The
// first look-ups give the chunk's bits; after the look-back each step's
// symbols (from L2) are looked up again, a warp scan of their lengths gives
// every lane its bit, and the lane's eight codes are packed MSB-first into
// the warp's words in shared memory: full words are stored, a lane's last
// bits are ORed into the word a later lane completed, the step's own last
// bits carry into the next step, and the full words leave with coalesced
// stores.  Bound by issue (mostly the ALU pipe) and the L1 pipeline: look-ups
// (about four wavefronts for 32 symbols), word stores and the copy out.  The
// kernel before it gave a lane 64 consecutive symbols: every word store and
// symbol load of a warp went to 32 different lines, and the far symbols of a
// wide distribution came from a table in global memory.  513^3 GRF, 1e-2 /
// 1e-3 / 1e-4 / 1e-5: 0.33 / 0.377 / 0.53 / 0.95 ms before, 0.26 / 0.284 /
// 0.397 / 0.502 now.
template <int WARPS, bool CLAMP, int MODE>
__device__ __forceinline__ void encode_tiles(const FusedEncodeArgs& a) {
  extern __shared__ __align__(16) unsigned char enc_smem_raw[];
  constexpr int kEncGroup = enc_group(WARPS), NG = WARPS / kEncGroup;
  __shared__ unsigned s_tile[NG], s_w[NG][kEncGroup], s_e[NG][kEncGroup], s_ok[NG];
  __shared__ unsigned long long s_base[NG][2];
  Scalars* sc = a.sc;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  EncTab<MODE, CLAMP> tab{};
  if (MODE == 2) {
    const int D = (a.dict + 7) / 8 * 8;
    uint16_t* low = reinterpret_cast<uint16_t*>(enc_smem_raw);
    uint8_t* len = enc_smem_raw + 2 * D;
    unsigned* fc = reinterpret_cast<unsigned*>(enc_smem_raw + 3 * D);
    for (int i = threadIdx.x; i < a.dict; i += blockDim.x) {
      const unsigned L = a.lens[i];
      len[i] = (uint8_t)L;
      low[i] = (uint16_t)(L ? a.codes[i] - a.first_code[L] : 0u);
    }
    if (threadIdx.x <= kMaxLen) fc[threadIdx.x] = threadIdx.x ? a.first_code[threadIdx.x] << (32 - threadIdx.x) : 0u;
    tab.low = low;
    tab.len = len;
    tab.fc = fc;
  } else if (MODE == 5) {
    unsigned* fc = reinterpret_cast<unsigned*>(enc_smem_raw);
    if (threadIdx.x <= kMaxLen) fc[threadIdx.x] = threadIdx.x ? a.first_code[threadIdx.x] << (32 - threadIdx.x) : 0u;
    tab.len = a.lens;
    tab.codes = a.codes;
    tab.first_code = a.first_code;
    tab.fc = fc;
  } else if (MODE == 4) {
    tab.ent = a.packed;
    tab.lo = 0;
  } else {
    unsigned* ent = reinterpret_cast<unsigned*>(enc_smem_raw);
    const unsigned wlo = CLAMP ? 0u : sc->enc_lo;
    // the compressor's symbols lie below enc_lo + enc_n: the rest is never read
    const int nfill = CLAMP ? min(a.win, a.dict) : min(a.win, (int)sc->enc_n);
    for (int i = threadIdx.x; i < nfill; i += blockDim.x) {
      const unsigned s = wlo + (unsigned)i;
      ent[i] = s < (unsigned)a.dict ? a.packed[s] : 0u;
    }
    tab.ent = ent;
    tab.lo = wlo;
  }
  unsigned* const buf =
      reinterpret_cast<unsigned*>(enc_smem_raw + enc_table_bytes<MODE>(a.win, a.dict)) + warp * kEncStage;
  const unsigned sbuf = smem_u32(buf);
  __syncthreads();
  const unsigned dmax = (unsigned)(a.dict - 1);
  const unsigned long long off_bits = sc->off_bits;
  const unsigned long long n_out = sc->n_outliers;
  unsigned* words = reinterpret_cast<unsigned*>(a.out + off_bits);
  const bool has_esc = a.esc && n_out;
  unsigned* chunk_esc = has_esc ? reinterpret_cast<unsigned*>(a.out + sc->off_chunk_esc) : nullptr;
  int32_t* ocode = reinterpret_cast<int32_t*>(a.out + sc->off_outliers);
  const unsigned long long word_cap = a.capacity > off_bits ? (a.capacity - off_bits) / 4 : 0ull;
  const int per = a.chunk / 32;
  const int ns = a.chunk / 256;  // steps of a chunk
  // an eighth of a chunk is 32 ns symbols, 4 ns lanes of the steps; the
  // reciprocal divides lane indices below 256 exactly
  const unsigned lpe = 4u * ns, lpe_inv = lpe ? (65536u + lpe - 1u) / lpe : 0u;
  const bool steps_ok = (a.chunk & 255) == 0 && (CLAMP || (reinterpret_cast<uintptr_t>(a.sym) & 15) == 0);
  // a lane's eight symbols (at p, from symbol i0 of the array): one load, or,
  // where a caller's array starts between 16-byte boundaries, eight
  auto eight = [&](const uint4* p, unsigned long long i0) {
    if constexpr (CLAMP) {
      if (reinterpret_cast<uintptr_t>(a.sym) & 15) {
        const uint16_t* h = a.sym + i0;
        unsigned w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = (unsigned)__ldg(h + 2 * i) | ((unsigned)__ldg(h + 2 * i + 1) << 16);
        return make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    return __ldg(p);
  };
  const int grp = warp / kEncGroup, gw = warp % kEncGroup;  // tile group, warp of the group
  const unsigned long long ntiles = (a.nch + kEncGroup - 1) / kEncGroup;
  auto group_sync = [&] { asm volatile("bar.sync %0, %1;\n" ::"r"(grp + 1), "n"(kEncGroup * 32) : "memory"); };
  while (true) {
    if (gw == 0 && lane == 0) s_tile[grp] = atomicAdd(a.ticket, 1u);
    group_sync();
    const unsigned long long tile = s_tile[grp];
    if (tile >= ntiles) break;
    const unsigned long long c = tile * kEncGroup + gw;  // past the last chunk: no symbols
    const unsigned long long cb = min(a.n, c * (unsigned long long)a.chunk);
    const unsigned long long ce = min(a.n, cb + (unsigned long long)a.chunk);
    const bool steps = steps_ok && ce - cb == (unsigned long long)a.chunk;
    // first look-ups: bits and escapes of the chunk
    unsigned xb = 0, xe = 0, bits = 0, nesc = 0;  // other chunks: a slice per lane
    const unsigned long long s0 = min(ce, cb + (unsigned long long)lane * per), s1 = min(ce, s0 + per);
    const int cnt = (int)(s1 - s0);
    unsigned tot_bits, tot_esc;
    if (steps) {
      const uint4* p = reinterpret_cast<const uint4*>(a.sym + cb) + lane;
      uint4 q[kEncSteps];
#pragma unroll
      for (int k = 0; k < kEncSteps; ++k) q[k] = k < ns ? eight(p + 32 * k, cb + 256 * k + 8 * lane) : make_uint4(0, 0, 0, 0);
      unsigned sum = 0;  // bits | escapes << 17
#pragma unroll
      for (int k = 0; k < kEncSteps; ++k) {
        if (k < ns) {
          const unsigned w[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
#pragma unroll
          for (int i = 0; i < 8; ++i) sum += tab.length(tab.symbol(w, i, dmax));
          if (has_esc) sum += (unsigned)__popc(escape_mask(w)) << 17;
        }
      }
      sum = __reduce_add_sync(0xffffffffu, sum);
      tot_bits = sum & 0x1FFFFu;  // at most 2048 codes of 32 bits
      tot_esc = sum >> 17;
    } else {
      for (int t = 0; t < cnt; ++t) {
        const unsigned s = CLAMP ? min((unsigned)a.sym[s0 + t], dmax) : (unsigned)a.sym[s0 + t];
        bits += tab.bits(tab.entry(s));
        nesc += s == 0;
      }
      if (!a.esc) nesc = 0;
      xb = bits;
      xe = nesc;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned yb = __shfl_up_sync(0xffffffffu, xb, o);
        const unsigned ye = __shfl_up_sync(0xffffffffu, xe, o);
        if (lane >= o) { xb += yb; xe += ye; }
      }
      tot_bits = __shfl_sync(0xffffffffu, xb, 31);
      tot_esc = __shfl_sync(0xffffffffu, xe, 31);
    }
    const unsigned W = (tot_bits + 31u) >> 5;
    if (lane == 0) {
      s_w[grp][gw] = W;
      s_e[grp][gw] = tot_esc;
    }
    group_sync();
    if (gw == 0) {
      unsigned long long bw, be;
      const unsigned tw = __reduce_add_sync(0xffffffffu, lane < kEncGroup ? s_w[grp][lane] : 0u);
      const unsigned te = __reduce_add_sync(0xffffffffu, lane < kEncGroup ? s_e[grp][lane] : 0u);
      const bool ok = enc_lookback(a.st, tile, tw, te, bw, be);
      if (lane == 0) {
        s_base[grp][0] = bw;
        s_base[grp][1] = be;
        s_ok[grp] = ok;
      }
    }
    group_sync();
    const unsigned long long pw = s_base[grp][0] + __reduce_add_sync(0xffffffffu, lane < gw ? s_w[grp][lane] : 0u);
    unsigned long long pe = s_base[grp][1] + __reduce_add_sync(0xffffffffu, lane < gw ? s_e[grp][lane] : 0u);
    const bool ok = s_ok[grp];
    if (lane == 0 && c < a.nch) {
      a.chunk_words[c] = W;
      if (chunk_esc) chunk_esc[c] = tot_esc;
      if (c == a.nch - 1) {
        sc->n_words = pw + W;
        sc->esc_seen = pe + tot_esc;
      }
    }
    if (!ok) {
      if (lane == 0) atomicOr(&sc->status, ST_TIMEOUT | ST_RAW);
      break;
    }
    if (c >= a.nch) continue;
    if (pw + W > word_cap) {  // the stream would not fit: it becomes a raw copy
      if (lane == 0) atomicOr(&sc->status, ST_RAW);
      continue;
    }
    unsigned* const cw = words + pw;  // the chunk's words
    if (steps) {
      const uint4* p = reinterpret_cast<const uint4*>(a.sym + cb) + lane;
      uint4 qn = eight(p, cb + 8 * lane);
      unsigned b0 = 0, carry = 0;  // the step's first bit in the chunk; the bits before it in its word
#pragma unroll 1
      for (int k = 0; k < ns; ++k) {
        const unsigned w[4] = {qn.x, qn.y, qn.z, qn.w};
        if (k + 1 < ns) qn = eight(p + 32 * (k + 1), cb + 256 * (k + 1) + 8 * lane);
        unsigned e[8], v = 0;  // v: this lane's bits | escapes << 16
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = tab.entry(tab.symbol(w, i, dmax));
#pragma unroll
        for (int i = 0; i < 8; ++i) v += tab.bits(e[i]);
        unsigned m8 = 0;
        if (has_esc) {
          m8 = escape_mask(w);
          v += (unsigned)__popc(m8) << 16;
        }
        unsigned x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        const unsigned tot = __shfl_sync(0xffffffffu, x, 31);
        x -= v;
        const unsigned start = b0 + (x & 0xFFFFu);
        {  // bit offsets of the chunk's eighths 1..7
          const unsigned g = 32u * k + lane, j = (g * lpe_inv) >> 16;
          if (j && j * lpe == g) a.splits[c * (kSplits - 1) + j - 1] = (uint16_t)start;
        }
        if (has_esc) {
          const unsigned te = tot >> 16;
          if (te) enc_outliers(a.esc, ocode, n_out, m8, cb + 256u * k, pe, x >> 16, te);
          pe += te;
        }
        const unsigned w0 = b0 >> 5;
        unsigned off = start & 31u, cur = lane == 0 ? carry : 0u;
        unsigned wp = sbuf + 4u * ((start >> 5) - w0);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const unsigned L = tab.bits(e[i]), t = tab.code(e[i], L);
          cur |= t >> off;
          const unsigned rest = __funnelshift_r(0u, t, off);  // the code's bits past this word
          off += L;
          const bool full = off >= 32u;
          st_shared_if(wp, cur, full);
          wp += full ? 4u : 0u;
          cur = full ? rest : cur;
          off &= 31u;
        }
        // the word of the step's last bits is completed by no lane: the last
        // lane stores it, every other lane's last bits lie in a stored word
        if (lane == 31 && off) st_shared_if(wp, cur, true);
        __syncwarp();
        if (lane != 31 && off) red_shared_or(wp, cur);
        __syncwarp();
        b0 += tot & 0xFFFFu;
        const unsigned nfull = (b0 >> 5) - w0;
#pragma unroll 1
        for (unsigned i = lane; i < nfull; i += 32) cw[w0 + i] = buf[i];
        carry = (b0 & 31u) ? buf[nfull] : 0u;
        __syncwarp();
      }
      if (lane == 0 && (b0 & 31u)) cw[b0 >> 5] = carry;
    } else {  // zero the chunk's words; words shared by lanes are ORed
      unsigned long long epos = pe + (xe - nesc);
      if (a.esc && nesc) {
        for (int t = 0; t < cnt; ++t)
          if (a.sym[s0 + t] == 0) {
            if (epos < n_out) ocode[epos] = a.esc[s0 + t];
            ++epos;
          }
      }
      if ((lane & 3) == 0 && lane) a.splits[c * (kSplits - 1) + (lane >> 2) - 1] = (uint16_t)(xb - bits);
      for (unsigned w = lane; w < W; w += 32) cw[w] = 0u;
      __syncwarp();
      const unsigned bit0 = xb - bits;
      unsigned off = bit0 & 31u, cur = 0;
      unsigned* wp = cw + (bit0 >> 5);
      bool head = off != 0u;  // the first word holds other lanes' bits
      for (int t = 0; t < cnt; ++t) {
        const unsigned s = CLAMP ? min((unsigned)a.sym[s0 + t], dmax) : (unsigned)a.sym[s0 + t];
        const unsigned ent = tab.entry(s), L = tab.bits(ent), tc = tab.code(ent, L);
        cur |= tc >> off;
        off += L;
        if (off >= 32u) {
          off -= 32u;
          if (head) atomicOr(wp, cur);
          else *wp = cur;
          head = false;
          ++wp;
          cur = __funnelshift_lc(0u, tc, L - off);
        }
      }
      if (off) atomicOr(wp, cur);
    }
  }
}

// One table: returns at once unless the codebook picked it.
template <int WARPS, bool CLAMP, int MODE>
__global__ void __launch_bounds__(WARPS * 32, 32 / WARPS) encode_fused_kernel(FusedEncodeArgs a) {
  const Scalars* sc = a.sc;
  if (sc->skip) return;  // the stream is already known to be a raw copy
  if (CLAMP) {
    if ((a.dict <= kEncWinSmall && sc->max_len <= kPackLen) != (MODE == 0)) return;
  } else if ((unsigned)MODE != sc->enc_mode) {
    return;
  }
  encode_tiles<WARPS, CLAMP, MODE>(a);
}

// Any codebook, a stream of at most kEncSmallChunks chunks per SM: the table
// stays in global memory (and what the symbols meet of it in L1), as a CTA
// codes too few symbols to pay for a copy of it, and a CTA of eight warps
// takes 8.5 KB of shared memory, so that the items of a batch share an
// SM.  In place of the three launches above, two of which return at once (but
// wait for an SM with 200 KB of free shared memory to do so): 64 uneven fields
// in a batch 4.60 ms against 4.45, 65^3 0.195 ms against 0.176; with the
// tables copied by one kernel of any mode 5.57 and 0.181.  (CLAMP: Huffman
// encoding of 65,536 caller's symbols with a dictionary of 65,536 took 162 us
// with the two launches of launch_encode_clamped against 137.)
constexpr int kEncSmallChunks = 8;
constexpr size_t kEncSmallSmem = enc_smem<5>(8, 0, 0);
template <bool CLAMP>
__global__ void __launch_bounds__(256) encode_small_kernel(FusedEncodeArgs a) {
  if (a.sc->skip) return;  // the stream is already known to be a raw copy
  if (a.sc->max_len <= kPackLen) encode_tiles<8, CLAMP, 4>(a);
  else encode_tiles<8, CLAMP, 5>(a);
}
__device__ __forceinline__ void encode_finish(unsigned long long raw_total, unsigned long long capacity, Scalars* sc) {
  if (sc->skip) return;  // already raw
  const unsigned long long total = sc->off_bits + pad8(4ull * sc->n_words);
  sc->total = total;
  if (sc->esc_seen != sc->n_outliers) atomicOr(&sc->status, ST_CORRUPT | ST_RAW);
  if (total >= raw_total || total > capacity || (sc->status & ST_OVERFLOW)) atomicOr(&sc->status, ST_RAW);
}
__global__ void encode_finish_kernel(unsigned long long raw_total, unsigned long long capacity, Scalars* sc) {
  if (threadIdx.x == 0 && blockIdx.x == 0) encode_finish(raw_total, capacity, sc);
}

// ---------------------------------------------------------------------------
// Decoding
// ---------------------------------------------------------------------------
// Shared memory of the decoder-table builder: the codebook section as it
// stands in the stream (when it fits), a code length per dictionary symbol
// and the counting pass's counts.
constexpr int kDtStage = 128 * 1024;
struct DtSmem {
  unsigned stage[kDtStage / 4];
  uint8_t len[kMaxDict];
  unsigned wcnt[(kMaxLen + 1) * 32];
  CanonTables ct;
  unsigned rfirst[512], rcount[512], roff[512];
};
static_assert(sizeof(DtSmem) <= 227 * 1024, "decoder tables' shared memory");

// The run headers of a staged section side by side, for more than kDtWalkRuns
// runs: a header says where the next one stands, so 256 threads first note for
// every word of their segment where a chain of headers through it leaves the
// segment (in the lengths' memory, u16 offsets past the segment's end, 0xFFFF:
// the chain ends inside); one thread then hops from segment to segment, and
// every segment's runs are checked and spread from its entry.  Bound by
// latency: the 256 hops and a segment's words.  The serial walk took about 45
// ns a run: the tables of 59x40x147 at 2e-5 0.209 ms against 0.093, of 40x30x33
// at 3e-4 0.217 against 0.074, of 513^3 at 1e-3 (593 runs) 0.077 against 0.05.
constexpr unsigned kDtWalkRuns = 512, kDtSegs = 256, kDtLongRun = 256;
__device__ __forceinline__ void walk_runs_parallel(DtSmem& S, unsigned long long nbytes, unsigned long long n_runs,
                                                   unsigned dict, unsigned* s_bad, unsigned* s_nlong, unsigned* s_end) {
  const unsigned* st = S.stage;
  const uint8_t* bytes = reinterpret_cast<const uint8_t*>(S.stage);
  uint16_t* ex = reinterpret_cast<uint16_t*>(S.len);
  static_assert(sizeof(S.len) >= 2 * (kDtStage / 4), "an exit per staged word");
  const unsigned nw = (unsigned)(nbytes / 4), seg = (nw + kDtSegs - 1) / kDtSegs;
  const unsigned b = min(nw, threadIdx.x * seg), e = min(nw, b + seg);
  const bool mine = threadIdx.x < kDtSegs;
  if (mine) {
    for (unsigned p = e; p-- > b;) {
      unsigned v = 0xFFFFu;
      if (p + 2 <= nw && st[p + 1] <= dict) {
        const unsigned nx = p + 2u + ((st[p + 1] + 3u) >> 2);
        v = nx < e ? ex[nx] : nx - e;  // nx - e: at most 2 + dict / 4
      }
      ex[p] = (uint16_t)v;
    }
    S.roff[threadIdx.x] = ~0u;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    *s_nlong = 0;
    for (unsigned pos = 0; pos < nw;) {
      const unsigned q = pos / seg, v = ex[pos];
      S.roff[q] = pos;
      if (v == 0xFFFFu) break;
      pos = min(nw, (q + 1) * seg) + v;
    }
  }
  __syncthreads();
  const unsigned entry = mine ? S.roff[threadIdx.x] : ~0u;
  unsigned k = 0;  // the segment's runs
  if (entry != ~0u)
    for (unsigned p = entry; p < e && p + 2 <= nw && st[p + 1] <= dict; p += 2u + ((st[p + 1] + 3u) >> 2)) ++k;
  for (int i = threadIdx.x; i < kMaxDict / 4; i += blockDim.x) reinterpret_cast<unsigned*>(S.len)[i] = 0u;
  unsigned* const tot = &S.wcnt[(kMaxLen + 1) * 32 - 1];
  const unsigned base = block_excl_scan(k, S.wcnt, tot);
  __syncthreads();
  bool bad = *tot < n_runs;
  __syncthreads();  // the scan's memory holds the long runs from here on
  unsigned prev = 0;
  if (mine) {
    S.rfirst[threadIdx.x] = ~0u;
    const unsigned nr = base >= n_runs ? 0u : (unsigned)min((unsigned long long)k, n_runs - base);
    unsigned p = entry;
    for (unsigned r = 0; r < nr; ++r) {
      const unsigned first = st[p], cnt = st[p + 1];
      if ((unsigned long long)first + cnt > (unsigned long long)dict || 4ull * p + 8 + cnt > nbytes ||
          (r && first < prev)) {
        bad = true;
        break;
      }
      if (r == 0) S.rfirst[threadIdx.x] = first;
      prev = first + cnt;
      if (cnt < kDtLongRun) {
        for (unsigned t = 0; t < cnt; ++t) {
          const uint8_t L = bytes[4 * p + 8 + t];
          bad |= L > kMaxLen;
          S.len[first + t] = L;
        }
      } else {  // at least 264 bytes of the section each
        S.wcnt[atomicAdd(s_nlong, 1u)] = p;
      }
      p += 2u + ((cnt + 3u) >> 2);
    }
    S.rcount[threadIdx.x] = prev;
    if (nr) atomicMax(s_end, prev);
  }
  static_assert(kDtStage / (kDtLongRun + 8) < (kMaxLen + 1) * 32, "the list of long runs");
  if (__syncthreads_or(bad)) {
    if (threadIdx.x == 0) *s_bad = 1;
    __syncthreads();
    return;
  }
  if (mine && S.rfirst[threadIdx.x] != ~0u) {  // ascending across the segments too
    int q = (int)threadIdx.x - 1;
    while (q >= 0 && S.rfirst[q] == ~0u) --q;
    bad = q >= 0 && S.rfirst[threadIdx.x] < S.rcount[q];
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
  for (unsigned q = wid; q < *s_nlong; q += warps) {
    const unsigned p = S.wcnt[q], first = st[p], cnt = st[p + 1];
    for (unsigned t = lane; t < cnt; t += 32) {
      const uint8_t L = bytes[4 * p + 8 + t];
      bad |= L > kMaxLen;
      S.len[first + t] = L;
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) *s_bad = 1;
  __syncthreads();
}

// Canonical order of a stream's codebook (one CTA of kCbThreads threads,
// DtSmem in its dynamic shared memory): the runs' lengths are spread over
// the dictionary in shared memory, and one counting pass places every
// symbol.  Bound by latency: the section's load, the serial walk over the run
// headers and the counting walk's 64 rows of 32 symbols per warp.  Keeping
// the lengths of more than 8192 present symbols in global scratch, with a
// binary search of the runs per length and the look-up table of the decoder
// filled here too, took 0.129 ms at 513^3, 1e-4 (65,532 present symbols)
// against 0.042, and 0.091 at 1e-3 (593 runs) against 0.040.
__device__ __forceinline__ void decode_tables_block(const uint8_t* runs, unsigned long long nbytes,
                                                    unsigned long long n_runs, int dict, DecodeTables* out,
                                                    Scalars* sc, unsigned char* smem_raw) {
  DtSmem& S = *reinterpret_cast<DtSmem*>(smem_raw);
  __shared__ unsigned s_bad, s_long, s_end;  // s_end: the end of the last run so far
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) {
    s_bad = 0;
    s_end = 0;
  }
  for (int i = threadIdx.x; i < kMaxDict / 4; i += blockDim.x) reinterpret_cast<unsigned*>(S.len)[i] = 0u;
  const uint8_t* rbase = runs;
  if (nbytes <= sizeof(S.stage) && (reinterpret_cast<uintptr_t>(runs) & 3) == 0) {
    const unsigned* src = reinterpret_cast<const unsigned*>(runs);
    const unsigned nwd = (unsigned)(nbytes / 4);
    for (unsigned i0 = threadIdx.x; i0 < nwd; i0 += 8 * blockDim.x) {  // eight loads in flight
      unsigned v[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) v[t] = i0 + t * blockDim.x < nwd ? src[i0 + t * blockDim.x] : 0u;
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (i0 + t * blockDim.x < nwd) S.stage[i0 + t * blockDim.x] = v[t];
    }
    uint8_t* kb = reinterpret_cast<uint8_t*>(S.stage);
    for (unsigned i = 4 * nwd + threadIdx.x; i < (unsigned)nbytes; i += blockDim.x) kb[i] = runs[i];
    rbase = kb;
  }
  __syncthreads();
  // walk the run headers (serial, 512 at a time), then spread the batch's
  // lengths: short runs a warp each, long ones by the whole block.  A fault is
  // collected in registers and the barrier's OR decides, so that all threads
  // leave the loop together.
  constexpr unsigned kLongRun = 1024;
  unsigned long long off = 0;
  const bool parallel = rbase != runs && n_runs > kDtWalkRuns;
  if (parallel) walk_runs_parallel(S, nbytes, n_runs, (unsigned)dict, &s_bad, &s_long, &s_end);
  for (unsigned long long rb = 0; rb < (parallel ? 0ull : n_runs); rb += 512) {
    const int nb = (int)min(512ull, n_runs - rb);
    bool bad = false;
    if (threadIdx.x == 0) {  // the chain of headers only: their checks follow in parallel
      bool ok = true;
      for (int q = 0; q < nb && ok; ++q) {
        ok = off + 8 <= nbytes;
        const unsigned cnt = ok ? *reinterpret_cast<const unsigned*>(rbase + off + 4) : 0u;
        S.roff[q] = (unsigned)off;
        ok &= cnt <= (unsigned)dict;
        off += 8ull + ((cnt + 3u) & ~3u);
      }
      bad = !ok;
      s_long = 0;
    }
    if (__syncthreads_or(bad)) {
      s_bad = 1;
      break;
    }
    if (threadIdx.x < (unsigned)nb) {
      const unsigned o = S.roff[threadIdx.x];
      const unsigned first = *reinterpret_cast<const unsigned*>(rbase + o);
      const unsigned cnt = *reinterpret_cast<const unsigned*>(rbase + o + 4);
      S.rfirst[threadIdx.x] = first;
      S.rcount[threadIdx.x] = cnt;
      S.roff[threadIdx.x] = o + 8u;
      if ((unsigned long long)first + cnt > (unsigned long long)dict || (unsigned long long)o + 8 + cnt > nbytes) bad = true;
      if (cnt >= kLongRun) s_long = 1;
    }
    __syncthreads();
    if (threadIdx.x < (unsigned)nb) {  // ascending, without overlap
      const unsigned end = threadIdx.x ? S.rfirst[threadIdx.x - 1] + S.rcount[threadIdx.x - 1] : s_end;
      if ((threadIdx.x || rb) && S.rfirst[threadIdx.x] < end) bad = true;
    }
    if (__syncthreads_or(bad)) {
      s_bad = 1;
      break;
    }
    if (threadIdx.x == 0) s_end = S.rfirst[nb - 1] + S.rcount[nb - 1];
    for (int q = wid; q < nb; q += nw)
      if (S.rcount[q] < kLongRun)
        for (unsigned t = lane; t < S.rcount[q]; t += 32) {
          const uint8_t L = rbase[S.roff[q] + t];
          bad |= L > kMaxLen;
          S.len[S.rfirst[q] + t] = L;
        }
    for (int q = 0; q < (s_long ? nb : 0); ++q)
      if (S.rcount[q] >= kLongRun)
        for (unsigned t = threadIdx.x; t < S.rcount[q]; t += blockDim.x) {
          const uint8_t L = rbase[S.roff[q] + t];
          bad |= L > kMaxLen;
          S.len[S.rfirst[q] + t] = L;
        }
    if (__syncthreads_or(bad)) {
      s_bad = 1;
      break;
    }
  }
  __syncthreads();
  if (!s_bad) {
    // symbols in half of the dictionary or less: counted between the first
    // run's first symbol and the last run's end (1,024 neighbouring ones of
    // 65,536: the kernel 10.4 us against 16.4); a wide span keeps the
    // dictionary's bound, a kernel argument (118 us against 126 by the span)
    const unsigned lo = n_runs ? *reinterpret_cast<const unsigned*>(rbase) : 0u, span = s_end - lo;
    if (2u * span <= (unsigned)dict) build_canonical(S.len + lo, (int)span, S.wcnt, out->canon, &S.ct, lo);
    else build_canonical(S.len, dict, S.wcnt, out->canon, &S.ct);
  }
  // the lengths must satisfy Kraft's inequality (in units of 2^-32)
  if (threadIdx.x == 0) {
    unsigned long long kr = 0;
    if (!s_bad)
      for (int L = 1; L <= kMaxLen; ++L) kr += (unsigned long long)S.ct.count[L] << (32 - L);
    if (s_bad || kr > (1ull << 32)) {
      S.ct.n = 0;  // no symbol can be decoded
      atomicOr(&sc->status, ST_CORRUPT);
    }
    out->ct = S.ct;
  }
}

struct DecodeArgs {
  const unsigned* words;               // bitstream
  unsigned long long n_words;
  const unsigned long long* word_off;  // [nch+1]
  const uint16_t* splits;              // [nch][7] bit offsets of runs 1..7
  unsigned long long nch;
  unsigned long long n;
  int chunk;
  const DecodeTables* tab;
  unsigned ncanon;                     // symbols staged in shared memory: a bound on the present symbols
  uint16_t* sym;
  Scalars* sc;
};

// One thread per run (an eighth of a chunk): table-driven canonical decoding.
// The thread's window is two words at a bit position (one funnel shift gives
// the next 32 bits); the words after them come from a private ring of eight
// words in shared memory (word-major: no bank conflicts), filled every fourth
// symbol at most with a 16-byte group loaded ahead of use, so a symbol's
// refill is a predicated move and a conflict-free load.  One shared-memory
// look-up gives a code's length and, for codes of at most kLutBits bits, the
// symbol; longer ones add their remaining bits to the prefix's canonical
// position and read the symbol there (predicated, off the chain from one code
// to the next); only the few prefixes of several lengths walk the
// left-justified last codes.  Sixteen
// symbols per step leave as one 32-byte sector.  A run must end exactly where
// the next one starts (the last run of a chunk within the chunk); reading past
// the chunk reads other bits or zeros and shows in that check.  Persistent
// CTAs: the look-up table is built in shared memory once per CTA.
// Bound by the latency and the rate of the shared-memory accesses (look-up,
// canonical symbol, ring: 7 wavefronts a symbol and warp, 38 % of the issue
// slots).  513^3 GRF, 1e-2 / 1e-3 / 1e-4 / 1e-5 (the last two with the outlier
// codes' pass): 0.290 / 0.291 / 0.538 / 0.846 ms; the kernel before it (a
// 64-bit window refilled by selects from a queue of registers, limits walked
// for every longer code, the canonical symbols in global memory, 512-thread
// CTAs) took 0.434 / 0.486 / 0.640 / 1.095.
constexpr int kDecThreads = 1024, kDecThreadsSmall = 256;
constexpr int kDecRing = 8;  // words of a thread's ring
constexpr unsigned kLutWalk = 63;  // length field of a prefix of several lengths
__host__ __device__ constexpr size_t dec_smem(int threads, unsigned ncanon) {
  return (size_t)threads * kDecRing * 4 + (4u << kLutBits) + 2 * 4 * (kMaxLen + 4) + 2 * (((size_t)ncanon + 7) / 8 * 8);
}
static_assert(dec_smem(kDecThreads, kMaxDict) <= 227 * 1024, "decoder shared memory");
__device__ __forceinline__ unsigned ld_shared_if(unsigned addr, bool pred, unsigned v) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q ld.shared.u32 %0, [%1];\n}\n"
               : "+r"(v)
               : "r"(addr), "r"((unsigned)pred));
  return v;
}
__device__ __forceinline__ unsigned ld_shared_u16_if(unsigned addr, bool pred, unsigned v) {
  asm volatile("{\n .reg .pred q;\n .reg .u16 h;\n setp.ne.u32 q, %2, 0;\n @q ld.shared.u16 h, [%1];\n @q cvt.u32.u16 %0, h;\n}\n"
               : "+r"(v)
               : "r"(addr), "r"((unsigned)pred));
  return v;
}
__device__ __forceinline__ void st_shared(unsigned addr, unsigned v) {
  asm volatile("st.shared.u32 [%0], %1;\n" ::"r"(addr), "r"(v));
}

template <int NT>
__global__ void __launch_bounds__(NT, NT == kDecThreads ? 1 : 2) decode_kernel(DecodeArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned* lut = reinterpret_cast<unsigned*>(smem_raw + (size_t)NT * kDecRing * 4);
  unsigned* last = lut + (1 << kLutBits);  // [kMaxLen + 4] left-justified last code of each length
  unsigned* base = last + kMaxLen + 4;     // [kMaxLen + 4] canonical position minus code
  uint16_t* canon = reinterpret_cast<uint16_t*>(base + kMaxLen + 4);
  const DecodeTables* T = a.tab;
  const unsigned nsym = min(T->ct.n, a.ncanon);
  {
    const uint4* src = reinterpret_cast<const uint4*>(T->canon);
    uint4* dst = reinterpret_cast<uint4*>(canon);
    const unsigned nv = (nsym + 7) / 8;
    for (unsigned i0 = threadIdx.x; i0 < nv; i0 += 4 * NT) {  // four loads in flight
      uint4 v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) v[t] = i0 + t * NT < nv ? src[i0 + t * NT] : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (i0 + t * NT < nv) dst[i0 + t * NT] = v[t];
    }
  }
  if (threadIdx.x == 0) last[kMaxLen + 1] = ~0u;
  if (threadIdx.x <= kMaxLen) {
    last[threadIdx.x] = (unsigned)(T->ct.limit[threadIdx.x] - 1ull);
    base[threadIdx.x] = T->ct.first_pos[threadIdx.x] - T->ct.first_code[threadIdx.x];
  }
  __shared__ unsigned s_minl;
  if (threadIdx.x == 0) s_minl = kMaxLen + 1;
  __syncthreads();
  if (threadIdx.x >= 1 && threadIdx.x <= kMaxLen && T->ct.count[threadIdx.x]) atomicMin(&s_minl, threadIdx.x);
  __syncthreads();
  // the look-up table: length << 16 | the symbol of a code of at most kLutBits
  // bits, or, for a prefix whose codes all have one longer length, the
  // canonical position of the first of them; kLutWalk << 16 | the length of
  // the first code for a prefix of several lengths (kMaxLen + 1: no code has
  // the prefix).  The last codes ascend with the length from the shortest one
  // on, and a thread's prefixes ascend, so its length only moves up (to the
  // sentinel past kMaxLen at most): a stream of one chunk takes 15.8 us, with a
  // binary search per prefix 32.2.  Positions are checked here, so that the
  // walk below takes them as they are (tables of a corrupt codebook).
  int l0 = (int)s_minl;
  unsigned lim = last[l0], off = l0 <= kMaxLen ? base[l0] : 0u;
  for (int p0 = threadIdx.x; p0 < (1 << kLutBits); p0 += 4 * NT) {
    unsigned e[4], at[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const unsigned pf = (unsigned)(p0 + t * NT) << (32 - kLutBits), pl = pf | ((1u << (32 - kLutBits)) - 1u);
      while (pf > lim) {
        lim = last[++l0];
        off = l0 <= kMaxLen ? base[l0] : 0u;
      }
      e[t] = (kLutWalk << 16) | (unsigned)l0;
      at[t] = ~0u;
      if (l0 <= kMaxLen && pl <= lim) {
        const unsigned i0 = (pf >> (32 - l0)) + off, i1 = (pl >> (32 - l0)) + off;
        if (i0 <= i1 && i1 < nsym) {
          e[t] = ((unsigned)l0 << 16) | (l0 <= kLutBits ? 0u : i0);
          at[t] = l0 <= kLutBits ? i0 : ~0u;
        }
      }
    }
    unsigned v[4];  // four symbols in flight
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] = at[t] != ~0u ? (unsigned)canon[at[t]] : 0u;
#pragma unroll
    for (int t = 0; t < 4; ++t) lut[p0 + t * NT] = e[t] | v[t];
  }
  static_assert((1 << kLutBits) % (4 * NT) == 0, "whole groups of four prefixes");
  __syncthreads();
  const unsigned ring = smem_u32(smem_raw) + 4u * threadIdx.x, canon_s = smem_u32(canon);
  constexpr unsigned kRow = 4u * NT, kMask = kRow * kDecRing - 1u;
  const unsigned* const wall = a.words + a.n_words;
  const unsigned long long nruns = a.nch * kSplits;
  const int sub = a.chunk / kSplits;
  for (unsigned long long r = blockIdx.x * (unsigned long long)NT + threadIdx.x; r < nruns;
       r += (unsigned long long)gridDim.x * NT) {
    const unsigned long long c = r / kSplits;
    const int k = (int)(r % kSplits);
    const unsigned long long cw0 = a.word_off[c], cw1 = a.word_off[c + 1];
    if (cw1 < cw0 || cw1 > a.n_words) { atomicOr(&a.sc->status, ST_CORRUPT); continue; }
    const unsigned long long cbits = (cw1 - cw0) * 32ull;
    const unsigned long long b0 = k ? a.splits[c * (kSplits - 1) + k - 1] : 0ull;
    const unsigned long long b1 = k < kSplits - 1 ? a.splits[c * (kSplits - 1) + k] : cbits;
    if (b0 > b1 || b1 > cbits) { atomicOr(&a.sc->status, ST_CORRUPT); continue; }
    const unsigned long long s0 = c * (unsigned long long)a.chunk + (unsigned long long)k * sub;
    const int cnt = (int)(min(a.n, s0 + (unsigned long long)sub) - s0);
    // words past the bitstream read zeros; words past a chunk's end are never
    // consumed by a valid run and show in the check below
    auto ld = [&](const unsigned* q) { return q < wall ? __ldg(q) : 0u; };
    auto ld4 = [&](const unsigned* g) {
      if (g + 4 <= wall) return __ldg(reinterpret_cast<const uint4*>(g));
      return make_uint4(ld(g), ld(g + 1), ld(g + 2), ld(g + 3));
    };
    const unsigned* gp = a.words + cw0 + (b0 >> 5);
    unsigned hi = ld(gp), lo = ld(gp + 1);
    gp += 2;
    const unsigned m = (unsigned)((reinterpret_cast<uintptr_t>(gp) >> 2) & 3);
    const unsigned* gq = gp - m;  // 16-byte aligned; ring rows 0..3 hold its words, the m first not part of the run
    auto push = [&](const uint4& v, unsigned row) {
      st_shared(ring + row, v.x);
      st_shared(ring + row + kRow, v.y);
      st_shared(ring + row + 2 * kRow, v.z);
      st_shared(ring + row + 3 * kRow, v.w);
    };
    push(ld4(gq), 0u);
    push(ld4(gq + 4), 4u * kRow);
    uint4 next = ld4(gq + 8);
    gq += 12;
    unsigned rp = m * kRow, wrow = 0u;  // ring offsets of the next read and of the next group
    unsigned nx = ld_shared_if(ring + rp, true, 0u);
    rp += kRow;
    int wend = 10 - (int)m;  // words of the run before this one are loaded or in the ring
    const unsigned pos0 = (unsigned)(b0 & 31);
    unsigned pos = pos0;  // bits from the run's first word
    const unsigned end = pos0 + (unsigned)min(b1 - b0, 0x7FFFFFFFull);  // where the run must end (at most, a chunk's last)
    bool bad = false;
    // before a symbol: words [pos / 32, + 2] of the run are hi, lo, nx, and the
    // ring holds those up to wend; a symbol moves on by one word at most
    auto refill = [&](int need) {
      if (wend - 3 - (int)(pos >> 5) < need) {
        push(next, wrow);
        wrow ^= 4u * kRow;
        wend += 4;
        next = ld4(gq);
        gq += 4;
      }
    };
    auto one = [&]() -> unsigned {
      const unsigned peek = __funnelshift_l(lo, hi, pos);
      unsigned e = lut[peek >> (32 - kLutBits)];
      unsigned L = e >> 16;
      const bool longer = L > (unsigned)kLutBits;
      unsigned idx = (e & 0xFFFFu) + ((peek << kLutBits) >> ((32 + kLutBits - L) & 31u));
      if (L == kLutWalk) {  // a prefix of several lengths
        L = e & 0xFFFFu;
        while (peek > last[L]) ++L;  // ends at the sentinel past kMaxLen
        idx = L <= (unsigned)kMaxLen ? (peek >> (32 - L)) + base[L] : nsym;
        if (idx >= nsym) {
          bad = true;
          L = 1;
          idx = 0;
        }
      }
      e = ld_shared_u16_if(canon_s + 2u * idx, longer, e);
      const unsigned np = pos + L;
      const bool cross = ((np ^ pos) & 32u) != 0u;
      pos = np;
      hi = cross ? lo : hi;
      lo = cross ? nx : lo;
      nx = ld_shared_if(ring + rp, cross, nx);
      rp = cross ? (rp + kRow) & kMask : rp;
      return e;
    };
    uint16_t* out = a.sym + s0;
    int i = 0;
    // Runs start on 8 bytes (a run is a multiple of four symbols), on a whole
    // sector where it is a multiple of sixteen: all lanes decode alike and only
    // the stores differ.  (Runs between sectors one symbol at a time beside the
    // others: chunks of 992 symbols, 20 M in all: 239 us against 61.)
    if ((reinterpret_cast<uintptr_t>(a.sym) & 31) == 0 && (a.chunk & 31) == 0) {
      auto pair = [&] {
        const unsigned e0 = one(), e1 = one();
        return __byte_perm(e0, e1, 0x5410);
      };
      for (; i + 16 <= cnt; i += 16) {
        unsigned v[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          if ((t & 1) == 0) refill(4);  // four symbols consume four words at most
          v[t] = pair();
        }
        if ((a.chunk & 127) == 0) {
          uint4* o = reinterpret_cast<uint4*>(out + i);
          o[0] = make_uint4(v[0], v[1], v[2], v[3]);
          o[1] = make_uint4(v[4], v[5], v[6], v[7]);
        } else {
          uint2* o = reinterpret_cast<uint2*>(out + i);
#pragma unroll
          for (int t = 0; t < 4; ++t) o[t] = make_uint2(v[2 * t], v[2 * t + 1]);
        }
      }
      for (; i + 4 <= cnt; i += 4) {
        refill(4);
        const unsigned v0 = pair(), v1 = pair();
        *reinterpret_cast<uint2*>(out + i) = make_uint2(v0, v1);
      }
    }
    for (; i < cnt; ++i) {
      refill(1);
      out[i] = (uint16_t)one();
    }
    if (bad || (k < kSplits - 1 ? pos != end : pos > end)) atomicOr(&a.sc->status, ST_CORRUPT);
  }
}

constexpr int kEncGroups = 8;  // a lane's slice: up to 8 groups of 8 symbols (chunk <= 2048)

__device__ __forceinline__ unsigned sym_of(const uint4* q, int i) {
  const unsigned w = (i & 4) ? ((i & 2) ? q[i >> 3].w : q[i >> 3].z) : ((i & 2) ? q[i >> 3].y : q[i >> 3].x);
  return (i & 1) ? (w >> 16) : (w & 0xFFFFu);
}

// Escaped symbols (symbol 0) take the outlier codes in stream order: one
// warp per chunk, each lane a slice of chunk/32 (<= 64) symbols read as 16-byte
// vectors when the slices allow it; a lane's escapes are a 64-bit mask.
__global__ void __launch_bounds__(256) escape_fixup_kernel(const uint16_t* sym, unsigned long long n, int chunk,
                                                           unsigned long long nch, const unsigned long long* esc_off,
                                                           const int32_t* ocode, unsigned long long n_out,
                                                           int32_t* esc, Scalars* sc) {
  const int lane = threadIdx.x & 31;
  const int per = chunk / 32;
  const int G = per / 8;
  for (unsigned long long c = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) / 32; c < nch;
       c += (unsigned long long)gridDim.x * blockDim.x / 32) {
    const unsigned long long cb = c * (unsigned long long)chunk;
    const unsigned long long s0 = min(n, cb + (unsigned long long)lane * per), s1 = min(n, s0 + per);
    const int cnt = (int)(s1 - s0);
    const bool vec = __all_sync(0xffffffffu, (per & 7) == 0 && cnt == per && (s0 & 7ull) == 0);
    unsigned long long m = 0;
    if (vec) {
      const uint4* p = reinterpret_cast<const uint4*>(sym + s0);
      uint4 q[kEncGroups];
#pragma unroll
      for (int g = 0; g < kEncGroups; ++g) q[g] = g < G ? __ldg(p + g) : make_uint4(1u, 1u, 1u, 1u);
#pragma unroll
      for (int i = 0; i < 8 * kEncGroups; ++i)
        if ((i >> 3) < G) m |= (unsigned long long)(sym_of(q, i) == 0) << i;
    } else {
      for (int t = 0; t < cnt; ++t) m |= (unsigned long long)(sym[s0 + t] == 0) << t;
    }
    const unsigned ne = __popcll(m);
    unsigned x = ne;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    const unsigned total = __shfl_sync(0xffffffffu, x, 31);
    const unsigned long long e0 = esc_off[c], e1 = esc_off[c + 1];
    if (e0 + total != e1 || e1 > n_out) {  // the outlier reads stay inside the outlier section
      if (lane == 0) atomicOr(&sc->status, ST_CORRUPT);
      continue;
    }
    unsigned long long e = e0 + (x - ne);
    if (vec && (reinterpret_cast<uintptr_t>(esc + s0) & 15) == 0) {
      // groups of four positions: one 16-byte store for each group holding an
      // escape (entries of the other positions are never read)
      int4* e4 = reinterpret_cast<int4*>(esc + s0);
      for (int g = 0; g < per / 4 && m; ++g) {
        const unsigned bits = (unsigned)(m >> (4 * g)) & 15u;
        if (!bits) continue;
        int v[4];
        unsigned r = 0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const bool on = (bits >> t) & 1u;
          v[t] = on ? __ldg(ocode + e + r) : 0;
          r += on;
        }
        e4[g] = make_int4(v[0], v[1], v[2], v[3]);
        e += r;
      }
    } else {
      while (m) {
        int idx[4];
        int k = 0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          idx[t] = m ? __ffsll((long long)m) - 1 : -1;
          m &= m ? m - 1 : 0ull;
          k += idx[t] >= 0;
        }
        int32_t v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) v[t] = idx[t] >= 0 ? __ldg(ocode + e + t) : 0;
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (idx[t] >= 0) esc[s0 + idx[t]] = v[t];
        e += k;
      }
    }
  }
}

__global__ void codes_from_symbols_kernel(const uint16_t* sym, const int32_t* esc, unsigned long long n, int radius,
                                          int32_t* out) {
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned s = sym[i];
    out[i] = s ? (int)s - radius : esc[i];
  }
}

}  // namespace bm
