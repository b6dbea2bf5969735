// In-cache Block kernels of coded double fields (MODE 0), which the
// double-precision unit bounds: it runs at two lanes a clock and SM, 16 cycles
// a warp's multiply-add and as much or more for an addition, a comparison or a
// conversion.  The lines of the first and last passes are taken by parity
// class, so that a line computes only what its class needs (all-coarse lines
// interpolate from their own values, one-odd lines from two neighbours, and the
// all-coarse nodes' zero coefficients are left out of the restriction), and the
// quantiser's range check, floor and conversions are integer arithmetic
// (bm_common.cuh).  Per 9^3 block 293 instead of 480 warp instructions of that
// unit.  385x385x257, B = 9, K = 2: forward 1.55 -> 1.04 ms, inverse 1.48 ->
// 1.22.  (Single precision keeps the general expression for every line: the
// classes' lines, every other one of every other plane, share shared-memory
// banks, and the same split took 0.494 against 0.446 ms forward and 0.701
// against 0.558 inverse at 513^3, B = 17.)
#pragma once

namespace bm {

// Blocks a CTA takes at once: the lines of four 9-node blocks fill the warps of
// each parity class (100, 160 and 64 lines; one block has 25, 40 and 16).
constexpr int block_group(int B) { return B == 9 ? 4 : 1; }

template <int B, int K>
struct GroupCfg {
  using Cfg = BlockCfg<double, B, K>;
  static constexpr int NB = block_group(B);
  static constexpr int NT_FWD = NB > 1 ? 192 : Cfg::NT_FWD, NT_INV = NB > 1 ? 192 : Cfg::NT_INV;
  static constexpr size_t fwd_stage_off = Cfg::up16(sizeof(double) * NB * (Cfg::A + Cfg::T1 + Cfg::CB0 + Cfg::CB1));
  static constexpr size_t fwd_smem = fwd_stage_off + Cfg::up16(2 * Cfg::PB * NB);
  static constexpr size_t inv_stage_off =
      Cfg::up16(sizeof(double) * NB * (Cfg::A + Cfg::T1 + Cfg::T2 + Cfg::CB0 + Cfg::CB1));
  static constexpr size_t inv_smem = inv_stage_off + Cfg::up16(4 * Cfg::PB * NB);
  static constexpr int fit(size_t bytes) {
    const int f = (int)((228u * 1024u) / (bytes + 1024u));
    return f < 1 ? 1 : f < 4 ? f : 4;
  }
  static constexpr int FWD_MIN_CTAS = fit(fwd_smem), INV_MIN_CTAS = fit(inv_smem);
};

// ---------------------------------------------------------------------------
// Lines of the first pass by parity class.  Line (i0, i1) of a level of N
// nodes is all-coarse (both indices even: its even nodes have no coefficient,
// and it interpolates from its own values), one-odd (from two neighbouring
// lines) or both-odd (from four).  Each class of NB blocks starts on a warp
// boundary, so a warp runs one class's code; the longest comes first.
// ---------------------------------------------------------------------------
template <int N, int NB>
struct Lines {
  static constexpr int C = (N + 1) / 2, H = (N - 1) / 2;
  static constexpr int up(int x) { return (x + 31) / 32 * 32; }
  static constexpr int n_both = NB * H * H, n_one = NB * 2 * H * C, n_cc = NB * C * C;
  static constexpr int s_one = up(n_both), s_cc = s_one + up(n_one), total = s_cc + n_cc;
  // Class of item `it` (2 both odd, 1 one odd, 0 all coarse; -1 none), its
  // block and its line.
  __device__ __forceinline__ static int of(int it, int& blk, int& i0, int& i1) {
    if (it < s_one) {
      blk = it / (H * H);
      const int q = it - blk * (H * H);
      i0 = 2 * (q / H) + 1;
      i1 = 2 * (q - q / H * H) + 1;
      return it < n_both ? 2 : -1;
    }
    if (it < s_cc) {
      const int k = it - s_one;
      blk = k / (2 * H * C);
      int q = k - blk * (2 * H * C);
      if (q < H * C) {
        i0 = 2 * (q / C) + 1;
        i1 = 2 * (q - q / C * C);
      } else {
        q -= H * C;
        i0 = 2 * (q / H);
        i1 = 2 * (q - q / H * H) + 1;
      }
      return k < n_one ? 1 : -1;
    }
    const int k = it - s_cc;
    blk = k / (C * C);
    const int q = k - blk * (C * C);
    i0 = 2 * (q / C);
    i1 = 2 * (q - q / C * C);
    return 0;
  }
};
// The quantisation codes of a line (all its nodes, or the odd ones of an
// all-coarse line), staged as in level_fwd.
template <int N, bool CC>
__device__ __forceinline__ void stage_line(const double (&d)[N], const double rq, const int base, uint16_t* stage,
                                           int32_t* esc_blk, bool& ovf, const bool full) {
  const unsigned sadd = full ? 1u : 0u, swide = full ? 0u : kStageWide;
  int codes[N];
  bool anyw = false;
#pragma unroll
  for (int k = CC ? 1 : 0; k < N; k += CC ? 2 : 1) {
    const int code = quantize(d[k], rq, ovf);
    const unsigned b = (unsigned)(code + kStageBias);
    const bool wide = b >= kStageWide;
    stage[base + (CC ? k / 2 : k)] = (uint16_t)(wide ? swide : b + sadd);
    codes[k] = code;
    anyw |= wide;
  }
  if (anyw) {
#pragma unroll
    for (int k = CC ? 1 : 0; k < N; k += CC ? 2 : 1) esc_blk[base + (CC ? k / 2 : k)] = codes[k];
  }
}

// First position of line (i0, i1) among a level's coefficients of one block.
template <int N>
__device__ __forceinline__ int line_base(int i0, int i1) {
  constexpr int C = (N + 1) / 2;
  const bool f0 = i0 & 1;
  return (i0 * N + i1) * N - (((i0 + 1) / 2) * C + (f0 ? 0 : (i1 + 1) / 2)) * C;
}

// Sums of the coarse values a line interpolates from, one per coarse node
// (the tensor-product interpolant is 1/2 of the sum for a one-odd line and
// 1/4 for a both-odd one: scalings by powers of two, folded exactly into the
// multiply-adds that use them).  row: distance of neighbouring lines, st:
// distance of coarse nodes in a line.
template <int C, int CLS>
__device__ __forceinline__ void coarse_sums(const double* r00, const double* r01, const double* r10, const double* r11,
                                            const int st, double (&v)[C]) {
#pragma unroll
  for (int J = 0; J < C; ++J) {
    if (CLS == 2) v[J] = (r00[st * J] + r01[st * J]) + (r10[st * J] + r11[st * J]);
    else if (CLS == 1) v[J] = r00[st * J] + r11[st * J];
    else v[J] = r00[st * J];
  }
}

// One line of the first forward pass: coefficients d = u - I(u|C), staged,
// then the restriction and solve along the line into T1.  The values are those
// of the general expression of level_fwd (field_huge excludes the fields whose
// sums could overflow here first).
template <int N, int CLS>
__device__ __forceinline__ void fwd_line(const double* X, double* T1, double* out, const int i0,
                                         const int i1, const int lvl_off, const double rq, uint16_t* stage,
                                         int32_t* esc_blk, bool& ovf, const bool full) {
  constexpr int C = (N + 1) / 2;
  const double* x = X + (i0 * N + i1) * N;
  const int lo0 = CLS && (i0 & 1) ? i0 - 1 : i0, hi0 = CLS && (i0 & 1) ? i0 + 1 : i0;
  const int lo1 = CLS && (i1 & 1) ? i1 - 1 : i1, hi1 = CLS && (i1 & 1) ? i1 + 1 : i1;
  double v[C];
  coarse_sums<C, CLS>(X + (lo0 * N + lo1) * N, X + (lo0 * N + hi1) * N, X + (hi0 * N + lo1) * N,
                         X + (hi0 * N + hi1) * N, 2, v);
  constexpr double se = CLS == 2 ? 0.25 : CLS == 1 ? 0.5 : 1.0;
  double d[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if (k & 1) d[k] = fma(-0.5 * se, v[k / 2] + v[k / 2 + 1], x[k]);
    else if (CLS) d[k] = fma(-se, v[k / 2], x[k]);
    else d[k] = 0.0;
  }
  if (CLS == 0) {  // u|C of this line: the start of the coarse values (the third pass adds z)
#pragma unroll
    for (int J = 0; J < C; ++J) out[((i0 / 2) * C + i1 / 2) * C + J] = v[J];
  }
  stage_line<N, CLS == 0>(d, rq, lvl_off + line_base<N>(i0, i1), stage, esc_blk, ovf, full);
  double z[C];
  restrict_solve<double, N, CLS == 0>(block_tab<double, N>(), d, z);
#pragma unroll
  for (int j = 0; j < C; ++j) T1[(i0 * C + j) * N + i1] = z[j];
}

// Second and third restriction passes of a level over NB blocks (array
// strides t1s, t2s, os): T1 -> T2 along dimension 1, T2 along dimension 0 added
// to (SIGN 1) or subtracted from (SIGN -1) the coarse values.
template <int N, int NB, int SIGN>
__device__ __forceinline__ void restrict_passes(const double* T1, const int t1s, double* T2,
                                                const int t2s, double* out, const int os) {
  constexpr int C = (N + 1) / 2;
  const auto& tb = block_tab<double, N>();
  for (int I = threadIdx.x; I < NB * N * C; I += blockDim.x) {
    const int blk = NB > 1 ? I / (N * C) : 0, L = I - blk * (N * C);  // L = i0*C + j2
    const int i0 = L / C, j2 = L - i0 * C;
    double d[N];
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = T1[blk * t1s + L * N + i];
    double z[C];
    restrict_solve<double, N>(tb, d, z);
#pragma unroll
    for (int j = 0; j < C; ++j) T2[blk * t2s + (j * C + j2) * N + i0] = z[j];
  }
  __syncthreads();
  for (int I = threadIdx.x; I < NB * C * C; I += blockDim.x) {
    const int blk = NB > 1 ? I / (C * C) : 0, L = I - blk * (C * C);  // L = j1*C + j2
    const int j1 = L / C, j2 = L - j1 * C;
    double d[N];
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = T2[blk * t2s + L * N + i];
    double z[C];
    restrict_solve<double, N>(tb, d, z);
#pragma unroll
    for (int J = 0; J < C; ++J) {
      double* o = out + blk * os + (J * C + j1) * C + j2;
      *o = SIGN > 0 ? *o + z[J] : *o - z[J];
    }
  }
  __syncthreads();
}

// Elements of level output j's buffer (the stride between a group's blocks).
template <int B>
constexpr int lvl_stride(int j) {
  return j == 0 ? cube(B) : (j & 1) ? cube((B + 1) / 2) : cube(((B + 1) / 2 + 1) / 2);
}

// Whether a field holds values of 2^960 or more: its lines then take the
// general expression, whose infinities make the stream raw.  A both-odd line
// adds eight values before it scales them, the general expression four, so the
// two part ways from values of 2^1021 on; a level's coarse values are at most
// 55 times its input's largest one (|z| <= 3^3 times the coefficients, which are
// at most twice the values), so no level of a smaller field comes near.
__device__ __forceinline__ bool field_huge(const Scalars* sc) {
  return __ldcg(&sc->maxabs_bits) >= 0x7BF0000000000000ull;  // 2^960
}

// ---------------------------------------------------------------------------
// Forward level of the first nv of NB blocks (array strides xs, t1s, os, ps;
// quantiser widths rq[blk * rqs]).  Levels below nine nodes have too few lines
// per class to fill warps, and a field of huge values takes the general
// expression for its overflows: there every line computes it.
// ---------------------------------------------------------------------------
template <int N, int NB>
__device__ __forceinline__ void group_level_fwd(double* X, const int xs, double* T1, const int t1s, double* out,
                                                const int os, const int lvl_off, const double* rq, const int rqs, uint16_t* stage,
                                                const int ps, int32_t* esc_blk, bool& ovf, const bool full,
                                                const bool huge, const int nv) {
  constexpr int C = (N + 1) / 2;
  if (N >= 9 && !huge) {
    using LN = Lines<N, NB>;
    for (int it = threadIdx.x; it < LN::total; it += blockDim.x) {
      int blk, i0, i1;
      const int cls = LN::of(it, blk, i0, i1);
      if (cls < 0 || blk >= nv) continue;
      double* x = X + blk * xs;
      double* t1 = T1 + blk * t1s;
      double* o = out + blk * os;
      const double q = rq[blk * rqs];
      if (cls == 2) fwd_line<N, 2>(x, t1, o, i0, i1, lvl_off, q, stage + blk * ps, esc_blk + blk * ps, ovf, full);
      else if (cls == 1) fwd_line<N, 1>(x, t1, o, i0, i1, lvl_off, q, stage + blk * ps, esc_blk + blk * ps, ovf, full);
      else fwd_line<N, 0>(x, t1, o, i0, i1, lvl_off, q, stage + blk * ps, esc_blk + blk * ps, ovf, full);
    }
  } else {
#pragma unroll 1
    for (int I = threadIdx.x; I < NB * N * N; I += blockDim.x) {
      const int blk = I / (N * N), L = I - blk * (N * N);
      if (blk >= nv) continue;
      const double* x = X + blk * xs;
      const int i0 = L / N, i1 = L - i0 * N;
      const bool f0 = i0 & 1, f1 = i1 & 1;
      const int lo0 = f0 ? i0 - 1 : i0, hi0 = f0 ? i0 + 1 : i0;
      const int lo1 = f1 ? i1 - 1 : i1, hi1 = f1 ? i1 + 1 : i1;
      const double* r00 = x + (lo0 * N + lo1) * N;
      const double* r01 = x + (lo0 * N + hi1) * N;
      const double* r10 = x + (hi0 * N + lo1) * N;
      const double* r11 = x + (hi0 * N + hi1) * N;
      double w[C];
#pragma unroll
      for (int J = 0; J < C; ++J) w[J] = 0.25 * ((r00[2 * J] + r01[2 * J]) + (r10[2 * J] + r11[2 * J]));
      double d[N];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const double e = (k & 1) ? 0.5 * (w[k / 2] + w[k / 2 + 1]) : w[k / 2];
        d[k] = x[L * N + k] - e;
      }
      const bool cc = !f0 && !f1;
      if (cc) {  // u|C of this line: the start of the coarse values (the third pass adds z)
#pragma unroll
        for (int J = 0; J < C; ++J) out[blk * os + ((i0 / 2) * C + i1 / 2) * C + J] = x[L * N + 2 * J];
      }
      const int base = lvl_off + line_base<N>(i0, i1);
      if (cc) stage_line<N, true>(d, rq[blk * rqs], base, stage + blk * ps, esc_blk + blk * ps, ovf, full);
      else stage_line<N, false>(d, rq[blk * rqs], base, stage + blk * ps, esc_blk + blk * ps, ovf, full);
      double z[C];
      restrict_solve<double, N>(block_tab<double, N>(), d, z);
#pragma unroll
      for (int j = 0; j < C; ++j) T1[blk * t1s + (i0 * C + j) * N + i1] = z[j];
    }
  }
  __syncthreads();
  restrict_passes<N, NB, 1>(T1, t1s, X, xs, out, os);  // T2 takes the place of the level's input
}

template <int N, int L, int K, int B>
struct GroupFwdLevels {
  __device__ __forceinline__ static void run(const LevelBufs<double>& bufs, double* T1, const double* rq,
                                             uint16_t* stage, int32_t* esc_blk, bool& ovf, const bool full,
                                             const bool huge, const int nv) {
    using Cfg = BlockCfg<double, B, K>;
    group_level_fwd<N, block_group(B)>(bufs(L), lvl_stride<B>(L), T1, Cfg::T1, bufs(L + 1),
                                               lvl_stride<B>(L + 1), lvl_offset(B, L), rq + L, K, stage, Cfg::PB,
                                               esc_blk, ovf, full, huge, nv);
    if constexpr (L + 1 < K)
      GroupFwdLevels<(N + 1) / 2, L + 1, K, B>::run(bufs, T1, rq, stage, esc_blk, ovf, full, huge, nv);
  }
};

// A group of blocks (nv of the NB consecutive ones from b on) of the forward
// pass: staged into shared memory (zero filled outside the domain), K levels
// with the codes quantised on the spot, the blocks' coarse values to the
// gathered grid G, their symbols and escapes out.  The quantiser table and
// max|u| are read around L1 (the batched kernel writes them in the same launch).
template <int B, int K>
__device__ __forceinline__ void fwd_group(const BlockArgs<double>& a, const int64_t b, const int nv,
                                          unsigned char* smem, bool& ovf) {
  using Cfg = BlockCfg<double, B, K>;
  using GC = GroupCfg<B, K>;
  constexpr int NB = GC::NB;
  __shared__ double s_rq[NB * K];
  double* A = reinterpret_cast<double*>(smem);
  double* T1 = A + NB * Cfg::A;
  double* cb0 = T1 + NB * Cfg::T1;
  double* cb1 = cb0 + NB * Cfg::CB0;
  uint16_t* stage = reinterpret_cast<uint16_t*>(smem + GC::fwd_stage_off);
  if (threadIdx.x < NB * K) {
    const int blk = threadIdx.x / K;
    const int tier = a.tier && blk < nv ? a.tier[b + blk] : 0;
    s_rq[threadIdx.x] = __ldcg(a.rq + tier * K + (threadIdx.x - blk * K));
  }
  for (int blk = 0; blk < nv; ++blk) {
    const BlockSpan<const double, B> sp(a.field, a.n0, a.n1, a.n2, BlockCoord(b + blk, a.nb1, a.nb2));
    issue_block_load<double, B>(A + blk * Cfg::A, a.field, sp, a.n1, a.n2);
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  const int64_t sbase = b * (int64_t)Cfg::PB;
  const LevelBufs<double> bufs{A, cb0, cb1};
  const bool full = a.radius == (1 << 15);
  GroupFwdLevels<B, 0, K, B>::run(bufs, T1, s_rq, stage, a.esc + sbase, ovf, full, field_huge(a.sc), nv);
  for (int blk = 0; blk < nv; ++blk) {  // block coarse values -> gathered grid G
    constexpr int M = Cfg::M;
    const BlockCoord bc(b + blk, a.nb1, a.nb2);
    const double* cf = bufs(K) + blk * lvl_stride<B>(K);
    double* g = a.G + (((int64_t)bc.b0 * M) * a.g1 + (int64_t)bc.b1 * M) * a.g2 + (int64_t)bc.b2 * M;
    for (int e = threadIdx.x; e < M * M * M; e += blockDim.x) {
      const int j0 = e / (M * M), r = e - j0 * M * M, j1 = r / M, j2 = r - j1 * M;
      g[((int64_t)j0 * a.g1 + j1) * a.g2 + j2] = cf[e];
    }
  }
  for (int blk = 0; blk < nv; ++blk) {
    const int64_t o = sbase + (int64_t)blk * Cfg::PB;
    if (full) copy_symbols<Cfg::PB>(a.sym + o, stage + blk * Cfg::PB);
    else store_codes<Cfg::PB>(a.sym + o, a.esc + o, stage + blk * Cfg::PB, a.radius);
  }
  __syncthreads();
}

template <int B, int K>
__global__ void __launch_bounds__(GroupCfg<B, K>::NT_FWD, GroupCfg<B, K>::FWD_MIN_CTAS)
    block_fwd_group_kernel(BlockArgs<double> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NB = block_group(B);
  bool ovf = false;
  for (int64_t b = (int64_t)blockIdx.x * NB; b < a.nblocks; b += (int64_t)gridDim.x * NB)
    fwd_group<B, K>(a, b, (int)(a.nblocks - b < NB ? a.nblocks - b : NB), smem_raw, ovf);
  if (ovf) atomicOr(&a.sc->status, ST_OVERFLOW);
}

// One line of the first inverse pass: its coefficients into X (all-coarse
// nodes have none), restriction and solve along the line into T1.
template <int N, bool CC>
__device__ __forceinline__ void inv_line(double* X, double* T1, const int i0, const int i1, const int lvl_off,
                                         const double q, const int32_t* codes) {
  constexpr int C = (N + 1) / 2;
  double* x = X + (i0 * N + i1) * N;
  const int base = lvl_off + line_base<N>(i0, i1);
  double d[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    d[k] = 0.0;
    if (!CC || (k & 1)) {
      d[k] = dequant(codes[base + (CC ? k / 2 : k)], q);
      x[k] = d[k];
    }
  }
  double z[C];
  restrict_solve<double, N, CC>(block_tab<double, N>(), d, z);
#pragma unroll
  for (int j = 0; j < C; ++j) T1[(i0 * C + j) * N + i1] = z[j];
}

// Whether a value is 2^1023 or more in magnitude, an infinity or NaN (on its
// bits: integer work, not the double unit's).
__device__ __forceinline__ bool top_binade(double v) { return ((unsigned)__double2hiint(v) << 1) >= 0xFFC00000u; }

// One line of the last inverse pass: u = I(u|C) + d in X.  A both-odd line adds
// two sums of four: where one lies in the top binade the sums are scaled first
// (exact), so that only the sum of four itself can overflow.
template <int N, int CLS>
__device__ __forceinline__ void interp_line(double* X, const double* cin, const int i0, const int i1) {
  constexpr int C = (N + 1) / 2;
  const int a0 = i0 >> 1, b0 = (i0 + 1) >> 1, a1 = i1 >> 1, b1 = (i1 + 1) >> 1;
  double v[C];
  coarse_sums<C, CLS>(cin + (a0 * C + a1) * C, cin + (a0 * C + b1) * C, cin + (b0 * C + a1) * C,
                         cin + (b0 * C + b1) * C, 1, v);
  double se = CLS == 2 ? 0.25 : CLS == 1 ? 0.5 : 1.0, ho = 0.5 * se;
  if (CLS == 2) {
    bool top = false;
#pragma unroll
    for (int J = 0; J < C; ++J) top |= top_binade(v[J]);
    if (top) {
#pragma unroll
      for (int J = 0; J < C; ++J) v[J] *= 0.25;
      se = 1.0;
      ho = 0.5;
    }
  }
  double* x = X + (i0 * N + i1) * N;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if (k & 1) x[k] = fma(ho, v[k / 2] + v[k / 2 + 1], x[k]);
    else if (CLS) x[k] = fma(se, v[k / 2], x[k]);
    else x[k] = v[k / 2];
  }
}

// Inverse level of the first nv of NB blocks: coarse values `cin` (C^3) and the
// level's codes give the N^3 values in X.  z = P D (three passes), u|C = c - z,
// u = I u|C + D.
template <int N, int NB>
__device__ __forceinline__ void group_level_inv(double* X, const int xs, double* T1, const int t1s, double* T2,
                                                const int t2s, double* cin, const int cs, const int lvl_off, const double* q, const int qs,
                                                const int32_t* codes, const int ps, const int nv) {
  constexpr int C = (N + 1) / 2;
  // the classes of a level of fewer than nine nodes share warps (they diverge)
  using LN = Lines<N, NB>;
  auto line_of = [&](int it, int& blk, int& i0, int& i1) {
    if (N >= 9) return LN::of(it, blk, i0, i1);
    blk = it / (N * N);
    const int L = it - blk * (N * N);
    i0 = L / N;
    i1 = L - i0 * N;
    return (i0 & 1) + (i1 & 1);
  };
  constexpr int total = N >= 9 ? LN::total : NB * N * N;
  for (int it = threadIdx.x; it < total; it += blockDim.x) {
    int blk, i0, i1;
    const int cls = line_of(it, blk, i0, i1);
    if (cls < 0 || blk >= nv) continue;
    if (cls) inv_line<N, false>(X + blk * xs, T1 + blk * t1s, i0, i1, lvl_off, q[blk * qs], codes + blk * ps);
    else inv_line<N, true>(X + blk * xs, T1 + blk * t1s, i0, i1, lvl_off, q[blk * qs], codes + blk * ps);
  }
  __syncthreads();
  restrict_passes<N, NB, -1>(T1, t1s, T2, t2s, cin, cs);
  for (int it = threadIdx.x; it < total; it += blockDim.x) {
    int blk, i0, i1;
    const int cls = line_of(it, blk, i0, i1);
    if (cls < 0 || blk >= nv) continue;
    if (cls == 2) interp_line<N, 2>(X + blk * xs, cin + blk * cs, i0, i1);
    else if (cls == 1) interp_line<N, 1>(X + blk * xs, cin + blk * cs, i0, i1);
    else interp_line<N, 0>(X + blk * xs, cin + blk * cs, i0, i1);
  }
  __syncthreads();
}

template <int N, int L, int K, int B>
struct GroupInvLevels {  // recompose levels L, L-1, ..., 0 (level L has N nodes)
  __device__ __forceinline__ static void run(const LevelBufs<double>& bufs, double* T1, double* T2, const double* q,
                                             const int32_t* codes, const int nv) {
    using Cfg = BlockCfg<double, B, K>;
    group_level_inv<N, block_group(B)>(bufs(L), lvl_stride<B>(L), T1, Cfg::T1, T2, Cfg::T2, bufs(L + 1),
                                               lvl_stride<B>(L + 1), lvl_offset(B, L), q + L, K, codes, Cfg::PB, nv);
    if constexpr (L > 0) GroupInvLevels<2 * N - 1, L - 1, K, B>::run(bufs, T1, T2, q, codes, nv);
  }
};

template <int B, int K>
__global__ void __launch_bounds__(GroupCfg<B, K>::NT_INV, GroupCfg<B, K>::INV_MIN_CTAS)
    block_inv_group_kernel(BlockArgs<double> a) {
  using Cfg = BlockCfg<double, B, K>;
  using GC = GroupCfg<B, K>;
  constexpr int NB = GC::NB, M = Cfg::M;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_q[NB * K];
  double* A = reinterpret_cast<double*>(smem_raw);
  double* T1 = A + NB * Cfg::A;
  double* T2 = T1 + NB * Cfg::T1;
  double* cb0 = T2 + NB * Cfg::T2;
  double* cb1 = cb0 + NB * Cfg::CB0;
  int32_t* codes = reinterpret_cast<int32_t*>(smem_raw + GC::inv_stage_off);
  const LevelBufs<double> bufs{A, cb0, cb1};
  for (int64_t b = (int64_t)blockIdx.x * NB; b < a.nblocks; b += (int64_t)gridDim.x * NB) {
    const int nv = (int)(a.nblocks - b < NB ? a.nblocks - b : NB);
    const int64_t sbase = b * (int64_t)Cfg::PB;
    if (threadIdx.x < NB * K) {
      const int blk = threadIdx.x / K;
      int tier = a.tier && blk < nv ? a.tier[b + blk] : 0;
      if (tier >= a.ntiers) {  // corrupt stream: keep the q reads inside the table
        if (a.sc) atomicOr(&a.sc->status, ST_CORRUPT);
        tier = 0;
      }
      s_q[threadIdx.x] = a.q[tier * K + (threadIdx.x - blk * K)];
    }
    for (int blk = 0; blk < nv; ++blk) {
      load_codes<Cfg::PB>(a.sym + sbase + blk * Cfg::PB, a.esc + sbase + blk * Cfg::PB, codes + blk * Cfg::PB, a.radius);
      const BlockCoord bc(b + blk, a.nb1, a.nb2);
      double* cf = bufs(K) + blk * lvl_stride<B>(K);
      const double* g = a.G + (((int64_t)bc.b0 * M) * a.g1 + (int64_t)bc.b1 * M) * a.g2 + (int64_t)bc.b2 * M;
      for (int e = threadIdx.x; e < M * M * M; e += blockDim.x) {
        const int j0 = e / (M * M), r = e - j0 * M * M, j1 = r / M, j2 = r - j1 * M;
        cf[e] = g[((int64_t)j0 * a.g1 + j1) * a.g2 + j2];
      }
    }
    __syncthreads();
    GroupInvLevels<M * 2 - 1, K - 1, K, B>::run(bufs, T1, T2, s_q, codes, nv);
    for (int blk = 0; blk < nv; ++blk)
      store_block<double, B>(BlockSpan<double, B>(a.field, a.n0, a.n1, a.n2, BlockCoord(b + blk, a.nb1, a.nb2)),
                             A + blk * Cfg::A, a.n1, a.n2);
    __syncthreads();
  }
}

}  // namespace bm
