// Tall-skinny dense kernels: Gram products (Eq. rreig's S^T S and S^T H S; Eq. bgs's V^T W),
// block-times-small-matrix products (Eqs. xupd, pupd; CholQR's X R^{-1}), the fused LOBPCG
// update, and deterministic reductions.  All are HBM-bound passes over n x nb blocks.
#include <type_traits>

#include "common.cuh"
#include "dense.cuh"
#include "vec.cuh"

namespace eig {

// ---------------------------------------------------------------------------------------
// Gram products
// ---------------------------------------------------------------------------------------
constexpr int kGramThreads = 256;
constexpr int kGramRows = 32;

struct PairList {
  int a[kMaxPairs], b[kMaxPairs];
  int n;
};

// 16-byte asynchronous global -> shared copy.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// A thread's values of a row: 16-byte loads where the tile is whole 16-byte pieces (tiles are
// TM-aligned in rows of a multiple of TM values, stages 16-byte aligned).
template <typename T, int TM>
__device__ __forceinline__ void gram_load(const T* p, T* v) {
  if constexpr ((TM * sizeof(T)) % 16 == 0) {
#pragma unroll
    for (int i = 0; i < TM; i += 16 / (int)sizeof(T)) {
      const Vec<T, 16 / (int)sizeof(T)> q = VecIO<T, 16 / (int)sizeof(T)>::ld(p + i);
#pragma unroll
      for (int k = 0; k < 16 / (int)sizeof(T); ++k) v[i + k] = q.v[k];
    }
  } else {
#pragma unroll
    for (int i = 0; i < TM; ++i) v[i] = p[i];
  }
}

// Accumulator of one element pair (j, j + 1) of a thread's tile: chunk sums c (fused multiply-adds
// over the chunk's rows), totals over the chunks.  FP32: totals in double-float, the two-sum of hi and c
// exact, its error and lo added and the pair normalised again, so that lo stays below half a unit of hi
// and a total loses at most 2^-48 of itself per chunk.  (Without the normalisation lo grows with the number
// of chunks, and so do its roundings: constant chunks lose 2e-8 after 5,000 of them.)  FP64: the chunk
// sums keep a total's chain short.
template <typename T> struct GramPair;
template <> struct GramPair<float> {
  float2 c, hi, lo;
  __device__ __forceinline__ void zero() { c = hi = lo = make_float2(0.0f, 0.0f); }
  __device__ __forceinline__ void fma(float a, float b0, float b1) {
    c = __ffma2_rn(make_float2(a, a), make_float2(b0, b1), c);
  }
  __device__ __forceinline__ void flush() {
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 s = __fadd2_rn(hi, c);
    const float2 bb = __ffma2_rn(hi, m1, s);                       // s - hi
    const float2 e1 = __ffma2_rn(__ffma2_rn(bb, m1, s), m1, hi);   // hi - (s - bb)
    const float2 e2 = __ffma2_rn(bb, m1, c);                       // c - bb
    const float2 e = __fadd2_rn(lo, __fadd2_rn(e1, e2));
    hi = __fadd2_rn(s, e);
    lo = __ffma2_rn(__ffma2_rn(s, m1, hi), m1, e);                 // e - (hi - s)
    c = make_float2(0.0f, 0.0f);
  }
  __device__ __forceinline__ double get(int k) const {
    return k ? (double)hi.y + (double)lo.y : (double)hi.x + (double)lo.x;
  }
};
template <> struct GramPair<double> {
  double c0, c1, t0, t1;
  __device__ __forceinline__ void zero() { c0 = c1 = t0 = t1 = 0.0; }
  __device__ __forceinline__ void fma(double a, double b0, double b1) {
    c0 = ::fma(a, b0, c0);
    c1 = ::fma(a, b1, c1);
  }
  __device__ __forceinline__ void flush() {
    t0 += c0;
    t1 += c1;
    c0 = c1 = 0.0;
  }
  __device__ __forceinline__ double get(int k) const { return k ? t1 : t0; }
};

// Pair and tile (first row ti, first column tj) of tile index `idx`; a pair of a block with itself
// has only the tiles that reach the upper triangle.  Returns false beyond the last tile.
template <int TMI, int TMJ>
__host__ __device__ inline bool gram_tile(const PairList& pairs, int nb, int idx, int* q, int* ti, int* tj) {
  for (int p = 0; p < pairs.n; ++p) {
    const bool sym = pairs.a[p] == pairs.b[p];
    for (int i = 0; i < nb; i += TMI) {
      const int j0 = sym ? i / TMJ * TMJ : 0, cnt = (nb - j0) / TMJ;
      if (idx < cnt) {
        *q = p;
        *ti = i;
        *tj = j0 + idx * TMJ;
        return true;
      }
      idx -= cnt;
    }
  }
  return false;
}

// G_q = A^T B of every pair.  A CTA stages chunks of 32 rows of every block; a group of threads
// (one thread per TMI x TMJ tile of the pairs) multiplies one chunk, and `groups` groups work on
// consecutive chunks side by side, so that a single narrow pair (16 tiles at nb = 16) still fills
// the CTA.  When one group does not fit (more than 256 tiles), a thread takes MAXT tiles in turn.
// PIPE: 16-byte cp.async copies into two stages, the next chunks' copies in flight while the
// current ones are multiplied (rows of nb values a multiple of 16 bytes and every block 16-byte
// aligned).  FP32 products are summed per 32-row chunk (chunks start at multiples of 32 rows), chunk
// sums in double-float, groups and CTAs in FP64 in a fixed order.
//
// What bounds it: one pair is an HBM pass; many pairs the shared-memory pipe (a 4 x 4 tile takes
// six clocks of loads for four clocks of multiply-adds per row, an 8 x 4 tile eight for eight), FP64
// the FP64 pipe (two lanes per clock per SM: hence only the upper tiles of a pair of a block with
// itself).  Measured: one FP32 pair at n = 2M, nb = 16 in 53 us (4.8 TB/s; 204 us when one group of 16
// threads multiplied), LOBPCG's twelve pairs there 441 us (515 us with 4 x 4 tiles); twelve FP64 pairs at
// n = 20,000, nb = 8 in 40 us (56 us).
template <typename T, int TMI, int TMJ, int MAXT, bool PIPE>
__global__ void __launch_bounds__(kGramThreads)
k_gram(BlockList blocks, PairList pairs, int nb, int64_t n, int64_t units, int tpg, int groups, double* part) {
  static_assert(TMJ % 2 == 0 || (TMI == 1 && TMJ == 1), "elements are accumulated in pairs");
  constexpr int NP = TMJ == 1 ? 1 : TMJ / 2;
  constexpr int kUnit = sizeof(T) == 4 ? kGramRows : 8;   // row granularity of the CTAs' shares
  extern __shared__ __align__(16) unsigned char sm_raw[];
  T* sm_base = reinterpret_cast<T*>(sm_raw);  // [stages][nblocks][groups * 32][nb]
  const int srows = groups * kGramRows;
  const size_t bl_elems = (size_t)srows * nb;
  const size_t stage_elems = (size_t)blocks.n * bl_elems;
  const int tid = threadIdx.x;
  const int grp = MAXT == 1 ? tid / tpg : 0;
  const int tile0 = MAXT == 1 ? tid % tpg : tid;
  GramPair<T> acc[MAXT][TMI][NP];
  int q[MAXT], ti[MAXT], tj[MAXT];
  bool on[MAXT];
#pragma unroll
  for (int s = 0; s < MAXT; ++s) {
    on[s] = grp < groups && gram_tile<TMI, TMJ>(pairs, nb, tile0 + s * kGramThreads, &q[s], &ti[s], &tj[s]);
#pragma unroll
    for (int i = 0; i < TMI; ++i)
#pragma unroll
      for (int j = 0; j < NP; ++j) acc[s][i][j].zero();
  }
  const int64_t r0 = units * blockIdx.x / gridDim.x * kUnit;
  const int64_t r1 = min64(n, units * (blockIdx.x + 1) / gridDim.x * kUnit);
  constexpr int EPC = 16 / sizeof(T);                // elements per 16-byte copy
  auto issue = [&](int64_t rc, T* stage) {           // copies of the chunks at row rc
    const int pieces = (int)min64(srows, r1 - rc) * nb / EPC;
    for (int b = 0; b < blocks.n; ++b) {
      const T* src = static_cast<const T*>(blocks.p[b]) + rc * nb;
      T* dst = stage + b * bl_elems;
      for (int i = tid; i < pieces; i += blockDim.x) cp_async16(dst + i * EPC, src + i * EPC);
    }
    cp_async_commit();
  };
  if (PIPE && r0 < r1) issue(r0, sm_base);
  int stage_i = 0;
  for (int64_t rc = r0; rc < r1; rc += srows) {
    const int rows = (int)min64(srows, r1 - rc);
    T* sm = sm_base + (PIPE ? (size_t)stage_i * stage_elems : 0);
    if (PIPE) {
      // the other stage was last read in the previous iteration: every thread is past it
      __syncthreads();
      if (rc + srows < r1) {
        issue(rc + srows, sm_base + (size_t)(stage_i ^ 1) * stage_elems);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
      stage_i ^= 1;
    } else {
      __syncthreads();
      for (int b = 0; b < blocks.n; ++b) {
        const T* src = static_cast<const T*>(blocks.p[b]) + rc * nb;
        T* dst = sm + b * bl_elems;
        for (int i = tid; i < rows * nb; i += blockDim.x) dst[i] = src[i];
      }
      __syncthreads();
    }
    const int crows = min(kGramRows, rows - grp * kGramRows);   // rows of this group's chunk (may be <= 0)
#pragma unroll
    for (int s = 0; s < MAXT; ++s) {
      if (on[s] && crows > 0) {
        const T* Ab = sm + pairs.a[q[s]] * bl_elems + (size_t)grp * kGramRows * nb + ti[s];
        const T* Bb = sm + pairs.b[q[s]] * bl_elems + (size_t)grp * kGramRows * nb + tj[s];
        auto row = [&](int r) {
          T av[TMI], bv[TMJ + 1];
          gram_load<T, TMI>(Ab + r * nb, av);
          gram_load<T, TMJ>(Bb + r * nb, bv);
          if (TMJ == 1) bv[1] = T(0);
#pragma unroll
          for (int i = 0; i < TMI; ++i)
#pragma unroll
            for (int j = 0; j < NP; ++j) acc[s][i][j].fma(av[i], bv[2 * j], bv[2 * j + 1]);
        };
        if (crows == kGramRows) {
#pragma unroll 4
          for (int r = 0; r < kGramRows; ++r) row(r);
        } else {
          for (int r = 0; r < crows; ++r) row(r);
        }
#pragma unroll
        for (int i = 0; i < TMI; ++i)
#pragma unroll
          for (int j = 0; j < NP; ++j) acc[s][i][j].flush();
      }
    }
  }
  // the groups' sums, in group order, then this CTA's partial; the lower triangle of a pair of a
  // block with itself mirrors the upper one (the same products in the same order)
  const int m = pairs.n * nb * nb;
  double* sred = reinterpret_cast<double*>(sm_raw);   // [groups][m]
  double* out = part + (size_t)blockIdx.x * m;
  double* dst = groups > 1 ? sred + (size_t)(grp < groups ? grp : 0) * m : out;
  __syncthreads();
#pragma unroll
  for (int s = 0; s < MAXT; ++s) {
    if (on[s]) {
      const bool sym = pairs.a[q[s]] == pairs.b[q[s]];
      double* d = dst + (size_t)q[s] * nb * nb;
#pragma unroll
      for (int i = 0; i < TMI; ++i)
#pragma unroll
        for (int j = 0; j < TMJ; ++j) {
          const int r = ti[s] + i, c = tj[s] + j;
          if (sym && r > c) continue;
          const double v = acc[s][i][j / 2].get(j & 1);
          d[r * nb + c] = v;
          if (sym && r < c) d[c * nb + r] = v;
        }
    }
  }
  if (groups > 1) {
    __syncthreads();
    for (int e = tid; e < m; e += blockDim.x) {
      double v = sred[e];
      for (int g = 1; g < groups; ++g) v += sred[(size_t)g * m + e];
      out[e] = v;
    }
  }
}

// out[j] = sum over parts in fixed order: one warp per output, lane l adds parts l, l+32, ...,
// then a fixed xor tree (bitwise reproducible, and the loads of a warp are independent).
__global__ void k_reduce_partials(const double* __restrict__ part, int nparts, int m, double* __restrict__ out) {
  const int j = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (j >= m) return;
  double s = 0.0;
  for (int b = lane; b < nparts; b += 32) s += part[(size_t)b * m + j];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[j] = s;
}

// Two CTAs per SM, each with a near-equal share of the rows in units of 32 rows (the FP32 chunks) or
// 8 (FP64, bound by its pipe: 20,000 rows are 66 per CTA instead of 96 in 209 of them).
// The grid also fixes how the rows are grouped into partial sums, and so the rounding of every Gram, to
// which the last iterations of the hybrid solve are sensitive: at n = 2M (tolerance 1e-6, 4 + 5 iterations)
// its largest residual is 9.8e-7 with two CTAs per SM, 9.9e-7 with one and a half, 6.7e-7 with one, and was
// 6.9e-7 with shares of equal whole chunks; another start took 7 RMM-DIIS iterations with two CTAs per SM
// and 21 with four.
static int gram_grid(int64_t n, eig_dtype vt, int64_t* units, int max_parts) {
  const int unit = vt == EIG_F32 ? kGramRows : 8;
  int64_t g = num_sms() * 2;
  if (max_parts > 0 && g > max_parts) g = max_parts;
  *units = (n + unit - 1) / unit;
  return (int)min64(g, *units);
}

size_t gram_scratch_bytes(int npairs, int nb) { return (size_t)num_sms() * 2 * npairs * nb * nb * 8 + 256; }

eig_status reduce_partials(const double* part, int nparts, int m, double* out, cudaStream_t st) {
  k_reduce_partials<<<(unsigned)(((int64_t)m * 32 + 255) / 256), 256, 0, st>>>(part, nparts, m, out);
  EIG_LAUNCH_CHECK("k_reduce_partials");
  return EIG_OK;
}

template <typename T, int TMI, int TMJ>
static eig_status gram_launch(const BlockList& blocks, const PairList& pl, int nb, int64_t n, double* G, void* part,
                              cudaStream_t st, int max_parts) {
  int64_t units;
  const int g = gram_grid(n, sizeof(T) == 4 ? EIG_F32 : EIG_F64, &units, max_parts);
  int q, ti, tj, ntiles = 0;
  while (gram_tile<TMI, TMJ>(pl, nb, ntiles, &q, &ti, &tj)) ++ntiles;
  const size_t chunk = (size_t)blocks.n * kGramRows * nb * sizeof(T);
  bool pipe = (nb * sizeof(T)) % 16 == 0;
  for (int b = 0; b < blocks.n; ++b) pipe = pipe && (reinterpret_cast<uintptr_t>(blocks.p[b]) % 16 == 0);
  pipe = pipe && 2 * chunk <= 200 * 1024;
  // groups: as many as the threads hold and two CTAs of two stages (and the groups' FP64 sums)
  // leave room for, and no more than a CTA's share has chunks
  const size_t m8 = (size_t)pl.n * nb * nb * 8;
  int64_t groups = ntiles <= kGramThreads ? kGramThreads / ntiles : 1;
  groups = min64(groups, (int64_t)(100 * 1024 / ((pipe ? 2 : 1) * chunk)));
  groups = min64(groups, (int64_t)(100 * 1024 / m8));
  groups = min64(groups, (n + (int64_t)g * kGramRows - 1) / ((int64_t)g * kGramRows));
  groups = max64(groups, 1);
  const int tpg = ntiles <= kGramThreads ? ntiles : kGramThreads;
  const int threads = (int)((groups * tpg + 31) / 32 * 32);
  size_t sm = (pipe ? 2 : 1) * (size_t)groups * chunk;
  if (groups > 1 && (size_t)groups * m8 > sm) sm = (size_t)groups * m8;
  auto kern = pipe ? k_gram<T, TMI, TMJ, 1, true> : k_gram<T, TMI, TMJ, 1, false>;
  if (ntiles > kGramThreads) {
    if constexpr (TMI == TMJ) {
      kern = pipe ? (ntiles <= 2 * kGramThreads ? k_gram<T, TMI, TMJ, 2, true> : k_gram<T, TMI, TMJ, 4, true>)
                  : (ntiles <= 2 * kGramThreads ? k_gram<T, TMI, TMJ, 2, false> : k_gram<T, TMI, TMJ, 4, false>);
    } else {
      return EIG_EUNSUPPORTED;   // the caller takes square tiles from here on
    }
  }
  if (sm > 48 * 1024) EIG_CUDA_TRY(::eig::ensure_dyn_smem(kern, (int)sm));
  kern<<<g, threads, sm, st>>>(blocks, pl, nb, n, units, tpg, (int)groups, static_cast<double*>(part));
  EIG_LAUNCH_CHECK("k_gram");
  return reduce_partials(static_cast<double*>(part), g, pl.n * nb * nb, G, st);
}

eig_status gram_multi(const BlockList& blocks, const int* pa, const int* pb, int npairs, int nb, int64_t n,
                      eig_dtype vt, double* G, void* part, cudaStream_t st, int max_parts) {
  if (npairs < 1 || npairs > kMaxPairs || nb < 1 || nb > 64 || n < 1 || blocks.n < 1 || blocks.n > 16) return EIG_EINVAL;
  PairList pl;
  pl.n = npairs;
  for (int q = 0; q < npairs; ++q) {
    if (pa[q] < 0 || pa[q] >= blocks.n || pb[q] < 0 || pb[q] >= blocks.n) return EIG_EINVAL;
    pl.a[q] = pa[q];
    pl.b[q] = pb[q];
  }
  const int TM = (nb % 4 == 0) ? 4 : ((nb % 2 == 0) ? 2 : 1);
  if ((size_t)npairs * (nb / TM) * (nb / TM) > 4 * kGramThreads) return EIG_EUNSUPPORTED;
  if (vt == EIG_F32) {
    // From 128 tiles of 4 x 4 on (of all pairs, a pair of a block with itself counted whole), 8 x 4 tiles:
    // two thirds of the loads from shared memory, but half the threads.  Set at LOBPCG's twelve pairs,
    // nb = 16, n = 2M (174 tiles): 441 us, 515 with 4 x 4.  One pair, n = 500,000, us with 4 x 4 / 8 x 4 tiles:
    // nb = 40 (below the line) 93 / 93, 48 136 / 124, 56 159 / 163, 64 163 / 166; a block with itself: 40 60 / 69,
    // 48 75 / 86, 56 97 / 102, 64 136 / 124.  n = 20,000: 48 30 / 39, 64 34 / 44: single pairs hardly gain.
    const int t8 = npairs * (nb / 8) * (nb / 4);
    if (nb % 8 == 0 && 2 * t8 > 128 && t8 <= kGramThreads)
      return gram_launch<float, 8, 4>(blocks, pl, nb, n, G, part, st, max_parts);
    if (TM == 4) return gram_launch<float, 4, 4>(blocks, pl, nb, n, G, part, st, max_parts);
    if (TM == 2) return gram_launch<float, 2, 2>(blocks, pl, nb, n, G, part, st, max_parts);
    return gram_launch<float, 1, 1>(blocks, pl, nb, n, G, part, st, max_parts);
  }
  if (vt == EIG_F64) {
    if (TM == 4) return gram_launch<double, 4, 4>(blocks, pl, nb, n, G, part, st, max_parts);
    if (TM == 2) return gram_launch<double, 2, 2>(blocks, pl, nb, n, G, part, st, max_parts);
    return gram_launch<double, 1, 1>(blocks, pl, nb, n, G, part, st, max_parts);
  }
  return EIG_EINVAL;
}

// ---------------------------------------------------------------------------------------
// Out = In M for a square M of the block's own width: CholQR's X <- X R^{-1}, in place
// ---------------------------------------------------------------------------------------
// A lane owns one 16-byte piece of a row: it loads it (coalesced), the warp exchanges whole rows
// through shared memory, and the lane computes its piece of the product with its columns of M held
// in registers, so nothing but the rows moves.  A row is read by its lanes before any of them writes
// it, hence In may be Out.  Sums run over k ascending, as k_block_apply's.  *skip (device, may be
// null) != 0 leaves Out untouched.  Bound by HBM in FP32: 50 us at n = 2M, NB = 16 (5.1 TB/s); the
// thread-per-element kernel took 187 us and a copy of the block (55 us) before it.
template <typename T, int NB>
__global__ void __launch_bounds__(256)
k_rows_apply(const T* In, const double* __restrict__ M, T* Out, int64_t n, const int* __restrict__ skip) {
  constexpr int VEC = 16 / (int)sizeof(T), LPR = NB / VEC, RPW = 32 / LPR, U = 4, LD = NB + VEC;
  __shared__ __align__(16) T buf[8][U][RPW][LD];
  if (skip && *skip != 0) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, pc = lane % LPR, rw = lane / LPR;
  T m[NB][VEC];
#pragma unroll
  for (int k = 0; k < NB; ++k)
#pragma unroll
    for (int c = 0; c < VEC; ++c) m[k][c] = (T)M[k * NB + pc * VEC + c];
  const int64_t step = (int64_t)gridDim.x * 8 * U * RPW;
  for (int64_t r0 = ((int64_t)blockIdx.x * 8 + w) * U * RPW; r0 < n; r0 += step) {
    Vec<T, VEC> in[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = r0 + u * RPW + rw;
      if (r < n) in[u] = VecIO<T, VEC>::ld(In + r * NB + pc * VEC);
      else in[u].zero();
    }
    __syncwarp();   // the previous rows have been read
#pragma unroll
    for (int u = 0; u < U; ++u) VecIO<T, VEC>::st(&buf[w][u][rw][pc * VEC], in[u]);
    __syncwarp();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const T* row = buf[w][u][rw];
      Vec<T, VEC> acc;
      acc.zero();
#pragma unroll
      for (int k0 = 0; k0 < NB; k0 += VEC) {
        const Vec<T, VEC> x = VecIO<T, VEC>::ld(row + k0);
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          if constexpr (sizeof(T) == 4) {
            const float2 xx = make_float2(x.v[v], x.v[v]);
#pragma unroll
            for (int c = 0; c < VEC; c += 2) {
              const float2 t = __ffma2_rn(xx, make_float2(m[k0 + v][c], m[k0 + v][c + 1]),
                                          make_float2(acc.v[c], acc.v[c + 1]));
              acc.v[c] = t.x;
              acc.v[c + 1] = t.y;
            }
          } else {
#pragma unroll
            for (int c = 0; c < VEC; ++c) acc.v[c] = fma(x.v[v], m[k0 + v][c], acc.v[c]);
          }
        }
      }
      const int64_t r = r0 + u * RPW + rw;
      if (r < n) VecIO<T, VEC>::st(Out + r * NB + pc * VEC, acc);
    }
  }
}

eig_status rows_apply(const void* In, int nb, const double* M, void* Out, int64_t n, eig_dtype vt, const int* skip,
                      cudaStream_t st) {
  if ((nb != 8 && nb != 16) || ((reinterpret_cast<uintptr_t>(In) | reinterpret_cast<uintptr_t>(Out)) & 15))
    return EIG_EUNSUPPORTED;
  const int rows = 8 * 4 * (32 / (nb * (vt == EIG_F64 ? 8 : 4) / 16));   // rows of one CTA pass
  const int grid = (int)max64(1, min64((n + rows - 1) / rows, (int64_t)num_sms() * 4));
  auto go = [&](auto kern, auto* out) {
    typedef std::remove_pointer_t<decltype(out)> T;
    kern<<<grid, 256, 0, st>>>(static_cast<const T*>(In), M, out, n, skip);
  };
  if (vt == EIG_F32 && nb == 8) go(k_rows_apply<float, 8>, static_cast<float*>(Out));
  else if (vt == EIG_F32) go(k_rows_apply<float, 16>, static_cast<float*>(Out));
  else if (vt == EIG_F64 && nb == 8) go(k_rows_apply<double, 8>, static_cast<double*>(Out));
  else if (vt == EIG_F64) go(k_rows_apply<double, 16>, static_cast<double*>(Out));
  else return EIG_EINVAL;
  EIG_LAUNCH_CHECK("k_rows_apply");
  return EIG_OK;
}

// ---------------------------------------------------------------------------------------
// Out = sum_s In_s M_s (+ beta Out): thread per (row, output column)
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void k_block_apply(BlockList in, int nb, const double* __restrict__ M, int m, T* __restrict__ Out,
                              double beta, int64_t n) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  T* sM = reinterpret_cast<T*>(sm_raw);  // K x m
  const int K = in.n * nb;
  for (int i = threadIdx.x; i < K * m; i += blockDim.x) sM[i] = (T)M[i];
  __syncthreads();
  const int64_t total = n * m;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = idx / m;
    const int j = (int)(idx % m);
    T acc = T(0);
    for (int s = 0; s < in.n; ++s) {
      const T* row = static_cast<const T*>(in.p[s]) + r * nb;
      const T* Ms = sM + (size_t)s * nb * m + j;
      for (int k = 0; k < nb; ++k) acc = fma(__ldg(row + k), Ms[(size_t)k * m], acc);
    }
    if (beta != 0.0) acc = fma((T)beta, Out[idx], acc);
    Out[idx] = acc;
  }
}

eig_status block_apply(const BlockList& in, int nb, const double* M, int m, void* Out, double beta, int64_t n,
                       eig_dtype vt, cudaStream_t st) {
  if (in.n < 1 || in.n > kMaxBlocks || nb < 1 || m < 1 || m > 64 || in.n * nb > 1024) return EIG_EINVAL;
  if (in.n == 1 && m == nb && beta == 0.0) {
    const eig_status s = rows_apply(in.p[0], nb, M, Out, n, vt, nullptr, st);
    if (s != EIG_EUNSUPPORTED) return s;
  }
  const int grid = num_sms() * 8;
  if (vt == EIG_F32) {
    const size_t sm = (size_t)in.n * nb * m * 4;
    if (sm > 48 * 1024) EIG_CUDA_TRY(::eig::ensure_dyn_smem(k_block_apply<float>, (int)sm));
    k_block_apply<float><<<grid, 256, sm, st>>>(in, nb, M, m, static_cast<float*>(Out), beta, n);
  } else if (vt == EIG_F64) {
    const size_t sm = (size_t)in.n * nb * m * 8;
    if (sm > 48 * 1024) EIG_CUDA_TRY(::eig::ensure_dyn_smem(k_block_apply<double>, (int)sm));
    k_block_apply<double><<<grid, 256, sm, st>>>(in, nb, M, m, static_cast<double*>(Out), beta, n);
  } else {
    return EIG_EINVAL;
  }
  EIG_LAUNCH_CHECK("k_block_apply");
  return EIG_OK;
}

// ---------------------------------------------------------------------------------------
// conversions, column sums of squares
// ---------------------------------------------------------------------------------------
template <typename A, typename B>
__global__ void k_convert(const A* __restrict__ s, B* __restrict__ d, int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    d[i] = (B)s[i];
}

eig_status convert(const void* src, eig_dtype st_, void* dst, eig_dtype dt_, int64_t count, cudaStream_t st) {
  const int grid = num_sms() * 8;
  if (st_ == EIG_F64 && dt_ == EIG_F32) k_convert<double, float><<<grid, 256, 0, st>>>((const double*)src, (float*)dst, count);
  else if (st_ == EIG_F32 && dt_ == EIG_F64) k_convert<float, double><<<grid, 256, 0, st>>>((const float*)src, (double*)dst, count);
  else if (st_ == EIG_F64 && dt_ == EIG_F64) k_convert<double, double><<<grid, 256, 0, st>>>((const double*)src, (double*)dst, count);
  else if (st_ == EIG_F32 && dt_ == EIG_F32) k_convert<float, float><<<grid, 256, 0, st>>>((const float*)src, (float*)dst, count);
  else return EIG_EINVAL;
  EIG_LAUNCH_CHECK("k_convert");
  return EIG_OK;
}

template <typename T>
__global__ void k_col_sumsq(const T* __restrict__ X, int k, int64_t n, double* __restrict__ part) {
  // thread handles column j = tid % k of rows tid/k, tid/k + stride...
  __shared__ double red[1024];
  const int rows_per_pass = blockDim.x / k;
  const int j = threadIdx.x % k, rr = threadIdx.x / k;
  double s = 0.0;
  if (rr < rows_per_pass) {
    for (int64_t r = blockIdx.x * (int64_t)rows_per_pass + rr; r < n; r += (int64_t)gridDim.x * rows_per_pass) {
      const double v = (double)X[r * k + j];
      s += v * v;
    }
  }
  red[threadIdx.x] = (rr < rows_per_pass) ? s : 0.0;
  __syncthreads();
  if (threadIdx.x < k) {
    double t = 0.0;
    for (int q = 0; q < rows_per_pass; ++q) t += red[q * k + threadIdx.x];
    part[(size_t)blockIdx.x * k + threadIdx.x] = t;
  }
}

size_t colsum_scratch_bytes(int k) { return (size_t)num_sms() * 4 * k * 8 + 256; }

eig_status col_sumsq(const void* X, int k, int64_t n, eig_dtype vt, double* out, void* part, cudaStream_t st) {
  if (k < 1 || k > 256) return EIG_EINVAL;
  const int grid = num_sms() * 4;
  const int threads = (256 / k) * k;
  if (vt == EIG_F32) k_col_sumsq<float><<<grid, threads, 0, st>>>((const float*)X, k, n, (double*)part);
  else if (vt == EIG_F64) k_col_sumsq<double><<<grid, threads, 0, st>>>((const double*)X, k, n, (double*)part);
  else return EIG_EINVAL;
  EIG_LAUNCH_CHECK("k_col_sumsq");
  return reduce_partials((const double*)part, grid, k, out, st);
}

// ---------------------------------------------------------------------------------------
// fused LOBPCG update: thread per (row, column j); a CTA covers rows_per_cta rows
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ double jacobi_den(double d, double th, double floor) {
  double den = d - th;
  const double mag = fmax(fabs(den), floor);
  return den < 0.0 ? -mag : mag;
}

// Jacobi denominator H_ii - theta, magnitude floored; FP32 is enough for a preconditioner.
__device__ __forceinline__ float jacobi_den_f(double d, double th, float floor) {
  const float den = (float)d - (float)th;
  const float mag = fmaxf(fabsf(den), floor);
  return den < 0.0f ? -mag : mag;
}

// Thread per (row, CPT adjacent columns), three CTAs per SM (80 registers); rows are read with
// 16-byte moves, the Rayleigh-Ritz coefficients come from shared memory as CPT-wide vectors.  In
// place: the lanes of a row (one warp) have read all their inputs before any of them writes
// (__syncwarp).
template <typename T, int NB>
__global__ void __launch_bounds__(256, 3)
k_lobpcg_update(T* __restrict__ X, T* __restrict__ W, T* __restrict__ P, T* __restrict__ HX,
                const T* __restrict__ HW, T* __restrict__ HP, const double* __restrict__ C, int k,
                const double* __restrict__ theta, const double* __restrict__ diagH, double floor, int precond,
                int64_t n, double* __restrict__ part) {
  constexpr int CPT = (NB * (int)sizeof(T) >= 16) ? 16 / (int)sizeof(T) : NB;
  constexpr int LPR = NB / CPT;           // lanes per row
  constexpr int RPP = 256 / LPR;          // rows per pass
  __shared__ __align__(16) T sC[3 * NB * NB];
  __shared__ double red[256 * CPT];
  for (int i = threadIdx.x; i < k * NB; i += blockDim.x) sC[i] = (T)C[i];
  __syncthreads();
  const int j0 = (threadIdx.x % LPR) * CPT, rr = threadIdx.x / LPR;
  double th[CPT];
#pragma unroll
  for (int c = 0; c < CPT; ++c) th[c] = theta[j0 + c];
  double rsq[CPT];
#pragma unroll
  for (int c = 0; c < CPT; ++c) rsq[c] = 0.0;
  float rh[CPT], rl[CPT];  // FP32 rows: double-float sums of squares
#pragma unroll
  for (int c = 0; c < CPT; ++c) rh[c] = rl[c] = 0.0f;
  // acc += A_row * Cblk[:, j0..j0+CPT) and hacc += HA_row * Cblk
  auto gemv2 = [&](const T* A, const T* HA, int cb, Vec<T, CPT>& acc, Vec<T, CPT>& hacc) {
#pragma unroll
    for (int l0 = 0; l0 < NB; l0 += CPT) {
      const Vec<T, CPT> a = VecIO<T, CPT>::ld(A + l0);
      const Vec<T, CPT> ha = VecIO<T, CPT>::ld(HA + l0);
#pragma unroll
      for (int v = 0; v < CPT; ++v) {
        const Vec<T, CPT> cv = VecIO<T, CPT>::ld(sC + (cb + l0 + v) * NB + j0);
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
          acc.v[c] = fma(a.v[v], cv.v[c], acc.v[c]);
          hacc.v[c] = fma(ha.v[v], cv.v[c], hacc.v[c]);
        }
      }
    }
  };
  // the loop bound is uniform across the CTA so that __syncwarp sees every lane
  for (int64_t base = blockIdx.x * (int64_t)RPP; base < n; base += (int64_t)gridDim.x * RPP) {
    const int64_t r = base + rr;
    const bool valid = r < n;
    Vec<T, CPT> xn, hxn, pn, hpn, wn;
    xn.zero(); hxn.zero(); pn.zero(); hpn.zero(); wn.zero();
    if (valid) {
      if (k == NB) {
        xn = VecIO<T, CPT>::ld(X + r * NB + j0);
        hxn = VecIO<T, CPT>::ld(HX + r * NB + j0);
      } else {
        gemv2(X + r * NB, HX + r * NB, 0, xn, hxn);
        gemv2(W + r * NB, HW + r * NB, NB, pn, hpn);
        if (k == 3 * NB) gemv2(P + r * NB, HP + r * NB, 2 * NB, pn, hpn);
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
          xn.v[c] += pn.v[c];
          hxn.v[c] += hpn.v[c];
        }
      }
      const double d = diagH[r];
#pragma unroll
      for (int c = 0; c < CPT; ++c) {
        const T res = hxn.v[c] - (T)th[c] * xn.v[c];
        if (sizeof(T) == 4) {
          // exact FP32 square summed in double-float
          const float f = (float)res, p = f * f, pe = fmaf(f, f, -p);
          const float s = rh[c] + p, bb = s - rh[c];
          rl[c] += ((rh[c] - (s - bb)) + (p - bb)) + pe;
          rh[c] = s;
          wn.v[c] = precond == 1 ? (T)(f / jacobi_den_f(d, th[c], (float)floor)) : res;
        } else {
          rsq[c] = fma((double)res, (double)res, rsq[c]);
          wn.v[c] = precond == 1 ? (T)((double)res / jacobi_den(d, th[c], floor)) : res;
        }
      }
    }
    __syncwarp();
    if (valid) {
      if (k != NB) {
        VecIO<T, CPT>::st(X + r * NB + j0, xn);
        VecIO<T, CPT>::st(HX + r * NB + j0, hxn);
        VecIO<T, CPT>::st(P + r * NB + j0, pn);
        VecIO<T, CPT>::st(HP + r * NB + j0, hpn);
      }
      VecIO<T, CPT>::st(W + r * NB + j0, wn);
    }
  }
#pragma unroll
  for (int c = 0; c < CPT; ++c) red[threadIdx.x * CPT + c] = rsq[c] + (double)rh[c] + (double)rl[c];
  __syncthreads();
  for (int j = threadIdx.x; j < NB; j += blockDim.x) {
    const int g = j / CPT, c = j % CPT;
    double t = 0.0;
    for (int q = 0; q < RPP; ++q) t += red[(q * LPR + g) * CPT + c];
    part[(size_t)blockIdx.x * NB + j] = t;
  }
}

int update_grid(int64_t n) {
  int64_t g = (n + 63) / 64;
  const int64_t cap = (int64_t)num_sms() * 8;
  return (int)(g < cap ? (g < 1 ? 1 : g) : cap);
}

eig_status lobpcg_update(void* X, void* W, void* P, void* HX, void* HW, void* HP, const double* C, int k, int nb,
                         const double* theta, const double* diagH, double floor, int precond, int64_t n,
                         eig_dtype vt, double* part, int nparts_max, int* nparts_out, cudaStream_t st) {
  if (nb < 1 || nb > 32 || 32 % nb != 0 || (k != nb && k != 2 * nb && k != 3 * nb)) return EIG_EINVAL;
  const int grid = update_grid(n);
  if (grid > nparts_max) return EIG_EINVAL;
#define EIG_UPD(T, NBV)                                                                                    \
  k_lobpcg_update<T, NBV><<<grid, 256, 0, st>>>((T*)X, (T*)W, (T*)P, (T*)HX, (const T*)HW, (T*)HP, C, k, theta, \
                                                diagH, floor, precond, n, part)
#define EIG_UPD_NB(T)                  \
  switch (nb) {                        \
    case 1: EIG_UPD(T, 1); break;      \
    case 2: EIG_UPD(T, 2); break;      \
    case 4: EIG_UPD(T, 4); break;      \
    case 8: EIG_UPD(T, 8); break;      \
    case 16: EIG_UPD(T, 16); break;    \
    default: EIG_UPD(T, 32); break;    \
  }
  if (vt == EIG_F32) {
    EIG_UPD_NB(float)
  } else if (vt == EIG_F64) {
    EIG_UPD_NB(double)
  } else {
    return EIG_EINVAL;
  }
#undef EIG_UPD_NB
#undef EIG_UPD
  EIG_LAUNCH_CHECK("k_lobpcg_update");
  *nparts_out = grid;
  return EIG_OK;
}

template <typename T>
__global__ void k_jacobi(T* __restrict__ R, const double* __restrict__ theta, const double* __restrict__ diagH,
                         double floor, int nb, int64_t n) {
  const int64_t total = n * nb;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / nb;
    const int j = (int)(i % nb);
    R[i] = (T)((double)R[i] / jacobi_den(diagH[r], theta[j], floor));
  }
}

eig_status jacobi_block(void* R, const double* theta, const double* diagH, double floor, int nb, int64_t n,
                        eig_dtype vt, cudaStream_t st) {
  const int grid = num_sms() * 8;
  if (vt == EIG_F32) k_jacobi<float><<<grid, 256, 0, st>>>((float*)R, theta, diagH, floor, nb, n);
  else if (vt == EIG_F64) k_jacobi<double><<<grid, 256, 0, st>>>((double*)R, theta, diagH, floor, nb, n);
  else return EIG_EINVAL;
  EIG_LAUNCH_CHECK("k_jacobi");
  return EIG_OK;
}

}  // namespace eig
