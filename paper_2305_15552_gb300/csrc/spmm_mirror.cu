// Mirrored row-stream SpMM: Y = H X with H = U + U_strict^T given by its stored upper triangle U
// (Sec. 1; Eqs. upd1-upd2; the half storage of Sec. 3.1 is the input format), GB300 layout.
//
// Why mirror.  In a half-stored kernel every stored h_ij feeds a gather y_i += h_ij x_j and a
// scatter z_j += h_ij x_i; on sm_103a both run out of shared memory and the scatter costs a
// read-modify-write of an nb-wide row per nonzero.  Here the plan expands U once, on the
// device, into both triangles, so the kernel only gathers.
//
// What bounds it.  Every entry of H costs one gather of an nb-wide X row from shared memory
// (64 bytes at nb = 16 in FP32), so at nb >= 16 the shared-memory pipe (128 bytes per clock
// per SM), not HBM, is the limit; at nb <= 8 it is HBM.  The layout is built so that the pipe
// moves little else and never stalls on bank conflicts, and so that HBM sees enough bytes in
// flight:
//   * one lane owns one row: per row block (256 rows, one CTA of 8 warps) and per panel of
//     column tiles, the rows are ranked by their entry count and warp w's lane l takes the
//     row of rank 32 w + l; the warp steps through its longest row's count, shorter rows
//     padded with zero-valued entries (a few percent);
//   * a matrix with fewer row blocks than SMs ranks its rows within two halves of the row block
//     instead, each half's warps a CTA of their own (row_groups);
//   * each step, lane l gathers its entry's whole X row in 16-byte pieces, starting at a
//     lane-dependent piece, and the entries are ordered so that lane l reads a row of class
//     (l + step) mod 8 (X row index mod 8): the 8 lanes of every shared-memory phase then hit
//     distinct banks for any nb;
//   * the entries (uint16 panel-local column + value) stream from HBM straight into registers,
//     several 8-step blocks ahead, bypassing L1 and evicted first from L2; each lane loads
//     only its own entries (16 + 32 bytes per block in FP32), a warp's 16-byte pieces side by side,
//     so that nothing is loaded twice and a load is four full wavefronts (with a lane's 32 bytes of
//     values side by side instead, n = 2M, 400 nonzeros a row took 1.80 ms at nb = 16 and 1.09 at
//     nb = 8, against 1.74 and 1.02);
//   * X: the X rows of the row block's column tiles (64 rows each) are staged in shared
//     memory by bulk copies (TMA) in panels of at most 24 tiles, evicted last from L2; a row
//     block whose tiles do not fit takes several panels, its rows' partial sums added in Y
//     in panel order.
// Every sum runs in a fixed order (steps in stream order, panels in order): Y is bitwise
// reproducible.
//
// Small FP64 matrices (FP64 values, n < 65,536: direct_plan) take the streams without row blocks
// and panels; see k_spmm_direct.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "spmm.cuh"
#include "tma.cuh"
#include "vec.cuh"

namespace eig {

namespace {

constexpr int kMR = 256;                 // rows per row block (one CTA)
constexpr int kMC = 64;                  // columns per tile (unit of X staging)
constexpr int kW = 8;                    // warps per CTA; warp w takes the rows of rank [32 w, 32 w + 32)
constexpr int kRW = kMR / kW;            // rows per warp
constexpr int kBS = 8;                   // steps per streamed block
constexpr int kBE = 32 * kBS;            // entries per block (32 lanes)
constexpr int kPT = 24;                  // tiles per panel at most (<= 32: one lane stages one tile)
constexpr int kPR = kPT * kMC;           // staged X rows per panel at most; 8 zero rows follow
constexpr int kL2 = 6;                   // streamed blocks prefetched into L2 ahead of use
constexpr int kDenseTile = 3000;         // mean stored entries of a tile (see dense_tiles)

// ---------------------------------------------------------------------------------------
// Plan: the strictly lower triangle as a CSR beside the upper one, built from U without sorting and
// without atomics on values.  A row of H is its row of the lower CSR, then its row of U.
// ---------------------------------------------------------------------------------------

// First of the ascending c[a, b) that is at least lim, expected near a.
__device__ __forceinline__ int64_t first_near(const int32_t* __restrict__ c, int64_t a, int64_t b, int64_t lim) {
  int64_t step = 1;
  while (a < b && (int64_t)c[min64(a + step, b) - 1] < lim) {
    a = min64(a + step, b);
    step *= 2;
  }
  for (int64_t e = min64(a + step, b); a < e;) {
    const int64_t m = (a + e) >> 1;
    if ((int64_t)c[m] < lim) a = m + 1; else e = m;
  }
  return a;
}

// First of the ascending c[a, b) that is at least lim.
__device__ __forceinline__ int64_t first_from(const int32_t* __restrict__ c, int64_t a, int64_t b, int64_t lim) {
  while (a < b) {
    const int64_t m = (a + b) >> 1;
    if ((int64_t)c[m] < lim) a = m + 1; else b = m;
  }
  return a;
}

// Index of tile column J among the nt <= 32 ascending columns tc, which hold it: slot[J mod 256] names
// one tile (J < 2^25 in the upper bits, its index in the lower five); where it names another, by search.
__device__ __forceinline__ int tile_index(const uint32_t* slot, const int32_t* tc, int nt, int32_t J) {
  const uint32_t x = slot[J & 255];
  if (x >> 5 == (uint32_t)J) return (int)(x & 31u);
  int lo = 0;
  for (int hi = nt - 1; lo < hi;) {
    const int mid = (lo + hi) >> 1;
    if (tc[mid] < J) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// CTA per row block, warp per row (32 rows each), the row block's upper tiles (256 rows x 64 columns) in
// groups of kCountTiles.  Per tile: seg[t * 256 + row] (unless seg is null), the offset in its row of the
// row's first entry in the tile (preset to "none" where there is none); cnt[t * 64 + j], the strictly-upper
// entries of each column (integer atomics in shared memory: order independent); the largest total of a
// tile; and, in the bitmap of the full matrix, the transposed tiles (64 rows of this row block as a column
// block of the row block that holds the tile's columns).  A group takes up each row where the group before
// it left it, so that a row is read once however many groups there are.
constexpr int kCountTiles = 32;
__global__ void __launch_bounds__(kMR) k_mir_colcounts(int64_t n, const int64_t* __restrict__ rowptr,
                                                       const int32_t* __restrict__ col,
                                                       const int64_t* __restrict__ tile_ptr,
                                                       const int32_t* __restrict__ tile_col, int64_t words_per_rb,
                                                       int32_t* __restrict__ seg, int32_t* __restrict__ cnt,
                                                       unsigned* __restrict__ bitmap, int* __restrict__ most) {
  __shared__ int s_cnt[kCountTiles][kMC];
  __shared__ int32_t s_tc[kCountTiles];
  __shared__ uint32_t s_slot[256];          // tile column and index, at the column mod 256 (one of them)
  __shared__ unsigned s_sub[kCountTiles];   // bit q: the 64 rows q have strictly-upper entries in the tile
  __shared__ int32_t s_next[kMR];           // per row: offset of the first chunk that the groups so far left
  const int64_t I = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  s_next[tid] = 0;
  const int64_t t0 = tile_ptr[I], t1 = tile_ptr[I + 1];
  for (int64_t g0 = t0; g0 < t1; g0 += kCountTiles) {
    const int nt = (int)min64(kCountTiles, t1 - g0);
    __syncthreads();
    for (int i = tid; i < kCountTiles * kMC; i += kMR) (&s_cnt[0][0])[i] = 0;
    if (tid < kCountTiles) {
      s_tc[tid] = tid < nt ? tile_col[g0 + tid] : INT32_MAX;
      s_sub[tid] = 0u;
    }
    s_slot[tid] = 0xffffffffu;
    __syncthreads();
    if (tid < nt) s_slot[s_tc[tid] & 255] = ((uint32_t)s_tc[tid] << 5) | tid;
    __syncthreads();
    const int32_t first = s_tc[0], last = s_tc[nt - 1];
    const bool again = g0 + nt < t1;   // another group follows
    for (int lr = w; lr < kMR; lr += kW) {
      const int64_t r = I * kMR + lr;
      if (r >= n) break;
      const int64_t e0 = rowptr[r], e1 = rowptr[r + 1];
      // tile column of the entry before the chunk, where it matters: an entry before the first chunk
      // belongs to an earlier group
      int32_t before = -1;
      int64_t q0 = e0 + s_next[lr];
      for (; q0 < e1; q0 += 128) {
        int32_t cs[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) cs[u] = q0 + 32 * u + lane < e1 ? col[q0 + 32 * u + lane] : INT32_MAX;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int32_t c = cs[u], J = c / kMC;
          const int32_t up = __shfl_up_sync(0xffffffffu, J, 1);
          if (c != INT32_MAX && J >= first && J <= last) {
            const int lo = tile_index(s_slot, s_tc, nt, J);
            if ((lane == 0 ? before : up) != J) {
              if (seg) seg[(g0 + lo) * kMR + lr] = (int32_t)(q0 + 32 * u + lane - e0);
              // a row whose only entry here is its diagonal has nothing strictly upper, but the tile
              // then belongs to this row block already
              if ((s_sub[lo] >> (lr / kMC) & 1u) == 0u) atomicOr(&s_sub[lo], 1u << (lr / kMC));
            }
            if ((int64_t)c != r) atomicAdd(&s_cnt[lo][c - J * kMC], 1);
          }
          before = __shfl_sync(0xffffffffu, J, 31);
        }
        if (before > last) {   // also after the row's end (INT32_MAX)
          bool more = false;
#pragma unroll
          for (int u = 0; u < 4; ++u) more = more || (cs[u] != INT32_MAX && cs[u] / kMC > last);
          if (again && !__any_sync(0xffffffffu, more)) q0 = e1;   // else the next group starts with this chunk
          break;
        }
      }
      if (again && lane == 0) s_next[lr] = (int32_t)(min64(q0, e1) - e0);
    }
    __syncthreads();
    for (int t = w; t < nt; t += kW) {
      int total = 0;
#pragma unroll
      for (int h = 0; h < kMC; h += 32) {
        const int x = s_cnt[t][h + lane];
        cnt[(g0 + t) * kMC + h + lane] = x;
        total += x;
      }
      total = warp_sum(total);
      if (lane == 0 && total) atomicMax(most, total);
      if (lane < 4 && (s_sub[t] >> lane & 1u)) {
        const int64_t Q = I * (kMR / kMC) + lane;
        atomicOr(bitmap + s_tc[t] / (kMR / kMC) * words_per_rb + (Q >> 5), 1u << (Q & 31));
      }
    }
  }
}

// Thread per column c: offsets of each upper tile's contribution to row c's lower part (tiles of
// c's column block in ascending row-block order), and the lower-part length of row c.
__global__ void k_mir_coloffsets(int64_t n, const int64_t* __restrict__ jt_ptr, const int32_t* __restrict__ jt_tile,
                                 const int32_t* __restrict__ cnt, int32_t* __restrict__ off,
                                 int64_t* __restrict__ lower) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= n) return;
  const int64_t J = c / kMC;
  const int j = (int)(c - J * kMC);
  int64_t run = 0;
  for (int64_t p = jt_ptr[J]; p < jt_ptr[J + 1]; ++p) {
    const int64_t t = jt_tile[p];
    off[t * kMC + j] = (int32_t)run;
    run += cnt[t * kMC + j];
  }
  lower[c] = run;
}

// Exclusive prefix sums in three passes over chunks of kScanChunk values: chunk sums, the sums'
// own prefix (one CTA), the chunks.
constexpr int kScanThreads = 256, kScanChunk = 4 * kScanThreads;

__device__ __forceinline__ int64_t scan_block(int64_t v, int64_t* total) {   // exclusive, over the CTA
  __shared__ int64_t s_w[kScanThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  __syncthreads();   // the previous use of s_w is over
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  int64_t base = 0, all = 0;
#pragma unroll
  for (int i = 0; i < kScanThreads / 32; ++i) {
    if (i < w) base += s_w[i];
    all += s_w[i];
  }
  *total = all;
  return base + x - v;
}
__global__ void __launch_bounds__(kScanThreads) k_scan_sums(const int64_t* __restrict__ v, int64_t n,
                                                            int64_t* __restrict__ sums) {
  int64_t s = 0, total;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t e = blockIdx.x * (int64_t)kScanChunk + i * kScanThreads + threadIdx.x;
    if (e < n) s += v[e];
  }
  scan_block(s, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}
__global__ void __launch_bounds__(kScanThreads) k_scan_tops(int64_t* __restrict__ sums, int64_t m) {
  int64_t run = 0;
  for (int64_t b = 0; b < m; b += kScanThreads) {
    const int64_t e = b + threadIdx.x;
    int64_t total;
    const int64_t x = scan_block(e < m ? sums[e] : 0, &total);
    if (e < m) sums[e] = run + x;
    run += total;
  }
}
// out[0..n]: out[n] is the total.
__global__ void __launch_bounds__(kScanThreads) k_scan_chunks(const int64_t* __restrict__ v, int64_t n,
                                                              const int64_t* __restrict__ sums,
                                                              int64_t* __restrict__ out) {
  int64_t run = sums[blockIdx.x];
  for (int i = 0; i < 4; ++i) {
    const int64_t e = blockIdx.x * (int64_t)kScanChunk + i * kScanThreads + threadIdx.x;
    int64_t total;
    const int64_t x = scan_block(e < n ? v[e] : 0, &total);
    if (e < n) out[e] = run + x;
    if (e == n - 1) out[n] = run + x + v[e];
    run += total;
  }
}
static eig_status exclusive_scan(const int64_t* v, int64_t n, int64_t* out, int64_t* sums, cudaStream_t st) {
  const int64_t m = (n + kScanChunk - 1) / kScanChunk;
  k_scan_sums<<<(unsigned)m, kScanThreads, 0, st>>>(v, n, sums);
  EIG_LAUNCH_CHECK("k_scan_sums");
  k_scan_tops<<<1, kScanThreads, 0, st>>>(sums, m);
  EIG_LAUNCH_CHECK("k_scan_tops");
  k_scan_chunks<<<(unsigned)m, kScanThreads, 0, st>>>(v, n, sums, out);
  EIG_LAUNCH_CHECK("k_scan_chunks");
  return EIG_OK;
}

// Strict lower part: entry (r, c) of upper tile t goes to row c, after the contributions of
// earlier row blocks, at its rank among the tile's entries of column c (rows ascending).  CTA per tile:
// eight lanes read a row's entries (up to 24 of them kept in registers, all loads in flight); ranks come
// from a column-major bitmap; the tile is transposed in shared memory and every column's entries,
// consecutive in row c, are written by one warp.  (A thread per row reading its entries and writing each
// to its row took 2.5 ms for 1.5e8 entries; this takes 1.8.)  Dynamic shared memory: `most` values and
// row bytes.
template <typename V>
__global__ void __launch_bounds__(kMR, 6) k_mir_lower(int64_t n, const int64_t* __restrict__ rowptr,
                                                   const int32_t* __restrict__ col, const V* __restrict__ val,
                                                   const int32_t* __restrict__ tile_rb,
                                                   const int32_t* __restrict__ tile_cb,
                                                   const int32_t* __restrict__ seg, const int32_t* __restrict__ off,
                                                   const int64_t* __restrict__ lptr, int most,
                                                   int32_t* __restrict__ lcol, V* __restrict__ lval) {
  constexpr int NW = kMR / 32, RP = kMR / 32, LD = 3;   // rows per lane group, entries kept per lane and row
  __shared__ unsigned bits[NW][kMC];    // bit b of word [w][j]: entry (row 32 w + b, column j)
  __shared__ uint8_t before[NW][kMC];   // entries of the column in earlier words (at most 224)
  __shared__ int start[kMC + 1];
  extern __shared__ __align__(16) unsigned char sm_tile[];
  V* sv = reinterpret_cast<V*>(sm_tile);
  uint8_t* sr = reinterpret_cast<uint8_t*>(sv + most);
  const int64_t t = blockIdx.x;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, sub = tid & 7, rr0 = tid >> 3;
  const int64_t r0 = (int64_t)tile_rb[t] * kMR, cb0 = (int64_t)tile_cb[t] * kMC;
  for (int i = tid; i < NW * kMC; i += kMR) (&bits[0][0])[i] = 0u;
  // rows rr0 + 32 u: first entry in the tile (this lane's), end of the row
  int64_t e0[RP];
  int left[RP];   // entries of the row from e0 on
#pragma unroll
  for (int u = 0; u < RP; ++u) {
    const int64_t r = r0 + rr0 + 32 * u;
    e0[u] = 0;
    left[u] = 0;
    if (r < n) {
      const int64_t a = rowptr[r], b = rowptr[r + 1];
      const int64_t e = a + seg[t * kMR + rr0 + 32 * u];
      if (e < b) {
        e0[u] = e;
        left[u] = (int)(b - e);
      }
    }
  }
  unsigned jp[RP];   // columns in the tile, a byte each (255: none)
#pragma unroll
  for (int u = 0; u < RP; ++u) {
    jp[u] = 0u;
#pragma unroll
    for (int d = 0; d < LD; ++d) {
      const int q = sub + 8 * d;
      const int64_t c = q < left[u] ? col[e0[u] + q] : INT64_MAX;
      jp[u] |= (c < cb0 + kMC && c != r0 + rr0 + 32 * u ? (unsigned)(c - cb0) : 255u) << (8 * d);
    }
  }
  auto jof = [&](int u, int d) { return (int)(jp[u] >> (8 * d) & 255u); };
  __syncthreads();
  // entries beyond the registers
  auto rest = [&](int u, auto f) {
    for (int q = sub + 8 * LD; q < left[u]; q += 8) {
      const int64_t c = col[e0[u] + q];
      if (c >= cb0 + kMC) break;
      if (c != r0 + rr0 + 32 * u) f((int)(c - cb0), q);
    }
  };
#pragma unroll
  for (int u = 0; u < RP; ++u) {
#pragma unroll
    for (int d = 0; d < LD; ++d)
      if (jof(u, d) != 255) atomicOr(&bits[u][jof(u, d)], 1u << rr0);
    rest(u, [&](int jj, int) { atomicOr(&bits[u][jj], 1u << rr0); });
  }
  __syncthreads();
  if (w == 0) {
    int x[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int total = 0;
#pragma unroll
      for (int q = 0; q < NW; ++q) {
        before[q][2 * lane + h] = (uint8_t)total;
        total += __popc(bits[q][2 * lane + h]);
      }
      x[h] = total;
    }
    int y = x[0] + x[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    start[2 * lane] = y - x[0] - x[1];
    start[2 * lane + 1] = y - x[1];
    if (lane == 31) start[kMC] = y;
  }
  __syncthreads();
  auto put = [&](int u, int jj, int q) {
    const int at = start[jj] + before[u][jj] + __popc(bits[u][jj] & ((1u << rr0) - 1u));
    sr[at] = (uint8_t)(rr0 + 32 * u);
    sv[at] = val[e0[u] + q];
  };
#pragma unroll
  for (int u = 0; u < RP; ++u) {
#pragma unroll
    for (int d = 0; d < LD; ++d)
      if (jof(u, d) != 255) put(u, jof(u, d), sub + 8 * d);
    rest(u, [&](int jj, int q) { put(u, jj, q); });
  }
  __syncthreads();
  for (int jj = w; jj < kMC; jj += NW) {
    const int q0 = start[jj], m = start[jj + 1] - q0;
    if (!m) continue;
    const int64_t pos = lptr[cb0 + jj] + off[t * kMC + jj];
    for (int i = lane; i < m; i += 32) {
      lcol[pos + i] = (int32_t)(r0 + sr[q0 + i]);
      lval[pos + i] = sv[q0 + i];
    }
  }
}

// The same for tiles of fewer entries (see dense_tiles): thread per row, which searches its row for the tile's
// first column instead of reading an offset kept per (tile, row), and writes each entry to its place.
template <typename V>
__global__ void __launch_bounds__(kMR) k_mir_lower_few(int64_t n, const int64_t* __restrict__ rowptr,
                                                       const int32_t* __restrict__ col, const V* __restrict__ val,
                                                       const int32_t* __restrict__ tile_rb,
                                                       const int32_t* __restrict__ tile_cb,
                                                       const int32_t* __restrict__ off,
                                                       const int64_t* __restrict__ lptr, int32_t* __restrict__ lcol,
                                                       V* __restrict__ lval) {
  constexpr int NW = kMR / 32;
  __shared__ unsigned bits[NW][kMC];   // bit b of word [w][j]: entry (row 32 w + b, column j)
  const int64_t t = blockIdx.x;
  const int tid = threadIdx.x, w = tid >> 5;
  for (int i = tid; i < NW * kMC; i += kMR) (&bits[0][0])[i] = 0u;
  const int64_t r = (int64_t)tile_rb[t] * kMR + tid, cb0 = (int64_t)tile_cb[t] * kMC;
  int64_t a = 0, b = 0;
  if (r < n) {
    b = rowptr[r + 1];
    a = first_from(col, rowptr[r], b, cb0);
  }
  __syncthreads();
  int64_t e = a;   // past the row's last entry in the tile
  for (; e < b; ++e) {
    const int64_t c = col[e];
    if (c >= cb0 + kMC) break;
    if (c != r) atomicOr(&bits[w][c - cb0], 1u << (tid & 31));
  }
  __syncthreads();
  for (int64_t k = a; k < e; ++k) {
    const int64_t c = col[k];
    if (c == r) continue;
    const int j = (int)(c - cb0);
    int rank = __popc(bits[w][j] & ((1u << (tid & 31)) - 1u));
    for (int q = 0; q < w; ++q) rank += __popc(bits[q][j]);
    const int64_t pos = lptr[c] + off[t * kMC + j] + rank;
    lcol[pos] = (int32_t)r;
    lval[pos] = val[k];
  }
}

// ---------------------------------------------------------------------------------------
// Plan: the row streams
// ---------------------------------------------------------------------------------------

// Last column block of panel p (-1 for a panel without tiles).
__device__ __forceinline__ int64_t panel_last_cb(const int32_t* __restrict__ pt0, const int32_t* __restrict__ pnt,
                                                 const int32_t* __restrict__ tcol, int64_t p) {
  return pnt[p] > 0 ? (int64_t)tcol[pt0[p] + pnt[p] - 1] : -1;
}

// Thread per row: entries the row has in each panel of its row block, and those of them left of the
// diagonal (binary searches per panel but the last).
__global__ void k_rs_counts(int64_t n, const int64_t* __restrict__ lptr, const int32_t* __restrict__ lcol,
                            const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                            const int32_t* __restrict__ rbp, const int32_t* __restrict__ pt0,
                            const int32_t* __restrict__ pnt, const int32_t* __restrict__ tcol,
                            uint16_t* __restrict__ cnt, uint16_t* __restrict__ cntl) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= n) return;
  const int64_t I = r / kMR;
  const int lr = (int)(r - I * kMR);
  int64_t kl = lptr[r], ku = rowptr[r];
  const int64_t el = lptr[r + 1], eu = rowptr[r + 1];
  const bool many = rbp[I + 1] - rbp[I] > 8;   // panels, with few entries of the row each
  for (int64_t p = rbp[I]; p < rbp[I + 1]; ++p) {
    const bool last = p + 1 == rbp[I + 1];
    const int64_t lim = (panel_last_cb(pt0, pnt, tcol, p) + 1) * kMC;   // first column past the panel
    const int64_t nl = last ? el : (many ? first_near(lcol, kl, el, lim) : first_from(lcol, kl, el, lim));
    const int64_t nu = last ? eu : (many ? first_near(col, ku, eu, lim) : first_from(col, ku, eu, lim));
    cnt[p * kMR + lr] = (uint16_t)(nl - kl + nu - ku);
    cntl[p * kMR + lr] = (uint16_t)(nl - kl);
    kl = nl;
    ku = nu;
  }
}

// CTA per panel: the panel's 256 rows ranked by entry count (descending, ties by row) within each
// group of `gr` consecutive rows (256: one group), so that each warp's 32 lanes take rows of
// near-equal length; steps of each warp = its longest row.
__global__ void __launch_bounds__(kMR) k_rs_rank(const uint16_t* __restrict__ cnt, int gr, uint8_t* __restrict__ perm,
                                                 int32_t* __restrict__ steps) {
  __shared__ uint16_t c[kMR];
  const int64_t p = blockIdx.x;
  const int t = threadIdx.x;
  c[t] = cnt[p * kMR + t];
  __syncthreads();
  const int mine = c[t];
  const int g0 = t / gr * gr;
  int rank = g0;
  for (int u = g0; u < g0 + gr; ++u) {
    const int o = c[u];
    rank += (o > mine) || (o == mine && u < t);
  }
  perm[p * kMR + rank] = (uint8_t)t;
  if (rank % kRW == 0) steps[p * kW + rank / kRW] = mine;
}

// Values of a streamed block: 16-byte pieces (kEpp consecutive steps of one lane), piece-major, so
// that a warp's load of one piece per lane is contiguous.  Columns: [lane][step] (16 bytes a lane).
template <typename V> struct BlkPiece { static constexpr int kEpp = 16 / (int)sizeof(V); };
template <typename V>
__device__ __forceinline__ int64_t blk_value_at(int lane, int step) {
  constexpr int E = BlkPiece<V>::kEpp;
  return (int64_t)(step / E) * 32 * E + lane * E + step % E;
}

// Order of a row's entries in its lane.  The entries of a panel fall into 8 classes (X row mod 8);
// lane l wants class (l + k) mod 8 at step k, so that the 8 lanes of a shared-memory phase read rows of
// 8 distinct classes.  The placement follows from the eight counts alone, level by level so that what
// cannot be had stays at the end of the stream: of the steps that want a parity, the first as many as
// the row has entries of it get one (the last ones take the other parity's surplus: the only steps that
// cost a conflict at nb >= 16 in FP32); of those that want a class mod 4 the same within the parity, of
// those that want a class mod 8 within the class mod 4.
// Step of entry i (columns ascending) of class c (16-byte aligned: two loads a place):
struct alignas(16) ClassPlace {
  int own;            // i < own: the i-th step that wants c
  int in8, base8;     // the next in8: steps that want c ^ 4, from its base8-th on
  int skip, in4;      // then the surplus of the class mod 4 (the c with bit 2 after the other one): its first
  int base4;          // in4 in steps that want (c ^ 2) mod 4, from the base4-th on,
  int base2;          // the rest in steps of the other parity, from the base2-th on
  int to_32_bytes;
};
__device__ __forceinline__ int half_from(int m, int first) { return m > first ? (m - first + 1) >> 1 : 0; }
__device__ __forceinline__ int class_step(const ClassPlace& g, int c, int l, int i) {
  if (i < g.own) return ((c - l) & 7) + 8 * i;
  int j = i - g.own;
  if (j < g.in8) return (((c ^ 4) - l) & 7) + 8 * (g.base8 + j);
  j += g.skip - g.in8;
  if (j < g.in4) return (((c ^ 2) - l) & 3) + 4 * (g.base4 + j);
  return (((c ^ 1) - l) & 1) + 2 * (g.base2 + j - g.in4);
}
// Places of class c = lane mod 8 from its count nc, for lane l's stream of m steps (warp-wide call).
__device__ __forceinline__ ClassPlace class_place(int c, int nc, int l, int m) {
  const unsigned all = 0xffffffffu;
  const int o1 = (c - l) & 1, o2 = (c - l) & 3, o3 = (c - l) & 7;
  const int nc4 = __shfl_xor_sync(all, nc, 4), nq = nc + nc4;             // entries of the class mod 4
  const int nq2 = __shfl_xor_sync(all, nq, 2), np = nq + nq2;             // of the parity
  const int np1 = __shfl_xor_sync(all, np, 1);
  const int mp = min(np, half_from(m, o1));                               // its steps that it keeps
  const int cap4 = half_from(mp, (o2 - o1) >> 1);                         // of these, wanted by c mod 4
  const int cap4x = __shfl_xor_sync(all, cap4, 2);
  const int mq = min(nq, cap4);
  const int in4 = min(nq - mq, max(0, cap4x - nq2)), rest = nq - mq - in4;
  const int restx = __shfl_xor_sync(all, rest, 2);
  const int cap8 = half_from(mq, (o3 - o2) >> 2);                         // wanted by c
  const int cap8x = __shfl_xor_sync(all, cap8, 4);
  const int in8 = min(max(0, nc - cap8), max(0, cap8x - nc4));
  const int left = max(0, nc - cap8) - in8, leftx = __shfl_xor_sync(all, left, 4);
  return ClassPlace{cap8, in8, nc4, (c & 4) ? leftx : 0, in4, nq2, np1 + ((c & 2) ? restx : 0), 0};
}

// Mask of the lanes of `in` whose class bits (ballots b0, b1, b2) equal c.
__device__ __forceinline__ unsigned class_mask(unsigned in, unsigned b0, unsigned b1, unsigned b2, int c) {
  return in & ((c & 1) ? b0 : ~b0) & ((c & 2) ? b1 : ~b1) & ((c & 4) ? b2 : ~b2);
}

// Rows of one stream that a warp places at a time: one, or four of at most kFewSteps steps.
constexpr int kFewSteps = 64;
// Panels of a row block from which on a row's first entry in a panel is searched for instead of summed up
// from the counts of the panels before it.
constexpr int kSumPanels = 32;

// The streams' arrays, and the panel's tiles in shared memory.
template <typename V> struct ScatterArgs {
  const int32_t* lcol;
  const V* lval;
  const int32_t* col;
  const V* val;
  uint16_t* bcol;
  V* bval;
  const int32_t* s_tc;
  const uint32_t* s_slot;
  int nt, pr;
};
// Rows of one stream: lane l's row, its entries in the panel and those left of the diagonal, the first of
// these and of the others.
struct StreamRow {
  int64_t r, el, eu;
  int len, nl;
};

// Places the 32 rows of a stream of nblk blocks from blk0 on, LR lanes a row (32, or 8: four rows at a
// time, which then have at most 8 * LR entries).  rv, rc: the warp's rows in shared memory, places: 8 each.
template <typename V, int LR>
__device__ __forceinline__ void scatter_rows(const ScatterArgs<V>& a, const StreamRow& mine, int64_t blk0, int nblk,
                                             V* rv0, uint16_t* rc0, ClassPlace* places) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int E = BlkPiece<V>::kEpp;
  const int lane = threadIdx.x & 31, sub = lane % LR, first = lane - sub, cls = lane & 7;
  const unsigned group = LR == 32 ? kAll : ((1u << (LR & 31)) - 1u) << first, below = (1u << lane) - 1u;
  ClassPlace* place_of = places + first / LR * 8;
  V* rv = rv0 + first / LR * (nblk * kBS);
  uint16_t* rc = rc0 + first / LR * (nblk * kBS);
  for (int l0 = 0; l0 < 32; l0 += 32 / LR) {
    const int l = l0 + first / LR;
    const int64_t r = __shfl_sync(kAll, mine.r, l);
    const int len = __shfl_sync(kAll, mine.len, l);
    const int longest = LR == 32 ? len : __shfl_sync(kAll, mine.len, l0);   // rows are ranked by length
    // entry q of the row: q < nl in the lower CSR, else in U
    const int nl = __shfl_sync(kAll, mine.nl, l);
    const int64_t el = __shfl_sync(kAll, mine.el, l), eu = __shfl_sync(kAll, mine.eu, l) - nl;
    auto col_at = [&](int q) { return q < nl ? a.lcol[el + q] : a.col[eu + q]; };
    auto val_at = [&](int q) { return q < nl ? a.lval[el + q] : a.val[eu + q]; };
    // class counts of the off-diagonal entries (class cls of each lane), then their placement
    int nc = 0, noff = 0, run = 0;
    auto count = [&](int32_t c) {
      const unsigned in = __ballot_sync(kAll, c >= 0 && (int64_t)c != r) & group;
      const unsigned b0 = __ballot_sync(kAll, c & 1), b1 = __ballot_sync(kAll, c & 2);
      const unsigned b2 = __ballot_sync(kAll, c & 4);
      nc += __popc(class_mask(in, b0, b1, b2, cls));
      noff += __popc(in);
    };
    auto place = [&](int32_t c, V v) {
      const bool valid = c >= 0, offd = valid && (int64_t)c != r;
      const unsigned in = __ballot_sync(kAll, offd) & group;
      const unsigned b0 = __ballot_sync(kAll, c & 1), b1 = __ballot_sync(kAll, c & 2);
      const unsigned b2 = __ballot_sync(kAll, c & 4);
      const int cl = c & 7;
      const int i = __shfl_sync(kAll, run, first + cl) + __popc(class_mask(in, b0, b1, b2, cl) & below);
      run += __popc(class_mask(in, b0, b1, b2, cls));
      if (valid) {
        const int k = offd ? class_step(place_of[cl], cl, l, i) : len - 1;
        const int32_t J = c / kMC;
        const int lo = tile_index(a.s_slot, a.s_tc, a.nt, J);
        rc[k] = (uint16_t)(lo * kMC + (c - J * kMC));
        rv[k] = v;
      }
    };
    auto set_places = [&]() {
      const ClassPlace p = class_place(cls, nc, l, noff);
      if (sub < 8) place_of[sub] = p;
      __syncwarp();
    };
    if (longest <= 8 * LR) {
      // read once, into registers, all loads in flight
      int32_t c[8];
      V v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const bool in = q * LR + sub < len;
        c[q] = in ? col_at(q * LR + sub) : -1;
        v[q] = V(0);
        if (in) v[q] = val_at(q * LR + sub);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q * LR < longest) count(c[q]);
      set_places();
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q * LR < longest) place(c[q], v[q]);
    } else if (LR == 32) {
      for (int q = lane; q - lane < len; q += 32) count(q < len ? col_at(q) : -1);
      set_places();
      for (int q = lane; q - lane < len; q += 32) {
        V v = V(0);
        if (q < len) v = val_at(q);
        place(q < len ? col_at(q) : -1, v);
      }
    }
    // padding: zero values on the zero row of the class the lane wants
    for (int k = len + sub; k < nblk * kBS; k += LR) {
      rc[k] = (uint16_t)(a.pr + ((l + k) & 7));
      rv[k] = V(0);
    }
    __syncwarp();
    for (int b = sub; b < nblk; b += LR) {
      const int64_t at = (blk0 + b) * kBE;
      *reinterpret_cast<uint4*>(a.bcol + at + l * kBS) = *reinterpret_cast<const uint4*>(rc + b * kBS);
#pragma unroll
      for (int u = 0; u < kBS; u += E)
        *reinterpret_cast<uint4*>(a.bval + at + blk_value_at<V>(l, u)) =
            *reinterpret_cast<const uint4*>(rv + b * kBS + u);
    }
    __syncwarp();
  }
}

// CTA per panel, warp per stream, its 32 rows in turn, or (FEW) four at a time where none has more than
// kFewSteps entries: a first pass over a row's entries counts its classes by ballots, a second one places every
// entry (the diagonal takes the row's last step: the small off-diagonal terms are summed before the
// typically much larger diagonal one) in a shared-memory row, padding included, which is written out in
// 16-byte pieces.  Reads are coalesced, every stream position is written once.  A thread per row (segments
// read in column order, class sequence chosen step by step, entries gathered in class order) took 8.3 ms
// for 3.0e8 entries; this takes 3.1.  Dynamic shared memory: per warp `cap` steps of columns and values
// (a multiple of 8, at least scatter_cap of the longest stream).
__host__ __device__ constexpr int scatter_cap(int steps) {
  const int few = 4 * (steps < kFewSteps ? steps : kFewSteps);
  return steps > few ? steps : few;
}
template <typename V, bool FEW>
__global__ void __launch_bounds__(kMR, 4)
k_rs_scatter(const int64_t* __restrict__ lptr, const int32_t* __restrict__ lcol, const V* __restrict__ lval,
             const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, const V* __restrict__ val, int64_t n,
             const int32_t* __restrict__ rbp, const int32_t* __restrict__ pan_rb, const int32_t* __restrict__ pt0,
             const int32_t* __restrict__ pnt, const int32_t* __restrict__ tcol, const uint16_t* __restrict__ cnt,
             const uint16_t* __restrict__ cntl, const uint8_t* __restrict__ perm, const int64_t* __restrict__ sboff,
             int pr, int cap, uint16_t* __restrict__ bcol, V* __restrict__ bval) {
  static_assert(kBS == 8 && (kBS * sizeof(V)) % 16 == 0 && kW == 8, "a lane's block is whole 16-byte pieces");
  extern __shared__ __align__(16) unsigned char sm_rows[];
  __shared__ int32_t s_tc[32];
  __shared__ uint32_t s_slot[256];      // tile column J and its index in the panel, at J mod 256 (one of them)
  __shared__ ClassPlace s_place[kW][FEW ? 32 : 8];
  const int64_t p = blockIdx.x;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nt = pnt[p];
  if (threadIdx.x < 32) s_tc[threadIdx.x] = (int)threadIdx.x < nt ? tcol[pt0[p] + threadIdx.x] : INT32_MAX;
  s_slot[threadIdx.x] = 0xffffffffu;
  __syncthreads();
  if ((int)threadIdx.x < nt) s_slot[s_tc[threadIdx.x] & 255] = ((uint32_t)s_tc[threadIdx.x] << 5) | threadIdx.x;
  __syncthreads();
  V* rv = reinterpret_cast<V*>(sm_rows) + (size_t)w * cap;
  uint16_t* rc = reinterpret_cast<uint16_t*>(reinterpret_cast<V*>(sm_rows) + (size_t)kW * cap) + (size_t)w * cap;
  const int64_t I = pan_rb[p], blk0 = sboff[p * kW + w];
  const int nblk = (int)(sboff[p * kW + w + 1] - blk0);
  if (nblk == 0) return;
  const int64_t p_first = rbp[I];
  const int my_lr = perm[p * kMR + w * 32 + lane];
  StreamRow mine = {I * kMR + my_lr, 0, 0, 0, 0};
  if (mine.r < n) {
    mine.len = cnt[p * kMR + my_lr];
    mine.nl = cntl[p * kMR + my_lr];
    mine.el = lptr[mine.r];
    mine.eu = rowptr[mine.r];
    if (p - p_first <= kSumPanels) {
      for (int64_t q = p_first; q < p; ++q) {
        const int nl = cntl[q * kMR + my_lr];
        mine.el += nl;
        mine.eu += cnt[q * kMR + my_lr] - nl;
      }
    } else {
      const int64_t lim = (panel_last_cb(pt0, pnt, tcol, p - 1) + 1) * kMC;
      mine.el = first_from(lcol, mine.el, lptr[mine.r + 1], lim);
      mine.eu = first_from(col, mine.eu, rowptr[mine.r + 1], lim);
    }
  }
  const ScatterArgs<V> a = {lcol, lval, col, val, bcol, bval, s_tc, s_slot, nt, pr};
  if constexpr (FEW) {
    if (nblk * kBS <= kFewSteps) {
      scatter_rows<V, 8>(a, mine, blk0, nblk, rv, rc, s_place[w]);
      return;
    }
  }
  scatter_rows<V, 32>(a, mine, blk0, nblk, rv, rc, s_place[w]);
}

// Row groups of a row block.  With fewer row blocks than SMs each half of a row block is a CTA of
// its own: ranking within a half pads one to two percent more and X is staged twice, but n = 20,000
// (79 row blocks, 100 nonzeros a row, FP32) takes 22.7 instead of 28.2 us at nb = 8 and 25.5 instead
// of 32.8 at nb = 16; at 196 row blocks it no longer gains, at 391 it loses.  At nb = 32, where one CTA's X
// fills an SM, it gains with long rows (300 a row 101 -> 71) and loses a little with short ones (n = 36,000,
// 140 a row: 58 -> 63).
int row_groups(int64_t nRB) { return nRB < num_sms() ? 2 : 1; }

// ---------------------------------------------------------------------------------------
// Plan: direct streams (no row blocks, no panels)
// ---------------------------------------------------------------------------------------
// FP64 products run at the FP64 pipe's rate (one warp multiply-add per 64 clocks per scheduler), so
// what matters is that every scheduler has the same number of them; with few rows, row blocks of
// unequal length on unequal numbers of CTAs per SM left the busiest scheduler with 2.6 times the
// average (n = 20,000, 100 nonzeros a row).  The bound on n is that of the streams' 16-bit columns, which
// are row indices of X here, and not where the panels catch up: at 65,000 rows with 100 or 400 nonzeros a
// row the direct streams take 0.60 and 0.66 of the panels' time at nb = 8 (105 against 175 us, 369
// against 563) and 0.54 and 0.56 at nb = 1 (23 against 42, 65 against 116), so a product of 65,536 rows
// takes that much longer than one of 65,535.
bool direct_plan(const SpmmPlan* P) { return P->val_type == EIG_F64 && P->n < 65536; }

// Warp per row: its entries, columns ascending and the diagonal last, dealt to its `split` lanes in
// turn (slot_of: the row's first slot).
__global__ void k_direct_fill(int64_t n, int split, const int64_t* __restrict__ lptr, const int32_t* __restrict__ lcol,
                              const double* __restrict__ lval, const int64_t* __restrict__ rowptr,
                              const int32_t* __restrict__ col, const double* __restrict__ val,
                              const int32_t* __restrict__ slot_of,
                              const int64_t* __restrict__ sboff, uint16_t* __restrict__ bcol,
                              double* __restrict__ bval) {
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= n) return;
  const int64_t el = lptr[r];
  const int before = (int)(lptr[r + 1] - el), len = before + (int)(rowptr[r + 1] - rowptr[r]);
  const int64_t eu = rowptr[r] - before;
  const int slot = slot_of[r];
  const int64_t blk0 = sboff[slot >> 5];
  const bool diag = before < len && (int64_t)col[eu + before] == r;
  for (int q = lane; q < len; q += 32) {
    const int i = !diag || q < before ? q : (q == before ? len - 1 : q - 1);
    const int k = i / split, sl = (slot & 31) + i % split;
    const int64_t at = (blk0 + k / kBS) * kBE;
    bcol[at + sl * kBS + k % kBS] = (uint16_t)(q < before ? lcol[el + q] : col[eu + q]);
    bval[at + blk_value_at<double>(sl, k % kBS)] = q < before ? lval[el + q] : val[eu + q];
  }
}

static eig_status reserve_streams(SpmmPlan* P, int64_t nent, size_t vb) {
  size_t at = 0;
  EIG_TRY(P->m_streams.reserve(DevBuf::part(nent * 2) + DevBuf::part(nent * vb)));
  P->m_bcol.borrow(P->m_streams, nent * 2, &at);
  P->m_bval.borrow(P->m_streams, nent * vb, &at);
  return EIG_OK;
}

// Rows ranked by length over the whole matrix (descending, ties by row): warp w takes ranks
// [32 w / split, 32 (w + 1) / split), each row on `split` adjacent lanes.
eig_status direct_fill(SpmmPlan* P, const int64_t* lptr, const int32_t* lcol, const double* lval, cudaStream_t st) {
  const int64_t n = P->n;
  std::vector<int64_t> h_len(n), h_l(n + 1), h_u(n + 1);
  EIG_CUDA_TRY(cudaMemcpyAsync(h_l.data(), lptr, (n + 1) * 8, cudaMemcpyDeviceToHost, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(h_u.data(), P->rowptr, (n + 1) * 8, cudaMemcpyDeviceToHost, st));
  EIG_CUDA_TRY(cudaStreamSynchronize(st));
  for (int64_t r = 0; r < n; ++r) h_len[r] = h_l[r + 1] - h_l[r] + h_u[r + 1] - h_u[r];
  // lanes per row: until a block of 8 (two slices) gives eight warps per scheduler
  int split = 1;
  while (split < 4 && (n * split + 31) / 32 * 2 < (int64_t)num_sms() * 32) split *= 2;
  const int64_t nw = (n * split + 31) / 32;
  int64_t longest = 0;
  for (int64_t l : h_len) longest = std::max(longest, l);
  std::vector<int64_t> start(longest + 2, 0);
  for (int64_t l : h_len) start[longest - l + 1]++;
  for (int64_t l = 0; l <= longest; ++l) start[l + 1] += start[l];
  std::vector<int32_t> slot_of(n), row(nw * 32, (int32_t)n), len(nw * 32, 0);
  for (int64_t r = 0; r < n; ++r) {
    const int64_t q = start[longest - h_len[r]]++ * split;
    slot_of[r] = (int32_t)q;
    for (int j = 0; j < split; ++j) {
      row[q + j] = (int32_t)r;
      len[q + j] = (int32_t)((h_len[r] - j + split - 1) / split);
    }
  }
  std::vector<int64_t> sboff(nw + 1, 0);
  for (int64_t w = 0; w < nw; ++w) sboff[w + 1] = sboff[w] + (len[w * 32] + kBS - 1) / kBS;
  P->m_dsplit = split;
  P->m_nblk = sboff[nw];
  DevBuf d_slot;
  EIG_TRY(d_slot.reserve(n * 4));
  EIG_TRY(P->m_drow.reserve(nw * 32 * 4));
  EIG_TRY(P->m_dlen.reserve(nw * 32 * 4));
  EIG_TRY(P->m_sboff.reserve((nw + 1) * 8));
  EIG_CUDA_TRY(cudaMemcpyAsync(d_slot.p, slot_of.data(), n * 4, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(P->m_drow.p, row.data(), nw * 32 * 4, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(P->m_dlen.p, len.data(), nw * 32 * 4, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(P->m_sboff.p, sboff.data(), (nw + 1) * 8, cudaMemcpyHostToDevice, st));
  const int64_t nent = std::max<int64_t>(P->m_nblk, 1) * kBE;
  EIG_TRY(reserve_streams(P, nent, 8));
  // padding: zero values, which the kernel multiplies by zeros of its own (its lengths bound the loads)
  EIG_CUDA_TRY(cudaMemsetAsync(P->m_bcol.p, 0, nent * 2, st));
  EIG_CUDA_TRY(cudaMemsetAsync(P->m_bval.p, 0, nent * 8, st));
  k_direct_fill<<<(unsigned)((n * 32 + 255) / 256), 256, 0, st>>>(
      n, split, lptr, lcol, lval, P->rowptr, P->col, static_cast<const double*>(P->val), d_slot.as<int32_t>(),
      P->m_sboff.as<int64_t>(), P->m_bcol.as<uint16_t>(), P->m_bval.as<double>());
  EIG_LAUNCH_CHECK("k_direct_fill");
  EIG_CUDA_TRY(cudaStreamSynchronize(st));  // temporaries go out of scope
  P->m_direct = true;
  return EIG_OK;
}

// Arrays over the upper tiles, which a plan needs until its lower CSR is built: tile row and column blocks,
// tiles by column block; entries per (tile, column) and their offsets; offsets per (tile, row), or null.
struct TileTemps {
  DevBuf mem, rb, cb, jptr, jt, cnt, off, seg, most;
};

// Tiles that hold many entries on average (of 16,384): their lower part is built by k_mir_lower, with an
// offset kept per (tile, row).  Else k_mir_lower_few searches the rows and no offsets are kept: 1 KB a tile
// would be several times the matrix where tiles hold a handful of entries, and the CTAs of nearly empty tiles
// would mostly set themselves up.  A whole plan with k_mir_lower / with k_mir_lower_few, FP32, ms, by mean
// entries of a tile: 8: 32.7 / 20.4, 156: 18.8 / 12.8, 1009: 5.26 / 4.74, 2446: 3.94 / 3.93, 3393 (n = 1M, 300
// a row): 8.56 / 9.05.
bool dense_tiles(const SpmmPlan* P) { return P->nnz >= kDenseTile * P->n_tiles; }

template <typename V>
eig_status rowstream_fill(SpmmPlan* P, TileTemps& tiles, PlanTemps& tmp, cudaStream_t st) {
  const int32_t *tile_rb = tiles.rb.as<int32_t>(), *tile_cb = tiles.cb.as<int32_t>();
  const int64_t n_up_tiles = P->n_tiles;
  const int64_t n = P->n;
  const int tb = 256;
  const int64_t gb = (n + tb - 1) / tb;
  const V* val = static_cast<const V*>(P->val);
  // 1. row lengths and offsets of the lower CSR
  const DevBuf &lower = tmp.lower, &lptr = tmp.lptr;
  unsigned* bitmap = tmp.bitmap.as<unsigned>();
  const int64_t nRB = P->nRB, wpr = (P->nCB + 31) / 32;
  int32_t *cnt = tiles.cnt.as<int32_t>(), *off = tiles.off.as<int32_t>(), *seg = tiles.seg.as<int32_t>();
  int* most_d = tiles.most.as<int>();
  EIG_CUDA_TRY(cudaMemsetAsync(most_d, 0, 4, st));
  if (seg) EIG_CUDA_TRY(cudaMemsetAsync(seg, 0x7F, tiles.seg.bytes, st));   // "none"
  k_mir_colcounts<<<(unsigned)nRB, kMR, 0, st>>>(n, P->rowptr, P->col, P->tile_ptr.as<int64_t>(),
                                                 P->tile_col.as<int32_t>(), wpr, seg, cnt, bitmap, most_d);
  EIG_LAUNCH_CHECK("k_mir_colcounts");
  k_mir_coloffsets<<<(unsigned)gb, tb, 0, st>>>(n, tiles.jptr.as<int64_t>(), tiles.jt.as<int32_t>(), cnt, off,
                                                lower.as<int64_t>());
  EIG_LAUNCH_CHECK("k_mir_coloffsets");
  EIG_TRY(exclusive_scan(lower.as<int64_t>(), n, lptr.as<int64_t>(), tmp.sums.as<int64_t>(), st));
  int64_t lnnz = 0;
  int most = 0;
  EIG_CUDA_TRY(cudaMemcpyAsync(&most, most_d, 4, cudaMemcpyDeviceToHost, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(&lnnz, lptr.as<int64_t>() + n, 8, cudaMemcpyDeviceToHost, st));
  EIG_CUDA_TRY(cudaStreamSynchronize(st));
  // 2. the lower CSR
  const size_t b_lcol = std::max<int64_t>(lnnz, 1) * 4, b_lval = std::max<int64_t>(lnnz, 1) * sizeof(V);
  DevBuf full, lcol, lval;
  size_t at = 0;
  EIG_TRY(full.reserve(DevBuf::part(b_lcol) + DevBuf::part(b_lval)));
  lcol.borrow(full, b_lcol, &at);
  lval.borrow(full, b_lval, &at);
  if (most > 0 && !seg) {
    k_mir_lower_few<V><<<(unsigned)n_up_tiles, kMR, 0, st>>>(n, P->rowptr, P->col, val, tile_rb, tile_cb, off,
                                                             lptr.as<int64_t>(), lcol.as<int32_t>(), lval.as<V>());
    EIG_LAUNCH_CHECK("k_mir_lower_few");
  } else if (most > 0) {
    const int cap = (most + 15) / 16 * 16;
    const size_t sm = (size_t)cap * (sizeof(V) + 1);
    if (sm > 40 * 1024) EIG_CUDA_TRY(::eig::ensure_dyn_smem(k_mir_lower<V>, sm));
    k_mir_lower<V><<<(unsigned)n_up_tiles, kMR, sm, st>>>(n, P->rowptr, P->col, val, tile_rb, tile_cb, seg, off,
                                                          lptr.as<int64_t>(), cap, lcol.as<int32_t>(), lval.as<V>());
    EIG_LAUNCH_CHECK("k_mir_lower");
  }
  if constexpr (sizeof(V) == 8) {
    if (direct_plan(P)) return direct_fill(P, lptr.as<int64_t>(), lcol.as<int32_t>(), lval.as<V>(), st);
  }
  // 3. tiles of the mirrored matrix per row block, cut into panels of at most kPT tiles
  //    (balanced: a row block of t tiles takes ceil(t / kPT) panels of near-equal size; a row
  //    block without tiles still gets one empty panel so that its rows are written)
  std::vector<int64_t> h_tptr;
  std::vector<int32_t> h_tcol;
  EIG_TRY(tile_lists_from_bitmap(nRB, wpr, bitmap, tmp.rb_cnt.as<int64_t>(), st, tmp.rb_ptr, P->m_tcol, h_tptr,
                                 h_tcol));
  tiles.mem.release();   // the lists' copies waited for the kernels above; the streams may need the room
  std::vector<int32_t> rbp(nRB + 1, 0), pt0, pnt;
  for (int64_t I = 0; I < nRB; ++I) {
    const int64_t t0 = h_tptr[I], nt = h_tptr[I + 1] - t0;
    const int64_t np = std::max<int64_t>(1, (nt + kPT - 1) / kPT);
    int64_t t = t0;
    for (int64_t q = 0; q < np; ++q) {
      const int64_t sz = nt / np + (q < nt % np ? 1 : 0);
      pt0.push_back((int32_t)t);
      pnt.push_back((int32_t)sz);
      t += sz;
    }
    rbp[I + 1] = rbp[I] + (int32_t)np;
  }
  const int64_t npan = rbp[nRB];
  P->m_npan = npan;
  // staged rows: those of the widest panel
  P->m_pr = std::max(1, *std::max_element(pnt.begin(), pnt.end())) * kMC;
  P->m_groups = row_groups(nRB);
  at = 0;
  EIG_TRY(P->m_own.reserve(DevBuf::part(nRB * 16) + DevBuf::part((nRB + 1) * 4) + 2 * DevBuf::part(npan * 4) +
                           DevBuf::part(npan * kMR) + DevBuf::part(npan * kW * 4) +
                           DevBuf::part((npan * kW + 1) * 8)));
  P->m_order.borrow(P->m_own, nRB * 16, &at);
  P->m_rbp.borrow(P->m_own, (nRB + 1) * 4, &at);
  P->m_pt0.borrow(P->m_own, npan * 4, &at);
  P->m_pnt.borrow(P->m_own, npan * 4, &at);
  P->m_perm.borrow(P->m_own, npan * kMR, &at);
  P->m_steps.borrow(P->m_own, npan * kW * 4, &at);
  P->m_sboff.borrow(P->m_own, (npan * kW + 1) * 8, &at);
  EIG_CUDA_TRY(cudaMemcpyAsync(P->m_rbp.p, rbp.data(), (nRB + 1) * 4, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(P->m_pt0.p, pt0.data(), npan * 4, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(P->m_pnt.p, pnt.data(), npan * 4, cudaMemcpyHostToDevice, st));
  // 4. entries per (panel, row); rows ranked per panel; steps per (panel, warp); stream offsets
  std::vector<int32_t> pan_rb(npan);
  for (int64_t I = 0; I < nRB; ++I)
    for (int32_t q = rbp[I]; q < rbp[I + 1]; ++q) pan_rb[q] = (int32_t)I;
  DevBuf pan, d_pan_rb, cntp, cntl;
  at = 0;
  EIG_TRY(pan.reserve(DevBuf::part(npan * 4) + 2 * DevBuf::part(npan * kMR * 2)));
  d_pan_rb.borrow(pan, npan * 4, &at);
  cntp.borrow(pan, npan * kMR * 2, &at);
  cntl.borrow(pan, npan * kMR * 2, &at);
  EIG_CUDA_TRY(cudaMemcpyAsync(d_pan_rb.p, pan_rb.data(), npan * 4, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemsetAsync(cntp.p, 0, npan * kMR * 2, st));
  k_rs_counts<<<(unsigned)gb, tb, 0, st>>>(n, lptr.as<int64_t>(), lcol.as<int32_t>(), P->rowptr, P->col,
                                           P->m_rbp.as<int32_t>(), P->m_pt0.as<int32_t>(), P->m_pnt.as<int32_t>(),
                                           P->m_tcol.as<int32_t>(), cntp.as<uint16_t>(), cntl.as<uint16_t>());
  EIG_LAUNCH_CHECK("k_rs_counts");
  k_rs_rank<<<(unsigned)npan, kMR, 0, st>>>(cntp.as<uint16_t>(), kMR / P->m_groups, P->m_perm.as<uint8_t>(),
                                            P->m_steps.as<int32_t>());
  EIG_LAUNCH_CHECK("k_rs_rank");
  std::vector<int32_t> h_steps(npan * kW);
  std::vector<int64_t> sboff(npan * kW + 1, 0);
  EIG_CUDA_TRY(cudaMemcpyAsync(h_steps.data(), P->m_steps.p, npan * kW * 4, cudaMemcpyDeviceToHost, st));
  EIG_CUDA_TRY(cudaStreamSynchronize(st));
  for (int64_t i = 0; i < npan * kW; ++i) sboff[i + 1] = sboff[i] + (h_steps[i] + kBS - 1) / kBS;
  const int64_t nblk = sboff[npan * kW];
  P->m_nblk = nblk;
  EIG_CUDA_TRY(cudaMemcpyAsync(P->m_sboff.p, sboff.data(), (npan * kW + 1) * 8, cudaMemcpyHostToDevice, st));
  // Row blocks in order of work, the longest first (a counting sort, stable): CTAs are started in this
  // order, so that the last ones to run are short.  In index order / in this order, us: n = 197,822 with
  // 1080 nonzeros a row, FP32, nb 16: 573 / 499, nb 8: 358 / 290; n = 663,527 with 300, FP64 vectors, nb 8:
  // 830 / 730; n = 2M with 400, FP32, nb 16: 1750 / 1709.  A row block's panels stand beside its number, so
  // that a CTA starts with one load and not two in a row.
  {
    std::vector<int64_t> work(nRB);
    int64_t longest = 0;
    for (int64_t I = 0; I < nRB; ++I) {
      work[I] = sboff[(int64_t)rbp[I + 1] * kW] - sboff[(int64_t)rbp[I] * kW];
      longest = std::max(longest, work[I]);
    }
    std::vector<int64_t> start(longest + 2, 0);
    for (int64_t x : work) start[longest - x + 1]++;
    for (int64_t l = 0; l <= longest; ++l) start[l + 1] += start[l];
    std::vector<int4> order(nRB);
    for (int64_t I = 0; I < nRB; ++I) order[start[longest - work[I]]++] = make_int4((int)I, rbp[I], rbp[I + 1], 0);
    EIG_CUDA_TRY(cudaMemcpyAsync(P->m_order.p, order.data(), nRB * 16, cudaMemcpyHostToDevice, st));
  }
  // 5. the streams
  const int64_t nent = std::max<int64_t>(nblk, 1) * kBE;
  EIG_TRY(reserve_streams(P, nent, sizeof(V)));
  if (nblk > 0) {
    // four rows at a time where half of the streams that have entries at all are short (without that path the
    // kernel is a fiftieth faster)
    int64_t some = 0, few = 0;
    for (int32_t x : h_steps) {
      some += x > 0;
      few += x > 0 && x <= kFewSteps;
    }
    const bool by_four = 2 * few >= some;
    const int steps = (*std::max_element(h_steps.begin(), h_steps.end()) + kBS - 1) / kBS * kBS;
    const int cap = by_four ? scatter_cap(steps) : steps;
    const size_t sm = (size_t)kW * cap * (2 + sizeof(V));
    auto scatter = by_four ? k_rs_scatter<V, true> : k_rs_scatter<V, false>;
    if (sm > 40 * 1024) EIG_CUDA_TRY(::eig::ensure_dyn_smem(scatter, sm));
    scatter<<<(unsigned)npan, kMR, sm, st>>>(
        lptr.as<int64_t>(), lcol.as<int32_t>(), lval.as<V>(), P->rowptr, P->col, val, n, P->m_rbp.as<int32_t>(),
        d_pan_rb.as<int32_t>(), P->m_pt0.as<int32_t>(), P->m_pnt.as<int32_t>(), P->m_tcol.as<int32_t>(),
        cntp.as<uint16_t>(), cntl.as<uint16_t>(), P->m_perm.as<uint8_t>(), P->m_sboff.as<int64_t>(), P->m_pr, cap,
        P->m_bcol.as<uint16_t>(), P->m_bval.as<V>());
    EIG_LAUNCH_CHECK("k_rs_scatter");
  }
  EIG_CUDA_TRY(cudaStreamSynchronize(st));  // temporaries go out of scope
  return EIG_OK;
}

// ---------------------------------------------------------------------------------------
// Kernel
// ---------------------------------------------------------------------------------------
struct RsArgs {
  int64_t n;
  const int4* order;
  const int32_t* pt0;
  const int32_t* pnt;
  const int32_t* tcol;
  const uint8_t* perm;
  const int32_t* steps;
  const int64_t* sboff;
  const uint16_t* bcol;
  const void* bval;
  float minus_zero;   // -0 (see RsAcc<double, N, true>)
  int pr;        // staged rows of the widest panel; the zero rows follow them
  int* err;
};

// Fused epilogue of a Chebyshev step (Alg. 3, Eq. chebypoly): Y = a (H X - c X) - Qp (first: no
// Qp), and Y = X on inactive (locked) columns; the same double arithmetic on the same rounded
// product H X as the separate elementwise pass.
struct MirrorEpi {
  const void* Qp;
  const int* active;
  double a, c;
  int first;
};

// One product of a batched launch, and the batch (passed by value: at most kBatchJobs jobs).
struct MirrorJob {
  RsArgs a;
  const void* X;
  void* Y;
  int ld, col0, xj_bulk;
  MirrorEpi epi;
};
constexpr int kBatchJobs = 64;
struct MirrorBatch {
  int n;
  int64_t cta0[kBatchJobs + 1];
  MirrorJob jobs[kBatchJobs];
};

// Double-float accumulation applies to FP64 vectors with FP32 or BF16 values.
template <typename T, typename V> struct MirrorDF { static constexpr bool value = false; };
template <> struct MirrorDF<double, float> { static constexpr bool value = true; };
template <> struct MirrorDF<double, uint16_t> { static constexpr bool value = true; };

// Lane geometry for (vector type T, value type V, kernel block width NB).
//   ES: bytes of one staged X element (FP32; FP64; or a (hi, lo) FP32 pair for double-float);
//   RBY: bytes of one staged X row, gathered by each lane as NCH pieces of LDB bytes.
template <typename T, typename V, int NB> struct RsShape {
  static constexpr bool DF = MirrorDF<T, V>::value;
  static constexpr int ES = (int)sizeof(T);
  static constexpr int RBY = NB * ES;
  static constexpr int LDB = RBY >= 16 ? 16 : RBY;
  static constexpr int NCH = RBY / LDB;       // pieces per row
  static constexpr int EPC = LDB / ES;        // elements per piece
  // lanes of a phase reading the same bank-line offset class get distinct pieces
  static constexpr int ROTDIV = NCH >= 8 ? 1 : 8 / NCH;
  static constexpr size_t XBYTES = (size_t)(kPR + 8) * RBY;   // at most
  static constexpr int MINB0 = (int)(233472 / (XBYTES + 1024 + 128));
  // register budget: up to 4 CTAs per SM for rows of <= 16 bytes, 3 for 32, else (and for
  // FP64 values, whose blocks take twice the registers) 2
  static constexpr int MAXB = sizeof(typename ValLoad<V>::storage) == 8 ? 2 : (RBY <= 16 ? 4 : (RBY <= 32 ? 3 : 2));
  static constexpr int MINB = MINB0 < 1 ? 1 : (MINB0 > MAXB ? MAXB : MINB0);   // resident CTAs per SM
  // streamed blocks held in registers: the next block loads while the current one runs
  static constexpr int PF = 2;
  static constexpr int VW = (kBS * (int)sizeof(typename ValLoad<V>::storage)) / 4;   // value words per block
};

// Streamed loads: bypass L1, evict first from L2 (each entry is read once per product).
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint4 ldg_stream(const void* p, uint64_t pol) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p), "l"(pol));
  return v;
}
// Bulk prefetch of a global range into L2 (no registers, no shared memory).
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_load_1d_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                                 uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}

// Shared-memory piece loads of 4, 8 or 16 bytes (raw words).
template <int B> struct SLd;
template <> struct SLd<4> {
  __device__ __forceinline__ static void ld(uint32_t a, uint32_t* w) {
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w[0]) : "r"(a));
  }
};
template <> struct SLd<8> {
  __device__ __forceinline__ static void ld(uint32_t a, uint32_t* w) {
    asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(a));
  }
};
template <> struct SLd<16> {
  __device__ __forceinline__ static void ld(uint32_t a, uint32_t* w) {
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(a));
  }
};

// y += v * x over a lane's N elements, x given as raw staged words.
template <typename T, int N, bool DF> struct RsAcc;
template <int N> struct RsAcc<float, N, false> {
  typedef float VT;
  typedef float OT;
  static constexpr int N2 = (N + 1) / 2;
  float2 y[N2];
  __device__ __forceinline__ void zero(float) {
#pragma unroll
    for (int e = 0; e < N2; ++e) y[e] = make_float2(0.0f, 0.0f);
  }
  __device__ __forceinline__ void add(int slot0, float v, const uint32_t* w, int nw) {
    if (nw % 2 == 0) {
      // packed FP32x2 multiply-add (sm_100+): two elements of y per instruction
      const float2 vv = make_float2(v, v);
#pragma unroll
      for (int e = 0; e < nw; e += 2) {
        const int s = (slot0 + e) / 2;
        y[s] = __ffma2_rn(vv, make_float2(__uint_as_float(w[e]), __uint_as_float(w[e + 1])), y[s]);
      }
    } else {
      y[slot0 / 2].x = fmaf(v, __uint_as_float(w[0]), y[slot0 / 2].x);
    }
  }
  __device__ __forceinline__ OT get(int e) const { return (e & 1) ? y[e / 2].y : y[e / 2].x; }
};
template <int N> struct RsAcc<double, N, false> {
  typedef double VT;
  typedef double OT;
  double y[N];
  __device__ __forceinline__ void zero(float) {
#pragma unroll
    for (int e = 0; e < N; ++e) y[e] = 0.0;
  }
  __device__ __forceinline__ void add(int slot0, double v, const uint32_t* w, int nw) {
#pragma unroll
    for (int e = 0; e < nw / 2; ++e) y[slot0 + e] = fma(v, __hiloint2double(w[2 * e + 1], w[2 * e]), y[slot0 + e]);
  }
  __device__ __forceinline__ OT get(int e) const { return y[e]; }
};
// Double-float: X staged as (hi, lo) FP32 pairs (8 bytes per element, like FP64); each product
// v * xh is summed into hi by two-sum, every error term and v * xl into lo: ~2^-44 relative per step, at
// FP32 instruction rate.  With p = v xh rounded, t = hi + p rounded and b = t - hi, the error of both
// roundings is (hi - (t - b)) + (v xh - b): the first difference is exact and the second is one fused
// multiply-add, which takes the product's rounding along (v xh - p need not be formed by itself: nine
// operations instead of eleven, 2.88 -> 2.60 ms at n = 2M, 400 nonzeros a row, nb = 8).  A 16-byte piece
// holds two elements as (hi_e, hi_e+1, lo_e, lo_e+1), so a step is FP32x2 arithmetic on element pairs;
// every operation is an explicit round-to-nearest (a subtraction a - b is fma(b, -1, a)).  A one-element
// piece (block width 1) holds (hi, lo).  The rounded product is fma(v, xh, nz) with nz = -0 from the
// kernel's arguments: the compiler contracts a packed multiplication and a following packed addition
// into one fused operation even where both have explicit roundings (also through a constant -0), and
// the two-sum would then lose its low word (errors of 1e-10 instead of 2e-15).
template <int N> struct RsAcc<double, N, true> {
  typedef float VT;
  typedef double OT;
  static constexpr int N2 = (N + 1) / 2;
  float2 hi[N2], lo[N2];
  float nz;
  __device__ __forceinline__ void zero(float minus_zero) {
    nz = minus_zero;
#pragma unroll
    for (int e = 0; e < N2; ++e) hi[e] = lo[e] = make_float2(0.0f, 0.0f);
  }
  __device__ __forceinline__ void add(int slot0, float v, const uint32_t* w, int nw) {
    if (nw == 4) {
      const int s = slot0 / 2;
      const float2 vv = make_float2(v, v), m1 = make_float2(-1.0f, -1.0f);
      const float2 xh = make_float2(__uint_as_float(w[0]), __uint_as_float(w[1]));
      const float2 xl = make_float2(__uint_as_float(w[2]), __uint_as_float(w[3]));
      const float2 t = __fadd2_rn(hi[s], __ffma2_rn(vv, xh, make_float2(nz, nz)));
      const float2 nb = __ffma2_rn(t, m1, hi[s]);                       // hi - t = -b
      const float2 e1 = __ffma2_rn(__fadd2_rn(t, nb), m1, hi[s]);       // hi - (t - b)
      const float2 e2 = __ffma2_rn(vv, xh, nb);                         // v xh - b
      hi[s] = t;
      lo[s] = __ffma2_rn(vv, xl, __fadd2_rn(lo[s], __fadd2_rn(e1, e2)));
    } else {
      float& h = (slot0 & 1) ? hi[slot0 / 2].y : hi[slot0 / 2].x;
      float& l = (slot0 & 1) ? lo[slot0 / 2].y : lo[slot0 / 2].x;
      const float xh = __uint_as_float(w[0]), xl = __uint_as_float(w[1]);
      const float t = __fadd_rn(h, __fmaf_rn(v, xh, nz));
      const float nb = __fsub_rn(h, t);
      const float e1 = __fsub_rn(h, __fadd_rn(t, nb));
      const float e2 = __fmaf_rn(v, xh, nb);
      h = t;
      l = __fmaf_rn(v, xl, __fadd_rn(l, __fadd_rn(e1, e2)));
    }
  }
  __device__ __forceinline__ OT get(int e) const {
    return (e & 1) ? (double)hi[e / 2].y + (double)lo[e / 2].y : (double)hi[e / 2].x + (double)lo[e / 2].x;
  }
};

// Value k (0..7) of a lane's streamed block, widened to the arithmetic type.
template <typename VS, typename VT> struct BlkVal;
template <typename VT> struct BlkVal<float, VT> {
  __device__ __forceinline__ static VT get(const uint32_t* w, int i) { return (VT)__uint_as_float(w[i]); }
};
template <typename VT> struct BlkVal<uint16_t, VT> {
  __device__ __forceinline__ static VT get(const uint32_t* w, int i) {
    const uint32_t u = w[i >> 1];
    return (VT)__uint_as_float((i & 1) ? (u & 0xFFFF0000u) : (u << 16));
  }
};
template <typename VT> struct BlkVal<double, VT> {
  __device__ __forceinline__ static VT get(const uint32_t* w, int i) {
    return (VT)__hiloint2double(w[2 * i + 1], w[2 * i]);
  }
};

// One staged X element of type T (FP32, FP64; double-float pairs are staged from FP64).
template <typename T, bool DF> struct Stage;
template <> struct Stage<float, false> {
  __device__ __forceinline__ static void put(unsigned char* row, int e, int, float x) {
    reinterpret_cast<float*>(row)[e] = x;
  }
};
template <> struct Stage<double, false> {
  __device__ __forceinline__ static void put(unsigned char* row, int e, int, double x) {
    reinterpret_cast<double*>(row)[e] = x;
  }
};
template <> struct Stage<double, true> {
  // element e of a staged row: hi and lo words in the piece layout of the double-float
  // accumulator (pairs of elements per 16-byte piece, or (hi, lo) for one-element rows)
  __device__ __forceinline__ static void put(unsigned char* row, int e, int nb, double x) {
    const float h = __double2float_rn(x);
    float* d = reinterpret_cast<float*>(row);
    const int ih = nb == 1 ? 0 : (e >> 1) * 4 + (e & 1);
    const int il = nb == 1 ? 1 : ih + 2;
    d[ih] = h;
    d[il] = __double2float_rn(x - (double)h);
  }
};

// Double-float staging of whole rows (ld == NB >= 2): a thread converts 16-byte pieces (two elements,
// the accumulator's piece layout), eight loads in flight.  One element at a time each panel waited
// for ~30 round trips to L2: 3.21 ms instead of 2.95 at n = 2M (400 nonzeros a row), nb = 8.
template <int NB>
__device__ __forceinline__ void stage_df_rows(unsigned char* xs, const double* __restrict__ X, const int32_t* tcol,
                                              int npt, int64_t n) {
  constexpr int PPR = NB / 2, U = 8;   // pieces per row, loads in flight
  const int total = npt * kMC * PPR;
  for (int i0 = threadIdx.x; i0 < total; i0 += U * kW * 32) {
    double2 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * kW * 32;
      x[u] = make_double2(0.0, 0.0);
      if (i < total) {
        const int64_t row = (int64_t)tcol[i / (kMC * PPR)] * kMC + i / PPR % kMC;
        if (row < n) x[u] = __ldg(reinterpret_cast<const double2*>(X + row * NB) + i % PPR);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * kW * 32;
      if (i >= total) break;
      const float h0 = __double2float_rn(x[u].x), h1 = __double2float_rn(x[u].y);
      reinterpret_cast<float4*>(xs)[i] = make_float4(h0, h1, __double2float_rn(x[u].x - (double)h0),
                                                     __double2float_rn(x[u].y - (double)h1));
    }
  }
}

// Warps [w0, w0 + blockDim.x / 32) of the slot-th longest row block of one product.  Y (and X, Qp) rows have stride ld
// elements; the product covers elements [col0, col0 + NB).
template <typename T, typename V, int NB, bool CHEB>
__device__ __forceinline__ void mirror_row_block(const RsArgs& a, const T* __restrict__ X, T* __restrict__ Y, int ld,
                                                 int col0, int xj_bulk, const MirrorEpi& epi, int64_t slot, int w0) {
  typedef RsShape<T, V, NB> Sh;
  constexpr bool DF = Sh::DF;
  constexpr int RBY = Sh::RBY, LDB = Sh::LDB, NCH = Sh::NCH, EPC = Sh::EPC, PF = Sh::PF, VW = Sh::VW;
  constexpr int NW = LDB / 4;  // words per piece
  typedef typename ValLoad<V>::storage VS;
  typedef RsAcc<T, NB, DF> Acc;
  typedef typename Acc::VT VT;
  typedef typename Acc::OT OT;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* xs = smem;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + (size_t)(a.pr + 8) * RBY);
  __shared__ int s_abort;

  // warps of a scheduler (every fourth) take a long and a short stream: 0 1 2 3 7 6 5 4
  const int tid = threadIdx.x, lane = tid & 31, wi = tid >> 5;
  const int w = w0 + (wi < 4 ? wi : 11 - wi);
  const int4 blk = a.order[slot];
  const int64_t r0 = (int64_t)blk.x * kMR;
  const int p0 = blk.y, p1 = blk.z;

  // zero rows (one per class) for the padding entries; never overwritten by staging
  for (int i = tid; i < 8 * RBY / 4; i += blockDim.x) reinterpret_cast<uint32_t*>(xs + (size_t)a.pr * RBY)[i] = 0u;
  if (tid == 0) {
    s_abort = 0;
    mbar_init(bar, 1);
    mbar_init_fence();
  }
  // this lane's pieces start at piece `rot` of the row (distinct among the lanes of a phase
  // whose rows share a bank-line offset)
  const int rot = (lane / Sh::ROTDIV) % NCH;
  uint32_t poff[NCH];
#pragma unroll
  for (int j = 0; j < NCH; ++j) poff[j] = (uint32_t)(((j + rot) % NCH) * LDB);
  const uint32_t xs_a = smem_u32(xs);
  const uint64_t pol_stream = policy_evict_first();
  const uint64_t pol_keep = policy_evict_last();
  uint32_t xphase = 0;

  for (int p = p0; p < p1; ++p) {
    __syncthreads();  // the previous panel's gathers are done
    const int t0 = a.pt0[p], npt = a.pnt[p];
    if (xj_bulk) {
      // one bulk copy per tile, issued by one lane each (at most kPT <= 32 tiles)
      if (tid < 32 && npt > 0) {
        const int64_t cb0 = lane < npt ? (int64_t)a.tcol[t0 + lane] * kMC : 0;
        const uint32_t bytes = lane < npt ? (uint32_t)(min64(kMC, a.n - cb0) * RBY) : 0u;
        const uint32_t tot = __reduce_add_sync(0xffffffffu, bytes);
        if (lane == 0) mbar_arrive_expect_tx(bar, tot);
        __syncwarp();
        if (lane < npt) tma_load_1d_hint(xs + (size_t)lane * kMC * RBY, X + cb0 * NB, bytes, bar, pol_keep);
      }
    } else if (DF && NB >= 2 && ld == NB) {
      if constexpr (DF && NB >= 2) stage_df_rows<NB>(xs, X, a.tcol + t0, npt, a.n);
    } else {
      // a whole CTA (the host does not split row blocks here): a constant stride, with which the divisions
      // below fold (FP64 values, nb = 32, scattered entries, n = 200,000: 29.5 ms, 63.9 with blockDim.x)
      for (int64_t i = tid; i < (int64_t)npt * kMC * NB; i += kW * 32) {
        const int t = (int)(i / (kMC * NB));
        const int rr = (int)((i / NB) % kMC), e = (int)(i % NB);
        const int64_t row = (int64_t)a.tcol[t0 + t] * kMC + rr;
        if (row < a.n) Stage<T, DF>::put(xs + (size_t)(t * kMC + rr) * RBY, e, NB, X[row * ld + col0 + e]);
      }
    }

    // this lane's row and the warp's stream; its first blocks load while X is staged
    const int64_t r = r0 + a.perm[(int64_t)p * kMR + w * 32 + lane];
    const int L = a.steps[(int64_t)p * kW + w];
    const int64_t b0 = a.sboff[(int64_t)p * kW + w];
    const int nb = (L + kBS - 1) / kBS;
    Acc acc;
    acc.zero(a.minus_zero);
    uint4 bc[PF];
    uint32_t bv[PF][VW];
    // a lane's pieces of a block, of columns and values alike, are 16 bytes at its number (blk_value_at): one
    // base each, so that a block's addresses take no index arithmetic of their own (with it, one dense row
    // of 60,000 at nb = 16, whose chain of blocks is the product, took 4.26 ms instead of 3.83, and n = 2M, 400
    // nonzeros a row, 1740 us instead of 1704)
    const unsigned char* cb = reinterpret_cast<const unsigned char*>(a.bcol) + b0 * (kBE * 2) + lane * 16;
    const unsigned char* vb = static_cast<const unsigned char*>(a.bval) + b0 * (kBE * (int)sizeof(VS)) + lane * 16;
    auto load_blk = [&](int b, int s) {
      bc[s] = ldg_stream(cb + (int64_t)b * (kBE * 2), pol_stream);
#pragma unroll
      for (int u = 0; u < VW; u += 4) {
        const uint4 t = ldg_stream(vb + (int64_t)b * (kBE * (int)sizeof(VS)) + u * 128, pol_stream);
        bv[s][u] = t.x; bv[s][u + 1] = t.y; bv[s][u + 2] = t.z; bv[s][u + 3] = t.w;
      }
    };
    // blocks kL2 ahead of the one running are prefetched into L2 by lane 0, so that the
    // register loads one block ahead see L2 rather than HBM latency
    auto prefetch_blk = [&](int b) {
      if (lane == 0 && b < nb) {
        prefetch_l2(cb + (int64_t)b * (kBE * 2), kBE * 2);
        prefetch_l2(vb + (int64_t)b * (kBE * (int)sizeof(VS)), kBE * (uint32_t)sizeof(VS));
      }
    };
    for (int b = 0; b < kL2; ++b) prefetch_blk(b);
#pragma unroll
    for (int s = 0; s < PF; ++s)
      if (s < nb) load_blk(s, s);
    if (xj_bulk) {
      if (npt > 0) {
        if (!mbar_wait_bounded(bar, xphase)) {
          atomicOr(a.err, 1);
          s_abort = 1;
        }
        __syncthreads();
        if (s_abort) break;
        xphase ^= 1u;
      }
    } else {
      __syncthreads();
    }
    for (int b = 0; b < nb; b += PF) {
#pragma unroll
      for (int s = 0; s < PF; ++s) {
        if (b + s < nb) {
          prefetch_blk(b + s + kL2);
          const uint32_t cw[4] = {bc[s].x, bc[s].y, bc[s].z, bc[s].w};
          uint32_t vw[VW];
#pragma unroll
          for (int u = 0; u < VW; ++u) vw[u] = bv[s][u];
          if (b + s + PF < nb) load_blk(b + s + PF, s);
          const int ks = min(kBS, L - (b + s) * kBS);   // steps in this block (warp-uniform)
          auto step = [&](int k) {
            const uint32_t c = (k & 1) ? (cw[k >> 1] >> 16) : (cw[k >> 1] & 0xFFFFu);
            const VT v = BlkVal<VS, VT>::get(vw, k);
            const uint32_t rowa = xs_a + c * (uint32_t)RBY;
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
              uint32_t xw[NW];
              SLd<LDB>::ld(rowa + poff[j], xw);
              acc.add(j * EPC, v, xw, NW);
            }
          };
          if (ks == kBS) {
            // a whole block: straight-line code, so the gathers of later steps can be issued
            // ahead of the multiply-adds of earlier ones
#pragma unroll
            for (int k = 0; k < kBS; ++k) step(k);
          } else {
#pragma unroll
            for (int k = 0; k < kBS; ++k)
              if (k < ks) step(k);
          }
        }
      }
    }
    // the row's sum over this panel: stored (first panel) or added to the earlier panels'
    if (r < a.n) {
      const bool first_panel = (p == p0), last_panel = (p == p1 - 1);
#pragma unroll
      for (int j = 0; j < NCH; ++j) {
        const int jc0 = col0 + ((j + rot) % NCH) * EPC;   // first element of the piece
        T* yp = Y + r * ld + jc0;
        OT v[EPC];
#pragma unroll
        for (int e = 0; e < EPC; ++e) v[e] = acc.get(j * EPC + e);
        if (!first_panel) {
          const Vec<T, EPC> old = VecIO<T, EPC>::ld(yp);
#pragma unroll
          for (int e = 0; e < EPC; ++e) v[e] += (OT)old.v[e];
        }
        Vec<T, EPC> out;
        if (CHEB && last_panel) {
          const Vec<T, EPC> xv = VecIO<T, EPC>::ld(X + r * ld + jc0);
          Vec<T, EPC> qv;
          qv.zero();
          if (!epi.first) qv = VecIO<T, EPC>::ld(static_cast<const T*>(epi.Qp) + r * ld + jc0);
#pragma unroll
          for (int e = 0; e < EPC; ++e) {
            if (!epi.active[jc0 + e]) {
              out.v[e] = xv.v[e];
            } else {
              // explicit roundings, as the separate elementwise step (k_cheb) takes them: the
              // single and the batched launch then agree bit for bit
              double yv = __dmul_rn(epi.a, __fma_rn(-epi.c, (double)xv.v[e], (double)(T)v[e]));
              if (!epi.first) yv = __dsub_rn(yv, (double)qv.v[e]);
              out.v[e] = (T)yv;
            }
          }
        } else {
#pragma unroll
          for (int e = 0; e < EPC; ++e) out.v[e] = (T)v[e];
        }
        VecIO<T, EPC>::st(yp, out);
      }
    }
  }
  if (s_abort) {
    // leave no bulk copy in flight into this CTA's shared memory (bounded wait on the phase
    // that gave up)
    if (tid == 0) (void)mbar_wait_bounded(bar, xphase);
    __syncthreads();
  }
}

// One product: CTA = row block, or one of its row groups.
template <typename T, typename V, int NB, bool CHEB>
__global__ void __launch_bounds__(kW * 32, RsShape<T, V, NB>::MINB)
k_spmm_mirror(const __grid_constant__ RsArgs a, const T* __restrict__ X, T* __restrict__ Y, int ld, int col0,
              int xj_bulk, const __grid_constant__ MirrorEpi epi) {
  const int g = kW * 32 / blockDim.x;   // CTAs per row block
  mirror_row_block<T, V, NB, CHEB>(a, X, Y, ld, col0, xj_bulk, epi, blockIdx.x / g, (int)(blockIdx.x % g) * (kW / g));
}

// Several products of one shape in one launch over their concatenated row blocks (the
// (instance, row block) work list of a batch): job j owns CTAs [cta0[j], cta0[j + 1]).
template <typename T, typename V, int NB, bool CHEB>
__global__ void __launch_bounds__(kW * 32, RsShape<T, V, NB>::MINB)
k_spmm_mirror_batch(const __grid_constant__ MirrorBatch B) {
  int j = 0;
  while (j + 1 < B.n && B.cta0[j + 1] <= (int64_t)blockIdx.x) ++j;
  const MirrorJob& J = B.jobs[j];
  mirror_row_block<T, V, NB, CHEB>(J.a, static_cast<const T*>(J.X), static_cast<T*>(J.Y), J.ld, J.col0, J.xj_bulk,
                                   J.epi, (int64_t)blockIdx.x - B.cta0[j], 0);
}

// Product of a direct plan, FP64: a warp takes 32 lanes' worth of rows (a row on `split` adjacent
// lanes) and NB <= 4 of the block's columns, gathering its rows of X through L1 and L2 (32 bytes per
// entry: one sector, one load).
//
// What bounds it: the FP64 pipe, and for few rows the longest row's chain of gathers and
// multiply-adds.  Column slices and split rows multiply the warps, so that the longest group (twice the
// average) is not the makespan; the launch order pairs long with short ones on an SM: CTAs (four warps,
// one per scheduler, of near-equal length) come in order of length, and every second round of one CTA
// per SM in the reverse order.  n = 20,000, 100 nonzeros a row: 41 us at nb = 8 (27 us of FP64
// multiply-adds), 76 at nb = 16, 14 at nb = 1; with row blocks and panels 108, 195 and 34.
struct DirectArgs {
  int64_t n;
  int32_t nw;            // warps' worth of slots
  int32_t split;         // lanes per row
  const int32_t* row;    // row of each slot (n: none)
  const int32_t* len;    // entries of each slot
  const int64_t* sboff;
  const uint16_t* bcol;
  const double* bval;
  int sms;
};
constexpr int kDirectWarps = 4;
// Four doubles (32 bytes, one sector) in one load; p 32-byte aligned.
__device__ __forceinline__ Vec<double, 4> ld_sector(const double* p) {
  Vec<double, 4> r;
  asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
               : "=d"(r.v[0]), "=d"(r.v[1]), "=d"(r.v[2]), "=d"(r.v[3]) : "l"(p));
  return r;
}

// SECTOR (NB = 4): every gathered piece starts on a 32-byte boundary.  The products' inputs are only
// aligned to 16 bytes, and a 32-byte load from such an address faults, so the host looks at X.  Two 16-byte
// loads cost little (n = 20,000, 100 nonzeros a row, X aligned / off by 16 bytes: nb = 8 43 / 44 us, 16 76 / 79).
template <int NB, bool CHEB, bool SECTOR>
__global__ void __launch_bounds__(kDirectWarps * 32, 4)
k_spmm_direct(const __grid_constant__ DirectArgs a, const double* __restrict__ X, double* __restrict__ Y, int ld,
              int col0, int slices, const __grid_constant__ MirrorEpi epi) {
  constexpr int VEC = NB >= 2 ? 2 : 1, NCH = NB / VEC;
  const int lane = threadIdx.x & 31;
  const int full = (int)gridDim.x / a.sms * a.sms, round = (int)blockIdx.x / a.sms;
  const int cta = (int)blockIdx.x < full && (round & 1) ? 2 * round * a.sms + a.sms - 1 - (int)blockIdx.x
                                                        : (int)blockIdx.x;
  const int task = cta * kDirectWarps + (threadIdx.x >> 5);
  const int g = task / slices;
  if (g >= a.nw) return;
  const int c0 = col0 + task % slices * NB;
  const int slot = g * 32 + lane;
  const int len = a.len[slot], L = a.len[g * 32];
  const int64_t r = a.row[slot];
  const int64_t b0 = a.sboff[g];
  const int nb = (L + kBS - 1) / kBS;
  const uint64_t pol = policy_evict_first();
  const double* Xc = X + c0;
  double y[NB];
#pragma unroll
  for (int e = 0; e < NB; ++e) y[e] = 0.0;
  uint4 cw;
  uint4 vw[4];
  auto load = [&](int b) {
    cw = ldg_stream(a.bcol + (b0 + b) * kBE + lane * kBS, pol);
#pragma unroll
    for (int u = 0; u < 4; ++u) vw[u] = ldg_stream(a.bval + (b0 + b) * kBE + blk_value_at<double>(lane, 2 * u), pol);
  };
  if (nb > 0) load(0);
  for (int b = 0; b < nb; ++b) {
    const uint32_t c4[4] = {cw.x, cw.y, cw.z, cw.w};
    double v[kBS];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[2 * u] = __hiloint2double((int)vw[u].y, (int)vw[u].x);
      v[2 * u + 1] = __hiloint2double((int)vw[u].w, (int)vw[u].z);
    }
    // the block's gathers all start before the first multiply-add; the next block's entries after them
    Vec<double, VEC> x[kBS][NCH];
#pragma unroll
    for (int k = 0; k < kBS; ++k) {
      const int64_t c = (k & 1) ? (c4[k >> 1] >> 16) : (c4[k >> 1] & 0xFFFFu);
      if constexpr (SECTOR) {
        static_assert(NB == 4, "a piece is one sector");
        Vec<double, 4> t;
        t.zero();
        if (b * kBS + k < len) t = ld_sector(Xc + c * ld);
        x[k][0].v[0] = t.v[0]; x[k][0].v[1] = t.v[1]; x[k][1].v[0] = t.v[2]; x[k][1].v[1] = t.v[3];
      } else {
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
          x[k][j].zero();
          if (b * kBS + k < len) x[k][j] = VecIO<double, VEC>::ld(Xc + c * ld + j * VEC);
        }
      }
    }
    if (b + 1 < nb) load(b + 1);
#pragma unroll
    for (int k = 0; k < kBS; ++k)
      if (b * kBS + k < L) {
#pragma unroll
        for (int j = 0; j < NCH; ++j)
#pragma unroll
          for (int e = 0; e < VEC; ++e) y[j * VEC + e] = fma(v[k], x[k][j].v[e], y[j * VEC + e]);
      }
  }
  for (int o = 1; o < a.split; o <<= 1)
#pragma unroll
    for (int e = 0; e < NB; ++e) y[e] += __shfl_xor_sync(0xffffffffu, y[e], o);
  if (r >= a.n || lane % a.split) return;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    const int jc = c0 + j * VEC;
    Vec<double, VEC> out;
    if (CHEB) {
      const Vec<double, VEC> xv = VecIO<double, VEC>::ld(X + r * ld + jc);
      Vec<double, VEC> qv;
      qv.zero();
      if (!epi.first) qv = VecIO<double, VEC>::ld(static_cast<const double*>(epi.Qp) + r * ld + jc);
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        double yv = __dmul_rn(epi.a, __fma_rn(-epi.c, xv.v[e], y[j * VEC + e]));
        if (!epi.first) yv = __dsub_rn(yv, qv.v[e]);
        out.v[e] = epi.active[jc + e] ? yv : xv.v[e];
      }
    } else {
#pragma unroll
      for (int e = 0; e < VEC; ++e) out.v[e] = y[j * VEC + e];
    }
    VecIO<double, VEC>::st(Y + r * ld + jc, out);
  }
}

}  // namespace

// ---------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------
size_t mirror_bytes_estimate(const SpmmPlan* P) {
  // lower CSR (temporary) + streams of 2-byte columns and values with ~5% padding
  const double fnnz = 2.0 * double(P->nnz);
  const double vb = double(dtype_size(P->val_type));
  return (size_t)(0.5 * fnnz * (4.0 + vb) + 1.1 * fnnz * (2.0 + vb) + 64.0 * double(P->n));
}

size_t mirror_tiles_bytes(const SpmmPlan* P) {
  const size_t per_tile = 3 * 4 + 2 * kMC * 4 + (dense_tiles(P) ? kMR * 4 : 0);
  return (size_t)P->n_tiles * per_tile + (size_t)P->nnz * (4 + dtype_size(P->val_type));
}

eig_status spmm_plan_build_mirror(SpmmPlan* P, const std::vector<int64_t>& h_tptr,
                                  const std::vector<int32_t>& h_tcol, PlanTemps& tmp, cudaStream_t st) {
  if (P->R != kMR || P->C != kMC) return EIG_EUNSUPPORTED;
  const int64_t nRB = P->nRB, nCB = P->nCB, nt = P->n_tiles;
  // row block of each upper tile, and the upper tiles grouped by column block (ascending row block)
  std::vector<int32_t> trb(std::max<int64_t>(nt, 1)), tcb(std::max<int64_t>(nt, 1));
  std::vector<int64_t> jptr(nCB + 1, 0);
  for (int64_t I = 0; I < nRB; ++I)
    for (int64_t t = h_tptr[I]; t < h_tptr[I + 1]; ++t) {
      trb[t] = (int32_t)I;
      tcb[t] = h_tcol[t];
      jptr[h_tcol[t] + 1]++;
    }
  for (int64_t J = 0; J < nCB; ++J) jptr[J + 1] += jptr[J];
  std::vector<int32_t> jt(std::max<int64_t>(nt, 1));
  {
    std::vector<int64_t> fill(jptr.begin(), jptr.end() - 1);
    for (int64_t t = 0; t < nt; ++t) jt[fill[tcb[t]]++] = (int32_t)t;
  }
  const size_t t4 = std::max<int64_t>(nt, 1) * 4;
  const size_t b_seg = dense_tiles(P) ? t4 * kMR : 0;
  TileTemps T;
  size_t at = 0;
  EIG_TRY(T.mem.reserve(3 * DevBuf::part(t4) + DevBuf::part(jptr.size() * 8) + 2 * DevBuf::part(t4 * kMC) +
                        DevBuf::part(4) + DevBuf::part(b_seg)));
  T.rb.borrow(T.mem, t4, &at);
  T.cb.borrow(T.mem, t4, &at);
  T.jt.borrow(T.mem, t4, &at);
  T.jptr.borrow(T.mem, jptr.size() * 8, &at);
  T.cnt.borrow(T.mem, t4 * kMC, &at);
  T.off.borrow(T.mem, t4 * kMC, &at);
  T.most.borrow(T.mem, 4, &at);
  if (b_seg) T.seg.borrow(T.mem, b_seg, &at);
  EIG_CUDA_TRY(cudaMemcpyAsync(T.rb.p, trb.data(), trb.size() * 4, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(T.cb.p, tcb.data(), tcb.size() * 4, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(T.jptr.p, jptr.data(), jptr.size() * 8, cudaMemcpyHostToDevice, st));
  EIG_CUDA_TRY(cudaMemcpyAsync(T.jt.p, jt.data(), jt.size() * 4, cudaMemcpyHostToDevice, st));
  eig_status s;
  if (P->val_type == EIG_F32) s = rowstream_fill<float>(P, T, tmp, st);
  else if (P->val_type == EIG_F64) s = rowstream_fill<double>(P, T, tmp, st);
  else s = rowstream_fill<uint16_t>(P, T, tmp, st);
  EIG_TRY(s);
  P->mirrored = true;
  return EIG_OK;
}

// Kernel block width for (T, V, NB): NB itself while one panel of staged X rows fits in a
// CTA's shared memory, else a column slice of it (the product then runs as several launches
// over column slices, each reading the matrix once).
template <typename T, typename V, int NB> struct RsSlice {
  static constexpr int value =
      (RsShape<T, V, NB>::XBYTES + 1024 <= 232448 || NB == 1) ? NB : RsSlice<T, V, NB / 2>::value;
};
template <typename T, typename V> struct RsSlice<T, V, 1> { static constexpr int value = 1; };

// The plan's row streams as kernel arguments.
static RsArgs rs_args(SpmmPlan* P) {
  RsArgs a;
  a.n = P->n;
  a.order = P->m_order.as<int4>();
  a.pt0 = P->m_pt0.as<int32_t>();
  a.pnt = P->m_pnt.as<int32_t>();
  a.tcol = P->m_tcol.as<int32_t>();
  a.perm = P->m_perm.as<uint8_t>();
  a.steps = P->m_steps.as<int32_t>();
  a.sboff = P->m_sboff.as<int64_t>();
  a.bcol = P->m_bcol.as<uint16_t>();
  a.bval = P->m_bval.p;
  a.minus_zero = -0.0f;
  a.pr = P->m_pr;
  a.err = P->err.as<int>();
  return a;
}

// X tiles by bulk copy: plain staging of whole, 16-byte aligned rows of a 16-byte multiple.
template <typename T, typename V, int NBK>
static int rs_xj_bulk(const T* X, int ld) {
  typedef RsShape<T, V, NBK> Sh;
  return !Sh::DF && ld == NBK && (Sh::RBY % 16 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15u) == 0);
}

template <typename T, typename V, int NBK, bool CHEB>
static eig_status rs_launch(SpmmPlan* P, const T* X, T* Y, int ld, int col0, const MirrorEpi& epi, cudaStream_t st) {
  typedef RsShape<T, V, NBK> Sh;
  int dev = 0, maxsm = 0;
  EIG_CUDA_TRY(cudaGetDevice(&dev));
  EIG_CUDA_TRY(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const size_t sm = (size_t)(P->m_pr + 8) * Sh::RBY + 16;
  if (sm > (size_t)maxsm) return EIG_EUNSUPPORTED;
  const RsArgs a = rs_args(P);
  const int xj_bulk = rs_xj_bulk<T, V, NBK>(X, ld);
  auto kern = k_spmm_mirror<T, V, NBK, CHEB>;
  EIG_CUDA_TRY(::eig::ensure_dyn_smem(kern, (int)sm));
  // the threads themselves stage double-float X: a whole CTA per row block then
  const int groups = xj_bulk ? P->m_groups : 1;
  kern<<<(unsigned)(P->nRB * groups), kW * 32 / groups, sm, st>>>(a, X, Y, ld, col0, xj_bulk, epi);
  EIG_LAUNCH_CHECK(CHEB ? "k_spmm_mirror_cheb" : "k_spmm_mirror");
  return EIG_OK;
}

// Columns [col0, col0 + nb) of a direct plan's product, in slices of at most four.  Slices of four
// start on 32-byte boundaries when X does (ld and col0 are then multiples of four); an X that is only
// 16-byte aligned is gathered in 16-byte pieces.
template <int NB, bool CHEB>
static eig_status direct_launch(SpmmPlan* P, const double* X, double* Y, int ld, int col0, const MirrorEpi& epi,
                                cudaStream_t st) {
  constexpr int NS = NB < 4 ? NB : 4;
  const bool sector = NS == 4 && (reinterpret_cast<uintptr_t>(X + col0) & 31u) == 0 && ld % 4 == 0;
  DirectArgs a;
  a.n = P->n;
  a.split = P->m_dsplit;
  a.nw = (int32_t)((P->n * a.split + 31) / 32);
  a.row = P->m_drow.as<int32_t>();
  a.len = P->m_dlen.as<int32_t>();
  a.sboff = P->m_sboff.as<int64_t>();
  a.bcol = P->m_bcol.as<uint16_t>();
  a.bval = P->m_bval.as<double>();
  a.sms = num_sms();
  const int tasks = a.nw * (NB / NS);
  auto kern = sector ? k_spmm_direct<NS, CHEB, NS == 4> : k_spmm_direct<NS, CHEB, false>;
  kern<<<(unsigned)((tasks + kDirectWarps - 1) / kDirectWarps), kDirectWarps * 32, 0, st>>>(a, X, Y, ld, col0, NB / NS,
                                                                                           epi);
  EIG_LAUNCH_CHECK(CHEB ? "k_spmm_direct_cheb" : "k_spmm_direct");
  return EIG_OK;
}

template <typename T, typename V, int NB>
eig_status mirror_launch(SpmmPlan* P, const T* X, T* Y, cudaStream_t st) {
  if constexpr (sizeof(V) == 8) {
    if (P->m_direct) return direct_launch<NB, false>(P, X, Y, NB, 0, MirrorEpi(), st);
  }
  constexpr int NBK = RsSlice<T, V, NB>::value;
  for (int c0 = 0; c0 < NB; c0 += NBK) EIG_TRY((rs_launch<T, V, NBK, false>(P, X, Y, NB, c0, MirrorEpi(), st)));
  return EIG_OK;
}

// Several products of one shape, each Y_i = H_i X_i (CHEB: the fused Chebyshev step with its
// own Qp_i, active_i, alpha_i, c_i), in one launch per at most kBatchJobs column slices over
// their concatenated row blocks; the sums are those of the single launch.
template <typename T, typename V, int NB, bool CHEB>
eig_status mirror_launch_batch(const SpmmJob* jobs, int count, cudaStream_t st) {
  constexpr int NBK = RsSlice<T, V, NB>::value;
  typedef RsShape<T, V, NBK> Sh;
  int dev = 0, maxsm = 0;
  EIG_CUDA_TRY(cudaGetDevice(&dev));
  EIG_CUDA_TRY(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  int pr = 0;
  for (int i = 0; i < count; ++i) {
    if (!jobs[i].P->mirrored) return EIG_EUNSUPPORTED;
    pr = std::max(pr, jobs[i].P->m_pr);
  }
  const size_t sm = (size_t)(pr + 8) * Sh::RBY + 16;
  if (sm > (size_t)maxsm) return EIG_EUNSUPPORTED;
  auto kern = k_spmm_mirror_batch<T, V, NBK, CHEB>;
  EIG_CUDA_TRY(::eig::ensure_dyn_smem(kern, (int)sm));
  MirrorBatch B;
  B.n = 0;
  int64_t ctas = 0;
  auto flush = [&]() -> eig_status {
    if (B.n == 0) return EIG_OK;
    B.cta0[B.n] = ctas;
    kern<<<(unsigned)ctas, kW * 32, sm, st>>>(B);
    EIG_LAUNCH_CHECK(CHEB ? "k_spmm_mirror_batch_cheb" : "k_spmm_mirror_batch");
    B.n = 0;
    ctas = 0;
    return EIG_OK;
  };
  for (int i = 0; i < count; ++i) {
    const SpmmJob& q = jobs[i];
    for (int c0 = 0; c0 < NB; c0 += NBK) {
      MirrorJob& J = B.jobs[B.n];
      J.a = rs_args(q.P);
      J.X = q.X;
      J.Y = q.Y;
      J.ld = NB;
      J.col0 = c0;
      J.xj_bulk = rs_xj_bulk<T, V, NBK>(static_cast<const T*>(q.X), NB);
      J.epi = MirrorEpi();
      if (CHEB) {
        J.epi.Qp = q.Qp;
        J.epi.active = q.active;
        J.epi.a = q.alpha;
        J.epi.c = q.c;
        J.epi.first = q.first;
      }
      B.cta0[B.n] = ctas;
      ctas += q.P->nRB;
      if (++B.n == kBatchJobs) EIG_TRY(flush());
    }
  }
  return flush();
}

#define EIG_MIRROR_BATCH_INST(T, V)                                                                    \
  template eig_status mirror_launch_batch<T, V, 8, false>(const SpmmJob*, int, cudaStream_t);           \
  template eig_status mirror_launch_batch<T, V, 16, false>(const SpmmJob*, int, cudaStream_t);          \
  template eig_status mirror_launch_batch<T, V, 8, true>(const SpmmJob*, int, cudaStream_t);            \
  template eig_status mirror_launch_batch<T, V, 16, true>(const SpmmJob*, int, cudaStream_t);
EIG_MIRROR_BATCH_INST(float, float)
EIG_MIRROR_BATCH_INST(double, float)

// One column of X (row stride ld, column col) times H into the same column of Y: the SpMV of
// a decoupled RMM-DIIS vector (Sec. 4.3), summed in the order of the block product's column.
template <typename T, typename V>
eig_status mirror_launch_column(SpmmPlan* P, const T* X, T* Y, int ld, int col, cudaStream_t st) {
  if constexpr (sizeof(V) == 8) {
    if (P->m_direct) return direct_launch<1, false>(P, X, Y, ld, col, MirrorEpi(), st);
  }
  return rs_launch<T, V, 1, false>(P, X, Y, ld, col, MirrorEpi(), st);
}

// The Chebyshev-step variant (same kernel, fused epilogue).
template <typename T, typename V, int NB>
eig_status mirror_launch_cheb(SpmmPlan* P, const T* X, T* Y, const T* Qp, const int* active, double alpha, double c,
                              int first, cudaStream_t st) {
  MirrorEpi epi;
  epi.Qp = Qp;
  epi.active = active;
  epi.a = alpha;
  epi.c = c;
  epi.first = first;
  if constexpr (sizeof(V) == 8) {
    if (P->m_direct) return direct_launch<NB, true>(P, X, Y, NB, 0, epi, st);
  }
  constexpr int NBK = RsSlice<T, V, NB>::value;
  for (int c0 = 0; c0 < NB; c0 += NBK) EIG_TRY((rs_launch<T, V, NBK, true>(P, X, Y, NB, c0, epi, st)));
  return EIG_OK;
}

#define EIG_MIRROR_CHEB_INST(T, V)                                                                               \
  template eig_status mirror_launch_cheb<T, V, 8>(SpmmPlan*, const T*, T*, const T*, const int*, double, double,  \
                                                  int, cudaStream_t);                                            \
  template eig_status mirror_launch_cheb<T, V, 16>(SpmmPlan*, const T*, T*, const T*, const int*, double, double, \
                                                   int, cudaStream_t);                                           \
  template eig_status mirror_launch_cheb<T, V, 32>(SpmmPlan*, const T*, T*, const T*, const int*, double, double, \
                                                   int, cudaStream_t);
EIG_MIRROR_CHEB_INST(float, float)
EIG_MIRROR_CHEB_INST(double, double)
EIG_MIRROR_CHEB_INST(double, float)

#define EIG_MIRROR_INST(T, V)                                                           \
  template eig_status mirror_launch<T, V, 1>(SpmmPlan*, const T*, T*, cudaStream_t);    \
  template eig_status mirror_launch<T, V, 2>(SpmmPlan*, const T*, T*, cudaStream_t);    \
  template eig_status mirror_launch<T, V, 4>(SpmmPlan*, const T*, T*, cudaStream_t);    \
  template eig_status mirror_launch<T, V, 8>(SpmmPlan*, const T*, T*, cudaStream_t);    \
  template eig_status mirror_launch<T, V, 16>(SpmmPlan*, const T*, T*, cudaStream_t);   \
  template eig_status mirror_launch<T, V, 32>(SpmmPlan*, const T*, T*, cudaStream_t);
EIG_MIRROR_INST(float, float)
EIG_MIRROR_INST(float, uint16_t)
EIG_MIRROR_INST(double, double)
EIG_MIRROR_INST(double, float)
EIG_MIRROR_INST(double, uint16_t)

template eig_status mirror_launch_column<float, float>(SpmmPlan*, const float*, float*, int, int, cudaStream_t);
template eig_status mirror_launch_column<float, uint16_t>(SpmmPlan*, const float*, float*, int, int, cudaStream_t);
template eig_status mirror_launch_column<double, double>(SpmmPlan*, const double*, double*, int, int, cudaStream_t);
template eig_status mirror_launch_column<double, float>(SpmmPlan*, const double*, double*, int, int, cudaStream_t);
template eig_status mirror_launch_column<double, uint16_t>(SpmmPlan*, const double*, double*, int, int,
                                                           cudaStream_t);

}  // namespace eig
