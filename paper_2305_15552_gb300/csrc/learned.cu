// Learned per-row preconditioner: features, MLP inference (weights in the kernel-parameter
// constant bank), fused loss + backward with deterministic reductions, Adam.
//
// The preconditioner K^{-1} of Eq. (wblock) is left open by the paper (Sec. 2.3: K only has to
// approximate H); this one replaces the Jacobi scaling by a per-entry factor m_ij = MLP(f_ij)
// learned from the solver's own residuals (the feature list and the network are in learned.cuh).
#include <cmath>
#include <vector>

#include "dense.cuh"
#include "learned.cuh"

namespace eig {
namespace {

constexpr int kApplyThreads = 256;

// ---------------------------------------------------------------------------------------
// (|H| 1)_i: sum over the full row of |h_ij|, from the upper triangle.  Each stored entry adds
// to its row and, off the diagonal, to its column's row.  Integer (fixed-point) atomics make
// the sum exact and order-independent; scale = 2^e with every row sum < 2^61 / scale.
// ---------------------------------------------------------------------------------------
template <typename V>
__global__ void k_lp_abs_total(const V* __restrict__ val, int64_t nnz, double* __restrict__ part) {
  __shared__ double red[256];
  double s = 0.0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
    s += fabs((double)ValLoad<V>::get(val, e));
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

template <typename V>
__global__ void k_lp_abs_accumulate(int64_t n, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                    const V* __restrict__ val, double scale,
                                    unsigned long long* __restrict__ acc) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
    unsigned long long own = 0;
    for (int64_t e = rowptr[i] + lane; e < rowptr[i + 1]; e += 32) {
      const unsigned long long q = __double2ull_rn(fabs((double)ValLoad<V>::get(val, e)) * scale);
      own += q;
      const int64_t j = col[e];
      if (j != i) atomicAdd(acc + j, q);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) own += __shfl_xor_sync(0xffffffffu, own, o);
    if (lane == 0 && own) atomicAdd(acc + i, own);
  }
}

__global__ void k_lp_abs_finish(int64_t n, const unsigned long long* __restrict__ acc, double inv_scale,
                                double* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (double)acc[i] * inv_scale;
}

// ---------------------------------------------------------------------------------------
// Features and the network
// ---------------------------------------------------------------------------------------
template <typename T> struct LpAcc { typedef float type; };
template <> struct LpAcc<double> { typedef double type; };

// f0..f5 of row i / column j; sc = sqrt(n) / ||r_j|| (0 for a zero column).
template <typename A>
__device__ __forceinline__ void lp_feature_row(double d, double th, double ra, A r, A hr, A sc, float f[kLpFeat]) {
  f[0] = (float)d;
  f[1] = (float)th;
  f[2] = (float)(d - th);
  f[3] = (float)ra;
  f[4] = (float)(r * sc);
  f[5] = (float)((hr - (A)d * r) * sc);
}

// J = 1 / floor(f2), the Jacobi scale the network corrects.
__device__ __forceinline__ float lp_jscale(float f2) {
  const float mag = fmaxf(fabsf(f2), kLpJacobiFloor);
  return 1.0f / (f2 < 0.0f ? -mag : mag);
}

// ReLU that keeps a NaN (so that a broken network reaches the Jacobi fallback).
__device__ __forceinline__ float lp_relu(float a) { return a > 0.0f ? a : (a == a ? 0.0f : a); }

// Weights from the kernel-parameter bank (compile-time offsets after unrolling).
struct LpConstW {
  const LpParams& P;
  __device__ __forceinline__ float operator()(int i) const { return P.p[i]; }
};
// Inference: max(a, 0) (one instruction); a parameter vector with a non-finite entry is
// caught on the host before the launch (it makes every output non-finite, as the network
// arithmetic would).
template <class WA>
__device__ __forceinline__ float lp_infer(const WA& w, const float f[kLpFeat]) {
  float u[kLpFeat];
#pragma unroll
  for (int q = 0; q < kLpFeat; ++q) u[q] = (f[q] - w(kLpOffMu + q)) / w(kLpOffSigma + q);
  float h1[kLpHid];
#pragma unroll
  for (int k = 0; k < kLpHid; ++k) {
    float a = w(kLpOffB1 + k);
#pragma unroll
    for (int q = 0; q < kLpFeat; ++q) a = fmaf(w(kLpOffW1 + k * kLpFeat + q), u[q], a);
    h1[k] = fmaxf(a, 0.0f);
  }
  float m = w(kLpOffB3);
#pragma unroll
  for (int k = 0; k < kLpHid; ++k) {
    float a = w(kLpOffB2 + k);
#pragma unroll
    for (int l = 0; l < kLpHid; ++l) a = fmaf(w(kLpOffW2 + k * kLpHid + l), h1[l], a);
    m = fmaf(w(kLpOffW3 + k), fmaxf(a, 0.0f), m);
  }
  return m;
}

// Per-column constants of a block (theta_j, sqrt(n)/||r_j||, active) into shared memory.
template <typename A>
__device__ __forceinline__ void lp_column_consts(const double* theta, const double* rsq, const int* active, int m,
                                                 int64_t n, double* sTh, A* sSc, int* sAct) {
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    sTh[j] = theta[j];
    const double q = rsq[j];
    sSc[j] = q > 0.0 ? (A)sqrt((double)n / q) : (A)0;
    sAct[j] = active ? active[j] : 1;
  }
  __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(kApplyThreads)
k_lp_apply(const __grid_constant__ LpParams prm, const T* R, const T* HR, int ld, int m, int64_t n,
           const double* __restrict__ diagH, const double* __restrict__ rowabs, const double* __restrict__ theta,
           const double* __restrict__ rsq, float floor_, const int* __restrict__ active, T* W, int* nonfinite,
           int broken) {
  typedef typename LpAcc<T>::type A;
  __shared__ double sTh[32];
  __shared__ A sSc[32];
  __shared__ int sAct[32];
  lp_column_consts<A>(theta, rsq, active, m, n, sTh, sSc, sAct);
  const LpConstW w{prm};
  int bad = 0;
  const int64_t cnt = n * m;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < cnt; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / m;
    const int j = (int)(e - i * m);
    const size_t o = (size_t)i * ld + j;
    const A r = (A)R[o], hr = (A)HR[o];
    const double d = diagH[i];
    A out = (A)0;
    if (sAct[j]) {
      float f[kLpFeat];
      lp_feature_row<A>(d, sTh[j], rowabs[i], r, hr, sSc[j], f);
      out = broken ? (A)NAN : (A)(lp_jscale(f[2]) * (1.0f + lp_infer(w, f))) * r;
      if (!isfinite(out)) {
        A den = (A)(d - sTh[j]);
        const A mag = den < (A)0 ? -den : den;
        const A fl = mag > (A)floor_ ? mag : (A)floor_;
        den = den < (A)0 ? -fl : fl;
        out = r / den;
        ++bad;
      }
    }
    W[o] = (T)out;
  }
  if (nonfinite && bad) atomicAdd(nonfinite, bad);
}

template <typename T>
__global__ void __launch_bounds__(kApplyThreads)
k_lp_features(const T* __restrict__ R, const T* __restrict__ HR, int ld, int m, int64_t n,
              const double* __restrict__ diagH, const double* __restrict__ rowabs, const double* __restrict__ theta,
              const double* __restrict__ rsq, float* __restrict__ F, float* __restrict__ rout) {
  typedef typename LpAcc<T>::type A;
  __shared__ double sTh[32];
  __shared__ A sSc[32];
  __shared__ int sAct[32];
  lp_column_consts<A>(theta, rsq, nullptr, m, n, sTh, sSc, sAct);
  const int64_t cnt = n * m;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < cnt; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / m;
    const int j = (int)(e - i * m);
    const size_t o = (size_t)i * ld + j;
    const A r = (A)R[o];
    float f[kLpFeat];
    lp_feature_row<A>(diagH[i], sTh[j], rowabs[i], r, (A)HR[o], sSc[j], f);
#pragma unroll
    for (int q = 0; q < kLpFeat; ++q) F[e * kLpFeat + q] = f[q];
    rout[e] = (float)r;
  }
}

__global__ void __launch_bounds__(kApplyThreads)
k_lp_forward(const __grid_constant__ LpParams prm, const float* __restrict__ F, int64_t count, float* __restrict__ mo,
             int broken) {
  const LpConstW w{prm};
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
    float f[kLpFeat];
#pragma unroll
    for (int q = 0; q < kLpFeat; ++q) f[q] = F[e * kLpFeat + q];
    mo[e] = broken ? NAN : lp_jscale(f[2]) * (1.0f + lp_infer(w, f));
  }
}

int params_broken(const LpParams& prm) {
  for (int i = 0; i < kLpParams; ++i)
    if (!std::isfinite(prm.p[i])) return 1;
  return 0;
}

int apply_grid(int64_t count) {
  const int64_t want = (count + kApplyThreads - 1) / kApplyThreads;
  return (int)min64(max64(want, 1), (int64_t)num_sms() * 8);
}

}  // namespace

// ---------------------------------------------------------------------------------------
// Loss of the correction targets and its gradient.  A CTA of four warps takes tiles of
// kGradThreads entries: forward, dL/dm, backward to the per-entry layer deltas, all staged in
// shared memory, then the products that make up each parameter's gradient, summed over the tile
// in entry order (FP32) and added to FP64 totals held by the thread that owns the parameter; CTA
// partials are reduced in a fixed order, so the result is deterministic.
//
// What bounds it: the shared-memory pipe and the FP32 pipe at about the same level (~3600 multiply-
// adds an entry; a 128-bit shared load takes two clocks when adjacent lanes share its address and
// four otherwise).  One thread per entry, as inference runs, would load every weight once per 32
// entries and staging rows of 32 words puts a warp's stores into one bank.  So:
//   * layers: warp w computes outputs [8 w, 8 w + 8) for all 128 entries, four entries a lane, so
//     eight weights (uniform, two loads) serve 32 multiply-adds a lane, issued as FP32x2 pairs;
//   * W2 gradient: two warps, each thread a 4 x 4 block of parameters in registers (two loads per
//     16 multiply-adds); the other two take W1, the biases and b3;
//   * rows are padded to 36 words: a lane's 16-byte piece of its own row is conflict free;
//   * the output layer's gradient is summed before the backward pass overwrites the second
//     layer's activations with the first layer's deltas; three CTAs per SM then fit.
// Every sum keeps its order (entries ascending, FP32, one tile of 128), so each tile's FP32 sums
// are those of a thread-per-entry kernel.  Measured at 8e6 entries (1M rows x 8 columns): 1.85 ms;
// the thread-per-entry kernel took 7.48 ms.
// ---------------------------------------------------------------------------------------
namespace {

constexpr int kGradThreads = 128;                                             // entries per tile
constexpr int kGradOut = kLpTrained + 1;                                      // + loss
constexpr int kGS = 36;                                                       // row stride of the staged blocks
constexpr int kGradCtas = 3;                                                  // per SM

struct GradSmem {
  float W2[kLpHid * kLpHid];            // [k][l]
  float W2T[kLpHid * kLpHid];           // [l][k]
  float W1[kLpHid * 8];                 // [k][6 weights, bias, 0]
  float b2[kLpHid], w3[kLpHid];
  float mu[8], sigma[8];                // [6], [7]: padding; mu[7] holds b3
  float U[kGradThreads * 8];            // features u0..u5, f2 (raw), 0
  float H1[kGradThreads * kGS];         // layer 1 activations
  float H2[kGradThreads * kGS];         // layer 2 activations, then the layer 1 deltas
  float Da2[kGradThreads * kGS];        // layer 2 deltas
  float dm[kGradThreads];
};
static_assert(sizeof(GradSmem) + 1024 <= 233472 / kGradCtas, "three CTAs per SM");

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// acc[i][2q..2q+1] += w[2q..2q+1] * x_i for the four entries i of a lane, eight outputs
__device__ __forceinline__ void grad_rank1(float2 (&acc)[4][4], const float* w, const float (&x)[4]) {
  const float4 wa = ld4(w), wb = ld4(w + 4);
  const float2 wp[4] = {make_float2(wa.x, wa.y), make_float2(wa.z, wa.w), make_float2(wb.x, wb.y),
                        make_float2(wb.z, wb.w)};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 xx = make_float2(x[i], x[i]);
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[i][q] = __ffma2_rn(wp[q], xx, acc[i][q]);
  }
}

// acc[i][:] += sum_r M[r][col0 .. col0 + 8) * S[entry i][r], r = 0..31 ascending
__device__ __forceinline__ void grad_layer(float2 (&acc)[4][4], const float* M, int col0, const float* S, int lane) {
#pragma unroll 2
  for (int r0 = 0; r0 < kLpHid; r0 += 4) {
    float4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = ld4(S + (lane + 32 * i) * kGS + r0);
    const float x0[4] = {x[0].x, x[1].x, x[2].x, x[3].x}, x1[4] = {x[0].y, x[1].y, x[2].y, x[3].y};
    const float x2[4] = {x[0].z, x[1].z, x[2].z, x[3].z}, x3[4] = {x[0].w, x[1].w, x[2].w, x[3].w};
    grad_rank1(acc, M + (r0 + 0) * kLpHid + col0, x0);
    grad_rank1(acc, M + (r0 + 1) * kLpHid + col0, x1);
    grad_rank1(acc, M + (r0 + 2) * kLpHid + col0, x2);
    grad_rank1(acc, M + (r0 + 3) * kLpHid + col0, x3);
  }
}

__device__ __forceinline__ void grad_store8(float* row, const float (&v)[8]) {
  reinterpret_cast<float4*>(row)[0] = make_float4(v[0], v[1], v[2], v[3]);
  reinterpret_cast<float4*>(row)[1] = make_float4(v[4], v[5], v[6], v[7]);
}

__global__ void __launch_bounds__(kGradThreads, kGradCtas)
k_lp_grad(const float* __restrict__ params, const float* __restrict__ F, const float* __restrict__ rr,
          const float* __restrict__ zz, const double* __restrict__ colw, int64_t n, int m,
          double* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
  __shared__ double red[kGradThreads];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  for (int i = t; i < kLpHid * kLpHid; i += kGradThreads) {
    const float v = params[kLpOffW2 + i];
    S.W2[i] = v;
    S.W2T[(i % kLpHid) * kLpHid + i / kLpHid] = v;
  }
  for (int i = t; i < kLpHid * 8; i += kGradThreads) {
    const int k = i >> 3, q = i & 7;
    S.W1[i] = q < kLpFeat ? params[kLpOffW1 + k * kLpFeat + q] : (q == kLpFeat ? params[kLpOffB1 + k] : 0.0f);
  }
  if (t < kLpHid) {
    S.b2[t] = params[kLpOffB2 + t];
    S.w3[t] = params[kLpOffW3 + t];
  }
  if (t < 8) {
    S.mu[t] = t < kLpFeat ? params[kLpOffMu + t] : (t == 7 ? params[kLpOffB3] : 0.0f);
    S.sigma[t] = t < kLpFeat ? params[kLpOffSigma + t] : 1.0f;
  }
  // roles of the gradient sums: which two warps take W2 differs among the CTAs of an SM, so that
  // the work is spread over its four schedulers
  const int role = (w + (int)((int64_t)blockIdx.x * kGradCtas / gridDim.x)) & 3;
  const int kb = 4 * (((role & 1) * 32 + lane) >> 3), lb = 4 * (lane & 7);   // W2 block (roles 0, 1)
  double tot[16];       // roles 0, 1: the 4 x 4 block; roles 2, 3: W1 (3), bias
#pragma unroll
  for (int i = 0; i < 16; ++i) tot[i] = 0.0;
  double tot_w3 = 0.0, tot_b3 = 0.0, loss = 0.0;
  const int64_t cnt = n * m;
  const int64_t ntiles = (cnt + kGradThreads - 1) / kGradThreads;
  // the next tile's features (6 consecutive words a thread apart), residual and target
  float fn[kLpFeat], rn = 0.0f, zn = 0.0f;
  auto fetch = [&](int64_t tile) {
    const int64_t base = tile * kGradThreads;
    const int valid = (int)min64(kGradThreads, cnt - base);
#pragma unroll
    for (int i = 0; i < kLpFeat; ++i) {
      const int e = t + i * kGradThreads;
      fn[i] = e < valid * kLpFeat ? F[base * kLpFeat + e] : 0.0f;
    }
    rn = t < valid ? rr[base + t] : 0.0f;
    zn = t < valid ? zz[base + t] : 0.0f;
  };
  if ((int64_t)blockIdx.x < ntiles) fetch(blockIdx.x);
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    __syncthreads();   // the weights are staged; the previous tile's sums are done with its rows
    const int64_t base = tile * kGradThreads;
    const int valid = (int)min64(kGradThreads, cnt - base);
    // ---- standardised features
#pragma unroll
    for (int i = 0; i < kLpFeat; ++i) {
      const int e = t + i * kGradThreads, x = e / kLpFeat, q = e % kLpFeat;
      S.U[x * 8 + q] = x < valid ? (fn[i] - S.mu[q]) / S.sigma[q] : 0.0f;
      if (q == 2) S.U[x * 8 + 6] = fn[i];
    }
    const float r = rn, z = zn;
    if (tile + gridDim.x < ntiles) fetch(tile + gridDim.x);
    __syncthreads();
    // ---- layer 1, outputs [8 w, 8 w + 8) of entries lane + 32 i
    unsigned m1 = 0, m2 = 0;   // bit 8 i + o: activation of output 8 w + o is positive
    {
      float4 ua[4];
      float2 ub[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ua[i] = ld4(S.U + (lane + 32 * i) * 8);
        ub[i] = *reinterpret_cast<const float2*>(S.U + (lane + 32 * i) * 8 + 4);
      }
      float h[4][8];
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const float4 wa = ld4(S.W1 + (8 * w + o) * 8), wb = ld4(S.W1 + (8 * w + o) * 8 + 4);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float a = wb.z;
          a = fmaf(wa.x, ua[i].x, a);
          a = fmaf(wa.y, ua[i].y, a);
          a = fmaf(wa.z, ua[i].z, a);
          a = fmaf(wa.w, ua[i].w, a);
          a = fmaf(wb.x, ub[i].x, a);
          a = fmaf(wb.y, ub[i].y, a);
          if (a > 0.0f) m1 |= 1u << (8 * i + o);
          h[i][o] = lane + 32 * i < valid ? lp_relu(a) : 0.0f;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) grad_store8(S.H1 + (lane + 32 * i) * kGS + 8 * w, h[i]);
    }
    __syncthreads();
    // ---- layer 2
    float2 acc[4][4];
    {
      const float4 ba = ld4(S.b2 + 8 * w), bb = ld4(S.b2 + 8 * w + 4);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[i][0] = make_float2(ba.x, ba.y);
        acc[i][1] = make_float2(ba.z, ba.w);
        acc[i][2] = make_float2(bb.x, bb.y);
        acc[i][3] = make_float2(bb.z, bb.w);
      }
    }
    grad_layer(acc, S.W2T, 8 * w, S.H1, lane);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float h[8];
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const float a = (o & 1) ? acc[i][o >> 1].y : acc[i][o >> 1].x;
        if (a > 0.0f) m2 |= 1u << (8 * i + o);
        h[o] = lane + 32 * i < valid ? lp_relu(a) : 0.0f;
      }
      grad_store8(S.H2 + (lane + 32 * i) * kGS + 8 * w, h);
    }
    __syncthreads();
    // ---- output layer of entry t, loss, dL/dm and dL/do = dL/dm * J (m = J (1 + o))
    {
      float mo = S.mu[7];
#pragma unroll
      for (int k = 0; k < kLpHid; k += 4) {
        const float4 wv = ld4(S.w3 + k), hv = ld4(S.H2 + t * kGS + k);
        mo = fmaf(wv.x, hv.x, mo);
        mo = fmaf(wv.y, hv.y, mo);
        mo = fmaf(wv.z, hv.z, mo);
        mo = fmaf(wv.w, hv.w, mo);
      }
      float dm = 0.0f;
      if (t < valid) {
        const float jsc = lp_jscale(S.U[t * 8 + 6]);
        const int64_t e = base + t;
        const int j = cnt <= 0x7fffffff ? (int)((unsigned)e % (unsigned)m) : (int)(e % m);
        const double cw = colw[j];
        const float err = jsc * (1.0f + mo) * r - z;
        dm = (float)(2.0 * cw) * r * err * jsc;
        loss += cw * (double)err * (double)err;
      }
      S.dm[t] = dm;
    }
    __syncthreads();
    // ---- layer 2 deltas
    {
      const float4 wa = ld4(S.w3 + 8 * w), wb = ld4(S.w3 + 8 * w + 4);
      const float wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float dm = S.dm[lane + 32 * i];
        float d[8];
#pragma unroll
        for (int o = 0; o < 8; ++o) d[o] = (m2 >> (8 * i + o) & 1u) ? dm * wv[o] : 0.0f;
        grad_store8(S.Da2 + (lane + 32 * i) * kGS + 8 * w, d);
      }
    }
    // w3 and b3 (the layer 2 activations are overwritten below): one lane per output
    if (role == 3) {
      float a3 = 0.0f, ab = 0.0f;
#pragma unroll 8
      for (int x = 0; x < kGradThreads; ++x) {
        const float dm = S.dm[x];
        a3 = fmaf(dm, S.H2[x * kGS + lane], a3);
        ab += dm;
      }
      tot_w3 += (double)a3;
      tot_b3 += (double)ab;
    }
    __syncthreads();
    // ---- layer 1 deltas, into the layer 2 activations' rows
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][q] = make_float2(0.0f, 0.0f);
    grad_layer(acc, S.W2, 8 * w, S.Da2, lane);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float d[8];
#pragma unroll
      for (int o = 0; o < 8; ++o)
        d[o] = (m1 >> (8 * i + o) & 1u) ? ((o & 1) ? acc[i][o >> 1].y : acc[i][o >> 1].x) : 0.0f;
      grad_store8(S.H2 + (lane + 32 * i) * kGS + 8 * w, d);
    }
    __syncthreads();
    // ---- sums over the tile of (delta x activation)
    if (role < 2) {
      float2 g[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) g[i][0] = g[i][1] = make_float2(0.0f, 0.0f);
#pragma unroll 4
      for (int x = 0; x < kGradThreads; ++x) {
        const float4 a = ld4(S.Da2 + x * kGS + kb), b = ld4(S.H1 + x * kGS + lb);
        const float av[4] = {a.x, a.y, a.z, a.w};
        const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 aa = make_float2(av[i], av[i]);
          g[i][0] = __ffma2_rn(aa, b0, g[i][0]);
          g[i][1] = __ffma2_rn(aa, b1, g[i][1]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        tot[4 * i + 0] += (double)g[i][0].x;
        tot[4 * i + 1] += (double)g[i][0].y;
        tot[4 * i + 2] += (double)g[i][1].x;
        tot[4 * i + 3] += (double)g[i][1].y;
      }
    } else {
      // row `lane` of W1, columns [0, 3) and b1 (role 2) or columns [3, 6) and b2 (role 3)
      const int q0 = role == 2 ? 0 : 3;
      const float* bias = role == 2 ? S.H2 : S.Da2;
      float g0 = 0.0f, g1 = 0.0f, g2 = 0.0f, gb = 0.0f;
#pragma unroll 8
      for (int x = 0; x < kGradThreads; ++x) {
        const float d = S.H2[x * kGS + lane];
        g0 = fmaf(d, S.U[x * 8 + q0], g0);
        g1 = fmaf(d, S.U[x * 8 + q0 + 1], g1);
        g2 = fmaf(d, S.U[x * 8 + q0 + 2], g2);
        gb += bias[x * kGS + lane];
      }
      tot[0] += (double)g0;
      tot[1] += (double)g1;
      tot[2] += (double)g2;
      tot[3] += (double)gb;
    }
  }
  double* out = part + (size_t)blockIdx.x * kGradOut;
  if (role < 2) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) out[kLpOffW2 - kLpFixed + (kb + i) * kLpHid + lb + c] = tot[4 * i + c];
  } else {
    const int q0 = role == 2 ? 0 : 3;
#pragma unroll
    for (int c = 0; c < 3; ++c) out[kLpOffW1 - kLpFixed + lane * kLpFeat + q0 + c] = tot[c];
    out[(role == 2 ? kLpOffB1 : kLpOffB2) - kLpFixed + lane] = tot[3];
    if (role == 3) {
      out[kLpOffW3 - kLpFixed + lane] = tot_w3;
      if (lane == 0) out[kLpOffB3 - kLpFixed] = tot_b3;
    }
  }
  red[t] = loss;
  __syncthreads();
  for (int o = kGradThreads / 2; o > 0; o >>= 1) {
    if (t < o) red[t] += red[t + o];
    __syncthreads();
  }
  if (t == 0) out[kLpTrained] = red[0];
}

__global__ void k_lp_adam(float* __restrict__ p, const double* __restrict__ g, float* __restrict__ m1,
                          float* __restrict__ m2, double lr, double b1, double b2, double bc1, double bc2, double eps) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= kLpTrained) return;
  const int i = kLpFixed + q;
  const double gq = g[q];
  const double a = b1 * (double)m1[i] + (1.0 - b1) * gq;
  const double v = b2 * (double)m2[i] + (1.0 - b2) * gq * gq;
  m1[i] = (float)a;
  m2[i] = (float)v;
  p[i] = (float)((double)p[i] - lr * (a / bc1) / (sqrt(v / bc2) + eps));
}

int grad_grid() { return num_sms() * kGradCtas; }

template <typename V>
eig_status row_abs_sum_t(const SpmmPlan& P, double* out, cudaStream_t st) {
  const int64_t n = P.n;
  const int grid = num_sms() * 4;
  DevBuf part, acc;
  EIG_TRY(part.reserve((size_t)grid * 8 + 8));
  EIG_TRY(acc.reserve((size_t)n * 8));
  k_lp_abs_total<V><<<grid, 256, 0, st>>>((const V*)P.val, P.nnz, part.as<double>());
  EIG_LAUNCH_CHECK("k_lp_abs_total");
  double* total_d = part.as<double>() + grid;
  EIG_TRY(reduce_partials(part.as<double>(), grid, 1, total_d, st));
  double total = 0.0;
  EIG_CUDA_TRY(cudaMemcpyAsync(&total, total_d, 8, cudaMemcpyDeviceToHost, st));
  EIG_CUDA_TRY(cudaStreamSynchronize(st));
  if (!std::isfinite(total)) return EIG_EINVAL;
  // every full-row sum is <= total: choose 2^e with total * 2^e < 2^61
  int ex = 0;
  std::frexp(total > 0.0 ? total : 1.0, &ex);
  const double scale = std::ldexp(1.0, 61 - ex);
  EIG_CUDA_TRY(cudaMemsetAsync(acc.p, 0, (size_t)n * 8, st));
  const int ag = (int)min64((n * 32 + 255) / 256, (int64_t)num_sms() * 16);
  k_lp_abs_accumulate<V><<<ag, 256, 0, st>>>(n, P.rowptr, P.col, (const V*)P.val, scale,
                                             acc.as<unsigned long long>());
  EIG_LAUNCH_CHECK("k_lp_abs_accumulate");
  k_lp_abs_finish<<<(int)min64((n + 255) / 256, (int64_t)num_sms() * 8), 256, 0, st>>>(
      n, acc.as<unsigned long long>(), 1.0 / scale, out);
  EIG_LAUNCH_CHECK("k_lp_abs_finish");
  EIG_CUDA_TRY(cudaStreamSynchronize(st));   // part / acc are released on return
  return EIG_OK;
}

}  // namespace

eig_status lp_row_abs_sum(const SpmmPlan& P, double* out, cudaStream_t st) {
  if (!P.rowptr || !out || P.n < 1) return EIG_EINVAL;
  switch (P.val_type) {
    case EIG_F32: return row_abs_sum_t<float>(P, out, st);
    case EIG_F64: return row_abs_sum_t<double>(P, out, st);
    case EIG_BF16: return row_abs_sum_t<uint16_t>(P, out, st);
  }
  return EIG_EINVAL;
}

eig_status lp_apply(const LpParams& prm, const void* R, const void* HR, int ld, int m, int64_t n, eig_dtype vt,
                    const double* diagH, const double* rowabs, const double* theta, const double* rsq, double floor_,
                    const int* active, void* W, int* nonfinite, cudaStream_t st) {
  if (m < 1 || m > 32 || ld < m || n < 0) return EIG_EINVAL;
  if (n == 0) return EIG_OK;
  const int grid = apply_grid(n * m);
  const int broken = params_broken(prm);
  if (vt == EIG_F32)
    k_lp_apply<float><<<grid, kApplyThreads, 0, st>>>(prm, (const float*)R, (const float*)HR, ld, m, n, diagH, rowabs,
                                                      theta, rsq, (float)floor_, active, (float*)W, nonfinite, broken);
  else if (vt == EIG_F64)
    k_lp_apply<double><<<grid, kApplyThreads, 0, st>>>(prm, (const double*)R, (const double*)HR, ld, m, n, diagH,
                                                       rowabs, theta, rsq, (float)floor_, active, (double*)W,
                                                       nonfinite, broken);
  else
    return EIG_EINVAL;
  EIG_LAUNCH_CHECK("k_lp_apply");
  return EIG_OK;
}

eig_status lp_features(const void* R, const void* HR, int ld, int m, int64_t n, eig_dtype vt, const double* diagH,
                       const double* rowabs, const double* theta, const double* rsq, float* F, float* r,
                       cudaStream_t st) {
  if (m < 1 || m > 32 || ld < m || n < 0) return EIG_EINVAL;
  if (n == 0) return EIG_OK;
  const int grid = apply_grid(n * m);
  if (vt == EIG_F32)
    k_lp_features<float><<<grid, kApplyThreads, 0, st>>>((const float*)R, (const float*)HR, ld, m, n, diagH, rowabs,
                                                         theta, rsq, F, r);
  else if (vt == EIG_F64)
    k_lp_features<double><<<grid, kApplyThreads, 0, st>>>((const double*)R, (const double*)HR, ld, m, n, diagH,
                                                          rowabs, theta, rsq, F, r);
  else
    return EIG_EINVAL;
  EIG_LAUNCH_CHECK("k_lp_features");
  return EIG_OK;
}

eig_status lp_forward(const LpParams& prm, const float* F, int64_t count, float* m_out, cudaStream_t st) {
  if (count < 0) return EIG_EINVAL;
  if (count == 0) return EIG_OK;
  k_lp_forward<<<apply_grid(count), kApplyThreads, 0, st>>>(prm, F, count, m_out, params_broken(prm));
  EIG_LAUNCH_CHECK("k_lp_forward");
  return EIG_OK;
}

size_t lp_grad_workspace_bytes() { return (size_t)grad_grid() * kGradOut * 8 + 256; }

eig_status lp_grad(const float* params, const float* F, const float* r, const float* z, const double* colw,
                   int64_t n, int m, double* out, void* workspace, cudaStream_t st) {
  if (m < 1 || n < 0 || !params || !out || !workspace) return EIG_EINVAL;
  const int64_t ntiles = (n * m + kGradThreads - 1) / kGradThreads;
  const int grid = (int)max64(1, min64(ntiles, grad_grid()));
  // set on every call: the attribute belongs to the current device
  EIG_CUDA_TRY(::eig::ensure_dyn_smem(k_lp_grad, (int)sizeof(GradSmem)));
  k_lp_grad<<<grid, kGradThreads, sizeof(GradSmem), st>>>(params, F, r, z, colw, n, m, (double*)workspace);
  EIG_LAUNCH_CHECK("k_lp_grad");
  return reduce_partials((const double*)workspace, grid, kGradOut, out, st);
}

eig_status lp_adam(float* params, const double* grad, float* m1, float* m2, int t, double lr, double beta1,
                   double beta2, double eps, cudaStream_t st) {
  if (t < 1 || !params || !grad || !m1 || !m2) return EIG_EINVAL;
  const double bc1 = 1.0 - std::pow(beta1, t), bc2 = 1.0 - std::pow(beta2, t);
  k_lp_adam<<<(kLpTrained + 255) / 256, 256, 0, st>>>(params, grad, m1, m2, lr, beta1, beta2, bc1, bc2, eps);
  EIG_LAUNCH_CHECK("k_lp_adam");
  return EIG_OK;
}

}  // namespace eig
