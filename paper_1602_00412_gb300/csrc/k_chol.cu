// Cholesky factor and its inverse for CholeskyQR (the GramSchmidt step of
// Alg. 1): G + shift I = L L^T and Rinv = L^-T, one CTA, k <= 256.
//
// In-place elimination on 4 x 4 tiles of the lower triangle. M starts as G and ends
// as L^-1: after pivot tile p, the tile rows <= p hold rows of L^-1, and of the tile
// rows I > p the columns <= p hold the partial right-hand sides of the inverse and
// the columns > p the trailing matrix, so factor and inverse share one triangle and
// one update. With X the rows 4 p .. 4 p + 3 of M (columns past the pivot by
// symmetry) and x the inverse of the pivot's factor, the four elimination rows are
//   W = x X,  x itself in the pivot's columns,
// whose columns > p are also L^T, and the update is M[I][J] -= W_I^T W_J.
// One barrier per pivot. Between two barriers
//  - the chain's warps, a lane per column of the matrix, bring X up to date with the
//    previous W, factor and invert the pivot (every lane does, so nothing is
//    broadcast) and leave the next W, which is four finished rows of L^-1;
//  - the tiles' warps, each thread holding its tiles in registers, apply the
//    previous W and put the next pivot's X into shared memory.
// What bounds it is the chain of k / 4 pivots on one SM: about 150 dependent
// instructions each, four roots among them. (Holding the tiles in shared memory made
// the update's loads and stores the bound; 16-wide panels with one warp on the
// diagonal block left 250 clocks per column on its shuffles.)
//
// Measured (GB300, back-to-back launches; column-at-a-time and 16-wide panel forms
// with FP64 before): fp32 k = 50 / 100 / 200: 8 / 20 / 71 us (20 / 47 / 893), accurate
// k = 50 / 100 / 200: 30 / 76 / 345 us (about 110 / 387 / 2408). The error of Rinv
// against a double-precision factor of the same matrix is, in the accurate form, that of
// the final rounding to fp32 (2.1e-8 to 2.6e-8, as the FP64 factor's) up to condition
// number 1e6 of G; in fp32 0.8e-7 to 1.4e-7 at condition 10 and 1e-3 to 1.8e-3 at 1e6
// (0.8e-7 to 3.2e-7 and 1.5e-3 to 2.6e-3 before).
//
// The accurate passes (see chol_inv) hold every value as an unevaluated sum of
// two floats (48 significant bits; sums and products by the error-free
// transformations of Dekker and Knuth): GB300 does 2 FP64 multiply-adds per clock
// per SM against 128 in FP32, so an FP64 multiply-add costs as much as 64
// FP32 instructions and the two-float one 12.
#include <atomic>

#include "sfd_internal.cuh"

namespace sfd {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ------------------------------------------------------- two-float arithmetic
// v = h + l with |l| <= ulp(h) / 2. The _rn intrinsics keep the compiler from
// contracting the error terms away.
struct DF {
  float h, l;
};
__device__ __forceinline__ DF df_fast(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ DF df_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
// a * b as (rounded product, its error with the cross terms), not normalised
__device__ __forceinline__ DF df_prod(DF a, DF b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return {p, e};
}

// Operations shared by the float and the two-float instantiation.
__device__ __forceinline__ float c_mul(float a, float b) { return a * b; }
__device__ __forceinline__ DF c_mul(DF a, DF b) {
  const DF p = df_prod(a, b);
  return df_fast(p.h, p.l);
}
// acc += a b; the two-float accumulator is normalised by c_norm after a run of terms
__device__ __forceinline__ void c_acc(float& acc, float a, float b) { acc = fmaf(a, b, acc); }
__device__ __forceinline__ void c_acc(DF& acc, DF a, DF b) {
  const DF p = df_prod(a, b), s = df_two_sum(acc.h, p.h);
  acc.h = s.h;
  acc.l = __fadd_rn(acc.l, __fadd_rn(s.l, p.l));
}
__device__ __forceinline__ float c_norm(float a) { return a; }
__device__ __forceinline__ DF c_norm(DF a) { return df_fast(a.h, a.l); }
__device__ __forceinline__ float c_neg(float a) { return -a; }
__device__ __forceinline__ DF c_neg(DF a) { return {-a.h, -a.l}; }
__device__ __forceinline__ float c_sub(float a, float b) { return a - b; }
__device__ __forceinline__ DF c_sub(DF a, DF b) {
  const DF s = df_two_sum(a.h, -b.h);
  return df_fast(s.h, __fadd_rn(s.l, __fsub_rn(a.l, b.l)));
}
__device__ __forceinline__ float c_shfl(float v, int lane) { return __shfl_sync(kFull, v, lane); }
__device__ __forceinline__ DF c_shfl(DF v, int lane) {
  return {__shfl_sync(kFull, v.h, lane), __shfl_sync(kFull, v.l, lane)};
}
__device__ __forceinline__ bool c_pos(float v) { return v > 0.f; }
__device__ __forceinline__ bool c_pos(DF v) { return v.h > 0.f; }
// 1 / sqrt of a pivot (scaled into the normal range): the hardware estimate in fp32
__device__ __forceinline__ float c_rsqrt(float p) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(p));
  return y;
}
// 1 / sqrt(p): the fp32 estimate y and one third-order correction
// y (1 + r / 2 + 3 r^2 / 8) with r = 1 - p y^2 formed to fp32 accuracy
__device__ __forceinline__ DF c_rsqrt(DF p) {
  const float y = c_rsqrt(p.h);
  const float th = __fmul_rn(p.h, y);
  const float tl = __fmaf_rn(p.l, y, __fmaf_rn(p.h, y, -th));
  const float r = __fsub_rn(__fmaf_rn(-th, y, 1.f), __fmul_rn(tl, y));
  return df_fast(y, __fmul_rn(__fmul_rn(y, r), __fmaf_rn(0.375f, r, 0.5f)));
}

// Four matrix rows in shared memory, [4][n] (two-float: then their low parts).
template <typename T>
struct Rows;
template <>
struct Rows<float> {
  float* p;
  __device__ float get(int o) const { return p[o]; }
  __device__ void put(int o, float v) const { p[o] = v; }
  __device__ void get4(int o, float (&v)[4]) const {
    const float4 a = *reinterpret_cast<const float4*>(p + o);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  }
  __device__ void put4(int o, const float (&v)[4]) const {
    *reinterpret_cast<float4*>(p + o) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <>
struct Rows<DF> {
  float *p, *q;
  __device__ DF get(int o) const { return {p[o], q[o]}; }
  __device__ void put(int o, DF v) const {
    p[o] = v.h;
    q[o] = v.l;
  }
  __device__ void get4(int o, DF (&v)[4]) const {
    const float4 a = *reinterpret_cast<const float4*>(p + o);
    const float4 b = *reinterpret_cast<const float4*>(q + o);
    v[0] = {a.x, b.x}; v[1] = {a.y, b.y}; v[2] = {a.z, b.z}; v[3] = {a.w, b.w};
  }
  __device__ void put4(int o, const DF (&v)[4]) const {
    *reinterpret_cast<float4*>(p + o) = make_float4(v[0].h, v[1].h, v[2].h, v[3].h);
    *reinterpret_cast<float4*>(q + o) = make_float4(v[0].l, v[1].l, v[2].l, v[3].l);
  }
};
template <typename T>
constexpr bool kTwo = sizeof(T) == 2 * sizeof(float);
template <typename T>
__device__ __forceinline__ T c_val(float h) {
  if constexpr (kTwo<T>) return {h, 0.f};
  else return h;
}
__device__ __forceinline__ float c_out(float v) { return v; }
__device__ __forceinline__ float c_out(DF v) { return __fadd_rn(v.h, v.l); }
__device__ __forceinline__ float c_times(float a, float s) { return a * s * s; }

__host__ __device__ constexpr int tri(int I) { return I * (I + 1) / 2; }

// The shift 2^-20 trace(G) / k keeps the factorisation defined for a rank-deficient
// block. G is taken times 2^-2e with trace / k in [1, 4) (the result is scaled back
// by 2^-e, both exact), which keeps pivots and low parts in the normal range.
template <typename T>
struct Scale {
  float sc;  // M = G sc sc + shift I, Rinv = L^-T sc
  T shift;
};
// red: 2 floats per warp
__device__ __forceinline__ void scale_of(const float* G, int k, float* red, Scale<float>& S) {
  const int nw = blockDim.x >> 5;
  float tr = 0.f;
  for (int i = threadIdx.x; i < k; i += blockDim.x) tr += G[(int64_t)i * k + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(kFull, tr, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = tr;
  __syncthreads();
  tr = 0.f;
  for (int w = 0; w < nw; ++w) tr += red[w];
  const float mean = tr / (float)k;
  const int e2 = mean > 0.f && isfinite(mean) ? ilogbf(mean) >> 1 : 0;
  S = {ldexpf(1.f, -e2), tr > 0.f ? ldexpf(mean, -20 - 2 * e2) : 1e-30f};
}
// The trace of the accurate form is a two-float sum of the diagonal times 2^-e, with e
// the exponent of its largest entry: a trace may exceed the largest float where no entry
// of G does.
__device__ __forceinline__ void scale_of(const float* G, int k, float* red, Scale<DF>& S) {
  const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float big = 0.f;
  for (int i = threadIdx.x; i < k; i += blockDim.x) big = fmaxf(big, fabsf(G[(int64_t)i * k + i]));
  const unsigned bits = __reduce_max_sync(kFull, __float_as_uint(big));
  if (lane == 0) red[warp] = __uint_as_float(bits);
  __syncthreads();
  for (int w = 0; w < nw; ++w) big = fmaxf(big, red[w]);
  const int e = big > 0.f && isfinite(big) ? ilogbf(big) : 0;
  __syncthreads();
  auto add = [](DF a, DF b) {
    const DF s = df_two_sum(a.h, b.h);
    return df_fast(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
  };
  DF tr = {0.f, 0.f};
  for (int i = threadIdx.x; i < k; i += blockDim.x)
    tr = add(tr, {ldexpf(G[(int64_t)i * k + i], -e), 0.f});
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    tr = add(tr, {__shfl_xor_sync(kFull, tr.h, o), __shfl_xor_sync(kFull, tr.l, o)});
  if (lane == 0) {
    red[2 * warp] = tr.h;
    red[2 * warp + 1] = tr.l;
  }
  __syncthreads();
  tr = {0.f, 0.f};
  for (int w = 0; w < nw; ++w) tr = add(tr, {red[2 * w], red[2 * w + 1]});
  const float kf = (float)k, q = __fdiv_rn(tr.h, kf);
  const DF mean = df_fast(q, __fdiv_rn(__fadd_rn(__fmaf_rn(-q, kf, tr.h), tr.l), kf));
  const bool pos = tr.h > 0.f;
  const int e2 = pos && isfinite(tr.h) ? (ilogbf(mean.h) + e) >> 1 : 0;
  const int es = e - 20 - 2 * e2;
  S.sc = ldexpf(1.f, -e2);
  S.shift = pos ? DF{ldexpf(mean.h, es), ldexpf(mean.l, es)} : DF{1e-30f, 0.f};
}

// CW chain warps (a lane per column), NTW tile warps with TPT tiles per thread.
template <typename T, int CW, int NTW, int TPT>
__global__ void __launch_bounds__(32 * (CW + NTW))
    k_chol_inv_tiles(const float* __restrict__ G, int k, float* __restrict__ Rinv,
                     int* __restrict__ flags) {
  constexpr int kLd = 32 * CW;  // columns of X and W
  constexpr int kPl = kTwo<T> ? 2 : 1;
  __shared__ __align__(16) float xw[4][kPl][4 * kLd];  // X and W of the even and odd pivots
  __shared__ float red[2 * (CW + NTW)];
  const int NB = (k + 3) >> 2;
  const int tid = threadIdx.x, warp = tid >> 5;
  auto rows = [&](int i) {
    Rows<T> r;
    r.p = xw[i][0];
    if constexpr (kTwo<T>) r.q = xw[i][1];
    return r;
  };

  // this thread's tiles (I < 0: none)
  int I[TPT], J[TPT];
  T m[TPT][4][4];
#pragma unroll
  for (int n = 0; n < TPT; ++n) {
    const int e = tid - 32 * CW + n * 32 * NTW;
    I[n] = -1;
    J[n] = 0;
    if (warp >= CW && e < tri(NB)) {
      int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
      while (tri(i) > e) --i;
      while (tri(i + 1) <= e) ++i;
      I[n] = i;
      J[n] = e - tri(i);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = 4 * I[n] + r, j = 4 * J[n] + q, a = max(i, j), b = min(i, j);
        m[n][r][q] = c_val<T>(I[n] < 0 ? 0.f : a < k ? G[(int64_t)a * k + b] : i == j ? 1.f : 0.f);
      }
  }
  Scale<T> S;
  scale_of(G, k, red, S);
  const float sc = S.sc;
  const T shift = S.shift;
  const float least = c_out(shift);  // in place of a pivot that is not positive
  // tiles of pivot P's row and column into X
  auto publish = [&](int n, int P) {
    const Rows<T> X = rows(P & 1);
    if (I[n] == P) {
#pragma unroll
      for (int r = 0; r < 4; ++r) X.put4(r * kLd + 4 * J[n], m[n][r]);
    } else if (J[n] == P) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const T t[4] = {m[n][0][r], m[n][1][r], m[n][2][r], m[n][3][r]};
        X.put4(r * kLd + 4 * I[n], t);
      }
    }
  };
#pragma unroll
  for (int n = 0; n < TPT; ++n) {
    if (I[n] < 0) continue;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (max(4 * I[n] + r, 4 * J[n] + q) >= k) continue;  // padding: the identity
        if constexpr (kTwo<T>) m[n][r][q].h = c_times(m[n][r][q].h, sc);
        else m[n][r][q] = c_times(m[n][r][q], sc);
        if (I[n] == J[n] && r == q) m[n][r][q] = c_sub(m[n][r][q], c_neg(shift));
      }
    publish(n, 0);
  }
  __syncthreads();

  int clamped = 0;
#pragma unroll 1
  for (int P = 0; P < NB; ++P) {
    const Rows<T> Wo = rows(2 + ((P + 1) & 1));  // of pivot P - 1
    if (warp < CW) {
      const Rows<T> X = rows(P & 1), Wn = rows(2 + (P & 1));
      const int g = tid, c = g >> 2;
      T d[4][4], v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        X.get4(r * kLd + 4 * P, d[r]);
        v[r] = X.get(r * kLd + g);
      }
      if (P > 0) {
        T lp[4][4], w[4];  // lp[u][r] = L[4 P + r][4 (P - 1) + u]
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          Wo.get4(u * kLd + 4 * P, lp[u]);
          w[u] = Wo.get(u * kLd + g);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {  // the pivot's lower triangle, and this column
#pragma unroll
          for (int q = 0; q <= r; ++q) {
            T acc = c_mul(lp[0][r], lp[0][q]);
#pragma unroll
            for (int u = 1; u < 4; ++u) c_acc(acc, lp[u][r], lp[u][q]);
            d[r][q] = c_sub(d[r][q], c_norm(acc));
          }
          T acc = c_mul(lp[0][r], w[0]);
#pragma unroll
          for (int u = 1; u < 4; ++u) c_acc(acc, lp[u][r], w[u]);
          if (c == P - 1) v[r] = c_val<T>(0.f);  // the inverse's new columns start from zero
          v[r] = c_sub(v[r], c_norm(acc));
        }
      }
      // factor the pivot (d: its L below the diagonal, inv: 1 / diagonal) and invert
      // the factor row by row (x)
      T inv[4], x[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool pos = c_pos(d[j][j]);
        clamped += !pos;
        inv[j] = c_rsqrt(pos ? d[j][j] : c_val<T>(least));
#pragma unroll
        for (int r = j + 1; r < 4; ++r) d[r][j] = c_mul(d[r][j], inv[j]);
#pragma unroll
        for (int r = j + 1; r < 4; ++r)
#pragma unroll
          for (int q = j + 1; q <= r; ++q) d[r][q] = c_sub(d[r][q], c_mul(d[r][j], d[q][j]));
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        x[r][r] = inv[r];
#pragma unroll
        for (int q = 0; q < r; ++q) {
          T acc = c_mul(d[r][q], x[q][q]);
#pragma unroll
          for (int t = q + 1; t < r; ++t) c_acc(acc, d[r][t], x[t][q]);
          x[r][q] = c_neg(c_mul(c_norm(acc), inv[r]));
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (c == P) v[r] = c_val<T>(r == (g & 3) ? 1.f : 0.f);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        T y = c_mul(x[r][0], v[0]);
#pragma unroll
        for (int t = 1; t <= r; ++t) c_acc(y, x[r][t], v[t]);
        y = c_norm(y);
        Wn.put(r * kLd + g, y);
        // row 4 P + r of L^-1: column 4 P + r of Rinv
        if (g < k && 4 * P + r < k) Rinv[(int64_t)g * k + 4 * P + r] = c <= P ? c_out(y) * sc : 0.f;
      }
    } else {
#pragma unroll
      for (int n = 0; n < TPT; ++n) {
        if (I[n] <= P) continue;
        if (J[n] == P) {  // taken by the chain; the inverse's columns start from zero
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) m[n][r][q] = c_val<T>(0.f);
          continue;
        }
        if (P > 0) {
          T acc[4][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            T l[4], w[4];
            Wo.get4(u * kLd + 4 * I[n], l);
            Wo.get4(u * kLd + 4 * J[n], w);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                if (u == 0) acc[r][q] = c_mul(l[r], w[q]);
                else c_acc(acc[r][q], l[r], w[q]);
              }
          }
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) m[n][r][q] = c_sub(m[n][r][q], c_norm(acc[r][q]));
        }
        publish(n, P + 1);
      }
    }
    __syncthreads();
  }
  if (tid == 0 && clamped) atomicAdd(&flags[1], clamped);
}

// ------------------------------------------------------------------ panel form
constexpr int kCB = 16;  // panel width
constexpr int kLiLd = kCB + 4;
constexpr int kPanelThreads = 512;
constexpr int kPanelSmemMax = 226 * 1024;  // dynamic; the kernel has a little static too

// block row I of M: 16 rows of 16 (I + 1) columns, leading dimension 16 (I + 1) + 4
// (16-byte rows; eight consecutive rows start in eight different bank quads)
__host__ __device__ constexpr int m_off(int I) { return 128 * I * (I + 1) + 64 * I; }
__host__ __device__ constexpr int m_ld(int I) { return 16 * (I + 1) + 4; }
// leading dimension of the pivot rows (reads down a column: two rows per bank)
__host__ __device__ constexpr int r_ld(int KP) { return KP + 4; }

// Steps c (diagonal block of row I only, after panel I - 1; nothing for I = 0) and a:
// factor and invert the block, L^-1 to Li. One warp: lane i + 16 h holds columns
// t = 2 s + h of row i of the block (d, shifted down by one s every two columns) and
// of the inverse (x). The next pivot is formed from values fetched before the
// current one's reciprocal root is known, so a column costs one root and two
// multiply-adds in sequence, and the shuffles of the updates overlap the next root.
template <typename T>
__device__ __forceinline__ void diag_block(Rows<T> M, Rows<T> R, int ldr, Rows<T> Li, int I, float least,
                                           int& clamped) {
  const int lane = threadIdx.x & 31, i = lane & 15, h = lane >> 4;
  T d[8], x[8];
  {
    const int o = m_off(I) + i * m_ld(I) + I * kCB + h;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      d[s] = M.get(o + 2 * s);
      x[s] = c_val<T>(i == 2 * s + h ? 1.f : 0.f);
    }
  }
  if (I > 0) {
    T acc[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) acc[s] = c_val<T>(0.f);
#pragma unroll(kTwo<T> ? 1 : 4)
    for (int u = 0; u < kCB; ++u) {
      const T a = R.get(u * ldr + I * kCB + i);
#pragma unroll
      for (int s = 0; s < 8; ++s) c_acc(acc[s], a, R.get(u * ldr + I * kCB + 2 * s + h));
    }
#pragma unroll
    for (int s = 0; s < 8; ++s) d[s] = c_sub(d[s], c_norm(acc[s]));
  }
  T piv = c_shfl(d[0], 0);
#pragma unroll(kTwo<T> ? 1 : 8)
  for (int jj = 0; jj < 8; ++jj) {
#pragma unroll
    for (int sub = 0; sub < 2; ++sub) {
      const int j = 2 * jj + sub, own = sub << 4;  // the half that holds column j
      const T dj = c_shfl(d[0], i | own);
      const T c = c_shfl(d[0], ((j + 1) & 15) | own);
      const T q = c_shfl(d[sub], ((j + 1) & 15) | (own ^ 16));
      const bool pos = c_pos(piv);
      clamped += !pos;
      const T inv = c_rsqrt(pos ? piv : c_val<T>(least));
      const T l = i > j ? c_mul(dj, inv) : c_val<T>(0.f);
      const T nl = c_neg(l), ln = c_mul(c, inv);
      piv = q;
      c_acc(piv, c_neg(ln), ln);
      piv = c_norm(piv);
#pragma unroll
      for (int s = 0; s < 8; ++s) {  // lanes <= j hold l = 0; columns past 15 are dead
        c_acc(d[s], nl, c_shfl(l, (j - sub + 2 * s + h) & 31));
        d[s] = c_norm(d[s]);
      }
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        if (i == j) x[s] = c_mul(x[s], inv);
        c_acc(x[s], nl, c_shfl(x[s], j | (h << 4)));
        x[s] = c_norm(x[s]);
      }
    }
#pragma unroll
    for (int s = 0; s < 7; ++s) d[s] = d[s + 1];
    d[7] = c_val<T>(0.f);
  }
#pragma unroll
  for (int s = 0; s < 8; ++s) Li.put(i * kLiLd + 2 * s + h, x[s]);
}

// One 16 x 32 tile of step c: block row I, columns 32 jt .. (a warp; 4 x 4 per lane).
template <typename T>
__device__ __forceinline__ void update_tile(Rows<T> M, Rows<T> R, int ldr, int p, int I, int jt) {
  const int lane = threadIdx.x & 31;
  const int r0 = (lane >> 3) * 4, col = jt * 32 + (lane & 7) * 4;
  // the next diagonal block is warp 0's: it leaves M there as it was
  if (col >= kCB * (I + 1) || (I == p + 1 && col >= kCB * I)) return;
  T acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = c_val<T>(0.f);
#pragma unroll(kTwo<T> ? 1 : 4)
  for (int t = 0; t < kCB; ++t) {
    T a[4], b[4];
    R.get4(t * ldr + I * kCB + r0, a);
    R.get4(t * ldr + col, b);
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) c_acc(acc[u][v], a[u], b[v]);
  }
  const bool fresh = (col >> 4) == p;  // the inverse's column block p starts from zero
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int o = m_off(I) + (r0 + u) * m_ld(I) + col;
    T m[4];
    M.get4(o, m);
#pragma unroll
    for (int v = 0; v < 4; ++v)
      m[v] = fresh ? c_neg(c_norm(acc[u][v])) : c_sub(m[v], c_norm(acc[u][v]));
    M.put4(o, m);
  }
}

// Step b for 16 columns c (rows c below the panel) of group g, pivot rows 8 part + h,
// + 2, + 4, + 6 of them: a half-warp per h.
template <typename T>
__device__ __forceinline__ void pivot_rows(Rows<T> M, Rows<T> R, int ldr, Rows<T> Li, int p, int g,
                                           int part) {
  const int lane = threadIdx.x & 31, h = lane >> 4, cc = lane & 15, c = g * kCB + cc;
  T in[kCB];
  if (g < p) {
#pragma unroll
    for (int u = 0; u < kCB; ++u) in[u] = M.get(m_off(p) + u * m_ld(p) + c);
  } else {
    const int o = m_off(g) + cc * m_ld(g) + p * kCB;
#pragma unroll
    for (int u = 0; u < kCB; u += 4) {
      T q[4];
      M.get4(o + u, q);
      in[u] = q[0]; in[u + 1] = q[1]; in[u + 2] = q[2]; in[u + 3] = q[3];
    }
  }
#pragma unroll 1
  for (int s = 0; s < 4; ++s) {
    const int t = 8 * part + 2 * s + h;
    T a0 = c_val<T>(0.f), a1 = c_val<T>(0.f);
    if (g == p) {
      a0 = Li.get(t * kLiLd + cc);
    } else {
#pragma unroll
      for (int u = 0; u < kCB; u += 4) {  // Li[t][u] is 0 for u > t
        if (u < 8 * part + 8) {
          T q[4];
          Li.get4(t * kLiLd + u, q);
          c_acc(a0, q[0], in[u]);
          c_acc(a1, q[1], in[u + 1]);
          c_acc(a0, q[2], in[u + 2]);
          c_acc(a1, q[3], in[u + 3]);
        }
      }
      a0 = c_sub(c_norm(a0), c_neg(c_norm(a1)));
    }
    R.put(t * ldr + c, a0);
  }
}

// Panel form, for triangles that do not fit the registers: M in shared memory, 16-wide
// panels, two barriers each. Per panel p:
//   a. one warp factors the 16 x 16 diagonal block and inverts it in registers;
//   b. the pivot rows R (16 x KP): Li times the block row p (columns < p), Li
//      itself, and the panel below times Li^T, which is L21^T (columns > p);
//   c. every block row i > p takes M[i][j] -= R[.][i]^T R[.][j] for all j <= i, in
//      16 x 32 warp tiles (4 x 4 per lane), while warp 0 updates the next diagonal
//      block in its registers and goes on to (a).
// lo_work: the low parts of M when they do not fit beside the rest (two-float form
// for k > 208), m_off(NB) floats of global memory; else null.
template <typename T, bool kLoGlobal>
__global__ void __launch_bounds__(kPanelThreads)
    k_chol_panel(const float* __restrict__ G, int k, float* __restrict__ Rinv, float* lo_work,
                   int* __restrict__ flags) {
  extern __shared__ __align__(16) float chol_sm[];
  const int NB = (k + kCB - 1) / kCB, KP = NB * kCB, ldr = r_ld(KP);
  const int msz = m_off(NB), rsz = kCB * ldr;
  Rows<T> M, R, Li;  // M: m_off(NB); R: 16 x ldr; Li: 16 x kLiLd
  M.p = chol_sm;
  R.p = M.p + msz;
  Li.p = R.p + rsz;
  if constexpr (kTwo<T>) {
    R.q = Li.p + kCB * kLiLd;
    Li.q = R.q + rsz;
    M.q = kLoGlobal ? lo_work : Li.q + kCB * kLiLd;
  }
  __shared__ float red[2 * (kPanelThreads / 32)];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;

  Scale<T> S;
  scale_of(G, k, red, S);
  const T shift = S.shift;
  const float least = c_out(shift);  // in place of a pivot that is not positive
  // the lower triangle of G, a warp per row; padding rows are the identity
  for (int i = warp; i < KP; i += nw) {
    const int I = i >> 4, o = m_off(I) + (i & 15) * m_ld(I), w = kCB * (I + 1);
    for (int j = lane; j < w; j += 32) {
      const int a = max(i, j), b = min(i, j);  // columns past the diagonal mirror it
      T x = c_val<T>(a < k ? c_times(G[(int64_t)a * k + b], S.sc) : (i == j ? 1.f : 0.f));
      if (i == j && i < k) x = c_sub(x, c_neg(shift));
      M.put(o + j, x);
    }
  }
  __syncthreads();

  int clamped = 0;
  for (int p = 0; p <= NB; ++p) {
    // ---- c for panel p - 1 (block row I has (I + 2) / 2 tiles), a for panel p
    if (warp == 0) {
      if (p < NB) diag_block<T>(M, R, ldr, Li, p, least, clamped);
    } else if (p > 0) {
      int I = p, nt = (p + 1) / 2, rem = warp - 1;  // row p without its diagonal block
      for (;;) {
        while (I < NB && rem >= nt) {
          rem -= nt;
          ++I;
          nt = (I + 2) / 2;
        }
        if (I >= NB) break;
        update_tile<T>(M, R, ldr, p - 1, I, rem);
        rem += nw - 1;
      }
      // rows 16 (p - 1) + t of L^-1 are R: column i = 16 (p - 1) + t of Rinv = L^-T
      const int t = lane & 15, i = (p - 1) * kCB + t;
      for (int c = 2 * (warp - 1) + (lane >> 4); c < k; c += 2 * (nw - 1)) {
        float v = 0.f;
        if (c < p * kCB) {
          v = c_out(R.get(t * ldr + c)) * S.sc;
        }
        if (i < k) Rinv[(int64_t)c * k + i] = v;
      }
    }
    __syncthreads();
    if (p == NB) break;
    // ---- b
    for (int it = warp; it < 2 * NB; it += nw) pivot_rows<T>(M, R, ldr, Li, p, it >> 1, it & 1);
    __syncthreads();
  }
  if (warp == 0 && lane == 0 && clamped) atomicAdd(&flags[1], clamped);
}

size_t panel_smem_bytes(int k, bool two, bool lo_global) {
  const int NB = (k + kCB - 1) / kCB;
  const size_t small = kCB * r_ld(NB * kCB) + kCB * kLiLd;
  return ((size_t)m_off(NB) * (two && !lo_global ? 2 : 1) + small * (two ? 2 : 1)) * sizeof(float);
}

template <typename T, bool kLoGlobal>
void launch_panel(const float* G, int k, float* Rinv, float* work, int* flags, cudaStream_t s) {
  auto f = k_chol_panel<T, kLoGlobal>;
  static std::atomic<unsigned> attr{0};
  int dev = 0;
  SFD_CUDA(cudaGetDevice(&dev));
  if (dev < 32 && !(attr.load() & (1u << dev))) {
    SFD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kPanelSmemMax));
    attr.fetch_or(1u << dev);
  }
  f<<<1, kPanelThreads, panel_smem_bytes(k, sizeof(T) == 8, kLoGlobal), s>>>(G, k, Rinv, work, flags);
}

}  // namespace

void chol_inv_blk(const float* G, int k, float* Rinv, float* work, int* flags, cudaStream_t s,
                  bool accurate) {
  // the triangle in registers, a tile per thread, up to k = 128 (136 / 406 / 528 tiles
  // for k = 64 / 112 / 128), in fp32 two tiles up to k = 160; the panel form above
  // (fp32 k = 160: 51 us in registers against 57 for the panels; k = 200, where two
  // tiles spill: 88 against 74; two-float k = 128: 129 against 166 at k = 129)
  if (accurate) {
    if (k <= 64) k_chol_inv_tiles<DF, 2, 5, 1><<<1, 224, 0, s>>>(G, k, Rinv, flags);
    else if (k <= 112) k_chol_inv_tiles<DF, 4, 13, 1><<<1, 544, 0, s>>>(G, k, Rinv, flags);
    else if (k <= 128) k_chol_inv_tiles<DF, 4, 17, 1><<<1, 672, 0, s>>>(G, k, Rinv, flags);
    else if (panel_smem_bytes(k, true, false) <= (size_t)kPanelSmemMax)
      launch_panel<DF, false>(G, k, Rinv, work, flags, s);
    else launch_panel<DF, true>(G, k, Rinv, work, flags, s);
  } else {
    if (k <= 64) k_chol_inv_tiles<float, 2, 5, 1><<<1, 224, 0, s>>>(G, k, Rinv, flags);
    else if (k <= 112) k_chol_inv_tiles<float, 4, 13, 1><<<1, 544, 0, s>>>(G, k, Rinv, flags);
    else if (k <= 128) k_chol_inv_tiles<float, 4, 17, 1><<<1, 672, 0, s>>>(G, k, Rinv, flags);
    else if (k <= 160) k_chol_inv_tiles<float, 5, 13, 2><<<1, 576, 0, s>>>(G, k, Rinv, flags);
    else launch_panel<float, false>(G, k, Rinv, nullptr, flags, s);
  }
  SFD_LAUNCH_CHECK();
}

}  // namespace sfd
