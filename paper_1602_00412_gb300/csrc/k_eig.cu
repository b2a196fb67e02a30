// Symmetric eigensolver for the small matrices of the method: P P^T (l x l)
// in SparseShrink (Alg. 3, svd(P, l)) and [B; B'][B; B']^T (2l x 2l) in
// DenseShrink (Alg. 5, svd([B; B'], l)). Only the `nwant` largest eigenpairs
// are formed, in fp32:
//  1. Householder tridiagonalisation A = Q T Q^T, A in registers (one CTA up to
//     n = 128, a cluster of 2 up to 256, of 8 up to 512).
//  2. Multisection on Sturm counts of T for eigenvalues n-1 .. n-nwant (a warp per
//     eigenvalue), and the 4 x 4 factors that join every four reflectors.
//  3. Inverse iteration for their eigenvectors of T (one thread per vector,
//     LU with partial pivoting of T - lambda I), then CholeskyQR2 of the block (a
//     classical Gram-Schmidt repair path takes over when vectors are dependent).
//  4. Back-transformation Z <- Q Z, four reflectors at a time.
// Every stage is a chain of n short steps on few SMs, so its latencies bound it. Kernel
// time 251 us for n = 100 (all vectors), 616 for n = 200 (100 of them) and 1.83 ms for n =
// 400 (200). Before, with the matrix in shared (n > 223: global) memory, the update and the
// product two passes, and one reflector at a time applied from global memory: 487 us,
// 1259 us and 12.4 ms. Results keep their accuracy for largest eigenvalues from 1e-12 to
// 1e18 (columns below a norm of 8.7e-19 are taken as zero). Gram matrices up to n = 64
// take one-sided Jacobi in one CTA.
#include <cooperative_groups.h>
#include <float.h>

#include <algorithm>
#include <atomic>

#include "sfd_internal.cuh"

namespace sfd {

namespace {

constexpr int kThreads = 1024;
constexpr int kSmemLimit = 200 * 1024;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ float block_reduce(float v, float* red, int op /*0 sum, 1 max, 2 min*/) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float t = __shfl_xor_sync(0xffffffffu, v, o);
    v = op == 0 ? v + t : (op == 1 ? fmaxf(v, t) : fminf(v, t));
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    float t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : (op == 0 ? 0.f : red[0]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      float u = __shfl_xor_sync(0xffffffffu, t, o);
      t = op == 0 ? t + u : (op == 1 ? fmaxf(t, u) : fminf(t, u));
    }
    if (threadIdx.x == 0) red[32] = t;
  }
  __syncthreads();
  return red[32];
}

__device__ __forceinline__ float hash_unit(int i, int j) {
  uint32_t h = (uint32_t)i * 0x9E3779B1u ^ ((uint32_t)j + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; h ^= h >> 15;
  return (float)(h >> 8) * (2.0f / 16777216.0f) - 1.0f;   // [-1, 1)
}

// One inverse-iteration step on column z (stride nwp): solve with the stored
// LU of T - lambda I (row swaps P, multipliers Lm, U with three diagonals),
// then scale to max |z| = 1 and finally to unit length.
__device__ void tri_solve_scaled(const float* U0, const float* U1, const float* U2,
                                 const float* Lm, const float* P, float* Z, int n, int nwp) {
  for (int i = 0; i + 1 < n; ++i) {
    float ri = Z[i * nwp], rn = Z[(i + 1) * nwp];
    if (P[i * nwp] != 0.f) { float t = ri; ri = rn; rn = t; }
    Z[i * nwp] = ri;
    Z[(i + 1) * nwp] = rn - Lm[i * nwp] * ri;
  }
  // back substitution; near a cluster the solution can outgrow fp32, so when
  // an entry passes 2^100 the whole system (solved part, neighbours and the
  // remaining right-hand side) is scaled by 2^-100 and the entry redone
  float zmax = 0.f, z1 = 0.f, z2 = 0.f;
  for (int i = n - 1; i >= 0; --i) {
    float z = (Z[i * nwp] - U1[i * nwp] * z1 - U2[i * nwp] * z2) / U0[i * nwp];
    if (!(fabsf(z) <= 0x1p100f)) {
      for (int k = 0; k < n; ++k) Z[k * nwp] *= 0x1p-100f;
      z1 *= 0x1p-100f;
      z2 *= 0x1p-100f;
      zmax *= 0x1p-100f;
      z = (Z[i * nwp] - U1[i * nwp] * z1 - U2[i * nwp] * z2) / U0[i * nwp];
      if (!(fabsf(z) <= 0x1p100f)) z = 0.f;
    }
    Z[i * nwp] = z;
    z2 = z1;
    z1 = z;
    zmax = fmaxf(zmax, fabsf(z));
  }
  float inv = zmax > 0.f ? 1.f / zmax : 1.f;
  float nrm = 0.f;
  for (int i = 0; i < n; ++i) {
    float z = Z[i * nwp] * inv;
    nrm = fmaf(z, z, nrm);
  }
  inv *= nrm > 0.f ? rsqrtf(nrm) : 0.f;
  for (int i = 0; i < n; ++i) Z[i * nwp] *= inv;
}

// LU with partial pivoting of the tridiagonal T - lam I (diagonal d, off
// diagonal e): U has three diagonals (U0, U1, U2), Lm the multipliers, P the
// row swaps; pivots below tiny_piv are raised to +-tiny_piv.
__device__ void tri_factor(const float* d, const float* e, float lam, float* U0, float* U1,
                           float* U2, float* Lm, float* P, int n, int st, float tiny_piv) {
  float a_i = d[0] - lam, c_i = n > 1 ? e[0] : 0.f;
  for (int i = 0; i + 1 < n; ++i) {
    const float b = e[i];
    const float an = d[i + 1] - lam;
    const float cn = (i + 2 < n) ? e[i + 1] : 0.f;
    float a_nx, c_nx;
    if (fabsf(b) > fabsf(a_i)) {
      const float l = a_i / b;
      U0[i * st] = b; U1[i * st] = an; U2[i * st] = cn; P[i * st] = 1.f; Lm[i * st] = l;
      a_nx = c_i - l * an;
      c_nx = -l * cn;
    } else {
      float piv = a_i;
      if (fabsf(piv) < tiny_piv) piv = piv < 0.f ? -tiny_piv : tiny_piv;
      const float l = b / piv;
      U0[i * st] = piv; U1[i * st] = c_i; U2[i * st] = 0.f; P[i * st] = 0.f; Lm[i * st] = l;
      a_nx = an - l * c_i;
      c_nx = cn;
    }
    a_i = a_nx;
    c_i = c_nx;
  }
  // the last row has no super-diagonals, multiplier or swap; they are written
  // (not left as whatever the memory held) because the solve reads U1 and U2
  // of that row times 0, and a leftover NaN / Inf pattern would make it NaN
  U0[(n - 1) * st] = a_i;
  U1[(n - 1) * st] = 0.f;
  U2[(n - 1) * st] = 0.f;
  Lm[(n - 1) * st] = 0.f;
  P[(n - 1) * st] = 0.f;
  for (int i = 0; i < n; ++i) {
    float u = U0[i * st];
    if (fabsf(u) < tiny_piv) U0[i * st] = u < 0.f ? -tiny_piv : tiny_piv;
  }
}

// Sturm count: how many eigenvalues of the tridiagonal (d, e2 = e^2) lie below x.
// The quotient uses the fast reciprocal (2 ulp): a count is only wrong for x
// within a few ulps of an eigenvalue, which moves the bisection result by as
// much and no more. |q| >= pivmin keeps the divisor in range.
__device__ int sturm_count(const float* d, const float* e2, int n, float x, float pivmin) {
  int cnt = 0;
  float q = d[0] - x;
  if (fabsf(q) < pivmin) q = -pivmin;
  cnt += q < 0.f;
  for (int i = 1; i < n; ++i) {
    q = (d[i] - x) - __fdividef(e2[i - 1], q);
    if (fabsf(q) < pivmin) q = -pivmin;
    cnt += q < 0.f;
  }
  return cnt;
}

// acc += a b on two neighbouring columns in one instruction (the same rounding as fmaf)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

// acc + (a b + c d) on two neighbouring columns: the products are summed first, so that
// acc, which may be far larger, is rounded once
__device__ __forceinline__ float2 add_products(float2 acc, float2 a, float2 b, float2 c, float2 d) {
  float2 r;
  asm("{\n\t.reg .b64 ra, rb, rc, rd, re;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "mov.b64 rd, {%8, %9};\n\tmov.b64 re, {%10, %11};\n\t"
      "mul.rn.f32x2 rc, rc, rd;\n\tfma.rn.f32x2 ra, ra, rb, rc;\n\t"
      "add.rn.f32x2 re, re, ra;\n\tmov.b64 {%0, %1}, re;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y), "f"(d.x), "f"(d.y), "f"(acc.x),
        "f"(acc.y));
  return r;
}

// Sum of v[0..RW) over the warp's lanes, each element in the lanes of one group:
// afterwards lane L holds element elem_of(L) (halving exchanges, so 9 shuffles for 8
// elements and 8 for 4).
template <int RW>
__device__ __forceinline__ float reduce_rows(float (&v)[RW]) {
  const int lane = threadIdx.x & 31;
  int off = 16;
#pragma unroll
  for (int half = RW / 2; half > 0; half >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int t = 0; t < half; ++t) {
      const float keep = up ? v[t + half] : v[t], send = up ? v[t] : v[t + half];
      v[t] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  float x = v[0];
  for (; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

// 1. Householder tridiagonalisation. Step k reflects column k below the diagonal:
// A22 -= u w^T + w u^T with p = beta A22 u, w = p - (beta u^T p / 2) u. The matrix
// stays in registers: warp W of all 16 NC holds rows i = W + 16 NC r, lane j of it
// columns j + 32 q (cyclic, so the shrinking trailing matrix stays spread), and one
// pass applies the previous step's update and multiplies by the new u. Between
// passes a thread per index forms w and the next column from p and the row that the
// pass left in shared memory. NC CTAs of a cluster leave p and the row in each
// other's shared memory (two buffers, so a CTA may run ahead by half a step); each
// forms the vectors for itself. What bounds it is that chain: two barriers, two warp
// sums, a square root and the lane sums of p per step. Reflector k goes to
// house[k n + i] (zero for i <= k) and beta[k].
template <int NC, int RW, int QP>
__global__ void __cluster_dims__(NC, 1, 1) __launch_bounds__(512)
    k_tridiag(const float* __restrict__ S, int n, float* __restrict__ house,
              float* __restrict__ beta_g, float* __restrict__ dg, float* __restrict__ eg,
              int* __restrict__ flags) {
  namespace cg = cooperative_groups;
  constexpr int kN = 64 * QP;  // columns held
  __shared__ float2 uw[512];   // (u, w) of the step before, by index
  __shared__ float xn[512];    // this step's column below the diagonal, by index
  __shared__ float p_s[2][kN], row_s[2][kN];
  __shared__ __align__(16) float kp_s[2][16 * NC];
  __shared__ __align__(16) float npart[16];
  __shared__ float amax_s[16 * NC], last_s;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = NC > 1 ? (int)cl.block_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = rank * 16 + warp;
  auto to_all = [&](float* at, float v) {  // the same address in every CTA
    if constexpr (NC == 1) {
      *at = v;
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) *cl.map_shared_rank(at, c) = v;
    }
  };
  auto sync_all = [&] {
    if constexpr (NC == 1) __syncthreads();
    else cl.sync();
  };
  if (rank == 0 && tid == 0) flags[3] = 0;
  if constexpr (NC > 1) cl.sync();  // every CTA runs before any writes to another

  float2 A[RW][QP];
  float amax = 0.f;
#pragma unroll
  for (int r = 0; r < RW; ++r)
#pragma unroll
    for (int q = 0; q < QP; ++q) {
      const int i = W + 16 * NC * r, j = lane + 64 * q;
      A[r][q].x = i < n && j < n ? S[(size_t)i * n + j] : 0.f;
      A[r][q].y = i < n && j + 32 < n ? S[(size_t)i * n + j + 32] : 0.f;
      amax = fmaxf(amax, fmaxf(fabsf(A[r][q].x), fabsf(A[r][q].y)));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if (lane == 0) to_all(&amax_s[W], amax);
  if (n <= 2 && tid == 0) last_s = S[(size_t)n * n - 1];
  sync_all();
  amax = 0.f;
  for (int c = 0; c < 16 * NC; ++c) amax = fmaxf(amax, amax_s[c]);
  // a column below this squared norm is at fp32 resolution of the matrix: its
  // reflector is skipped (and 2 / |u|^2 cannot overflow)
  const float negligible2 = fmaxf(1e-30f * amax * amax, 64.f * FLT_MIN);

  float u0 = 0.f, bt = 0.f, x = 0.f;  // of the step before (x: this thread's entry of its column)
  for (int k = 0;; ++k) {
    // ---- vectors: thread i forms w_i of the step before and entry i of column k
    const int i = tid, b = (k - 1) & 1;
    float ui = 0.f, wi = 0.f, col = 0.f;
    if (k == 0) {
      if (i < n) col = S[i];
    } else {
      float ks;  // u^T p
      if constexpr (NC <= 2) {
        float4 t[4 * NC];
#pragma unroll
        for (int c = 0; c < 4 * NC; ++c) t[c] = *reinterpret_cast<const float4*>(&kp_s[b][4 * c]);
#pragma unroll
        for (int h = 2 * NC; h > 0; h >>= 1)
#pragma unroll
          for (int c = 0; c < h; ++c) {
            t[c].x += t[c + h].x; t[c].y += t[c + h].y;
            t[c].z += t[c + h].z; t[c].w += t[c + h].w;
          }
        ks = (t[0].x + t[0].y) + (t[0].z + t[0].w);
      } else {
        ks = 0.f;
#pragma unroll
        for (int c = 0; c < NC / 2; ++c) ks += kp_s[b][lane + 32 * c];
        ks = warp_sum(ks);
      }
      const float K = 0.5f * bt * ks;
      const float wk = p_s[b][k] - K * u0;
      if (i >= k && i < n) {
        ui = i == k ? u0 : x;
        wi = p_s[b][i] - K * ui;
        col = row_s[b][i] - (ui * wk + wi * u0);
      }
    }
    if (i == k && rank == 0) dg[k] = col;
    if (k + 2 >= n) {  // the last 2 x 2 block
      if (rank == 0) {
        if (i == k + 1 && i < n) {
          eg[k] = col;
          dg[i] = last_s - 2.f * ui * wi;
        }
        if (i == n - 1) eg[n - 1] = 0.f;
      }
      break;
    }
    x = i > k && i < n ? col : 0.f;
    uw[i] = make_float2(ui, wi);
    xn[i] = x;
    const float ns = warp_sum(x * x);
    if (lane == 0) npart[warp] = ns;
    __syncthreads();
    // ---- the reflector
    float norm2 = 0.f;
#pragma unroll
    for (int c = 0; c < 16; c += 4) {
      const float4 t = *reinterpret_cast<const float4*>(&npart[c]);
      norm2 += (t.x + t.y) + (t.z + t.w);
    }
    const float x0 = xn[k + 1];
    float alpha = x0;
    u0 = x0;
    bt = 0.f;
    if (norm2 - x0 * x0 > negligible2) {
      alpha = -copysignf(sqrtf(norm2), x0);
      u0 = x0 - alpha;
      bt = 2.f / (norm2 - x0 * x0 + u0 * u0);
    }
    if (rank == k % NC) {
      if (i < n) house[(size_t)k * n + i] = i == k + 1 ? u0 : x;
      if (tid == 0) {
        beta_g[k] = bt;
        eg[k] = alpha;
      }
    }
    // ---- A -= u w^T + w u^T of the step before; p = A u
    float2 uq[QP], wq[QP], nq[QP];
#pragma unroll
    for (int q = 0; q < QP; ++q) {
      const int j = lane + 64 * q;
      const float2 s0 = uw[j], s1 = uw[j + 32];
      uq[q] = make_float2(s0.x, s1.x);
      wq[q] = make_float2(s0.y, s1.y);
      nq[q] = make_float2(j == k + 1 ? u0 : xn[j], j + 32 == k + 1 ? u0 : xn[j + 32]);
    }
    float acc[RW];
    float* row_out = row_s[k & 1];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const int ir = W + 16 * NC * r;
      acc[r] = 0.f;
      if (ir <= k || ir >= n) continue;
      const float2 s = uw[ir];
      const float2 nu = make_float2(-s.x, -s.x), nw = make_float2(-s.y, -s.y);
      float2 a2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < QP; ++q) {
        if (64 * q + 63 <= k || 64 * q >= n) continue;
        // (two multiply-adds onto A would round it twice: residuals 1.07 to 1.12 times
        // these, for 1.5 % of the call at n = 200)
        A[r][q] = add_products(A[r][q], nw, uq[q], nu, wq[q]);
        a2 = fma2(A[r][q], nq[q], a2);
      }
      acc[r] = a2.x + a2.y;
      if (ir == k + 1) {
#pragma unroll
        for (int q = 0; q < QP; ++q) {
          to_all(&row_out[lane + 64 * q], A[r][q].x);
          to_all(&row_out[lane + 64 * q + 32], A[r][q].y);
        }
      }
      if (k + 3 == n && ir == n - 1) {
#pragma unroll
        for (int q = 0; q < QP; ++q) {
          if (lane + 64 * q == n - 1) to_all(&last_s, A[r][q].x);
          if (lane + 64 * q + 32 == n - 1) to_all(&last_s, A[r][q].y);
        }
      }
    }
    // beta joins here, before the next product with u: u^T A u alone is of the size of
    // the eigenvalue cubed and leaves fp32's range near 1e14 and below 1e-11
    const float pr = bt * reduce_rows<RW>(acc);
    // lane L holds row W + 16 NC r with r from its top bits
    constexpr int kSh = RW == 8 ? 2 : 3;
    const int re = RW == 8 ? ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)
                           : ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1);
    const int ip = W + 16 * NC * re;
    float kp = 0.f;
    if (ip > k && ip < n) {
      const float un = ip == k + 1 ? u0 : xn[ip];
      kp = un * pr;
      if ((lane & ((1 << kSh) - 1)) == 0) to_all(&p_s[k & 1][ip], pr);
    }
#pragma unroll
    for (int o = 16; o >= (1 << kSh); o >>= 1) kp += __shfl_xor_sync(0xffffffffu, kp, o);
    if (lane == 0) to_all(&kp_s[k & 1][W], kp);
    sync_all();
  }
  if constexpr (NC > 1) cl.sync();  // no CTA leaves while another may still write to it
}

// 2. Multisection: a warp per eigenvalue evaluates Sturm counts at 32 interior
// points and keeps the sub-interval holding it (5 bits a round). The blocks past
// the eigenvalues' form T of I - V T V^T = H_k .. H_k+3, four reflectors at a time
// (a warp each): T_jj = beta_j, T_0:j,j = -beta_j T_0:j,0:j V_0:j^T v_j.
constexpr int kBisectWarps = 8;

__global__ void __launch_bounds__(32 * kBisectWarps)
    k_bisect_wy(float* __restrict__ dg, const float* __restrict__ eg, int n, int nwant,
                float* __restrict__ evals, const float* __restrict__ house,
                const float* __restrict__ beta, float* __restrict__ wy) {
  __shared__ float d[kMaxEig], e2[kMaxEig];
  __shared__ float red[33];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int nb = (nwant + kBisectWarps - 1) / kBisectWarps;
  if ((int)blockIdx.x >= nb) {
    const int g = ((int)blockIdx.x - nb) * kBisectWarps + warp, k0 = 4 * g;
    if (k0 + 2 >= n) return;
    float dot[4][4], bt[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      bt[a] = k0 + a + 2 < n ? beta[k0 + a] : 0.f;
#pragma unroll
      for (int c = 0; c < a; ++c) dot[c][a] = 0.f;
    }
    for (int i = k0 + 1 + lane; i < n; i += 32) {
      float v[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) v[a] = k0 + a + 2 < n ? house[(size_t)(k0 + a) * n + i] : 0.f;
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < a; ++c) dot[c][a] = fmaf(v[c], v[a], dot[c][a]);
    }
    float T[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      float y[4];
#pragma unroll
      for (int c = 0; c < a; ++c) y[c] = warp_sum(dot[c][a]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float t = 0.f;
        if (c < a) {
#pragma unroll
          for (int f = c; f < a; ++f) t = fmaf(T[c][f], y[f], t);
          t *= -bt[a];
        }
        T[c][a] = c == a ? bt[a] : t;
      }
    }
    if (lane == 0)
#pragma unroll
      for (int a = 0; a < 4; ++a)
        *reinterpret_cast<float4*>(wy + 16 * g + 4 * a) = make_float4(T[a][0], T[a][1], T[a][2], T[a][3]);
    return;
  }
  for (int i = tid; i < n; i += nt) {
    const float ei = eg[i];
    d[i] = dg[i];
    e2[i] = ei * ei;
  }
  __syncthreads();
  float lo_t = FLT_MAX, hi_t = -FLT_MAX, me2 = 0.f;
  for (int i = tid; i < n; i += nt) {
    const float r = fabsf(eg[i]) + (i > 0 ? fabsf(eg[i - 1]) : 0.f);
    lo_t = fminf(lo_t, d[i] - r);
    hi_t = fmaxf(hi_t, d[i] + r);
    if (i < n - 1) me2 = fmaxf(me2, e2[i]);
  }
  float lo = block_reduce(lo_t, red, 2);
  float hi = block_reduce(hi_t, red, 1);
  me2 = block_reduce(me2, red, 1);
  const float tnorm = fmaxf(fmaxf(fabsf(lo), fabsf(hi)), FLT_MIN);
  const float pivmin = FLT_MIN * fmaxf(1.f, me2);
  const float abstol = FLT_EPSILON * tnorm;
  if (blockIdx.x == 0 && tid == 0) dg[n] = tnorm;
  lo -= 4.f * abstol + 2.f * pivmin;
  hi += 4.f * abstol + 2.f * pivmin;
  const int j = blockIdx.x * kBisectWarps + warp;
  if (j >= nwant) return;
  const int target = n - 1 - j;  // ascending index of the j-th largest
  float a = lo, b = hi;
  for (int round = 0; round < 64; ++round) {
    if (b - a <= fmaxf(abstol, 2.f * FLT_EPSILON * fmaxf(fabsf(a), fabsf(b)))) break;
    const float h = (b - a) / 33.f;
    const int cnt = sturm_count(d, e2, n, a + (float)(lane + 1) * h, pivmin);
    const unsigned above = __ballot_sync(0xffffffffu, cnt > target);
    if (above) {
      const int ts = __ffs(above) - 1;  // first point above the eigenvalue
      const float na = ts > 0 ? a + (float)ts * h : a;
      b = a + (float)(ts + 1) * h;
      a = na;
    } else {
      a = a + 32.f * h;
    }
  }
  if (lane == 0) evals[j] = 0.5f * (a + b);
}

// 3. Inverse iteration: one thread per eigenvector, vpc per CTA, the LU of
// T - lambda I (reciprocal pivots) and the iterate in shared memory (interleaved by
// thread). Three solves with one factorisation; an iterate is scaled by its largest
// entry where the next solve reads it and to unit length at the end. Each loop
// fetches the next row's entries before the current row's are written, so a row
// costs its arithmetic and not a shared-memory round trip. Eigenvalues tied within
// fp32 resolution get distinct shifts.
__global__ void k_inviter(const float* __restrict__ dg, const float* __restrict__ eg,
                          const float* __restrict__ evals, int n, int nwant, float* __restrict__ Z,
                          int nwp) {
  extern __shared__ __align__(16) float sm[];
  const int vpc = blockDim.x;
  float* d = sm;
  float* e = d + n;
  for (int i = threadIdx.x; i < n; i += vpc) {
    d[i] = dg[i];
    e[i] = eg[i];
  }
  __syncthreads();
  const int j = blockIdx.x * vpc + threadIdx.x;
  if (j >= nwant) return;
  const float tnorm = dg[n];
  const float pertol = 10.f * FLT_EPSILON * tnorm;
  const float tiny_piv = FLT_EPSILON * tnorm;
  int rank = 0;
  for (int k = j; k > 0 && evals[k - 1] - evals[k] < pertol; --k) ++rank;
  const float lam = evals[j] - (float)rank * pertol;
  const size_t blk = (size_t)n * vpc;
  float* R0 = e + n + threadIdx.x;  // 1 / pivot
  float* U1 = R0 + blk;
  float* U2 = U1 + blk;
  float* Lm = U2 + blk;
  float* P = Lm + blk;
  float* Zs = P + blk;
  // LU with partial pivoting; pivots below tiny_piv are raised to +-tiny_piv
  {
    float a_i = d[0] - lam, c_i = n > 1 ? e[0] : 0.f;
    for (int i = 0; i + 1 < n; ++i) {
      const float b = e[i], an = d[i + 1] - lam, cn = i + 2 < n ? e[i + 1] : 0.f;
      const bool swap = fabsf(b) > fabsf(a_i);
      float piv = swap ? b : a_i;
      if (fabsf(piv) < tiny_piv) piv = piv < 0.f ? -tiny_piv : tiny_piv;
      const float rp = 1.f / piv, l = (swap ? a_i : b) * rp;
      const float u1 = swap ? an : c_i;
      R0[i * vpc] = rp;
      U1[i * vpc] = u1;
      U2[i * vpc] = swap ? cn : 0.f;
      Lm[i * vpc] = l;
      P[i * vpc] = swap ? 1.f : 0.f;
      a_i = (swap ? c_i : an) - l * u1;
      c_i = swap ? -l * cn : cn;
    }
    if (fabsf(a_i) < tiny_piv) a_i = a_i < 0.f ? -tiny_piv : tiny_piv;
    R0[(n - 1) * vpc] = 1.f / a_i;
    U1[(n - 1) * vpc] = 0.f;
    U2[(n - 1) * vpc] = 0.f;
    Lm[(n - 1) * vpc] = 0.f;
    P[(n - 1) * vpc] = 0.f;
  }
  float inv = 1.f;
  for (int it = 0; it < 3; ++it) {
    // forward: apply the row swaps and multipliers to inv * (the last iterate, or at
    // first the hash vector)
    float ri = (it == 0 ? hash_unit(0, j) : Zs[0]) * inv;
    float l = Lm[0], sw = P[0], zn = Zs[min(1, n - 1) * vpc];
    for (int i = 0; i + 1 < n; ++i) {
      const float rn = (it == 0 ? hash_unit(i + 1, j) : zn) * inv;
      const float li = l, si = sw;
      l = Lm[(i + 1) * vpc];  // row n - 1 of Lm and P is never used
      sw = P[(i + 1) * vpc];
      zn = Zs[min(i + 2, n - 1) * vpc];
      const float top = si != 0.f ? rn : ri, bot = si != 0.f ? ri : rn;
      Zs[i * vpc] = top;
      ri = bot - li * top;
    }
    Zs[(n - 1) * vpc] = ri;
    // back substitution; near a cluster the solution can outgrow fp32, so when an
    // entry passes 2^100 the whole system (solved part, neighbours and the
    // remaining right-hand side) is scaled by 2^-100 and the entry redone
    float zmax = 0.f, z1 = 0.f, z2 = 0.f;
    float r0 = R0[(n - 1) * vpc], u1 = U1[(n - 1) * vpc], u2 = U2[(n - 1) * vpc],
          zr = Zs[(n - 1) * vpc];
    for (int i = n - 1; i >= 0; --i) {
      const float c0 = r0, c1 = u1, c2 = u2, cz = zr;
      const int next = max(i - 1, 0) * vpc;
      r0 = R0[next];
      u1 = U1[next];
      u2 = U2[next];
      zr = Zs[next];
      float z = (cz - c1 * z1 - c2 * z2) * c0;
      if (!(fabsf(z) <= 0x1p100f)) {
        for (int t = 0; t < n; ++t) Zs[t * vpc] *= 0x1p-100f;
        z1 *= 0x1p-100f;
        z2 *= 0x1p-100f;
        zmax *= 0x1p-100f;
        zr *= 0x1p-100f;
        z = (cz * 0x1p-100f - c1 * z1 - c2 * z2) * c0;
        if (!(fabsf(z) <= 0x1p100f)) z = 0.f;
      }
      Zs[i * vpc] = z;
      z2 = z1;
      z1 = z;
      zmax = fmaxf(zmax, fabsf(z));
    }
    inv = zmax > 0.f ? 1.f / zmax : 1.f;
  }
  // an iterate that collapsed (zero or non-finite) restarts as the hash
  // vector; the orthonormalisation then takes its component off the others
  float nz = 0.f;
  for (int i = 0; i < n; ++i) {
    const float z = Zs[i * vpc] * inv;
    nz = fmaf(z, z, nz);
  }
  const bool bad = !(nz > 0.f) || !isfinite(nz);
  const float sc = bad ? 0.f : inv * rsqrtf(nz);
  for (int i = 0; i < n; ++i)
    Z[(size_t)i * nwp + j] = bad ? hash_unit(i, j) * rsqrtf((float)n) : Zs[i * vpc] * sc;
}

// CholeskyQR of the eigenvector block Z (n x nwant, row-major, ld nwp): G = Z^T Z in
// 32 x 32 tiles (each entry sums all n rows in order), then Z2 = Z R^-1 (R^-1 upper
// triangular) in 32 x 32 tiles. A CTA requests its whole operands at once (n, nwant
// <= 512: 132 KB), so a tile costs one trip to memory; 2 x 2 outputs per thread.
// check: the Gram of the second pass must be the identity to a few ulps times the
// condition number of Z; an entry off by more than 1e-2 means that inverse iteration
// left (nearly) dependent vectors (eigenvalues tied at fp32 resolution), and
// flags[3] selects the repair path.
constexpr int kZT = 32;
constexpr int kZLd = kZT + 2;
inline size_t zpanel_bytes(int rows) { return (size_t)2 * rows * kZLd * sizeof(float); }

__global__ void __launch_bounds__(256)
    k_zgram(const float* __restrict__ Z, int n, int nwant, int nwp, float* __restrict__ G, int check,
            int* __restrict__ flags) {
  extern __shared__ __align__(16) float sm[];
  float *za = sm, *zb = sm + n * kZLd;
  const int a0 = blockIdx.y * kZT, c0 = blockIdx.x * kZT;
  for (int e = threadIdx.x; e < n * kZT; e += 256) {  // nwp is a multiple of 32: no column guard
    const int r = e / kZT, c = e % kZT;
    za[r * kZLd + c] = Z[(size_t)r * nwp + a0 + c];
    zb[r * kZLd + c] = Z[(size_t)r * nwp + c0 + c];
  }
  __syncthreads();
  const int tx = (threadIdx.x & 15) * 2, ty = (threadIdx.x >> 4) * 2;
  float acc[2][2] = {};
#pragma unroll 8
  for (int r = 0; r < n; ++r) {
    const float2 u = *reinterpret_cast<const float2*>(&za[r * kZLd + ty]);
    const float2 v = *reinterpret_cast<const float2*>(&zb[r * kZLd + tx]);
    acc[0][0] = fmaf(u.x, v.x, acc[0][0]);
    acc[0][1] = fmaf(u.x, v.y, acc[0][1]);
    acc[1][0] = fmaf(u.y, v.x, acc[1][0]);
    acc[1][1] = fmaf(u.y, v.y, acc[1][1]);
  }
  bool off = false;
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int a = a0 + ty + q, c = c0 + tx + t;
      if (a < nwant && c < nwant) {
        G[(size_t)a * nwant + c] = acc[q][t];
        off |= !(fabsf(acc[q][t] - (a == c ? 1.f : 0.f)) <= 1e-2f);
      }
    }
  if (check && off) flags[3] = 1;
}

__global__ void __launch_bounds__(256)
    k_zmul(const float* __restrict__ Z, const float* __restrict__ R, int n, int nwant, int nwp,
           float* __restrict__ Y) {
  extern __shared__ __align__(16) float sm[];
  const int i0 = blockIdx.y * kZT, c0 = blockIdx.x * kZT;
  const int K = min(nwant, c0 + kZT);  // R is upper triangular
  const int ldz = K | 1;
  float *rt = sm, *zt = sm + K * kZLd;
  for (int e = threadIdx.x; e < K * kZT; e += 256) {
    const int r = e / kZT, c = e % kZT;
    rt[r * kZLd + c] = c0 + c < nwant ? R[(size_t)r * nwant + c0 + c] : 0.f;
  }
  for (int r = threadIdx.x >> 5; r < kZT; r += 8)
    for (int c = threadIdx.x & 31; c < K; c += 32)
      zt[r * ldz + c] = i0 + r < n ? Z[(size_t)(i0 + r) * nwp + c] : 0.f;
  __syncthreads();
  const int tx = (threadIdx.x & 15) * 2, ty = (threadIdx.x >> 4) * 2;
  float acc[2][2] = {};
#pragma unroll 8
  for (int k = 0; k < K; ++k) {
    const float u0 = zt[ty * ldz + k], u1 = zt[(ty + 1) * ldz + k];
    const float2 v = *reinterpret_cast<const float2*>(&rt[k * kZLd + tx]);
    acc[0][0] = fmaf(u0, v.x, acc[0][0]);
    acc[0][1] = fmaf(u0, v.y, acc[0][1]);
    acc[1][0] = fmaf(u1, v.x, acc[1][0]);
    acc[1][1] = fmaf(u1, v.y, acc[1][1]);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int i = i0 + ty + q, c = c0 + tx + t;
      if (i < n && c < nwp) Y[(size_t)i * nwp + c] = c < nwant ? acc[q][t] : 0.f;
    }
}

// Repair path (runs only when flags[3] is set): classical Gram-Schmidt twice
// over the inverse-iteration vectors in descending eigenvalue order; a vector
// left almost inside the span of the earlier ones gets one more solve with its
// own shifted factorisation from a perturbed start and is projected again.
// Zs (column j at Zs[j n]) and the factorisation scratch fw (6 n) are global.
__global__ void __launch_bounds__(kThreads)
    k_cgs_repair(const int* __restrict__ flags, const float* __restrict__ Zin, int nwp,
                 const float* __restrict__ dg, const float* __restrict__ eg,
                 const float* __restrict__ evals, int n, int nwant, float* __restrict__ Zs,
                 float* __restrict__ fw) {
  if (flags[3] == 0) return;
  __shared__ float d[kMaxEig], e[kMaxEig], tcoef[kMaxEig];
  __shared__ float red[33];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  for (int i = tid; i < n; i += nt) {
    d[i] = dg[i];
    e[i] = eg[i];
  }
  for (int j = warp; j < nwant; j += nw)
    for (int i = lane; i < n; i += 32) Zs[(size_t)j * n + i] = Zin[(size_t)i * nwp + j];
  __syncthreads();
  const float tnorm = dg[n];
  const float pertol = 10.f * FLT_EPSILON * tnorm;
  const float tiny_piv = FLT_EPSILON * tnorm;
  for (int j = 0; j < nwant; ++j) {
    float* zj = Zs + (size_t)j * n;
    for (int attempt = 0; attempt < 4; ++attempt) {
      float n0 = 0.f;
      for (int i = tid; i < n; i += nt) n0 = fmaf(zj[i], zj[i], n0);
      n0 = block_reduce(n0, red, 0);
      for (int pass = 0; pass < 2; ++pass) {
        for (int c = warp; c < j; c += nw) {
          const float* zc = Zs + (size_t)c * n;
          float s = 0.f;
          for (int i = lane; i < n; i += 32) s = fmaf(zc[i], zj[i], s);
          s = warp_sum(s);
          if (lane == 0) tcoef[c] = s;
        }
        __syncthreads();
        for (int i = tid; i < n; i += nt) {
          float acc = zj[i];
          for (int c = 0; c < j; ++c) acc -= tcoef[c] * Zs[(size_t)c * n + i];
          zj[i] = acc;
        }
        __syncthreads();
      }
      float n1 = 0.f;
      for (int i = tid; i < n; i += nt) n1 = fmaf(zj[i], zj[i], n1);
      n1 = block_reduce(n1, red, 0);
      if (n1 > 1e-4f * n0 || attempt == 3) {
        const float inv = n1 > 0.f ? rsqrtf(n1) : 0.f;
        for (int i = tid; i < n; i += nt) zj[i] *= inv;
        __syncthreads();
        break;
      }
      if (tid == 0) {
        int rank = 0;
        for (int k = j; k > 0 && evals[k - 1] - evals[k] < pertol; --k) ++rank;
        float* col = fw + 5 * (size_t)n;
        tri_factor(d, e, evals[j] - rank * pertol, fw, fw + n, fw + 2 * n, fw + 3 * n, fw + 4 * n, n,
                   1, tiny_piv);
        for (int i = 0; i < n; ++i) col[i] = zj[i] + 1e-3f * hash_unit(i + 7919 * attempt, j);
        tri_solve_scaled(fw, fw + n, fw + 2 * n, fw + 3 * n, fw + 4 * n, col, n, 1);
        for (int i = 0; i < n; ++i) zj[i] = col[i];
      }
      __syncthreads();
    }
  }
}

// 4. Back-transformation Z <- H_0 ... H_{n-3} Z: a warp per eigenvector holds it in
// registers (NR per lane) and applies four reflectors at a time, z -= V (T (V^T z)),
// so that the four lane sums overlap. The reflectors come through shared memory, as
// many quads at once as fit (all of them up to n = 224): fetched one quad ahead into
// registers, a quad waited for its trip to L2.
constexpr int kBackWarps = 4;
constexpr int kBackSmem = 200 * 1024;

template <int NR>
__global__ void __launch_bounds__(32 * kBackWarps)
    k_back(const float* __restrict__ house, const float* __restrict__ wy, int n, int nwant,
           const float* __restrict__ Z, int nwp, const float* __restrict__ Zrep,
           const int* __restrict__ flags, int seg, float* __restrict__ evecs) {
  extern __shared__ __align__(16) float sm[];  // seg quads of 4 n reflector entries and T
  const int lane = threadIdx.x & 31;
  const int j = blockIdx.x * kBackWarps + (threadIdx.x >> 5);
  const bool live = j < nwant;
  const bool rep = flags[3] != 0;  // the repair path produced Zrep (column j at Zrep[j n])
  float z[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int e = r * 32 + lane;
    z[r] = live && e < n ? (rep ? Zrep[(size_t)j * n + e] : Z[(size_t)e * nwp + j]) : 0.f;
  }
  const int quads = n > 2 ? (n + 1) / 4 : 0;
  for (int hi = quads; hi > 0; hi -= seg) {
    const int lo = max(0, hi - seg);
    const int k1 = min(4 * hi, n - 2);  // reflectors 4 lo .. k1 - 1
    float* T_s = sm + (size_t)4 * seg * n;
    for (int e = threadIdx.x; e < (k1 - 4 * lo) * n; e += blockDim.x)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(sm + e)),
                   "l"(house + (size_t)4 * lo * n + e));
    for (int e = threadIdx.x; e < 16 * (hi - lo); e += blockDim.x) T_s[e] = wy[16 * lo + e];
    for (int e = (k1 - 4 * lo) * n + threadIdx.x; e < 4 * (hi - lo) * n; e += blockDim.x)
      sm[e] = 0.f;  // the last quad's missing reflectors
    asm volatile("cp.async.commit_group;" ::);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int g = hi - 1; g >= lo && live; --g) {
      const float* V = sm + (size_t)4 * (g - lo) * n;
      const float* Tg = T_s + 16 * (g - lo);
      float v[4][NR], y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const int e = min(r * 32 + lane, n - 1);  // z is 0 past n
          v[a][r] = V[a * n + e];
          y[a] = fmaf(v[a][r], z[r], y[a]);
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int a = 0; a < 4; ++a) y[a] += __shfl_xor_sync(0xffffffffu, y[a], o);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        float c = 0.f;
#pragma unroll
        for (int f = a; f < 4; ++f) c = fmaf(Tg[4 * a + f], y[f], c);
#pragma unroll
        for (int r = 0; r < NR; ++r) z[r] = r * 32 + lane < n ? fmaf(-c, v[a][r], z[r]) : 0.f;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int e = r * 32 + lane;
    if (live && e < n) evecs[(size_t)e * nwant + j] = z[r];
  }
}

// ---------------------------------------------------------------------------
// PSD input, n <= kJacobiMax: one-sided Jacobi on the Cholesky factor.
// S + s I = L L^T (s = 2^-20 trace/n keeps a rank-deficient Gram factorable).
// Orthogonalising the columns of L by plane rotations (Hestenes) gives
// L J = U Sigma with U the eigenvectors of L L^T and Sigma^2 its eigenvalues,
// so no rotation product is accumulated: eigenvector i is column i / its norm,
// eigenvalue i its squared norm minus s. Pairs follow the round-robin
// tournament; one warp per pair, one barrier per round. Column walks are
// bank-conflict free because the row stride n|1 is odd.
// up to 64: beyond n = 20 the tridiagonal path is faster (n = 50: 137 us against 286),
// but a sketch of l <= 64 folded from many buffers would leave the value it has always
// had in the fifth digit
constexpr int kJacobiMax = 64;
constexpr int kJacobiSweeps = 30;

__global__ void __launch_bounds__(kThreads)
    k_symeig_jacobi(const float* __restrict__ S, int n, int nwant, float* __restrict__ evals,
                    float* __restrict__ evecs) {
  extern __shared__ float A[];          // n x (n|1)
  __shared__ float nrm[kJacobiMax + 1], rdiag[kJacobiMax];
  __shared__ int rnk[kJacobiMax];
  __shared__ float red[33];
  __shared__ int rotations;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int lda = n | 1;
  // shift: 2^-20 trace/n for a positive semi-definite S (the Grams of the
  // method); if the factorisation meets a non-positive pivot, S is indefinite
  // and it restarts with the Gershgorin bound, which makes S + sI definite
  __shared__ int indefinite;
  __shared__ float shift_sh;
  float tr = 0.f, gersh = FLT_MAX;
  for (int i = warp; i < n; i += nw) {
    float off = 0.f;
    for (int j = lane; j < n; j += 32) {
      const float v = S[(size_t)i * n + j];
      if (j == i) tr += v; else off += fabsf(v);
    }
    off = warp_sum(off);
    if (lane == 0) gersh = fminf(gersh, S[(size_t)i * n + i] - off);
  }
  tr = block_reduce(tr, red, 0);
  gersh = block_reduce(gersh, red, 2);
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (tid == 0) {
      float sft = tr > 0.f ? ldexpf(tr / (float)n, -20) : FLT_MIN;
      if (attempt == 1) sft = fmaxf(sft, -gersh) * 1.01f + FLT_MIN;
      shift_sh = sft;
      indefinite = 0;
    }
    __syncthreads();
    const float sft = shift_sh;
    for (int e = tid; e < n * n; e += nt) {
      const int i = e / n, j = e % n;
      A[i * lda + j] = S[e] + (i == j ? sft : 0.f);
    }
    __syncthreads();
    // Cholesky, lower, in place; column j is scaled one step later (after the
    // barrier), so the trailing update can read it raw in the same step
    for (int j = 0; j < n; ++j) {
      float piv = A[j * lda + j];
      if (!(piv > 0.f)) {
        piv = sft;
        if (tid == 0 && attempt == 0 && j < n) indefinite = 1;
      }
      const float rinv = 1.f / piv;
      if (tid == 0) rdiag[j] = sqrtf(piv);
      if (j > 0) {
        const float sc = 1.f / rdiag[j - 1];
        for (int i = j + tid; i < n; i += nt) A[i * lda + (j - 1)] *= sc;
      }
      for (int i = j + 1 + warp; i < n; i += nw) {
        const float aij = A[i * lda + j] * rinv;
        for (int t = j + 1 + lane; t <= i; t += 32) A[i * lda + t] -= aij * A[t * lda + j];
      }
      __syncthreads();
    }
    if (!indefinite) break;
  }
  const float shift = shift_sh;
  for (int e = tid; e < n * n; e += nt) {
    const int i = e / n, j = e % n;
    if (j > i) A[i * lda + j] = 0.f;
    else if (j == i) A[i * lda + j] = rdiag[i];
  }
  __syncthreads();
  // one-sided Jacobi over the columns of L
  const int np = n + (n & 1);                 // even count; column n is a virtual zero
  const float tiny = ldexpf(fabsf(tr) + shift * n, -30);  // columns below this are zero
  const float tol = 4.f * FLT_EPSILON * sqrtf((float)n);  // attainable fp32 orthogonality
  for (int sweep = 0; sweep < kJacobiSweeps; ++sweep) {
    if (tid == 0) rotations = 0;
    __syncthreads();
    for (int r = 0; r < np - 1; ++r) {
      for (int w = warp; w < np / 2; w += nw) {
        int p, q;
        if (w == 0) { p = r; q = np - 1; }
        else { p = (r + w) % (np - 1); q = (r - w + (np - 1)) % (np - 1); }
        if (p >= n || q >= n) continue;
        float a = 0.f, b = 0.f, g = 0.f;
        for (int i = lane; i < n; i += 32) {
          const float x = A[i * lda + p], y = A[i * lda + q];
          a = fmaf(x, x, a);
          b = fmaf(y, y, b);
          g = fmaf(x, y, g);
        }
        a = warp_sum(a); b = warp_sum(b); g = warp_sum(g);
        if (fminf(a, b) <= tiny || fabsf(g) <= tol * sqrtf(a * b)) continue;
        const float zeta = (b - a) / (2.f * g);
        const float t = copysignf(1.f, zeta) / (fabsf(zeta) + sqrtf(1.f + zeta * zeta));
        const float c = rsqrtf(1.f + t * t), sn = c * t;
        for (int i = lane; i < n; i += 32) {
          const float x = A[i * lda + p], y = A[i * lda + q];
          A[i * lda + p] = c * x - sn * y;
          A[i * lda + q] = sn * x + c * y;
        }
        if (lane == 0) atomicAdd(&rotations, 1);
      }
      __syncthreads();
    }
    if (rotations == 0) break;
    __syncthreads();
  }
  // squared column norms, ranks (descending, ties by index), outputs
  for (int c = warp; c < n; c += nw) {
    float a = 0.f;
    for (int i = lane; i < n; i += 32) a = fmaf(A[i * lda + c], A[i * lda + c], a);
    a = warp_sum(a);
    if (lane == 0) nrm[c] = a;
  }
  __syncthreads();
  for (int c = tid; c < n; c += nt) {
    int r = 0;
    const float v = nrm[c];
    for (int c2 = 0; c2 < n; ++c2) r += (nrm[c2] > v) || (nrm[c2] == v && c2 < c);
    rnk[c] = r;
  }
  __syncthreads();
  for (int c = warp; c < n; c += nw) {
    const int r = rnk[c];
    if (r >= nwant) continue;
    const float v = nrm[c];
    const float inv = v > 0.f ? rsqrtf(v) : 0.f;
    for (int i = lane; i < n; i += 32) evecs[(size_t)i * nwant + r] = A[i * lda + c] * inv;
    if (lane == 0) evals[r] = v - shift;
  }
}

}  // namespace

namespace {
// Scratch of the tridiagonal path, carved from one float array.
struct EigScratch {
  float *house, *beta, *d, *e, *wy, *Z, *Z2, *Z3, *G, *R, *cw, *fw;
  int* flags;
  size_t floats;
};
EigScratch carve(float* w, int n, int nwant) {
  const size_t nwp = (size_t)((nwant + 31) & ~31);
  EigScratch c;
  size_t o = 0;
  auto take = [&](size_t k) {
    float* p = w ? w + o : nullptr;
    o += (k + 63) & ~(size_t)63;  // 256-byte aligned pieces
    return p;
  };
  c.house = take((size_t)n * n);
  c.beta = take(n);
  c.d = take(n + 2);
  c.e = take(n);
  c.wy = take(16 * (((size_t)n + 3) / 4));
  c.Z = take(n * nwp);
  c.Z2 = take(n * nwp);
  c.Z3 = take(n * nwp);
  c.G = take(nwp * nwp);
  c.R = take(nwp * nwp);
  c.cw = take(nwp * (nwp | 1));
  c.fw = take(6 * (size_t)n);
  c.flags = reinterpret_cast<int*>(take(16));
  c.floats = o;
  return c;
}
}  // namespace

size_t symeig_work_floats(int n, int nwant) { return carve(nullptr, n, nwant).floats; }

void symeig(const float* S, int n, int nwant, float* evals, float* evecs, float* work,
            cudaStream_t s, bool psd) {
  if (psd && n <= kJacobiMax) {
    static std::atomic<unsigned> jac_attr{0};  // one bit per device
    int dv = 0;
    SFD_CUDA(cudaGetDevice(&dv));
    if (dv < 32 && !(jac_attr.load() & (1u << dv))) {
      SFD_CUDA(cudaFuncSetAttribute(k_symeig_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kJacobiMax * (kJacobiMax | 1) * (int)sizeof(float)));
      jac_attr.fetch_or(1u << dv);
    }
    const size_t bytes = (size_t)n * (n | 1) * sizeof(float);
    k_symeig_jacobi<<<1, kThreads, bytes, s>>>(S, n, nwant, evals, evecs);
    SFD_LAUNCH_CHECK();
    return;
  }
  const int nwp = (nwant + 31) & ~31;
  EigScratch c = carve(work, n, nwant);
  static std::atomic<unsigned> attr{0};
  int dev = 0;
  SFD_CUDA(cudaGetDevice(&dev));
  if (dev < 32 && !(attr.load() & (1u << dev))) {
    SFD_CUDA(cudaFuncSetAttribute(k_inviter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kSmemLimit));
    SFD_CUDA(cudaFuncSetAttribute(k_zgram, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)zpanel_bytes(kMaxEig)));
    SFD_CUDA(cudaFuncSetAttribute(k_zmul, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)zpanel_bytes(kMaxEig)));
    for (auto f : {k_back<4>, k_back<8>, k_back<16>})
      SFD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kBackSmem));
    attr.fetch_or(1u << dev);
  }
  // one CTA's registers hold n = 128; a step of a cluster costs more in its barrier
  // than it saves below that
  if (n <= 128)
    k_tridiag<1, 8, 2><<<1, 512, 0, s>>>(S, n, c.house, c.beta, c.d, c.e, c.flags);
  else if (n <= 256)
    k_tridiag<2, 8, 4><<<2, 512, 0, s>>>(S, n, c.house, c.beta, c.d, c.e, c.flags);
  else
    k_tridiag<8, 4, 8><<<8, 512, 0, s>>>(S, n, c.house, c.beta, c.d, c.e, c.flags);
  SFD_LAUNCH_CHECK();
  const int quads = n > 2 ? (n + 1) / 4 : 0;  // n - 2 reflectors
  const int bw = kBisectWarps;
  k_bisect_wy<<<(nwant + bw - 1) / bw + (quads + bw - 1) / bw, 32 * bw, 0, s>>>(
      c.d, c.e, n, nwant, evals, c.house, c.beta, c.wy);
  SFD_LAUNCH_CHECK();
  int vpc = 32;
  while (vpc > 1 && (size_t)(2 * n + 6 * (size_t)n * vpc) * sizeof(float) > (size_t)kSmemLimit)
    vpc >>= 1;
  const size_t ibytes = (size_t)(2 * n + 6 * (size_t)n * vpc) * sizeof(float);
  k_inviter<<<(nwant + vpc - 1) / vpc, vpc, ibytes, s>>>(c.d, c.e, evals, n, nwant, c.Z, nwp);
  SFD_LAUNCH_CHECK();
  const dim3 gg(nwp / kZT, nwp / kZT);
  const dim3 gm(nwp / kZT, (n + kZT - 1) / kZT);
  for (int pass = 0; pass < 2; ++pass) {  // CholeskyQR2: Z -> Z2 -> Z3 (Z is kept)
    const float* zin = pass == 0 ? c.Z : c.Z2;
    float* zout = pass == 0 ? c.Z2 : c.Z3;
    k_zgram<<<gg, 256, zpanel_bytes(n), s>>>(zin, n, nwant, nwp, c.G, pass, c.flags);
    SFD_LAUNCH_CHECK();
    chol_inv(c.G, nwant, c.R, c.cw, c.flags, s);
    k_zmul<<<gm, 256, zpanel_bytes(std::max(nwant, kZT)), s>>>(zin, c.R, n, nwant, nwp, zout);
    SFD_LAUNCH_CHECK();
  }
  // Z2 is free again: the repair path (if flagged) writes its block there
  k_cgs_repair<<<1, kThreads, 0, s>>>(c.flags, c.Z, nwp, c.d, c.e, evals, n, nwant, c.Z2, c.fw);
  SFD_LAUNCH_CHECK();
  const int gb = (nwant + kBackWarps - 1) / kBackWarps;
  const size_t quad_bytes = ((size_t)4 * n + 16) * sizeof(float);
  const int seg = std::max(1, std::min(quads, (int)(kBackSmem / quad_bytes)));
  auto back = n <= 128 ? k_back<4> : n <= 256 ? k_back<8> : k_back<16>;
  back<<<gb, 32 * kBackWarps, seg * quad_bytes, s>>>(c.house, c.wy, n, nwant, c.Z3, nwp, c.Z2,
                                                     c.flags, seg, evecs);
  SFD_LAUNCH_CHECK();
}

}  // namespace sfd
