// Dense kernels of the SparseShrink / DenseShrink path:
//  - Philox4x64-10 Gaussian draws (G of Alg. 1, x of Alg. 6)
//  - Gram X^T X of tall-skinny blocks (CholeskyQR of Alg. 1's GramSchmidt,
//    P P^T of Alg. 3, [B; B'][B; B']^T of Alg. 5)
//  - tall-skinny products X * T (apply R^-1, H diag(s), U_l diag(s))
//  - Cholesky of a shifted Gram and the inverse of its factor (one CTA)
//  - shrink weights sqrt(1 - lambda_l^2 / lambda_i^2) (Alg. 3 / Alg. 5)
// All arithmetic is fp32; the small k x k factorisations live in one CTA.
#include <algorithm>
#include <atomic>

#include "sfd_internal.cuh"

namespace sfd {

namespace {

// ---------------------------------------------------------------- Philox
// Philox4x64-10 (Salmon et al., SC'11): 64x64->128 multiplies with the two
// published multipliers, key bumped by the two Weyl constants each round.
__device__ __forceinline__ void philox_round(uint64_t& x0, uint64_t& x1, uint64_t& x2, uint64_t& x3,
                                             uint64_t k0, uint64_t k1) {
  const uint64_t m0 = 0xD2E7470EE14C6C93ull, m1 = 0xCA5A826395121157ull;
  uint64_t p0_lo = m0 * x0, p0_hi = __umul64hi(m0, x0);
  uint64_t p1_lo = m1 * x2, p1_hi = __umul64hi(m1, x2);
  uint64_t n0 = p1_hi ^ x1 ^ k0;
  uint64_t n2 = p0_hi ^ x3 ^ k1;
  x0 = n0; x1 = p1_lo; x2 = n2; x3 = p0_lo;
}

__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t key0, uint64_t key1) {
  uint64_t k0 = key0, k1 = key1;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    philox_round(c[0], c[1], c[2], c[3], k0, k1);
    k0 += 0x9E3779B97F4A7C15ull;
    k1 += 0xBB67AE8584CAA73Bull;
  }
}

__device__ __forceinline__ float u24(uint64_t w) {
  return ((float)(uint32_t)(w >> 40) + 0.5f) * 5.9604644775390625e-8f;  // 2^-24
}

__global__ void k_gauss_fill(float* __restrict__ out, int64_t rows, int cols, int ld, uint64_t seed,
                             uint64_t b, uint64_t r, uint64_t tag) {
  int64_t blk = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t count = rows * (int64_t)cols;
  if (blk * 4 >= count) return;
  uint64_t c[4] = {(uint64_t)blk, b, r, tag};
  philox4x64_10(c, seed, 0ull);
  float z[4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float ua = u24(c[2 * h]), ub = u24(c[2 * h + 1]);
    float rad = sqrtf(-2.f * logf(ua));
    float sn, cs;
    sincospif(2.f * ub, &sn, &cs);
    z[2 * h] = rad * cs;
    z[2 * h + 1] = rad * sn;
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    int64_t e = blk * 4 + t;
    if (e < count) {
      int64_t row = e / cols;
      int col = (int)(e - row * cols);
      out[row * ld + col] = z[t];
    }
  }
}

// ------------------------------------------------------------------ Gram
// 8 x 8 register tiles of the upper triangle of G, one per thread: 7 (7 + 1) / 2 = 28
// of them for n = 50, 325 for n = 200, where 128 x 128 tiles computed 2.4 times as many
// products. Tile column g of ng stands for columns 4 g .. 4 g + 3 and 4 (ng + g) ..
// 4 (ng + g) + 3, so that neighbouring tiles' float4 loads use different banks with the
// rows as they lie in memory. Rows arrive 16 at a time through a ring of cp.async
// stages, as a straight copy where rows are contiguous (k_gram_tri). The multiply-adds
// are packed two columns at a time (half the issue slots; each is rounded as fmaf), 64
// per thread and row against 4 shared float4 loads. What bounds it is latency: with 64
// accumulators a thread there are two warps per scheduler, and at 200,000 x 200 the FMA
// pipe is 55 % busy, the shared-memory pipe 59 %.
// Cold, with its reduction: 100,000 x 200 128 us (31 TFLOP/s, one triangle counted; 438
// in 128 x 128 tiles, 168 with row by row copies), 20,000 x 100 23 us (49, 25), 2,000 x
// 50 11 us (15 with row by row copies). Rows of any other alignment go row by row, their
// copies spread over all threads: 200,000 x 33 at a pitch of 33 107 us (200 in 128 x 128
// tiles, 267 with a warp per row), 400,000 x 1 104 (333, 435).
constexpr int kT = 128;  // output tile of the tensor-core Grams' partials
constexpr int kG8 = 8;
constexpr int kGRows = 16;    // rows per stage
constexpr int kGStages = 3;
constexpr int kGramBlocks = 304;  // CTAs of a Gram, about 2 per SM

// acc[0..1] += a (b0, b1)
__device__ __forceinline__ void pair_fma(float2& acc, float a, float b0, float b1) {
  asm("{\n\t.reg .b64 ra, rb, rc;\n\t"
      "mov.b64 ra, {%2, %2};\n\tmov.b64 rb, {%3, %4};\n\tmov.b64 rc, {%0, %1};\n\t"
      "fma.rn.f32x2 rc, ra, rb, rc;\n\tmov.b64 {%0, %1}, rc;\n\t}"
      : "+f"(acc.x), "+f"(acc.y)
      : "f"(a), "f"(b0), "f"(b1));
}

__device__ __forceinline__ void async_copy4(float* dst, const float* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(in ? 4 : 0));
}
__device__ __forceinline__ void async_copy8(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(bytes));
}
__device__ __forceinline__ void async_copy16(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(bytes));
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::); }
template <int N>
__device__ __forceinline__ void async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Columns 4 c4 .. 4 c4 + 3 of row g of the operand (zero past n columns or when !in) to
// dst, in copies of vec columns: 4 (or 2) when rows of both blocks start on 16- (8-)
// byte boundaries and the first block's width is a multiple of that, or it is the
// only one; else 1.
__device__ __forceinline__ void async_cols(float* dst, const float* X, int ldx, const ColMap& map,
                                           int64_t g, int c4, bool in, int vec) {
  const int n = map.total(), c = 4 * c4;
  auto src_of = [&](int cc) {
    return cc < map.k0 ? X + g * ldx + cc : map.x1 + g * map.ld1 + (cc - map.k0);
  };
  auto left = [&](int cc) { return in && cc < n ? (cc < map.k0 ? map.k0 : n) - cc : 0; };
  if (vec == 4) {
    const int w = min(4, left(c));
    async_copy16(dst, w > 0 ? src_of(c) : X, 4 * w);
  } else if (vec == 2) {
#pragma unroll
    for (int t = 0; t < 4; t += 2) {
      const int w = min(2, left(c + t));
      async_copy8(dst + t, w > 0 ? src_of(c + t) : X, 4 * w);
    }
  } else {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const bool ok = left(c + t) > 0;
      async_copy4(dst + t, ok ? src_of(c + t) : X, ok);
    }
  }
}

// The indices i, i + step, .. as (row r, column c) of rows of w, without a division each.
struct Grid2 {
  int r, c, dr, dc, w;
  __device__ __forceinline__ Grid2(int i, int step, int width)
      : r(i / width), c(i % width), dr(step / width), dc(step % width), w(width) {}
  __device__ __forceinline__ void next() {
    r += dr;
    c += dc;
    if (c >= w) {
      c -= w;
      ++r;
    }
  }
};

// partial[chunk][tile][64]: tiles of the upper triangle in row-major order.
// pitch: floats between rows, of both blocks, when a stage is 16 pitch floats of each
// block as they lie (both start on 16 bytes, pitch and the first block's width are
// multiples of 4): a float4 per thread and step, 6 instructions each where the row by
// row copies of pitch = 0 need 25 and took as long as the products.
__global__ void __launch_bounds__(512)
    k_gram_tri(const float* __restrict__ X, int ldx, ColMap map, int64_t rows,
               int64_t rows_per_chunk, int ntiles, int vec, int pitch, float* __restrict__ partial) {
  extern __shared__ __align__(16) float sm[];
  const int n = map.total(), ng = (n + kG8 - 1) / kG8;
  const int rs = pitch ? pitch : ng * kG8;  // floats between rows of a stage
  const int split = pitch && map.k1 ? kGRows * rs : 0;  // where its second block begins
  const int stage = split ? 2 * split : kGRows * rs;
  const int tid = threadIdx.x;
  const int slot = (int)(blockIdx.y * blockDim.x) + tid, e = min(slot, ntiles - 1);
  int ti = 0, start = 0;
  {  // row ti of the triangle starts at ti ng - ti (ti - 1) / 2
    const float h = (float)ng + 0.5f;
    ti = max(0, (int)(h - sqrtf(fmaxf(h * h - 2.f * (float)e, 0.f))) - 1);
    start = ti * ng - ti * (ti - 1) / 2;
    while (start + (ng - ti) <= e) { start += ng - ti; ++ti; }
  }
  const int tj = ti + (e - start);
  // offset in a stage of columns 4 q .. 4 q + 3 (of the last ones when there are none:
  // those products are dropped, as those of columns past n are)
  auto quad = [&](int q) {
    const int c = 4 * min(q, (n - 1) >> 2);
    return split && c >= map.k0 ? split + c - map.k0 : c;
  };
  const int qa = quad(ti), qb = quad(ng + ti), qc = quad(tj), qd = quad(ng + tj);
  const int64_t r_beg = (int64_t)blockIdx.x * rows_per_chunk;
  const int64_t r_end = min(rows, r_beg + rows_per_chunk);
  const int nst = (int)((r_end - r_beg + kGRows - 1) / kGRows);
  auto load = [&](int st) {
    float* buf = sm + (st % kGStages) * stage;
    const int64_t r0 = r_beg + (int64_t)st * kGRows;
    if (pitch) {
      const int before = ((int)min((int64_t)kGRows, r_end - r0) - 1) * rs;  // the last row
      const float* src = X + r0 * ldx;
      const int valid = before + map.k0;
      for (int i = 4 * tid; i < kGRows * rs; i += 4 * blockDim.x) {
        const int w = max(0, min(4, valid - i));
        async_copy16(buf + i, w ? src + i : X, 4 * w);
      }
      if (split) {
        const float* src1 = map.x1 + r0 * map.ld1;
        const int valid1 = before + map.k1;
        for (int i = 4 * tid; i < kGRows * rs; i += 4 * blockDim.x) {
          const int w = max(0, min(4, valid1 - i));
          async_copy16(buf + split + i, w ? src1 + i : X, 4 * w);
        }
      }
    } else {
      Grid2 at(tid, blockDim.x, 2 * ng);  // c: group of four columns
      for (; at.r < kGRows; at.next())
        async_cols(buf + at.r * rs + 4 * at.c, X, ldx, map, r0 + at.r, at.c, r0 + at.r < r_end, vec);
    }
  };
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll
  for (int st = 0; st < kGStages - 1; ++st) {
    if (st < nst) load(st);
    async_commit();
  }
  for (int st = 0; st < nst; ++st) {
    async_wait<kGStages - 2>();
    __syncthreads();  // stage st has landed, and everyone is done with stage st - 1
    if (st + kGStages - 1 < nst) load(st + kGStages - 1);
    async_commit();
    const float* buf = sm + (st % kGStages) * stage;
    // the next row's operands are on their way while this row's products are formed
    float4 f[2][4];
    auto fetch = [&](int r, float4 (&q)[4]) {
      const float* row = buf + r * rs;
      q[0] = *reinterpret_cast<const float4*>(row + qa);
      q[1] = *reinterpret_cast<const float4*>(row + qb);
      q[2] = *reinterpret_cast<const float4*>(row + qc);
      q[3] = *reinterpret_cast<const float4*>(row + qd);
    };
    fetch(0, f[0]);
#pragma unroll 2
    for (int i = 0; i < kGRows; ++i) {
      const float4(&q)[4] = f[i & 1];
      fetch(min(i + 1, kGRows - 1), f[(i + 1) & 1]);
      const float a[8] = {q[0].x, q[0].y, q[0].z, q[0].w, q[1].x, q[1].y, q[1].z, q[1].w};
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        pair_fma(acc[c][0], a[c], q[2].x, q[2].y);
        pair_fma(acc[c][1], a[c], q[2].z, q[2].w);
        pair_fma(acc[c][2], a[c], q[3].x, q[3].y);
        pair_fma(acc[c][3], a[c], q[3].z, q[3].w);
      }
    }
  }
  async_wait<0>();
  if (slot >= ntiles) return;
  float4* out = reinterpret_cast<float4*>(partial + ((int64_t)blockIdx.x * ntiles + e) * 64);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    out[2 * i] = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
    out[2 * i + 1] = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
  }
}

// G = sum over chunks of a tile's partials, written to both triangles. A block takes
// one tile; group g of its eight groups of 64 threads adds the chunks g, g + 16, ..
// and g + 8, g + 24, .. in two sums (eight loads before their adds), and the groups
// are added in order.
__global__ void __launch_bounds__(512)
    k_gram_tri_reduce(const float* __restrict__ partial, int nchunks, int n, float* __restrict__ G) {
  __shared__ float sums[8][64];
  const int el = threadIdx.x & 63, grp = threadIdx.x >> 6, ng = (n + kG8 - 1) / kG8;
  const int64_t stride = (int64_t)gridDim.x * 64;
  const float* p = partial + (int64_t)blockIdx.x * 64 + el;
  float s0 = 0.f, s1 = 0.f;
  int ch = grp;
  for (; ch + 56 < nchunks; ch += 64) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = __ldg(p + (int64_t)(ch + 8 * u) * stride);
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      s0 += v[u];
      s1 += v[u + 1];
    }
  }
  for (; ch + 8 < nchunks; ch += 16) {
    s0 += p[(int64_t)ch * stride];
    s1 += p[(int64_t)(ch + 8) * stride];
  }
  if (ch < nchunks) s0 += p[(int64_t)ch * stride];
  sums[grp][el] = s0 + s1;
  __syncthreads();
  if (grp) return;
  int ti = 0, start = 0;
  while (start + (ng - ti) <= (int)blockIdx.x) { start += ng - ti; ++ti; }
  const int tj = ti + ((int)blockIdx.x - start);
  auto col = [&](int g, int i) { return i < 4 ? 4 * g + i : 4 * (ng + g) + i - 4; };
  const int a = col(ti, el >> 3), c = col(tj, el & 7);
  if (a >= n || c >= n || (ti == tj && a > c)) return;
  float t = 0.f;
#pragma unroll
  for (int g = 0; g < 8; ++g) t += sums[g][el];
  G[(int64_t)a * n + c] = t;
  G[(int64_t)c * n + a] = t;
}

// G[e] = sum over chunks of the tensor-core Grams' partial tiles (one 128 x 128 tile
// each). A block takes 32 consecutive output elements; its 8 warps each sum every 8th
// chunk (coalesced 128-byte reads per chunk), and the 8 warp sums are added in a fixed
// order, so the result does not depend on scheduling.
constexpr int kRedGroups = 8;

__global__ void __launch_bounds__(32 * kRedGroups)
    k_gram_reduce(const float* __restrict__ partial, int nchunks, int n, float* __restrict__ G) {
  __shared__ float sums[kRedGroups][33];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int64_t e = (int64_t)blockIdx.x * 32 + lane;
  const bool live = e < (int64_t)n * n;
  float acc = 0.f;
  if (live) {
    const int a = (int)(e / n), c = (int)(e % n);
    const float* p = partial + a * kT + c;
    constexpr int64_t stride = kT * kT;
    // chunks grp, grp + 16, ... into s0 and grp + 8, grp + 24, ... into s1,
    // in that order; eight loads are issued before their adds
    float s0 = 0.f, s1 = 0.f;
    int ch = grp;
    for (; ch + 7 * kRedGroups < nchunks; ch += 8 * kRedGroups) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldg(p + (int64_t)(ch + u * kRedGroups) * stride);
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        s0 += v[u];
        s1 += v[u + 1];
      }
    }
    for (; ch + kRedGroups < nchunks; ch += 2 * kRedGroups) {
      s0 += p[ch * stride];
      s1 += p[(ch + kRedGroups) * stride];
    }
    if (ch < nchunks) s0 += p[ch * stride];
    acc = s0 + s1;
  }
  sums[grp][lane] = acc;
  __syncthreads();
  if (grp == 0 && live) {
    float t = 0.f;
#pragma unroll
    for (int g = 0; g < kRedGroups; ++g) t += sums[g][lane];
    G[e] = t;
  }
}

// ---------------------------------------------------------------- X * T
// Y[rows, 0:kout] = X[rows, map] T, RT x 8 outputs per thread. A warp's lanes are 8 row
// groups by 4 column groups (lane row lr of warp row wr has rows wr 8 RT + lr + 8 i),
// so its loads of X and T from shared memory are one wavefront each, 16 per 4 inner
// columns against 256 multiply-adds per lane at RT = 8. X and T arrive 16 inner
// columns at a time through a ring of cp.async stages (T from L2), T's rows split in
// halves as the Gram's. Each output adds its products in column order. Where
// there are rows enough 50,000 x 200 x 200 takes 131 us (31 TFLOP/s; 205 in 128 x 128
// tiles, a fifth of their products padding), 20,000 x 100 x 100 27 us (46): the FMA pipe
// is 58 % busy (200,000 x 200 x 200), because the warps come to it together after each
// barrier and each step of four columns' loads.
constexpr int kMK = 16;        // inner columns per stage
constexpr int kMLd = kMK + 4;  // X stage leading dimension: 8 rows start in 8 bank quads
constexpr int kMStages = 3;
constexpr int kMWideSmem = 226 * 1024;

// acc += the stage's 16 inner columns: xs this lane's first row, tb its columns of T
template <int RT>
__device__ __forceinline__ void gemm_stage(float2 (&acc)[RT][4], const float* xs, const float* tb,
                                           int ts, int ps) {
#pragma unroll 1
  for (int k = 0; k < kMK; k += 4) {
    float4 a[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) a[i] = *reinterpret_cast<const float4*>(xs + i * 8 * kMLd + k);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 b0 = *reinterpret_cast<const float4*>(tb + (k + u) * ts);
      const float4 b1 = *reinterpret_cast<const float4*>(tb + (k + u) * ts + ps);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const float x = u == 0 ? a[i].x : u == 1 ? a[i].y : u == 2 ? a[i].z : a[i].w;
        pair_fma(acc[i][0], x, b0.x, b0.y);
        pair_fma(acc[i][1], x, b0.z, b0.w);
        pair_fma(acc[i][2], x, b1.x, b1.y);
        pair_fma(acc[i][3], x, b1.z, b1.w);
      }
    }
  }
}

// rows r0 + 8 i (< r_end) of this lane's column group tc
template <int RT>
__device__ __forceinline__ void gemm_store(const float2 (&acc)[RT][4], float* Y, int ldy, int64_t r0,
                                           int64_t r_end, int tc, int kout, bool vec_y) {
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int64_t g = r0 + 8 * i;
    if (g >= r_end) break;
    float* y = Y + g * ldy + tc * 8;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 p = acc[i][2 * h], q = acc[i][2 * h + 1];
      const int c = tc * 8 + 4 * h;
      if (vec_y && c + 4 <= kout) {
        *reinterpret_cast<float4*>(y + 4 * h) = make_float4(p.x, p.y, q.x, q.y);
      } else {
        if (c < kout) y[4 * h] = p.x;
        if (c + 1 < kout) y[4 * h + 1] = p.y;
        if (c + 2 < kout) y[4 * h + 2] = q.x;
        if (c + 3 < kout) y[4 * h + 3] = q.y;
      }
    }
  }
}

// rows k0 .. k0 + count - 1 of T (zero past n rows and kout columns), ts floats apart at
// dst, by all threads in copies of vec_t columns
__device__ __forceinline__ void async_t_rows(float* dst, const float* T, int k0, int count, int n,
                                             int kout, int wcols, int vec_t) {
  const int ps = wcols * 16, ts = 2 * ps;
  if (vec_t == 1) {  // neighbouring threads take neighbouring columns
    for (Grid2 at(threadIdx.x, blockDim.x, wcols * 32); at.r < count; at.next()) {
      const int kk = k0 + at.r, c = at.c;
      const bool ok = kk < n && c < kout;
      async_copy4(dst + at.r * ts + ((c >> 2) & 1) * ps + (c >> 3) * 4 + (c & 3),
                  ok ? T + (int64_t)kk * kout + c : T, ok);
    }
    return;
  }
  for (Grid2 at(threadIdx.x, blockDim.x, wcols * 8); at.r < count; at.next()) {
    const int kk = k0 + at.r, c4 = at.c;
    float* d = dst + at.r * ts + (c4 & 1) * ps + (c4 >> 1) * 4;
    const float* src = T + (int64_t)kk * kout + 4 * c4;
#pragma unroll
    for (int t = 0; t < 4; t += 2) {
      if (t % vec_t) continue;
      const bool ok = kk < n && 4 * c4 + t < kout;
      if (vec_t == 4) async_copy16(d, ok ? src : T, ok ? 16 : 0);
      else async_copy8(d + t, ok ? src + t : T, ok ? 8 : 0);
    }
  }
}

template <int RT>
__global__ void __launch_bounds__(256)
    k_gemm_rows(const float* __restrict__ X, int ldx, ColMap map, int64_t rows,
                const float* __restrict__ T, int kout, int wcols, int vec_x, int vec_t,
                bool vec_y, float* __restrict__ Y, int ldy) {
  extern __shared__ __align__(16) float sm[];
  const int n = map.total();
  const int ps = wcols * 16, ts = 2 * ps;  // T stage: half and whole row, in floats
  constexpr int xfl = 8 * RT * kMLd;
  const int stage = xfl + kMK * ts;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r_lane = lane >> 2, tc = warp * 4 + (lane & 3);  // a warp per 32 columns
  const int64_t row0 = (int64_t)blockIdx.x * 8 * RT;
  const int nst = (n + kMK - 1) / kMK;
  auto load = [&](int st) {
    float* xs = sm + (st % kMStages) * stage;
    float* tb = xs + xfl;
    for (int i = tid; i < 8 * RT * (kMK / 4); i += blockDim.x) {
      const int r = i >> 2, q = i & 3;
      const int64_t g = row0 + r;
      async_cols(xs + r * kMLd + 4 * q, X, ldx, map, g, st * (kMK / 4) + q, g < rows, vec_x);
    }
    async_t_rows(tb, T, st * kMK, kMK, n, kout, wcols, vec_t);
  };
  float2 acc[RT][4];
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll
  for (int st = 0; st < kMStages - 1; ++st) {
    if (st < nst) load(st);
    async_commit();
  }
  for (int st = 0; st < nst; ++st) {
    async_wait<kMStages - 2>();
    __syncthreads();
    if (st + kMStages - 1 < nst) load(st + kMStages - 1);
    async_commit();
    const float* xs = sm + (st % kMStages) * stage + r_lane * kMLd;
    const float* tb = sm + (st % kMStages) * stage + xfl + tc * 4;
    gemm_stage<RT>(acc, xs, tb, ts, ps);
  }
  async_wait<0>();
  gemm_store<RT>(acc, Y, ldy, row0 + r_lane, rows, tc, kout, vec_y);
}

// The same product for few rows, where a call is one chain of latencies: T and 16 rows
// of X arrive as they lie in memory, in one round of straight copies (no stages, no
// arithmetic per element), then each thread forms 2 x 4 outputs. X as k_gram_tri's
// straight copies want it, T on 16 bytes; VT is the width of T's shared loads (4, 2
// or 1, a divisor of kout).
// Cold: 2,000 x 50 x 50 7.7 us (18 through the stages), 4,800 x 100 x 100 10 (22),
// 4,000 x 200 x 200 24 (43).
constexpr int kSRows = 16;

template <int VT>
__global__ void __launch_bounds__(512)
    k_gemm_small(const float* __restrict__ X, int ldx, ColMap map, int64_t rows,
                 const float* __restrict__ T, int kout, bool vec_y, float* __restrict__ Y, int ldy) {
  extern __shared__ __align__(16) float sm[];
  const int n = map.total(), tid = threadIdx.x;
  const int t_floats = (n * kout + 7) & ~3;  // the last row's unused columns included
  float* xs = sm + t_floats;
  const int split = map.k1 ? kSRows * ldx : 0;
  const int64_t row0 = (int64_t)blockIdx.x * kSRows;
  const int before = ((int)min((int64_t)kSRows, rows - row0) - 1) * ldx;
  const int valid = before + map.k0, valid1 = before + map.k1, t_valid = n * kout;
  const float* src = X + row0 * ldx;
  for (int i = 4 * tid; i < kSRows * ldx; i += 4 * blockDim.x) {
    const int w = max(0, min(4, valid - i));
    async_copy16(xs + i, w ? src + i : X, 4 * w);
    if (split) {
      const int w1 = max(0, min(4, valid1 - i));
      async_copy16(xs + split + i, w1 ? map.x1 + row0 * ldx + i : X, 4 * w1);
    }
  }
  for (int i = 4 * tid; i < t_floats; i += 4 * blockDim.x) {
    const int w = max(0, min(4, t_valid - i));
    async_copy16(sm + i, w ? T + i : T, 4 * w);
  }
  async_commit();
  async_wait<0>();
  __syncthreads();
  const int groups = (kout + 3) >> 2;
  if (tid >= groups * (kSRows / 2)) return;
  const int c = 4 * (tid % groups), r = 2 * (tid / groups);
  float2 acc[2][2] = {};
  const float* x0 = xs + r * ldx;
  const float* tc = sm + c;
  auto step = [&](float a0, float a1, int k) {
    const float* t = tc + k * kout;
    float b[4];
    if (VT == 4) {
      const float4 q = *reinterpret_cast<const float4*>(t);
      b[0] = q.x; b[1] = q.y; b[2] = q.z; b[3] = q.w;
    } else if (VT == 2) {
      const float2 q = *reinterpret_cast<const float2*>(t), p = *reinterpret_cast<const float2*>(t + 2);
      b[0] = q.x; b[1] = q.y; b[2] = p.x; b[3] = p.y;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = t[j];
    }
    pair_fma(acc[0][0], a0, b[0], b[1]);
    pair_fma(acc[0][1], a0, b[2], b[3]);
    pair_fma(acc[1][0], a1, b[0], b[1]);
    pair_fma(acc[1][1], a1, b[2], b[3]);
  };
  for (int k = 0; k < n; k += 4) {
    const float* x = x0 + (split && k >= map.k0 ? split + k - map.k0 : k);
    const float4 a0 = *reinterpret_cast<const float4*>(x);
    const float4 a1 = *reinterpret_cast<const float4*>(x + ldx);
    step(a0.x, a1.x, k);
    if (k + 1 < n) step(a0.y, a1.y, k + 1);
    if (k + 2 < n) step(a0.z, a1.z, k + 2);
    if (k + 3 < n) step(a0.w, a1.w, k + 3);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int64_t g = row0 + r + i;
    if (g >= rows) break;
    float* y = Y + g * ldy + c;
    const float2 p = acc[i][0], q = acc[i][1];
    if (vec_y && c + 4 <= kout) {
      *reinterpret_cast<float4*>(y) = make_float4(p.x, p.y, q.x, q.y);
    } else {
      y[0] = p.x;
      if (c + 1 < kout) y[1] = p.y;
      if (c + 2 < kout) y[2] = q.x;
      if (c + 3 < kout) y[3] = q.y;
    }
  }
}

// The same product with T kept in shared memory (n kout up to about 46,000, 200 x 200
// included): one CTA per SM, each with its own contiguous rows in tiles of wrows 8 RT,
// so that only X moves during the products and the tiles of a CTA follow each other
// through one ring of stages.
template <int RT>
__global__ void __launch_bounds__(512)
    k_gemm_wide(const float* __restrict__ X, int ldx, ColMap map, int64_t rows,
                int64_t rows_per_cta, const float* __restrict__ T, int kout, int wrows, int wcols,
                int vec_x, int vec_t, bool vec_y, float* __restrict__ Y, int ldy) {
  extern __shared__ __align__(16) float sm[];
  const int n = map.total();
  const int ps = wcols * 16, ts = 2 * ps;
  const int nst = (n + kMK - 1) / kMK, tile = wrows * 8 * RT, xfl = tile * kMLd;
  float* xbuf = sm + nst * kMK * ts;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r_lane = (warp / wcols) * 8 * RT + (lane >> 2), tc = (warp % wcols) * 4 + (lane & 3);
  const int64_t r_beg = (int64_t)blockIdx.x * rows_per_cta;
  const int64_t r_end = min(rows, r_beg + rows_per_cta);
  const int ntile = (int)((r_end - r_beg + tile - 1) / tile), total = ntile * nst;
  auto load = [&](int s) {  // stage s % nst of tile s / nst
    const int64_t row0 = r_beg + (int64_t)(s / nst) * tile;
    float* xs = xbuf + (s % kMStages) * xfl;
    for (int i = tid; i < tile * (kMK / 4); i += blockDim.x) {
      const int r = i >> 2, q = i & 3;
      async_cols(xs + r * kMLd + 4 * q, X, ldx, map, row0 + r, (s % nst) * (kMK / 4) + q,
                 row0 + r < r_end, vec_x);
    }
  };
  async_t_rows(sm, T, 0, nst * kMK, n, kout, wcols, vec_t);
  float2 acc[RT][4];
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll
  for (int s = 0; s < kMStages - 1; ++s) {  // T lands with the first stage
    if (s < total) load(s);
    async_commit();
  }
  int st = 0;  // stage within the tile
  int64_t row0 = r_beg;
  for (int s = 0; s < total; ++s) {
    async_wait<kMStages - 2>();
    __syncthreads();
    if (s + kMStages - 1 < total) load(s + kMStages - 1);
    async_commit();
    gemm_stage<RT>(acc, xbuf + (s % kMStages) * xfl + r_lane * kMLd, sm + st * kMK * ts + tc * 4, ts,
                   ps);
    if (++st == nst) {
      gemm_store<RT>(acc, Y, ldy, row0 + r_lane, r_end, tc, kout, vec_y);
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
      st = 0;
      row0 += tile;
    }
  }
  async_wait<0>();
}

// --------------------------------------------------- Cholesky + inverse
__device__ float block_sum_f(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  float t = 0.f;
  if (threadIdx.x < 32) {
    t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) red[32] = t;
  }
  __syncthreads();
  return red[32];
}

// The wide form (k > kMaxEll: eigenvector blocks): one CTA of kCholThreads
// threads, one column at a time. G + s I = R^T R with s = 2^-20 trace(G)/k
// (shifted CholeskyQR: keeps the factorisation defined for a rank-deficient
// block; X R^-1 then spans the same columns), then Rinv = R^-1.
// A is k x lda (lda odd, so column walks hit distinct banks).
//  - Cholesky, right-looking, one barrier per column: step j writes
//    R[j][t] = L[t][j] into the upper triangle (never read by the update),
//    R[j][j] into rdiag, and updates the trailing lower triangle with the
//    scaled column computed on the fly.
//  - Inverse, one barrier per row: R X = I is solved for all columns at once
//    by back-substitution from the last row; the running right-hand sides B
//    (upper triangular, B[i][c] stored at A[c][i]) take the freed lower
//    triangle. Rinv[r][c] = B[r][c] / R[r][r].
constexpr int kCholThreads = 256;

__global__ void __launch_bounds__(kCholThreads)
    k_chol_inv(const float* __restrict__ G, int k, float* __restrict__ Rinv, float* __restrict__ A,
               int* __restrict__ flags) {
  __shared__ float red[33];
  __shared__ float rdiag[kMaxEig];
  const int lda = k | 1;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  float tr = 0.f;
  for (int e = tid; e < k * k; e += nt) {
    int i = e / k, j = e % k;
    float v = G[e];
    A[i * lda + j] = v;
    if (i == j) tr += v;
  }
  tr = block_sum_f(tr, red);
  const float shift = tr > 0.f ? ldexpf(tr / (float)k, -20) : 1e-30f;
  for (int i = tid; i < k; i += nt) A[i * lda + i] += shift;
  __syncthreads();
  for (int j = 0; j < k; ++j) {
    float p = A[j * lda + j];
    if (!(p > 0.f)) p = shift;
    const float ljj = sqrtf(p);
    const float inv = 1.f / ljj;
    if (tid == 0) {
      rdiag[j] = ljj;
      if (!(A[j * lda + j] > 0.f)) atomicAdd(&flags[1], 1);
    }
    for (int t = j + 1 + tid; t < k; t += nt) A[j * lda + t] = A[t * lda + j] * inv;
    for (int i = j + 1 + warp; i < k; i += nw) {
      const float lij = A[i * lda + j] * inv;
      for (int t = j + 1 + lane; t <= i; t += 32) A[i * lda + t] -= lij * (A[t * lda + j] * inv);
    }
    __syncthreads();
  }
  // B = I in the lower triangle (B[i][c] at A[c][i], i <= c)
  for (int e = tid; e < k * k; e += nt) {
    int c = e / k, i = e % k;
    if (i <= c) A[c * lda + i] = i == c ? 1.f : 0.f;
  }
  __syncthreads();
  for (int j = k - 1; j > 0; --j) {
    const float rj = 1.f / rdiag[j];
    // B[i][c] -= R[i][j] * B[j][c] / R[j][j]   for i < j <= c
    for (int c = j + warp; c < k; c += nw) {
      const float xjc = A[c * lda + j] * rj;
      for (int i = lane; i < j; i += 32) A[c * lda + i] -= A[i * lda + j] * xjc;
    }
    __syncthreads();
  }
  for (int e = tid; e < k * k; e += nt) {
    int r = e / k, c = e % k;
    Rinv[e] = c >= r ? A[c * lda + r] / rdiag[r] : 0.f;
  }
}

// ------------------------------------------------------- shrink weights
__global__ void k_shrink_weights(const float* __restrict__ evals, const float* __restrict__ evecs,
                                 int n, int nwant, int nkeep, int thr_zero,
                                 float* __restrict__ T, double* __restrict__ scal) {
  __shared__ float s[kMaxEig];
  const float thr = thr_zero ? 0.f : fmaxf(evals[nkeep - 1], 0.f);
  for (int j = threadIdx.x; j < nkeep; j += blockDim.x) {
    float ev = evals[j];
    s[j] = (ev > thr && ev > 0.f) ? sqrtf(1.f - thr / ev) : 0.f;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n * nkeep; e += blockDim.x) {
    int i = e / nkeep, j = e % nkeep;
    T[e] = evecs[i * nwant + j] * s[j];
  }
  if (threadIdx.x == 0) {
    double acc = 0.0;
    for (int j = 0; j < nkeep; ++j) acc += fmax((double)evals[j] - (double)thr, 0.0);
    scal[0] = acc;
    scal[1] = thr;
  }
}

// --------------------------------------------------------------- transpose
__global__ void k_transpose(const float* __restrict__ in, int64_t rows, int cols, int ld_in,
                            float* __restrict__ out, int64_t ld_out) {
  __shared__ float t[32][33];
  int64_t r0 = (int64_t)blockIdx.x * 32;
  int c0 = blockIdx.y * 32;
  int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  for (int k = ty; k < 32; k += 8) {
    int64_t r = r0 + k;
    int c = c0 + tx;
    t[k][tx] = (r < rows && c < cols) ? in[r * ld_in + c] : 0.f;
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    int c = c0 + k;
    int64_t r = r0 + tx;
    if (c < cols && r < rows) out[(int64_t)c * ld_out + r] = t[tx][k];
  }
}

__global__ void k_csr_to_dense_t(const int* __restrict__ ptr, const int* __restrict__ idx,
                                 const float* __restrict__ val, int rows, float* __restrict__ out,
                                 int ld) {
  int r = blockIdx.x;
  if (r >= rows) return;
  for (int p = ptr[r] + threadIdx.x; p < ptr[r + 1]; p += blockDim.x)
    atomicAdd(&out[(int64_t)idx[p] * ld + r], val[p]);
}

}  // namespace

// ======================================================================= API
void launch_gauss_fill(float* out, int64_t rows, int cols, int ld, uint64_t seed, uint64_t b,
                       uint64_t r, uint64_t tag, cudaStream_t s) {
  int64_t nblk = (rows * cols + 3) / 4;
  if (nblk == 0) return;
  k_gauss_fill<<<(unsigned)((nblk + 255) / 256), 256, 0, s>>>(out, rows, cols, ld, seed, b, r, tag);
  SFD_LAUNCH_CHECK();
}

// columns per asynchronous copy: see async_cols
static int vec_cols(const float* X, int ldx, const ColMap& map) {
  for (int v = 4; v > 1; v >>= 1) {
    const bool first = ldx % v == 0 && (uintptr_t)X % (4 * v) == 0;
    if (first && (map.k1 == 0 || (map.k0 % v == 0 && map.ld1 % v == 0 &&
                                  (uintptr_t)map.x1 % (4 * v) == 0)))
      return v;
  }
  return 1;
}

// whether rows can be copied as they lie (vec: vec_cols), little of them being padding
static bool straight_rows(int ldx, const ColMap& map, int vec) {
  return vec == 4 && ldx <= ((map.total() + 7) & ~7) && (map.k1 == 0 || map.ld1 == ldx);
}

void gram(const float* X, int ldx, ColMap map, int64_t rows, float* G, Workspace& ws,
          cudaStream_t s) {
  const int n = map.total(), ng = (n + kG8 - 1) / kG8;
  const int ntiles = ng * (ng + 1) / 2;
  // chunks of rows and parts of the triangle: about two CTAs per SM. Rows are cut
  // into the same chunks, and chunks added in the same order, as with 128 x 128 tiles,
  // so a Gram keeps its bits; a chunk's tiles go to as many CTAs as it then had tiles.
  const int n128 = (n + kT - 1) / kT, parts = n128 * (n128 + 1) / 2;
  const int threads = ((ntiles + parts - 1) / parts + 31) & ~31;
  int nchunks = (int)std::max<int64_t>(
      1, std::min<int64_t>((rows + kGRows - 1) / kGRows, kGramBlocks / parts));
  int64_t rpc = (rows + nchunks - 1) / nchunks;
  rpc = ((rpc + kGRows - 1) / kGRows) * kGRows;
  nchunks = (int)std::max<int64_t>(1, (rows + rpc - 1) / rpc);
  float* partial = ws.gram_partial;
  if (rows > 0) {
    const int vec = vec_cols(X, ldx, map);
    const bool straight = straight_rows(ldx, map, vec);
    const int pitch = straight ? ldx : 0;
    const int row = straight ? (map.k1 ? 2 : 1) * ldx : ng * kG8;
    const size_t bytes = (size_t)kGStages * kGRows * row * sizeof(float);
    static std::atomic<unsigned> attr{0};
    int dev = 0;
    SFD_CUDA(cudaGetDevice(&dev));
    if (dev < 32 && !(attr.load() & (1u << dev))) {
      SFD_CUDA(cudaFuncSetAttribute(k_gram_tri, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    2 * kGStages * kGRows * kMaxEig * (int)sizeof(float)));
      attr.fetch_or(1u << dev);
    }
    k_gram_tri<<<dim3(nchunks, parts), threads, bytes, s>>>(X, ldx, map, rows, rpc, ntiles, vec,
                                                            pitch, partial);
    SFD_LAUNCH_CHECK();
  } else {
    nchunks = 0;
  }
  k_gram_tri_reduce<<<ntiles, 512, 0, s>>>(partial, nchunks, n, G);
  SFD_LAUNCH_CHECK();
}

void gram_reduce_tiles(const float* partial, int nchunks, int n, float* G, cudaStream_t s) {
  int64_t ne = (int64_t)n * n;
  k_gram_reduce<<<(unsigned)((ne + 31) / 32), 32 * kRedGroups, 0, s>>>(partial, nchunks, n, G);
  SFD_LAUNCH_CHECK();
}

void gemm_ts(const float* X, int ldx, ColMap map, int64_t rows, const float* T, int kout, float* Y,
             int ldy, cudaStream_t s) {
  if (rows <= 0 || kout <= 0) return;
  const int wcols = (kout + 31) / 32;  // <= 8 (kout <= 256)
  const int n = map.total();
  const int vec_x = vec_cols(X, ldx, map);
  int vec_t = 4;
  while (vec_t > 1 && (kout % vec_t || (uintptr_t)T % (4 * vec_t))) vec_t >>= 1;
  const bool vec_y = (ldy & 3) == 0 && ((uintptr_t)Y & 15) == 0;
  static std::atomic<unsigned> attr{0};
  int dev = 0;
  SFD_CUDA(cudaGetDevice(&dev));
  if (dev < 32 && !(attr.load() & (1u << dev))) {
    for (auto f : {k_gemm_wide<4>, k_gemm_wide<5>, k_gemm_wide<6>, k_gemm_wide<7>, k_gemm_wide<8>})
      SFD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMWideSmem));
    for (auto f : {k_gemm_small<1>, k_gemm_small<2>, k_gemm_small<4>})
      SFD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMWideSmem));
    const int most = kMStages * (128 * kMLd + kMK * kMaxEll) * (int)sizeof(float);
    for (auto f : {k_gemm_rows<2>, k_gemm_rows<8>})
      SFD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    attr.fetch_or(1u << dev);
  }
  // few rows: while their CTAs (up to four an SM, as shared memory allows) take at most
  // two turns; then T, loaded again for every 16 rows, costs more than the latencies.
  // us against the other forms, cold: 10,000 x 100 x 100 18 to 24 (two turns), 20,000 x
  // 100 x 100 26 to 27 (three), 20,000 x 200 x 100 53 to 43 (five).
  const size_t small_bytes =
      ((size_t)((n * kout + 7) & ~3) + (size_t)(map.k1 ? 2 : 1) * kSRows * ldx) * sizeof(float);
  const int64_t small_ctas = (rows + kSRows - 1) / kSRows;
  if (straight_rows(ldx, map, vec_x) && (uintptr_t)T % 16 == 0 &&
      small_ctas <= 2 * 152 * (int64_t)std::min<size_t>(4, kMWideSmem / small_bytes)) {
    const int threads = ((kout + 3) / 4 * (kSRows / 2) + 31) & ~31;
    auto k = kout % 4 == 0 ? k_gemm_small<4> : kout % 2 == 0 ? k_gemm_small<2> : k_gemm_small<1>;
    k<<<(unsigned)small_ctas, threads, small_bytes, s>>>(X, ldx, map, rows, T, kout, vec_y, Y, ldy);
    SFD_LAUNCH_CHECK();
    return;
  }
  // T in shared memory, one CTA per SM, where the rows fill the SMs (32 or more each; 130
  // against 180 us through the stages at 50,000 x 200 x 200, 24 against 36 at 10,000 x
  // 100 x 100), with the rows of warps and the rows per thread that waste least of the
  // last tile: narrow outputs, whose 16 warps would cover 512 rows and more, take fewer
  // (20,011 x 200 x 20: 30 us, 79 with 16; 10,000 x 50 x 3: 9 and 26)
  const size_t t_bytes = (size_t)((n + kMK - 1) / kMK) * kMK * wcols * 32 * sizeof(float);
  const int most_rows = std::max(1, 16 / wcols);
  const size_t x_row = (size_t)kMStages * kMLd * sizeof(float);
  if (rows >= 152 * 32 && t_bytes + most_rows * 64 * x_row <= (size_t)kMWideSmem) {
    const int64_t rpc = (rows + 151) / 152;
    int rt = 8, wr = most_rows;
    int64_t best = INT64_MAX;
    for (int w = most_rows; w >= 1; --w)
      for (int r = 8; r >= 4; --r) {
        // a tile's time goes with the rows of a thread, whatever the warps; of equal
        // ones that with the fewest rows (its padding is copied too)
        const int64_t cost = (rpc + w * 8 * r - 1) / (w * 8 * r) * r * 16 + w;
        if (cost < best) {
          best = cost;
          rt = r;
          wr = w;
        }
      }
    auto k = rt == 8 ? k_gemm_wide<8> : rt == 7 ? k_gemm_wide<7> : rt == 6 ? k_gemm_wide<6>
             : rt == 5 ? k_gemm_wide<5> : k_gemm_wide<4>;
    k<<<(unsigned)((rows + rpc - 1) / rpc), wr * wcols * 32, t_bytes + wr * 8 * rt * x_row, s>>>(
        X, ldx, map, rows, rpc, T, kout, wr, wcols, vec_x, vec_t, vec_y, Y, ldy);
    SFD_LAUNCH_CHECK();
    return;
  }
  // else T through the stages: 64 rows per CTA (8 x 8 outputs per thread), or 16 (2 x 8)
  // below two CTAs an SM of 64. T, which every CTA loads, outweighs empty SMs from 193
  // outputs on: 16 rows there only where 64 leave half of the SMs empty (256 x 256:
  // 10,000 rows 67 us, 100 with 16 rows; 4,900 rows 39 and 53; 4,801 x 150 x 150 32 and 23)
  const int64_t ctas64 = (rows + 63) / 64;
  const int rt = ctas64 < (wcols >= 7 ? 76 : 2 * 152) ? 2 : 8, tile = 8 * rt;
  const size_t bytes = (size_t)kMStages * (tile * kMLd + kMK * wcols * 32) * sizeof(float);
  auto k = rt == 2 ? k_gemm_rows<2> : k_gemm_rows<8>;
  k<<<(unsigned)((rows + tile - 1) / tile), wcols * 32, bytes, s>>>(
      X, ldx, map, rows, T, kout, wcols, vec_x, vec_t, vec_y, Y, ldy);
  SFD_LAUNCH_CHECK();
}

void chol_inv(const float* G, int k, float* Rinv, float* work, int* flags, cudaStream_t s,
              bool accurate) {
  // the in-place forms serve k <= 256 (every block the method orthonormalises): the
  // triangle in registers, above that in shared memory, its low parts in global memory
  // where both do not fit (two-float, k > 208); only eigenvector blocks (fp32) are
  // wider, and go a column at a time through global memory
  if (k <= kMaxEll) {
    chol_inv_blk(G, k, Rinv, work, flags, s, accurate);
    return;
  }
  if (accurate) throw CudaError{cudaErrorInvalidValue, "chol_inv: accurate form for k <= 256"};
  k_chol_inv<<<1, kCholThreads, 0, s>>>(G, k, Rinv, work, flags);
  SFD_LAUNCH_CHECK();
}

void shrink_weights(const float* evals, const float* evecs, int n, int nwant, int nkeep,
                    int thr_zero, float* T, double* scal, cudaStream_t s) {
  k_shrink_weights<<<1, 1024, 0, s>>>(evals, evecs, n, nwant, nkeep, thr_zero, T, scal);
  SFD_LAUNCH_CHECK();
}

void transpose(const float* in, int64_t rows, int cols, int ld_in, float* out, int64_t ld_out,
               cudaStream_t s) {
  if (rows <= 0 || cols <= 0) return;
  dim3 grid((unsigned)((rows + 31) / 32), (cols + 31) / 32);
  k_transpose<<<grid, dim3(32, 8), 0, s>>>(in, rows, cols, ld_in, out, ld_out);
  SFD_LAUNCH_CHECK();
}

void csr_to_dense_t(const int* ptr, const int* idx, const float* val, int rows, int64_t d,
                    float* out, int ld, cudaStream_t s) {
  (void)d;
  if (rows <= 0) return;
  k_csr_to_dense_t<<<rows, 128, 0, s>>>(ptr, idx, val, rows, out, ld);
  SFD_LAUNCH_CHECK();
}

}  // namespace sfd
