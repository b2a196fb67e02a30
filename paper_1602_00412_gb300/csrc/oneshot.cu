// Per-stage entry points of include/sfd.h (one buffer / one stack / one
// matrix), used to check each stage against the oracle. Each call runs
// synchronously, in a stream and memory that the last one left (ScratchLease);
// before that was kept, allocating and freeing took most of a call's time. On a GB300,
// per call and with inputs on the device:
//   sfd_csr_spmm, 50,000 x 50,000, 2.5e6 entries, k = 100           2329 -> 240 us
//   sfd_csr_spmm_ex, transposed, 30,011 x 20,000, 3e6, k = 50, fp16  2016 -> 457
//   sfd_gram, 50,000 x 100, tensor cores                              274 -> 43
//   sfd_gemm_ts, 49,999 x 200 x 200                                   418 -> 162
//   sfd_orthonormalize, 20,000 x 100                                  818 -> 439
//   sfd_dense_shrink, 200 x 20,000, l = 100                          1494 -> 966
//   sfd_bssh_buffer, 1,801 x 2,000, l = 50                           2850 -> 2248 (2030 with
//                                                          the few-row X T since)
#include <string.h>

#include <algorithm>
#include <new>

#include "engine.cuh"

using namespace sfd;

namespace {

// The body of a one-shot call: errors become status codes.
template <typename F>
int guarded(F&& f) {
  try {
    return f();
  } catch (const CudaError& e) {
    return e.err == cudaErrorMemoryAllocation ? SFD_ENOMEM : SFD_ECUDA;
  } catch (const std::bad_alloc&) {
    return SFD_ENOMEM;
  }
}

// out: [0] 1 if the row pointer does not start at 0, decreases or has a row of more than
// max_row entries, [1] its last entry, [2] its longest row; [0] and [2] start at 0.
__global__ void k_check_rowptr(const int* __restrict__ ptr, int64_t m, int64_t max_row,
                               int* __restrict__ out) {
  int bad = 0, most = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int a = ptr[i], b = ptr[i + 1];
    if ((i == 0 && a != 0) || b < a || (int64_t)b - a > max_row) bad = 1;
    else most = max(most, b - a);
    if (i == m - 1) out[1] = b;
  }
  bad = __any_sync(0xffffffffu, bad);
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0) {
    if (bad) atomicOr(out, 1);
    if (most) atomicMax(out + 2, most);
  }
}

struct RowptrCheck {
  int64_t nnz = -1;  // -1: not a row pointer
  int64_t max_row = 0;
};

// The device row pointer, checked where it is (400 KB to the host and a loop there
// took 150 us for 100,000 rows).
RowptrCheck checked_rowptr(Scratch& L, const int32_t* rowptr, int64_t m, int64_t max_row) {
  // through a copy, as the entries below: what is no device memory is refused by it
  int* copy = reinterpret_cast<int*>(L.reserve((m + 1) * sizeof(int)));
  SFD_CUDA(cudaMemcpyAsync(copy, rowptr, (m + 1) * sizeof(int), cudaMemcpyDeviceToDevice,
                           L.stream));
  SFD_CUDA(cudaMemsetAsync(L.head, 0, 3 * sizeof(int), L.stream));
  const int grid = (int)std::min<int64_t>((m + 255) / 256, 4 * 152);
  k_check_rowptr<<<grid, 256, 0, L.stream>>>(copy, m, max_row, L.head);
  SFD_LAUNCH_CHECK();
  int* h = reinterpret_cast<int*>(L.pinned);
  SFD_CUDA(cudaMemcpyAsync(h, L.head, 3 * sizeof(int), cudaMemcpyDeviceToHost, L.stream));
  SFD_CUDA(cudaStreamSynchronize(L.stream));
  RowptrCheck r;
  if (!h[0]) r = {h[1], h[2]};
  return r;
}

// copy a device CSR into csr (allocated)
void copy_csr(Csr& csr, int64_t m, int64_t nnz, const int32_t* rowptr, const int32_t* colidx,
              const float* vals, cudaStream_t s) {
  SFD_CUDA(cudaMemcpyAsync(csr.ptr, rowptr, (m + 1) * sizeof(int), cudaMemcpyDeviceToDevice, s));
  if (nnz > 0) {
    SFD_CUDA(cudaMemcpyAsync(csr.idx, colidx, nnz * sizeof(int), cudaMemcpyDeviceToDevice, s));
    SFD_CUDA(cudaMemcpyAsync(csr.val, vals, nnz * sizeof(float), cudaMemcpyDeviceToDevice, s));
  }
}

// whether no entry was marked bad; waits for the stream
bool entries_ok(Scratch& L, const int* flags) {
  int* h = reinterpret_cast<int*>(L.pinned);
  SFD_CUDA(cudaMemcpyAsync(h, flags, sizeof(int), cudaMemcpyDeviceToHost, L.stream));
  SFD_CUDA(cudaStreamSynchronize(L.stream));
  return *h == 0;
}

// copy a device CSR into a slot and build its CSC / work lists; false on bad entries
bool load_slot(Slot& S, Scratch& L, int64_t m, const RowptrCheck& r, const int32_t* rowptr,
               const int32_t* colidx, const float* vals) {
  copy_csr(S.csr, m, r.nnz, rowptr, colidx, vals, S.stream);
  S.build((int)m, r.nnz, r.max_row);
  return entries_ok(L, S.ws.flags);
}

// Y = A X or A^T X by product(c, partial, stream). Only the side asked for is built:
// the CSC costs a radix sort that A X does not need.
template <typename F>
int run_spmm(int64_t m, int64_t d, const int32_t* rowptr, const int32_t* colidx, const float* vals,
             int ld_max, bool transposed, F&& product) {
  return guarded([&]() -> int {
    ScratchLease L(true);
    const RowptrCheck r = checked_rowptr(*L.s, rowptr, m, INT32_MAX);
    if (r.nnz < 0 || (r.nnz > 0 && (!colidx || !vals))) return SFD_EINVAL;
    Csr csr, csc;
    SortBuffers sort;
    Workspace ws;
    double* fro2 = nullptr;
    float* partial = nullptr;
    const int64_t cap = std::max<int64_t>(r.nnz, 1);
    DevArena A;
    A.carve(L.s, [&](DevArena& a) {
      csr.ptr = a.alloc<int>(m + 1);
      csr.idx = a.alloc<int>(cap);
      csr.val = a.alloc<float>(cap);
      if (transposed) {
        csc.ptr = a.alloc<int>(d + 1);
        csc.idx = a.alloc<int>(cap);
        csc.val = a.alloc<float>(cap);
        alloc_sort(a, sort, ws, cap, d + m);
        alloc_work(a, csc.work, d, cap);
      } else {
        alloc_work(a, csr.work, m, cap);
      }
      fro2 = a.alloc<double>(1024 + 8);
      ws.flags = a.alloc<int>(16);
      partial = a.alloc<float>((size_t)(2 * (r.nnz / kSplit) + 4) * ld_max);
    });
    Csr& c = transposed ? csc : csr;
    clear_work(c.work, L->stream);
    SFD_CUDA(cudaMemsetAsync(ws.flags, 0, 16 * sizeof(int), L->stream));
    copy_csr(csr, m, r.nnz, rowptr, colidx, vals, L->stream);
    csr.nseg = (int)m;
    csr.nnz = r.nnz;
    csr.may_split = r.max_row > kSplit;
    launch_check_entries(csr.idx, csr.val, r.nnz, (int)d, nullptr, fro2, ws.flags, L->stream);
    if (transposed) build_csc(csr, csc, (int)d, sort, ws, L->stream);
    else build_work(csr, L->stream);
    if (!entries_ok(*L.s, ws.flags)) return SFD_EINVAL;
    product(c, partial, L->stream);
    SFD_CUDA(cudaStreamSynchronize(L->stream));
    return SFD_OK;
  });
}

// Shared body of the two dense products: scratch, stream, timeout flag.
template <typename F>
int run_dense(F&& f) {
  return guarded([&]() -> int {
    ScratchLease L;
    Workspace ws;
    DevArena A;
    A.carve(L.s, [&](DevArena& a) { alloc_dense_scratch(a, ws); });
    clear_dense_scratch(ws, L->stream);
    f(ws, L->stream);
    int* flags = reinterpret_cast<int*>(L->pinned);
    SFD_CUDA(cudaMemcpyAsync(flags, ws.flags, 4 * sizeof(int), cudaMemcpyDeviceToHost, L->stream));
    SFD_CUDA(cudaStreamSynchronize(L->stream));
    return flags[2] ? SFD_ETIMEOUT : SFD_OK;
  });
}

}  // namespace

extern "C" {

int sfd_bssh_buffer(int64_t m, int64_t d, int32_t ell, const int32_t* rowptr, const int32_t* colidx,
                    const float* vals, uint64_t seed, int64_t b, const sfd_options* opt,
                    float* Bp_out, sfd_shrink_info* info) {
  if (m < 1 || d < 1 || ell < 1 || ell > m || m > d || ell > kMaxEll || !rowptr || !Bp_out || b < 0)
    return SFD_EINVAL;
  sfd_options o;
  if (opt) o = *opt; else sfd_options_init(&o);
  return guarded([&]() -> int {
    ScratchLease L(true);
    const RowptrCheck rp = checked_rowptr(*L.s, rowptr, m, d);
    if (rp.nnz < 0 || (rp.nnz > 0 && (!colidx || !vals))) return SFD_EINVAL;
    Slot S(d, ell, m, rp.nnz, L.s);
    if (!load_slot(S, *L.s, m, rp, rowptr, colidx, vals)) return SFD_EINVAL;
    const int q = q_for(o, (int)m);
    int inject = o.inject_vs_fail, r = 0, p = 0;
    Verdict v{};
    bool ok = false;
    for (; r < std::max(1, o.retry_cap); ++r) {
      p = o.verify ? vs_steps(d, delta_br(o.delta, b, r)) : 0;
      S.enqueue_attempt((int)m, q, seed, (uint64_t)b, (uint64_t)r, std::max(p, 1), o.verify);
      SFD_CUDA(cudaEventSynchronize(S.done));
      v = *S.verdict_host;
      ok = v.ok != 0;
      if (o.verify && inject > 0) {
        ok = false;
        --inject;
      }
      if (ok) break;
    }
    transpose(S.Bpt, d, ell, S.ld, Bp_out, d, S.stream);
    SFD_CUDA(cudaStreamSynchronize(S.stream));
    if (info) {
      info->q = q;
      info->attempts = std::min(r + 1, std::max(1, o.retry_cap));
      info->verified = ok ? 1 : 0;
      info->vs_steps = p;
      info->delta_shrink = v.delta;
      info->logsum = v.logsum;
      info->fro2_a = v.fro2a;
      info->fro2_b = v.fro2b;
      info->captured = v.captured;
    }
    return SFD_OK;
  });
}

int sfd_q_features(int64_t m, int64_t d, int32_t ell, const int32_t* rowptr, const int32_t* colidx,
                   const float* vals, uint64_t seed, int64_t b, int32_t q_fixed, float* features) {
  if (m < 1 || d < 1 || ell < 1 || ell > m || m > d || ell > kMaxEll || !rowptr || !features ||
      b < 0 || q_fixed < 1)
    return SFD_EINVAL;
  return guarded([&]() -> int {
    ScratchLease L(true);
    const RowptrCheck rp = checked_rowptr(*L.s, rowptr, m, d);
    if (rp.nnz < 0 || (rp.nnz > 0 && (!colidx || !vals))) return SFD_EINVAL;
    Slot S(d, ell, m, rp.nnz, L.s);
    if (!load_slot(S, *L.s, m, rp, rowptr, colidx, vals)) return SFD_EINVAL;
    // S0 = (A'G)^T (A'G) for the G of attempt 0 (Alg. 1's start block)
    launch_gauss_fill(S.W, d, ell, S.ld, seed, (uint64_t)b, 0, 1, S.stream);
    spmm(S.csr, S.W, S.ld, S.ld, S.Y, S.ld, S.ws.partial_rows, S.stream);
    gram(S.Y, S.ld, single_map(ell), m, S.ws.small_a, S.ws, S.stream);
    q_features(S.csr, S.csc, d, ell, q_fixed, S.fro2, S.ws.small_a, S.qfeat, S.qacc, S.stream);
    SFD_CUDA(cudaMemcpyAsync(features, S.qfeat, kQF * sizeof(float), cudaMemcpyDeviceToHost,
                             S.stream));
    SFD_CUDA(cudaStreamSynchronize(S.stream));
    return SFD_OK;
  });
}

int sfd_dense_shrink(int64_t rows, int64_t d, int32_t ell, const float* M, float* B_out) {
  if (rows < 1 || d < 1 || ell < 1 || ell > kMaxEll || rows > 2 * (int64_t)ell || !M || !B_out ||
      d > 2000000)
    return SFD_EINVAL;
  return guarded([&]() -> int {
    ScratchLease L;
    Merger G(d, ell, L.s);
    // rows 0..min(rows,l) are the "B" block, the rest the stacked block
    const int k0 = (int)std::min<int64_t>(rows, ell);
    const int k1 = (int)(rows - k0);
    transpose(M, k0, (int)d, (int)d, G.B(), G.ld, G.stream);
    SFD_CUDA(cudaMemsetAsync(G.stack, 0, (size_t)d * G.ld * sizeof(float), G.stream));
    if (k1 > 0) transpose(M + (size_t)k0 * d, k1, (int)d, (int)d, G.stack, G.ld, G.stream);
    G.dense_shrink(G.stack, G.ld, k1);
    transpose(G.B(), d, ell, G.ld, B_out, d, G.stream);
    SFD_CUDA(cudaStreamSynchronize(G.stream));
    return SFD_OK;
  });
}

int sfd_csr_spmm(int64_t m, int64_t d, const int32_t* rowptr, const int32_t* colidx,
                 const float* vals, int32_t k, const float* X, int32_t ldx, float* Y, int32_t ldy,
                 int32_t transpose_flag) {
  if (m < 1 || d < 1 || k < 1 || k > kMaxEll || ldx < k || ldy < k || (ldx & 3) || (ldy & 3) ||
      !rowptr || !X || !Y)
    return SFD_EINVAL;
  return run_spmm(m, d, rowptr, colidx, vals, std::max(ldx, ldy), transpose_flag != 0,
                  [&](const Csr& c, float* partial, cudaStream_t s) {
                    spmm(c, X, ldx, k, Y, ldy, partial, s);
                  });
}

int sfd_spmm_variant_count(int32_t x_fp16) { return spmm_variants(x_fp16 != 0); }

int sfd_csr_spmm_ex(int64_t m, int64_t d, const int32_t* rowptr, const int32_t* colidx,
                    const float* vals, int32_t k, const void* X, int32_t x_fp16, int32_t ldx,
                    float* Y, int32_t ldy, int32_t transpose_flag, int32_t variant) {
  if (m < 1 || d < 1 || k < 1 || ldx < k || ldy < k || !rowptr || !X || !Y ||
      variant < 0 || variant >= spmm_variants(x_fp16 != 0))
    return SFD_EINVAL;
  if (x_fp16 ? (k > 128 || (ldx & 7) || (ldy & 7)) : (k > kMaxEll || (ldx & 3) || (ldy & 3)))
    return SFD_EINVAL;
  return run_spmm(m, d, rowptr, colidx, vals, std::max(ldx, ldy), transpose_flag != 0,
                  [&](const Csr& c, float* partial, cudaStream_t s) {
                    if (x_fp16)
                      spmm_h(c, static_cast<const __half*>(X), ldx, k, Y, ldy, partial, s, variant);
                    else
                      spmm(c, static_cast<const float*>(X), ldx, k, Y, ldy, partial, s, variant);
                  });
}

int sfd_orthonormalize(int64_t rows, int32_t k, float* X, int32_t ld) {
  if (rows < 1 || k < 1 || k > kMaxEll || ld < k || !X) return SFD_EINVAL;
  return guarded([&]() -> int {
    ScratchLease L;
    Workspace ws;
    float* tmp = nullptr;
    DevArena A;
    A.carve(L.s, [&](DevArena& a) {
      alloc_dense_scratch(a, ws);
      tmp = a.alloc<float>((size_t)rows * ld);
    });
    clear_dense_scratch(ws, L->stream);
    const ColMap map = single_map(k);
    // shifted CholeskyQR3: the first (shifted) pass leaves a block of condition
    // number about sqrt(||X||^2 / shift) <= 2^10 whatever cond(X) was; the
    // next two make it orthonormal to fp32 accuracy
    for (int pass = 0; pass < 3; ++pass) {
      const float* in = pass == 1 ? tmp : X;
      gram(in, ld, map, rows, ws.small_a, ws, L->stream);
      chol_inv(ws.small_a, k, ws.small_b, ws.eig_work, ws.flags, L->stream, true);
      gemm_ts(in, ld, map, rows, ws.small_b, k, pass == 1 ? X : tmp, ld, L->stream);
    }
    SFD_CUDA(cudaMemcpy2DAsync(X, ld * sizeof(float), tmp, ld * sizeof(float), k * sizeof(float),
                               rows, cudaMemcpyDeviceToDevice, L->stream));
    SFD_CUDA(cudaStreamSynchronize(L->stream));
    return SFD_OK;
  });
}

int sfd_set_wait_limit(int64_t spins) {
  return guarded([&]() -> int {
    set_wait_limit(spins);
    return SFD_OK;
  });
}

int sfd_wait_selftest(int64_t spins, float* ms_out) {
  return guarded([&]() -> int {
    return wait_selftest(spins, ms_out) ? SFD_ETIMEOUT : SFD_OK;
  });
}

int sfd_gram(int64_t rows, int32_t k, const float* X, int32_t ldx, float* G, int32_t precision) {
  if (rows < 0 || k < 1 || k > kMaxEll || ldx < k || !G || (rows > 0 && !X)) return SFD_EINVAL;
  if (precision != 0 && !((precision == 1 || precision == 2) && tc_supported(k, k)))
    return SFD_EINVAL;
  return run_dense([&](Workspace& ws, cudaStream_t s) {
    if (precision) gram_tc(X, ldx, single_map(k), rows, G, ws, s, precision == 2);
    else gram(X, ldx, single_map(k), rows, G, ws, s);
  });
}

int sfd_gemm_ts(int64_t rows, int32_t n, const float* X, int32_t ldx, const float* T, int32_t kout,
                float* Y, int32_t ldy, int32_t precision) {
  if (rows < 0 || n < 1 || n > kMaxEll || kout < 1 || kout > kMaxEll || ldx < n || ldy < kout ||
      !T || (rows > 0 && (!X || !Y)))
    return SFD_EINVAL;
  if (precision != 0 && !(precision == 1 && tc_supported(n, kout)) &&
      !(precision == 2 && tc_split_supported(n, kout)))
    return SFD_EINVAL;
  return run_dense([&](Workspace& ws, cudaStream_t s) {
    if (precision) gemm_ts_tc(X, ldx, single_map(n), rows, T, kout, Y, ldy, ws, s, nullptr,
                              precision == 2);
    else gemm_ts(X, ldx, single_map(n), rows, T, kout, Y, ldy, s);
  });
}

int sfd_symeig(int32_t n, const float* S, int32_t nwant, float* evals, float* evecs) {
  if (n < 1 || n > kMaxEig || nwant < 1 || nwant > n || !S || !evals || !evecs) return SFD_EINVAL;
  return guarded([&]() -> int {
    ScratchLease L;
    float* work =
        reinterpret_cast<float*>(L->reserve(symeig_work_floats(kMaxEig, kMaxEig) * sizeof(float)));
    symeig(S, n, nwant, evals, evecs, work, L->stream);
    SFD_CUDA(cudaStreamSynchronize(L->stream));
    return SFD_OK;
  });
}

}  // extern "C"
