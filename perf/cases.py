"""The workloads this framework is timed on: whole SFD streams through a kept
context, many streams through a batch, and the single stages through their own
entry points. Sizes are those of the repository's configurations and tests (the
C1, C2, C3 and C4 streams and the stage tests), thinned where a full stream
would only repeat the same buffers.

A sketch B is determined up to the signs of its rows (and a rotation inside a
cluster of singular values): what a program uses, and what two correct
implementations agree on, is the covariance estimate B^T B. A case that ends in
a sketch therefore returns B^T B itself (d <= 4096) or B^T B applied to a block
of 256 >= l directions, which determines it. Eigenvectors are returned as the
rank-nwant matrix V diag(w) V^T beside the eigenvalues, for the same reason.
"""
import math

import numpy as np
import torch

from paper_1602_00412_gb300 import sfd

PROBES = 256       # columns of the block a wide sketch's B^T B is applied to
FULL_COV = 4096    # up to this d the whole d x d matrix B^T B is returned
TAG_START = 1      # Philox tag of the start block of the power iteration


def listed():
    return [
        # The smallest configuration as a first-time user runs it: default options
        # (fp32), host arrays, one call, five buffers; latency and launches count.
        {"name": "stream c1 host", "kind": "stream", "rows": "zipf", "n": 10000, "d": 2000,
         "ell": 50, "mean": 20.0, "rank": 10, "decay": 0.7, "precision": 0, "where": "host"},
        # The benchmark configuration (mixed precision, device arrays), four of its
        # twenty 50,000-row buffers and a ragged rest that the sketch call flushes.
        {"name": "stream c2 mixed", "kind": "stream", "rows": "zipf", "n": 203333, "d": 50000,
         "ell": 100, "mean": 50.0, "rank": 20, "decay": 0.8, "precision": 1, "where": "device"},
        # Bag-of-words rows at l = 200 (the C3 configuration's sketch size), wider than
        # the 128 columns one tensor-core tile holds: one whole buffer and a flushed rest.
        {"name": "stream bow l200", "kind": "stream", "rows": "bow", "n": 130000, "d": 100000,
         "ell": 200, "mean": 66.7, "rank": 0, "decay": 0.0, "precision": 1, "where": "device"},
        # Many small independent streams side by side (the C4 configuration: d, l and
        # density differ per stream, uniform columns), the next block of rows of each.
        # In fp32: uniform columns leave a flat noise spectrum at l, on which mixed
        # precision's sketches differ by 1e-4 when any sum changes its order.
        {"name": "batch c4", "kind": "batch", "streams": 8, "shapes": 4, "d_lo": 1000,
         "d_hi": 8000, "n_lo": 3000, "n_hi": 8000, "precision": 0},
        # One buffer's BoostedSparseShrink by itself, ragged row count, mixed precision.
        {"name": "shrink one buffer", "kind": "bssh", "rows": "zipf", "m": 1801, "d": 2000,
         "ell": 50, "mean": 20.0, "rank": 10, "decay": 0.7, "precision": 1},
        # DenseShrink of two stacked sketches: folding sketches that were made elsewhere.
        {"name": "dense shrink", "kind": "dense", "rows": 200, "d": 20000, "ell": 100},
        # The product A X of the power iteration on a whole C2 buffer, fp32 block.
        {"name": "spmm c2", "kind": "spmm", "rows": "zipf", "m": 50000, "d": 50000, "mean": 50.0,
         "k": 100, "ld": 104, "half": 0, "transpose": 0},
        # The transposed product A^T X on a many-streams buffer, fp16 block, odd row count.
        {"name": "spmm transposed half", "kind": "spmm", "rows": "uniform", "m": 30011, "d": 20000,
         "mean": 100.0, "k": 50, "ld": 56, "half": 1, "transpose": 1},
        # Gram of a C2 block on the tensor cores (TF32 inputs).
        {"name": "gram tf32", "kind": "gram", "rows": 50000, "k": 100, "ld": 104, "precision": 1},
        # X T in fp32 at a width beyond the tensor-core tile, one row short of round.
        {"name": "gemm fp32 l200", "kind": "gemm", "rows": 49999, "k": 200, "kout": 200,
         "ld": 200, "precision": 0},
        # Orthonormalising a block (the Gram-Schmidt step), fp64 factors.
        {"name": "orthonormalize", "kind": "orth", "rows": 20000, "k": 100, "ld": 104},
        # The smallest call: the small symmetric eigenproblem of one sketch merge.
        {"name": "symeig 200", "kind": "eig", "n": 200, "nwant": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stream", "batch", "bssh", "dense", "spmm", "gram", "gemm", "orth", "eig"])
    rows = rng.choice(["zipf", "uniform", "bow"])
    if kind == "stream":
        d = _log(rng, 1000, 60000)
        ell = rng.choice([20, 33, 50, 77, 100, 128, 150, 200])
        n = max(2 * ell, min(_log(rng, 2000, 150000), 4 * d))
        return {"kind": kind, "rows": rows, "n": n, "d": d, "ell": ell,
                "mean": rng.uniform(10.0, 60.0), "rank": max(1, ell // 4), "decay": 0.85,
                "precision": 0 if rows == "uniform" else rng.choice([0, 1]),
                "where": rng.choice(["host", "device"])}
    if kind == "batch":
        return {"kind": kind, "streams": rng.randint(2, 12), "shapes": rng.randint(0, 1 << 20),
                "d_lo": 1000, "d_hi": _log(rng, 2000, 12000), "n_lo": 2000,
                "n_hi": _log(rng, 3000, 9000), "precision": 0}
    if kind == "bssh":
        d = _log(rng, 500, 30000)
        ell = rng.choice([20, 37, 50, 100, 128, 200])
        m = max(ell, min(d, _log(rng, 400, 30000)))
        return {"kind": kind, "rows": rows, "m": m, "d": d, "ell": ell,
                "mean": rng.uniform(10.0, 60.0), "rank": max(1, ell // 4), "decay": 0.85,
                "precision": 0 if rows == "uniform" else rng.choice([0, 1])}
    if kind == "dense":
        ell = rng.choice([20, 50, 77, 100, 128, 200, 256])
        return {"kind": kind, "rows": rng.randint(ell // 2, 2 * ell), "d": _log(rng, 500, 60000),
                "ell": ell}
    if kind == "spmm":
        half = rng.choice([0, 1])
        k = rng.randint(8, 128 if half else 256)
        return {"kind": kind, "rows": rows, "m": _log(rng, 500, 60000), "d": _log(rng, 500, 60000),
                "mean": rng.uniform(10.0, 60.0), "k": k, "ld": (k + 7) // 8 * 8, "half": half,
                "transpose": rng.choice([0, 1])}
    if kind == "gram":
        precision = rng.choice([0, 1, 2])
        k = rng.randint(8, 256 if precision == 0 else 128)
        return {"kind": kind, "rows": _log(rng, 500, 100000), "k": k,
                "ld": (k + 3) // 4 * 4 + rng.choice([0, 4]), "precision": precision}
    if kind == "gemm":
        precision = rng.choice([0, 1, 2])
        top = (256, 128, 112)[precision]
        k, kout = rng.randint(8, top), rng.randint(8, top)
        return {"kind": kind, "rows": _log(rng, 500, 100000), "k": k, "kout": kout,
                "ld": (max(k, kout) + 3) // 4 * 4, "precision": precision}
    if kind == "orth":
        k = rng.randint(8, 256)
        return {"kind": kind, "rows": _log(rng, 2 * k, 60000), "k": k, "ld": (k + 7) // 8 * 8}
    n = rng.randint(20, 256)
    return {"kind": "eig", "n": n, "nwant": rng.randint(n // 3, n)}


# ------------------------------------------------------------------ input data
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt * 7919 + 17) % (1 << 62))
    return g


def _zipf_cdf(d, s):
    c = np.cumsum(np.arange(1, d + 1, dtype=np.float64) ** (-s))
    return torch.from_numpy(c / c[-1]).cuda()


def _csr(g, n, d, rank, decay, mean, rows):
    """n sparse rows over d columns without repeats within a row, sorted by
    column: int64 row pointer, int32 columns, float32 values on the GPU."""
    ones = torch.ones(n, device="cuda")
    if rows == "bow":
        cnt = torch.exp(math.log(mean) + 0.8 * torch.randn(n, device="cuda", generator=g)).round()
        cnt = cnt.clamp(max=2000)
    else:
        cnt = torch.poisson(ones * mean, generator=g)
    cnt = cnt.clamp(max=max(1, d // 2)).long()
    r = torch.repeat_interleave(torch.arange(n, device="cuda"), cnt)
    cdf = None if rows == "uniform" else _zipf_cdf(d, 1.05 if rows == "bow" else 1.1)

    def cols(k):
        if cdf is None:
            return torch.randint(0, d, (k,), device="cuda", generator=g)
        u = torch.rand(k, device="cuda", generator=g, dtype=torch.float64)
        return torch.searchsorted(cdf, u, right=True).clamp(max=d - 1)

    key = torch.sort(r * d + cols(r.numel()))[0]
    for _ in range(24):               # a repeated column of a row is drawn again
        dup = torch.zeros(key.numel(), dtype=torch.bool, device="cuda")
        dup[1:] = key[1:] == key[:-1]
        k = int(dup.sum())
        if k == 0:
            break
        key[dup] = key[dup] // d * d + cols(k)
        key = torch.sort(key)[0]
    key = torch.unique_consecutive(key)
    r, c = key // d, key % d
    if rows == "bow":                 # log(1 + count), rows of unit length
        z = torch.poisson(torch.full((key.numel(),), 2.0, device="cuda"), generator=g).clamp(min=1)
        v = torch.log1p(z)
        nrm = torch.segment_reduce(v * v, "sum", lengths=torch.bincount(r, minlength=n))
        v = v / nrm.sqrt().clamp(min=1e-20)[r]
    else:                             # a planted low-rank signal and noise
        sig = 10.0 * decay ** torch.arange(rank, device="cuda", dtype=torch.float32)
        x = torch.randn((n, rank), device="cuda", generator=g) * sig
        y = torch.randn((d, rank), device="cuda", generator=g)
        v = 0.1 * torch.randn(key.numel(), device="cuda", generator=g)
        for a in range(0, key.numel(), 1 << 22):
            b = a + (1 << 22)
            v[a:b] += (x[r[a:b]] * y[c[a:b]]).sum(1)
    ip = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ip[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
    return ip, c.to(torch.int32), v.float()


def _shapes(case):
    """Per stream of a batch: d, l, density and rows (as the C4 configuration
    draws them, with fewer rows)."""
    rng = np.random.default_rng([case["shapes"], 4])
    out = []
    for _ in range(case["streams"]):
        out.append((int(rng.integers(case["d_lo"], case["d_hi"] + 1)),
                    int(rng.choice([20, 50, 100])), float(rng.uniform(0.005, 0.05)),
                    int(rng.integers(case["n_lo"], case["n_hi"] + 1))))
    return out


def _inputs(case, seed):
    """Everything that follows from the seed: the arrays a call is given."""
    g, k = _gen(seed), case["kind"]
    if k == "stream":
        return _csr(g, case["n"], case["d"], case["rank"], case["decay"], case["mean"],
                    case["rows"])
    if k == "batch":
        return [_csr(_gen(seed, 1 + i), n, d, max(1, ell // 4), 0.9, d * rho, "uniform")
                for i, (d, ell, rho, n) in enumerate(_shapes(case))]
    if k in ("bssh", "spmm"):
        rank = case.get("rank", 20)
        ip, ix, v = _csr(g, case["m"], case["d"], rank, case.get("decay", 0.8), case["mean"],
                         case["rows"])
        if k == "bssh":
            return ip.int(), ix, v
        rows_in = case["m"] if case["transpose"] else case["d"]
        X = torch.zeros((rows_in, case["ld"]), device="cuda")
        X[:, :case["k"]] = torch.rand((rows_in, case["k"]), device="cuda", generator=g) * 2 - 1
        return ip.int(), ix, v, X.half() if case["half"] else X
    if k == "dense":                  # two stacked blocks of decaying orthogonal-like rows
        M = torch.randn((case["rows"], case["d"]), device="cuda", generator=g)
        return (M * (0.97 ** torch.arange(case["rows"], device="cuda"))[:, None]).contiguous()
    if k in ("gram", "gemm"):
        X = torch.zeros((case["rows"], case["ld"]), device="cuda")
        X[:, :case["k"]] = torch.randn((case["rows"], case["k"]), device="cuda", generator=g)
        if k == "gram":               # columns of different length, as before an orthonormalisation
            X[:, :case["k"]] *= torch.logspace(0, 1, case["k"], device="cuda")
            return X
        T = torch.randn((case["k"], case["kout"]), device="cuda", generator=g).triu()
        return X, T.contiguous()
    if k == "orth":                   # condition number about 1e3, as a power step leaves it
        mix = torch.randn((case["k"], case["k"]), device="cuda", generator=g)
        mix = torch.linalg.qr(mix.cpu())[0].cuda()
        s = torch.logspace(0, -3, case["k"], device="cuda")
        X = torch.zeros((case["rows"], case["ld"]), device="cuda")
        X[:, :case["k"]] = torch.randn((case["rows"], case["k"]), device="cuda", generator=g) * s @ mix
        return X
    n = case["n"]                     # a decaying Gram matrix
    M = torch.randn((n, 3 * n), device="cuda", generator=g, dtype=torch.float64)
    M = M * (0.95 ** torch.arange(n, device="cuda", dtype=torch.float64))[:, None]
    return (M @ M.T).float().contiguous()


def _probe(seed, d):
    return None if d <= FULL_COV else torch.randn((d, PROBES), device="cuda", generator=_gen(seed, 99))


def _philox_seed(seed):
    return (int(seed) * 7 + 3) % (1 << 31)


# ------------------------------------------------------------- prepare and run
def prepare(case, seed):
    k = case["kind"]
    data = _inputs(case, seed)
    st = {"case": case, "kind": k}
    if k == "stream":
        if case["where"] == "host":
            data = [a.cpu().numpy() for a in data]
        st["data"] = data
        st["sketch"] = sfd.SFD(case["d"], case["ell"], _philox_seed(seed), precision=case["precision"])
        st["B"] = torch.empty((case["ell"], case["d"]), device="cuda")
        st["probe"] = _probe(seed, case["d"])
    elif k == "batch":
        sh = _shapes(case)
        st["data"] = data
        st["batch"] = sfd.Batch([s[0] for s in sh], [s[1] for s in sh], _philox_seed(seed),
                                precision=case["precision"])
        st["B"] = [torch.empty((s[1], s[0]), device="cuda") for s in sh]
        st["probe"] = [_probe(seed, s[0]) for s in sh]
    elif k == "bssh":
        st["data"] = data
        st["opts"] = sfd.options(precision=case["precision"])
        st["seed"] = _philox_seed(seed)
        st["B"] = torch.empty((case["ell"], case["d"]), device="cuda")
        st["probe"] = _probe(seed, case["d"])
    elif k == "dense":
        st["data"] = data
        st["B"] = torch.empty((case["ell"], case["d"]), device="cuda")
        st["probe"] = _probe(seed, case["d"])
    elif k == "spmm":
        st["data"] = data
        st["Y"] = torch.zeros((case["d"] if case["transpose"] else case["m"], case["ld"]), device="cuda")
    elif k == "gram":
        st["data"] = data
        st["G"] = torch.empty((case["k"], case["k"]), device="cuda")
    elif k == "gemm":
        st["data"] = data
        st["Y"] = torch.zeros((case["rows"], case["ld"]), device="cuda")
    elif k == "orth":
        st["data"] = data
        st["X"] = torch.empty_like(data)
    else:
        st["data"] = data
        st["w"] = torch.empty(case["nwant"], device="cuda")
        st["V"] = torch.empty((case["n"], case["nwant"]), device="cuda")
    return st


def _cov(B, probe):
    return B.T @ B if probe is None else B.T @ (B @ probe)


def run(st):
    case, k = st["case"], st["kind"]
    if k == "stream":
        s = st["sketch"]
        s.reset()
        s.append(*st["data"])
        return _cov(s.sketch(st["B"]), st["probe"])
    if k == "batch":
        b = st["batch"]
        for i, rows in enumerate(st["data"]):
            b.append(i, *rows)
        b.wait()
        return [_cov(b.sketch(i, B), p) for i, (B, p) in enumerate(zip(st["B"], st["probe"]))]
    if k == "bssh":
        info = sfd.sfd_bssh_buffer(case["m"], case["d"], case["ell"], *st["data"], st["seed"], 0,
                                   st["B"], st["opts"])
        return {"cov": _cov(st["B"], st["probe"]), "q": info["q"], "attempts": info["attempts"]}
    if k == "dense":
        sfd.sfd_dense_shrink(case["rows"], case["d"], case["ell"], st["data"], st["B"])
        return _cov(st["B"], st["probe"])
    if k == "spmm":
        ip, ix, v, X = st["data"]
        if case["half"]:
            sfd.sfd_csr_spmm_ex(case["m"], case["d"], ip, ix, v, case["k"], X, case["ld"], st["Y"],
                                case["ld"], case["transpose"], 0)
        else:
            sfd.sfd_csr_spmm(case["m"], case["d"], ip, ix, v, case["k"], X, case["ld"], st["Y"],
                             case["ld"], case["transpose"])
        return st["Y"][:, :case["k"]]
    if k == "gram":
        sfd.sfd_gram(case["rows"], case["k"], st["data"], case["ld"], st["G"], case["precision"])
        return st["G"]
    if k == "gemm":
        X, T = st["data"]
        sfd.sfd_gemm_ts(case["rows"], case["k"], X, case["ld"], T, case["kout"], st["Y"], case["ld"],
                        case["precision"])
        return st["Y"][:, :case["kout"]]
    if k == "orth":                   # in place: each pass starts from the same block
        st["X"].copy_(st["data"])
        sfd.sfd_orthonormalize(case["rows"], case["k"], st["X"], case["ld"])
        return st["X"][:, :case["k"]]
    sfd.sfd_symeig_noalloc(case["n"], st["data"], case["nwant"], st["w"], st["V"])
    return {"w": st["w"], "rebuilt": (st["V"] * st["w"]) @ st["V"].T}


# ------------------------------------------------------------------ work, exact
def _q(m):
    return max(0, math.ceil(math.log(4.0 * m)))   # the fixed power count schedule


def _stream_work(n, d, ell, nnz):
    """Bytes: the entries and row pointers read once, the sketch written once.
    Flops: the power iteration's sparse products, Grams and triangular
    products, the shrink and the fold of every buffer."""
    flops = 0.0
    left_n, left_nnz = n, nnz
    while left_n > 0:
        m = min(left_n, d, max(1, math.ceil(ell * d / max(1.0, nnz / n))))
        e = nnz * m / n
        q = _q(m)
        flops += 2.0 * e * ell * (2 * q + 2) + 3.0 * ell * ell * (m * (q + 2) + d * (q + 2))
        flops += 36.0 * e * 4 + 4.0 * d * ell * ell * 2 + 10.0 * (2 * ell) ** 3
        left_n -= m
        left_nnz -= e
    return 8.0 * nnz + 8.0 * (n + 1) + 4.0 * ell * d, flops


def work(case):
    k = case["kind"]
    if k == "stream":
        mean = case["mean"] * (math.exp(0.32) if case["rows"] == "bow" else 1.0)
        b, f = _stream_work(case["n"], case["d"], case["ell"], mean * case["n"])
    elif k == "batch":
        p = [_stream_work(n, d, ell, d * rho * n) for d, ell, rho, n in _shapes(case)]
        b, f = sum(x[0] for x in p), sum(x[1] for x in p)
    elif k == "bssh":
        mean = case["mean"] * (math.exp(0.32) if case["rows"] == "bow" else 1.0)
        b, f = _stream_work(case["m"], case["d"], case["ell"], mean * case["m"])
    elif k == "dense":
        r, d, ell = case["rows"], case["d"], case["ell"]
        b, f = 4.0 * d * (r + ell), 1.0 * d * r * r + 2.0 * d * r * ell + 10.0 * r ** 3
    elif k == "spmm":
        mean = case["mean"] * (math.exp(0.32) if case["rows"] == "bow" else 1.0)
        nnz, rin = mean * case["m"], case["m"] if case["transpose"] else case["d"]
        rout = case["d"] if case["transpose"] else case["m"]
        b = 8.0 * nnz + 4.0 * case["m"] + case["k"] * (rin * (2.0 if case["half"] else 4.0) + 4.0 * rout)
        f = 2.0 * nnz * case["k"]
    elif k == "gram":
        b, f = 4.0 * case["k"] * (case["rows"] + case["k"]), 1.0 * case["rows"] * case["k"] ** 2
    elif k == "gemm":
        b = 4.0 * (case["rows"] * (case["k"] + case["kout"]) + case["k"] * case["kout"])
        f = 2.0 * case["rows"] * case["k"] * case["kout"]
    elif k == "orth":
        b, f = 8.0 * case["rows"] * case["k"], 3.0 * 3.0 * case["rows"] * case["k"] ** 2
    else:
        n, w = case["n"], case["nwant"]
        b, f = 4.0 * (n * n + n * w + w), 4.0 / 3.0 * n ** 3 + 2.0 * n * n * w
    return {"bytes": b, "flops": f}


def _start_block(seed, b, d, ell):
    """The Gaussian start block of buffer b: Philox4x64-10 keyed (seed, 0),
    counter (block, b, 0, 1), 24-bit uniforms, Box-Muller; row-major d x l."""
    before = ((b << 64) + (TAG_START << 192)) - 1    # numpy steps the counter before it draws
    words = np.random.Philox(counter=before % (1 << 256), key=int(seed)).random_raw((d * ell + 3) // 4 * 4)
    u = torch.from_numpy((words >> np.uint64(40)).astype(np.float64)).cuda()
    u = (u + 0.5) * 2.0 ** -24
    u = u.reshape(-1, 2)
    rad, ang = torch.sqrt(-2.0 * torch.log(u[:, 0])), 2.0 * math.pi * u[:, 1]
    z = torch.stack([rad * torch.cos(ang), rad * torch.sin(ang)], 1).reshape(-1)
    return z[:d * ell].reshape(d, ell)


def _sparse(ip, ix, v, n, d):
    return torch.sparse_csr_tensor(ip.long(), ix.long(), v.double(), size=(n, d))


def _transposed(ip, ix, v, n, d):
    r = torch.repeat_interleave(torch.arange(n, device="cuda"), ip[1:] - ip[:-1])
    c, order = torch.sort(ix.long(), stable=True)
    tp = torch.zeros(d + 1, dtype=torch.int64, device="cuda")
    tp[1:] = torch.cumsum(torch.bincount(c, minlength=d), 0)
    return _sparse(tp, r[order], v[order], d, n)


def _shrunk(M, ell):
    """Rows sqrt(s_i^2 - s_l^2) v_i^T of the singular value decomposition of M."""
    lam, H = torch.linalg.eigh(M @ M.T)
    lam, H = lam.flip(0)[:ell].clamp(min=0), H.flip(1)[:, :ell]
    thr = lam[ell - 1] if lam.numel() >= ell else lam.new_zeros(())
    w = torch.where(lam > thr, torch.sqrt((1 - thr / lam.clamp(min=1e-300)).clamp(min=0)),
                    lam.new_zeros(()))
    return (H * w).T @ M


def _buffer(ip, ix, v, m, d, ell, seed, b):
    """SparseShrink of one buffer in float64 (accepted on its first attempt)."""
    A, At = _sparse(ip, ix, v, m, d), _transposed(ip, ix, v, m, d)
    Y = torch.linalg.qr(A @ _start_block(seed, b, d, ell))[0]
    for _ in range(_q(m)):
        W = torch.linalg.qr(At @ Y)[0]
        Y = torch.linalg.qr(A @ W)[0]
    return _shrunk((At @ Y).T.contiguous(), ell)


def _stream(ip, ix, v, n, d, ell, seed):
    """The whole stream in float64: buffers of l d entries or d rows, the rest flushed."""
    h = ip.cpu().numpy()
    B = torch.zeros((ell, d), dtype=torch.float64, device="cuda")
    start, b = 0, 0
    while start < n:
        end = int(np.searchsorted(h, h[start] + ell * d, side="left"))
        end = min(n, start + d, max(end, start + 1))
        e0, e1, m = int(h[start]), int(h[end]), end - start
        p, x, w = ip[start:end + 1] - e0, ix[e0:e1], v[e0:e1]
        if m >= ell:
            new = _buffer(p, x, w, m, d, ell, seed, b)
        else:
            new = _sparse(p, x, w, m, d).to_dense()
        B = _shrunk(torch.cat([B, new]), ell)
        start, b = end, b + 1
    return B


def exact(case, seed):
    k, data = case["kind"], _inputs(case, seed)
    if k == "stream":
        B = _stream(*data, case["n"], case["d"], case["ell"], _philox_seed(seed))
        p = _probe(seed, case["d"])
        return _cov(B, None if p is None else p.double())
    if k == "batch":
        out = []
        for i, ((d, ell, rho, n), rows) in enumerate(zip(_shapes(case), data)):
            B = _stream(*rows, n, d, ell, _philox_seed(seed) + i)
            p = _probe(seed, d)
            out.append(_cov(B, None if p is None else p.double()))
        return out
    if k == "bssh":
        B = _buffer(data[0].long(), data[1], data[2], case["m"], case["d"], case["ell"],
                    _philox_seed(seed), 0)
        p = _probe(seed, case["d"])
        return {"cov": _cov(B, None if p is None else p.double()), "q": None, "attempts": None}
    if k == "dense":
        B = _shrunk(data.double(), case["ell"])
        p = _probe(seed, case["d"])
        return _cov(B, None if p is None else p.double())
    if k == "spmm":
        ip, ix, v, X = data
        make = _transposed if case["transpose"] else _sparse
        return make(ip.long(), ix, v, case["m"], case["d"]) @ X[:, :case["k"]].double()
    if k == "gram":
        X = data[:, :case["k"]].double()
        return X.T @ X
    if k == "gemm":
        return data[0][:, :case["k"]].double() @ data[1].double()
    if k == "orth":
        Q, R = torch.linalg.qr(data[:, :case["k"]].double())
        return Q * torch.sign(torch.diagonal(R))
    lam, V = torch.linalg.eigh(data.double())
    lam, V = lam.flip(0)[:case["nwant"]], V.flip(1)[:, :case["nwant"]]
    return {"w": lam, "rebuilt": (V * lam) @ V.T}
