"""What the framework's users have it do, case by case, through its public calls.

The calls are those of paper_1503_05464_gb300: compress a dense matrix (alone
or many together), apply the compressed form to a block of vectors, factor it,
solve with the factors, and the two steps that the compression spends its time
in and that are public calls of their own (the fused sampling products and the
batched interpolative decomposition).  Matrices, tolerances, leaf sizes and
sample schedules are those of the repository's configurations: the Toeplitz
matrix 1/(1+|i-j|) (FP64, leaf 128, rtol 1e-6, 64/32), the Gaussian kernel in
the unit cube (FP32, leaf 256, rtol 1e-4, 128/64), the kernel 1/(4 pi r) on the
unit sphere (FP32, leaf 512, rtol 1e-6, 256/128), the quantum-chemistry
Toeplitz matrix and the Schur complements of the 7-point Laplacian that the
serving loop compresses (FP32, leaf 256, rtol 1e-6, 128/64).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1503_05464_gb300 as P

F64 = torch.float64
SETTINGS = {   # family: dtype, sampling arithmetic, leaf, rtol, first and further sample columns
    "toeplitz": (torch.float64, "native", 128, 1e-6, 64, 32),
    "qchem": (torch.float64, "native", 128, 1e-6, 64, 32),
    "gauss": (torch.float32, "bf16x3", 256, 1e-4, 128, 64),
    "bem": (torch.float32, "bf16x3", 512, 1e-6, 256, 128),
    "schur": (torch.float32, "bf16x3", 256, 1e-6, 128, 64),
}


def listed():
    return [
        # one product with a small compressed matrix: launches and host work count
        dict(name="matvec_toeplitz2k_1", kind="matvec", family="toeplitz", n=2000, nrhs=1),
        # the paper's power method: one product per iteration with a matrix of its Table 3
        dict(name="matvec_qchem80k_1", kind="matvec", family="qchem", n=80000, nrhs=1),
        # a large system of small ranks, a block of right-hand sides
        dict(name="solve_toeplitz80k_16", kind="solve", family="toeplitz", n=80000, nrhs=16),
        # a request of the serving loop against a resident factorization (ranks in the hundreds)
        dict(name="solve_schur5k_32", kind="solve", family="schur", n=71 * 71, nrhs=32),
        # the serving loop's factorization of a new request, and its first right-hand sides
        dict(name="factor_schur10k", kind="factor", family="schur", n=100 * 100, nrhs=8),
        # many matrices of uneven size together: compress, factor, solve 16 right-hand sides
        dict(name="batch24_mixed", kind="batch", count=24, nmin=1000, nmax=8000, nrhs=16),
        # whole compressions: the smallest, an ordinary one, and the headline
        dict(name="compress_toeplitz2k", kind="compress", family="toeplitz", n=2000, nrhs=16),
        dict(name="compress_gauss20k", kind="compress", family="gauss", n=20000, nrhs=16),
        dict(name="compress_bem60k", kind="compress", family="bem", n=60000, nrhs=16),
        # the fused sampling products of a first pass: tensor cores, and plain FP32 (the default)
        dict(name="sample_bf16x3_20k_128", kind="sample", mode="bf16x3", dtype="f32", n=20000,
             cols=128, leaf=256),
        dict(name="sample_native_10k_64", kind="sample", mode="native", dtype="f32", n=10000,
             cols=64, leaf=256),
        # the interpolative decompositions of a leaf level (both sides of 32 nodes)
        dict(name="id_64x512x256", kind="id", count=64, m=512, d=256, rtol=1e-6, dtype="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec", "matvec", "solve", "solve", "factor", "batch", "compress",
                       "compress", "sample", "sample", "sample", "id"])
    if kind == "batch":   # continuous batches hold a few to a few dozen matrices
        return dict(kind=kind, count=rng.randint(3, 24), nmin=1000, nmax=_log_int(rng, 2000, 8000),
                    nrhs=rng.randint(1, 32))
    if kind == "sample":
        mode = rng.choice(["native", "native", "bf16x3", "bf16x2", "tf32"])
        dtype = rng.choice(["f32", "f64"]) if mode == "native" else "f32"
        return dict(kind=kind, mode=mode, dtype=dtype,
                    n=_log_int(rng, 1000, 8000 if dtype == "f64" else 20000),
                    cols=rng.randint(16, 128), leaf=rng.choice([64, 128, 256]))
    if kind == "id":
        m = _log_int(rng, 48, 700)
        return dict(kind=kind, count=_log_int(rng, 2, 128), m=m, d=rng.randint(32, min(m, 320)),
                    rtol=rng.choice([1e-4, 1e-6]), dtype=rng.choice(["f32", "f64"]))
    nrhs = rng.choice([1, 1, rng.randint(2, 8), rng.randint(9, 64)])
    if kind == "compress":
        fam = rng.choice(["toeplitz", "gauss", "bem"])
        lo, hi = {"toeplitz": (1000, 8000), "gauss": (2000, 20000), "bem": (3000, 20000)}[fam]
        return dict(kind=kind, family=fam, n=_log_int(rng, lo, hi), nrhs=16)
    if kind == "matvec":
        fam = rng.choice(["toeplitz", "qchem", "gauss"])
        hi = 20000 if fam == "gauss" else 80000
        return dict(kind=kind, family=fam, n=_log_int(rng, 1000, hi), nrhs=nrhs)
    fam = rng.choice(["toeplitz", "schur"])
    if fam == "schur":
        return dict(kind=kind, family=fam, n=rng.randint(32, 100) ** 2, nrhs=nrhs)
    return dict(kind=kind, family=fam, n=_log_int(rng, 1000, 80000), nrhs=nrhs)


# ------------------------------------------------------------------- inputs
def _gen(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _randn(shape, seed, dtype):
    return torch.randn(shape, generator=_gen(seed), device="cuda", dtype=F64).to(dtype)


def _rcb(pts, leaf):
    """Points in recursive-coordinate-bisection order (the cluster tree's splits)."""
    perm = np.arange(len(pts))
    stack = [(0, len(pts))]
    while stack:
        lo, hi = stack.pop()
        if hi - lo <= leaf:
            continue
        sub = pts[perm[lo:hi]]
        axis = int(np.argmax(sub.max(axis=0) - sub.min(axis=0)))
        perm[lo:hi] = perm[lo:hi][np.argsort(sub[:, axis], kind="stable")]
        mid = lo + (hi - lo) // 2
        stack += [(lo, mid), (mid, hi)]
    return pts[perm]


def _points(family, n, leaf, seed):
    rng = np.random.default_rng(seed)
    if family == "gauss":
        pts = rng.random((n, 3))
    else:
        pts = rng.standard_normal((n, 3))
        pts /= np.linalg.norm(pts, axis=1, keepdims=True)
    return torch.as_tensor(_rcb(pts, leaf), device="cuda")


def _kernel_rows(family, x, r0, r1, h=0.2):
    """Rows [r0, r1) of a kernel matrix, FP64."""
    d2 = sum((x[r0:r1, a, None] - x[None, :, a]) ** 2 for a in range(3))
    at = (torch.arange(r1 - r0, device="cuda"), torch.arange(r0, r1, device="cuda"))
    if family == "gauss":
        k = torch.exp(-d2 / (2 * h * h))
        k[at] += 1.0
    else:
        d2[at] = 1.0
        k = 1.0 / (4 * math.pi * d2.sqrt())
        k[at] = math.sqrt(x.shape[0])
    return k


def _symbol(family, seed):
    """t(k) of a Toeplitz matrix a_ij = t(i - j); the seed moves the diagonal a little."""
    shift = 0.25 * float(np.random.default_rng(seed).random())

    def t(k):
        zero = k == 0
        if family == "toeplitz":
            return torch.where(zero, torch.full_like(k, 10.0 + shift), 1.0 / (1.0 + k.abs()))
        sgn = 1.0 - 2.0 * torch.remainder(k, 2.0)
        return torch.where(zero, torch.full_like(k, math.pi ** 2 / 6 + shift),
                           sgn / torch.where(zero, torch.ones_like(k), k * k))
    return t


def _toeplitz_product(t, n, X):
    """A X by a circulant embedding, FP64."""
    k = torch.arange(n, dtype=F64, device="cuda")
    c = torch.cat([t(k), k.new_zeros(1), t(-k)[1:].flip(0)])
    f = torch.fft.rfft(c)
    return torch.fft.irfft(f[:, None] * torch.fft.rfft(X.to(F64), n=2 * n, dim=0), n=2 * n, dim=0)[:n]


def _schur(n):
    k = math.isqrt(n)
    i = torch.arange(1, k + 1, dtype=F64, device="cuda")
    phi = math.sqrt(2.0 / (k + 1)) * torch.sin(torch.outer(i, i) * math.pi / (k + 1))
    mu = 2.0 - 2.0 * torch.cos(i * math.pi / (k + 1))
    a = 2.0 + mu[:, None] + mu[None, :]
    c = 1.0 / a
    for _ in range(k - 1):
        c = 1.0 / (a - c)
    M = torch.einsum("pq,iq,jq->pij", a - 2.0 * c, phi, phi).reshape(k, k * k)
    S = ((phi[:, None, :] * phi[None, :, :]).reshape(k * k, k) @ M)
    return S.reshape(k, k, k, k).permute(0, 2, 1, 3).reshape(n, n).to(torch.float32).contiguous()


def _dense(family, n, leaf, dtype, seed, h=0.2):
    if family == "schur":   # the seed sets the operator's zero-order term: S + shift I
        S = _schur(n)
        S.diagonal().add_(0.05 * float(np.random.default_rng(seed).random()))
        return S
    if family in ("toeplitz", "qchem"):
        t = _symbol(family, seed)
        i = torch.arange(n, dtype=F64, device="cuda")
        return t(i[:, None] - i[None, :]).to(dtype)
    x = _points(family, n, leaf, seed)
    A = torch.empty((n, n), dtype=dtype, device="cuda")
    for r0 in range(0, n, 2048):
        A[r0:r0 + 2048] = _kernel_rows(family, x, r0, min(n, r0 + 2048), h)
    return A


def _opts(family, seed, leaf=None):
    _, mode, lf, rtol, d0, step = SETTINGS[family]
    return P.hss_default_opts(leaf_size=leaf or lf, rtol=rtol, d0=d0, d_step=step,
                              sample_mode=mode, seed=seed)


def _handle(case, seed):
    """The compressed form that a program keeps: Toeplitz matrices through the
    matrix-free call (they need not be stored), the others from the dense matrix."""
    fam, n = case["family"], case["n"]
    dtype, _, leaf, _, _, _ = SETTINGS[fam]
    if fam not in ("toeplitz", "qchem"):
        return P.hss_compress(_dense(fam, n, leaf, dtype, seed), _opts(fam, seed))
    t = _symbol(fam, seed)

    def sample(R, Sr, Sc):
        Sr.copy_(_toeplitz_product(t, n, R))
        if Sc is not None:
            Sc.copy_(Sr)   # symmetric

    def extract(rows, cols, out):
        out.copy_(t(rows.double()[:, None] - cols.double()[None, :]))

    return P.hss_compress_matfree(n, sample, extract, dtype=dtype, opts=_opts(fam, seed))


def _batch_specs(case, seed):
    """Sizes, families and settings of a mixed batch: the sizes and families are the
    case's own, the seed moves the matrices' values."""
    rng = np.random.default_rng([case["count"], case["nmin"], case["nmax"], case["nrhs"]])
    out = []
    for q in range(case["count"]):
        n = int(rng.integers(case["nmin"], case["nmax"] + 1))
        out.append(dict(n=n, leaf=128 if n < 4000 else 256,
                        family="toeplitz" if rng.random() < 0.5 else "gauss",
                        h=float(rng.uniform(0.1, 0.4)), seed=seed * 1000 + q))
    return out


def _batch_opts(s):
    rtol, d0, step = (1e-6, 64, 32) if s["family"] == "toeplitz" else (1e-4, 128, 64)
    return P.hss_default_opts(leaf_size=s["leaf"], rtol=rtol, d0=d0, d_step=step,
                              sample_mode="bf16x3", seed=s["seed"])


def _id_inputs(case, seed):
    """Samples of far-field blocks: m points of a patch of the sphere against 1024
    points elsewhere, times a random matrix (rank well below m, decaying spectrum)."""
    rng = np.random.default_rng(seed)
    Ys = []
    for q in range(case["count"]):
        m = case["m"] - (37 * q) % (1 + case["m"] // 8)   # uneven sizes
        z = np.concatenate([0.4 * rng.standard_normal((m, 3)) + [0, 0, 1],
                            rng.standard_normal((1024, 3)) - [0, 0, 1.2]])
        x = torch.as_tensor(z / np.linalg.norm(z, axis=1, keepdims=True), device="cuda")
        K = 1.0 / (0.02 + torch.cdist(x[:m], x[m:], compute_mode="donot_use_mm_for_euclid_dist"))
        Y = K @ torch.randn((1024, case["d"]), generator=_gen(seed * 7919 + q), device="cuda", dtype=F64)
        Ys.append(Y.to(torch.float32 if case["dtype"] == "f32" else F64).contiguous())
    return Ys


def _sample_inputs(case, seed):
    n, c = case["n"], case["cols"]
    dtype = torch.float32 if case["dtype"] == "f32" else F64
    A = _dense("gauss", n, case["leaf"], dtype, seed)
    R = torch.empty((n, c), dtype=dtype, device="cuda")
    P.hss_random_gaussian(seed, n, 0, c, R)
    starts = list(range(0, n, case["leaf"])) + [n]
    return A, R, starts


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind in ("matvec", "solve", "factor"):
        dtype = SETTINGS[case["family"]][0]
        st["h"] = _handle(case, seed)
        st["X"] = _randn((case["n"], case["nrhs"]), seed + 1, dtype)
        if kind == "solve":
            P.hss_factor(st["h"])
    elif kind == "compress":
        dtype, _, leaf, _, _, _ = SETTINGS[case["family"]]
        st["A"] = _dense(case["family"], case["n"], leaf, dtype, seed)
        st["opts"] = _opts(case["family"], seed)
        st["X"] = _randn((case["n"], case["nrhs"]), seed + 1, dtype)
    elif kind == "batch":
        specs = _batch_specs(case, seed)
        st["As"] = [_dense(s["family"], s["n"], s["leaf"], torch.float32, s["seed"], s["h"])
                    for s in specs]
        st["opts"] = [_batch_opts(s) for s in specs]
        st["Bs"] = [_randn((s["n"], case["nrhs"]), s["seed"] + 1, torch.float32) for s in specs]
    elif kind == "sample":
        st["A"], st["R"], st["starts"] = _sample_inputs(case, seed)
        st["Sr"], st["Sc"] = torch.empty_like(st["R"]), torch.empty_like(st["R"])
        st["mode"] = case["mode"]
    else:
        st["Ys"] = _id_inputs(case, seed)
        st["rtol"] = case["rtol"]
        # the generators of every rank, end to end in one buffer
        st["E"] = torch.zeros(sum(y.shape[0] * min(y.shape) for y in st["Ys"]), dtype=F64, device="cuda")
    return st


def run(st):
    kind = st["kind"]
    if kind == "matvec":
        return P.hss_matvec(st["h"], st["X"])
    if kind == "solve":
        return P.hss_solve(st["h"], st["X"])
    if kind == "factor":
        P.hss_factor(st["h"])
        return P.hss_solve(st["h"], st["X"])
    if kind == "compress":   # the compressed form is opaque: its action on a block is what it holds
        h = P.hss_compress(st["A"], st["opts"])
        return P.hss_matvec(h, st["X"])
    if kind == "batch":
        hs, _ = P.hss_compress_batched(st["As"], st["opts"])
        P.hss_factor_batched(hs)
        return P.hss_solve_batched(hs, st["Bs"])[0]
    if kind == "sample":
        P.hss_sample(st["A"], st["R"], 0, st["R"].shape[1], st["Sr"], st["Sc"], st["starts"], st["mode"])
        return {"Sr": st["Sr"], "Sc": st["Sc"]}
    out = P.hss_id_batched(st["Ys"], st["rtol"])   # [(k, perm, E)] per matrix
    E = torch.cat([e.reshape(-1) for _, _, e in out])
    st["E"][:E.numel()] = E
    return {"k": np.array([k for k, _, _ in out], dtype=np.int64),
            "perm": torch.cat([p for _, p, _ in out]), "E": st["E"]}


# ------------------------------------------------------------ work and values
def _rank(family, n):
    """A typical generator rank of the family at these settings (for counting only)."""
    return {"toeplitz": 2.0 * math.log2(n), "qchem": 0.6 * math.sqrt(n), "gauss": 220,
            "bem": 0.9 * n ** 0.7, "schur": 6.5 * math.sqrt(n)}[family]


def _form(family, n):
    """(entries of the compressed form, leaves, leaf order, rank): D of every leaf, and per
    non-root node E of both sides and B, with ranks that halve with the level's block
    side until they meet the leaf's."""
    _, _, leaf, _, _, _ = SETTINGS[family]
    leaves = 1 << max(0, math.ceil(math.log2(n / leaf)))
    lo = n / leaves
    top, ent, nodes = _rank(family, n), n * lo, leaves
    while nodes > 1:
        r = min(lo / 3 if family in ("toeplitz", "qchem") else lo / 2, top)
        r = r if family in ("toeplitz", "qchem") else max(r, top / math.sqrt(nodes))
        m = min(n / nodes, 2 * r)
        ent += nodes * (2 * max(m - r, 0) * r + r * r)
        nodes //= 2
    return ent, leaves, lo, top


def _compress_work(family, n, es):
    top = _rank(family, n)
    return n * n * es, 4.0 * n * n * (top + 10)


def work(case):
    kind = case["kind"]
    if kind == "sample":
        n, c, es = case["n"], case["cols"], 4 if case["dtype"] == "f32" else 8
        return dict(bytes=n * n * es + 3 * n * c * es, flops=4.0 * n * n * c)
    if kind == "id":
        es, cnt, m, d = 4 if case["dtype"] == "f32" else 8, case["count"], 0.94 * case["m"], case["d"]
        k = min(m, d, 64.0)
        steps = 4 * (k * d * m - (d + m) * k * (k - 1) / 2 + (k - 1) * k * (2 * k - 1) / 6)
        return dict(bytes=cnt * (m * d * es + (m - k) * k * 8 + 4 * m),
                    flops=cnt * (steps + (m - k) * k * k))
    if kind == "batch":
        b = f = 0.0
        for s in _batch_specs(case, 0):
            n = s["n"]
            r = 25.0 if s["family"] == "toeplitz" else 200.0
            ent = n * s["leaf"] + 4 * n * r
            b += 4.0 * n * n + 8 * n * case["nrhs"]
            f += 4.0 * n * n * (r + 10) + 2 * n * s["leaf"] ** 2 + 4 * ent * case["nrhs"]
        return dict(bytes=b, flops=f)
    fam, n, q = case["family"], case["n"], case["nrhs"]
    es = 8 if SETTINGS[fam][0] == F64 else 4
    if kind == "compress":
        b, f = _compress_work(fam, n, es)
        return dict(bytes=b + 2 * n * q * es, flops=f)
    ent, leaves, lo, top = _form(fam, n)
    if kind == "matvec":   # the form once, X in, the product out
        return dict(bytes=ent * es + 2 * n * q * es, flops=2.0 * ent * q)
    if kind == "solve":    # the factors have the form's order of magnitude, in FP64
        return dict(bytes=2 * ent * 8 + 2 * n * q * es, flops=4.0 * ent * q)
    # factor: an LQ of every node (order m, m - k rows) and the root's LU
    f, nodes, m = 0.0, leaves, lo
    while nodes >= 1:
        f += nodes * (4.0 / 3.0 if nodes > 1 else 2.0 / 3.0) * m ** 3
        nodes //= 2
        m = 2 * max(min(lo / 2, top), top / math.sqrt(max(nodes, 1)) if fam == "schur" else 0)
    return dict(bytes=ent * es + 2 * ent * 8 + 2 * n * q * es, flops=f + 4.0 * ent * q)


def exact(case, seed):
    kind = case["kind"]
    if kind == "id":
        return None   # the pivots decide E: there is no value without them
    if kind == "sample":
        A, R, starts = _sample_inputs(case, seed)
        R = R.to(F64)
        Sr, Sc = torch.zeros_like(R), torch.zeros_like(R)
        for a, b in zip(starts, starts[1:]):
            blk = A[a:b].to(F64)
            blk[:, a:b] = 0.0
            Sr[a:b] = blk @ R
            Sc += blk.T @ R[a:b]
        return {"Sr": Sr, "Sc": Sc}
    if kind == "batch":
        out = []
        for s in _batch_specs(case, seed):
            A = _dense(s["family"], s["n"], s["leaf"], torch.float32, s["seed"], s["h"]).to(F64)
            out.append(torch.linalg.solve(A, _randn((s["n"], case["nrhs"]), s["seed"] + 1,
                                                    torch.float32).to(F64)))
        return out
    fam, n = case["family"], case["n"]
    dtype, _, leaf, _, _, _ = SETTINGS[fam]
    X = _randn((n, case["nrhs"]), seed + 1, dtype).to(F64)
    if kind in ("matvec", "compress"):
        if fam in ("toeplitz", "qchem"):
            return _toeplitz_product(_symbol(fam, seed), n, X)
        A = _dense(fam, n, leaf, dtype, seed)
        return torch.cat([A[r:r + 4096].to(F64) @ X for r in range(0, n, 4096)])
    if fam == "schur":
        return torch.linalg.solve(_dense(fam, n, leaf, dtype, seed).to(F64), X)
    # Toeplitz, eigenvalues between 9 and 9 + 2 ln n: conjugate gradients with FFT products
    t = _symbol(fam, seed)
    x = torch.zeros_like(X)
    r = X.clone()
    p, rs = r.clone(), (r * r).sum(0)
    for _ in range(200):
        Ap = _toeplitz_product(t, n, p)
        a = rs / (p * Ap).sum(0)
        x += a * p
        r -= a * Ap
        new = (r * r).sum(0)
        if float((new / (X * X).sum(0)).max()) < 1e-31:
            break
        p = r + (new / rs) * p
        rs = new
    return x
