"""Performance cases: what a user of this library runs, from single building blocks to
whole solves, each through a public entry point.

A case is a dict of plain values whose "kind" names the entry point:

  lanczos     blanczos on a resident matrix, FP64, one restart cycle from a given start
              block (warm starts and fixed budgets; the dense case converges in it)
  lanczos_tol blanczos on a small matrix with its defaults, to the tolerance
  rsvd        rsvd (RandSVD), FP64, from a given start block
  backward    svd_backward of sigma and U adjoints
  orth        cgs_cqr2, the re-orthogonalisation of a block against a basis, FP64
  small_svd   the SVD of a projected matrix, leading right vectors
  spmm        CSR times a block, FP64 or FP32 values
  transpose   CSR of the transpose
  project     dense_mm on FP32 blocks (P^T Y or P M), the mixed form's products
  mm_split    mm_bf16x6, the mixed form's product with a dense A whose pieces are laid
              out once

The mixed form appears through its products, whose outputs are FP32.  A whole mixed
solve returns FP64 triplets of FP32-accurate subspaces.
"""

import math

import numpy as np
import torch

import paper_2403_06218_gb300 as tsvd

DEV = "cuda"


# ---- the cases ---------------------------------------------------------------------
def listed():
    return [
        # the benchmark's default solve: 100 triplets of a 20,000 x 20,000 FP64 matrix
        dict(name="solve dense 20k", kind="lanczos", m=20_000, n=20_000, d=0, k=100, b=128, r=4),
        # one cycle of the sparse benchmark matrix (10 entries a row, flat spectrum)
        dict(name="solve sparse 100k", kind="lanczos", m=100_000, n=100_000, d=10, k=64, b=64, r=9),
        # a small interactive solve to the default tolerance
        dict(name="solve small 512x256", kind="lanczos_tol", m=512, n=256, k=10, b=16, r=4),
        # RandSVD of the sparse benchmark matrix with its benchmark parameters
        dict(name="rsvd sparse 100k", kind="rsvd", m=100_000, n=100_000, d=10, k=64, p=64, q=3),
        # the paper's dense experiment: a tall matrix, a narrow block
        dict(name="rsvd dense 100k x 10k", kind="rsvd", m=100_000, n=10_000, d=0, k=10, p=6, q=2),
        # gradient with respect to the values of a sparse matrix with weighted rows
        dict(name="backward sparse", kind="backward", m=100_001, n=80_003, d=10, k=32),
        # one late block of a Lanczos cycle against the basis before it
        dict(name="orth 100k 512+64", kind="orth", q=100_000, s=512, b=64),
        # the projected matrix of the dense solve
        dict(name="small svd 512", kind="small_svd", n=512, b=128, nv=100),
        # power-law rows, a ragged block, FP32 values (ratings, graphs)
        dict(name="spmm power-law f32", kind="spmm", m=500_000, n=250_000, law="power", nnz=12_000_000, w=100, f32=True),
        # the transpose build that every sparse solve begins with
        dict(name="transpose power-law", kind="transpose", m=500_000, n=250_000, law="power", nnz=12_000_000),
        # the mixed form's projection of a block on a basis
        dict(name="project f32 500k", kind="project", q=500_003, s=512, b=128, trans=True),
        # the mixed form's product with a dense matrix
        dict(name="mm split 20k", kind="mm_split", m=20_000, n=20_000, w=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lanczos", "lanczos", "lanczos_tol", "rsvd", "rsvd", "backward", "orth", "small_svd", "spmm",
                       "transpose", "project", "mm_split"])
    if kind == "lanczos":
        if rng.random() < 0.5:  # dense, square to 2:1 either way
            n = _log(rng, 2_000, 14_000)
            b = rng.choice([32, 48, 64, 100, 128])
            r = rng.randint(3, min(8, 640 // b))
            return dict(kind=kind, m=int(n * math.exp(rng.uniform(-0.7, 0.7))), n=n, d=0, k=rng.randint(10, min(100, b * r // 3)),
                        b=b, r=r)
        b = rng.choice([16, 32, 50, 64])
        return dict(kind=kind, m=_log(rng, 20_000, 120_000), n=_log(rng, 20_000, 120_000), d=rng.randint(5, 20), k=b, b=b,
                    r=rng.randint(5, 9))
    if kind == "lanczos_tol":
        n = _log(rng, 128, 600)
        return dict(kind=kind, m=_log(rng, n, 2_000), n=n, k=rng.randint(5, 12), b=rng.choice([8, 16, 20]), r=rng.randint(4, 6))
    if kind == "rsvd":
        if rng.random() < 0.5:
            n = _log(rng, 2_000, 8_000)
            return dict(kind=kind, m=_log(rng, n, 60_000), n=n, d=0, k=rng.randint(8, 12), p=rng.randint(4, 8), q=rng.randint(1, 3))
        return dict(kind=kind, m=_log(rng, 20_000, 120_000), n=_log(rng, 20_000, 120_000), d=rng.randint(5, 20),
                    k=rng.randint(10, 64), p=rng.randint(10, 64), q=rng.randint(1, 3))
    if kind == "backward":
        return dict(kind=kind, m=_log(rng, 20_000, 120_000), n=_log(rng, 20_000, 120_000), d=rng.randint(5, 15),
                    k=rng.randint(8, 40))
    if kind == "orth":
        b = rng.choice([16, 33, 64, 100, 128])
        return dict(kind=kind, q=_log(rng, 5_000, 150_000), s=rng.choice([0, b, 3 * b, rng.randint(1, 512)]), b=b)
    if kind == "small_svd":
        b = rng.choice([16, 32, 48, 64, 96, 128])
        n = b * rng.randint(2, max(2, 576 // b))
        return dict(kind=kind, n=n, b=b, nv=rng.randint(min(b, n - 1) // 2, min(b, n - 1)))
    if kind in ("spmm", "transpose"):
        law = rng.choice(["power", "uniform"])
        m, n = _log(rng, 10_000, 500_000), _log(rng, 10_000, 250_000)
        c = dict(kind=kind, m=m, n=n, law=law, nnz=m * rng.randint(5, 20))
        return dict(c, w=_log(rng, 1, 128), f32=rng.random() < 0.5) if kind == "spmm" else c
    if kind == "project":
        return dict(kind=kind, q=_log(rng, 10_000, 500_000), s=rng.randint(16, 512), b=rng.randint(8, 128),
                    trans=rng.random() < 0.5)
    return dict(kind=kind, m=_log(rng, 2_000, 20_000), n=_log(rng, 2_000, 20_000), w=_log(rng, 8, 128))


# ---- inputs --------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, dtype=dtype, device=DEV)


def _reflect(X, U):
    """(I - 2 u_1 u_1^T) .. (I - 2 u_L u_L^T) X in place."""
    for u in U.flip(0):
        X.addr_(u, u @ X, alpha=-2.0)
    return X


def _units(g, count, n):
    u = _randn(g, count, n)
    return u / u.norm(dim=1, keepdim=True)


def _dense(g, m, n, sigma, reflectors=8):
    """H_U diag(sigma) H_V^T with seeded products of Householder reflectors."""
    A = torch.zeros(m, n, dtype=torch.float64, device=DEV)
    i = torch.arange(sigma.numel(), device=DEV)
    A[i, i] = sigma
    _reflect(A, _units(g, reflectors, m))
    _reflect(A.t(), _units(g, reflectors, n))
    return A


def _decay(n):
    """sigma_i = 1 / (1 + i)^1.5"""
    return torch.arange(1, n + 1, dtype=torch.float64, device=DEV).pow(-1.5)


def _paper_spectrum(n):
    """The paper's dense experiment: 10 down to 1e-14 over the first half."""
    i = torch.arange(n, dtype=torch.float64, device=DEV)
    return torch.where(i < n // 2, 10.0 ** (1.0 - 15.0 * i / (n // 2)), torch.full_like(i, 1e-14))


def _coo(g, m, n, law, nnz):
    """Sorted distinct (row, column) pairs."""
    if law == "uniform":  # the same number of entries in each row, one in each of d column ranges
        d = max(1, nnz // m)
        j = torch.arange(d, device=DEV)
        lo, hi = j * n // d, (j + 1) * n // d
        cols = lo + (torch.rand(m, d, generator=g, dtype=torch.float64, device=DEV) * (hi - lo)).long()
        return torch.arange(m, device=DEV).repeat_interleave(d), cols.reshape(-1)
    # power law: degrees ~ z^-2.1 up to 20,000, columns by a popularity that falls as rank^-1.27;
    # more pairs than wanted are drawn, as popular columns repeat, and nnz of the distinct ones kept
    z = torch.rand(m, generator=g, dtype=torch.float64, device=DEV).clamp_min(1e-12).pow(-1 / 1.1).clamp_max(20_000)
    deg = (z * (1.5 * nnz / float(z.sum()))).ceil().clamp_max(n // 2).long()
    rows = torch.arange(m, device=DEV).repeat_interleave(deg)
    u = torch.rand(rows.numel(), generator=g, dtype=torch.float64, device=DEV)
    rank = ((1 - u * (1 - float(n) ** -0.27)).pow(-1 / 0.27) - 1).long().clamp_(0, n - 1)
    perm = torch.randperm(n, generator=g, device=DEV)
    key = torch.unique(rows * n + perm[rank])
    while key.numel() < nnz:
        more = torch.randint(m * n, (2 * (nnz - key.numel()),), generator=g, device=DEV)
        key = torch.unique(torch.cat([key, more]))
    key = key[torch.randperm(key.numel(), generator=g, device=DEV)[:nnz]].sort()[0]
    return torch.div(key, n, rounding_mode="floor"), key % n


def _csr(rows, cols, vals, m):
    rp = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.bincount(rows, minlength=m).cumsum(0)
    return rp.int(), cols.int(), vals


def _sparse(g, m, n, law, nnz, dtype=torch.float64, scale=None):
    rows, cols = _coo(g, m, n, law, nnz)
    vals = _randn(g, rows.numel(), dtype=dtype)
    if scale is not None:
        vals = vals * scale[rows]
    return (*_csr(rows, cols, vals, m), rows)


class _Op:
    """A and A^T applied with torch, for exact() and the triplets that backward starts from."""

    def __init__(self, x, m, n):
        if "A" in x:
            self.a, self.at = x["A"], x["A"].t()
            return
        rp, ci, va, rows = x["csr"]
        order = torch.argsort(ci.long() * m + rows)
        t = _csr(ci.long()[order], rows[order], va.double()[order], n)
        self.a = torch.sparse_csr_tensor(rp, ci, va.double(), size=(m, n))
        self.at = torch.sparse_csr_tensor(*t, size=(n, m))


def _inputs(c, seed):
    """The plain inputs of a case (tensors and index arrays)."""
    g = _gen(seed)
    kind = c["kind"]
    x = {}
    if kind in ("lanczos", "rsvd"):
        m, n = c["m"], c["n"]
        if c["d"]:
            x["csr"] = _sparse(g, m, n, "uniform", m * c["d"])
        else:
            x["A"] = _dense(g, m, n, _decay(min(m, n)) if kind == "lanczos" else _paper_spectrum(min(m, n)))
        x["start"] = _randn(g, max(m, n), c["b"]) if kind == "lanczos" else _randn(g, min(m, n), c["k"] + c["p"])
    elif kind == "lanczos_tol":
        m, n = c["m"], c["n"]
        i = torch.arange(n, dtype=torch.float64, device=DEV)
        x["s"] = 2.0 ** (-i / 8)
        x["U"] = torch.linalg.qr(_randn(g, m, n))[0]
        x["V"] = torch.linalg.qr(_randn(g, n, n))[0]
        x["A"] = (x["U"] * x["s"]) @ x["V"].t()
    elif kind == "backward":
        m, n, k = c["m"], c["n"], c["k"]
        rank = torch.randperm(m, generator=g, device=DEV).double()
        x["csr"] = _sparse(g, m, n, "uniform", m * c["d"], scale=1 + 9 * (1 + rank).pow(-0.25))
        op = _Op(x, m, n)
        V = _randn(g, n, 2 * k)  # subspace iteration: the triplets of an earlier solve
        for _ in range(30):
            V = torch.linalg.qr(op.at @ (op.a @ V))[0]
        Q = torch.linalg.qr(op.a @ V)[0]
        u, s, vh = torch.linalg.svd((op.at @ Q).t() @ V)
        x["s"], x["U"], x["V"] = s[:k].contiguous(), (Q @ u)[:, :k].contiguous(), (V @ vh.t())[:, :k].contiguous()
        x["sb"], x["Ub"] = torch.ones(k, dtype=torch.float64, device=DEV), _randn(g, m, k)
    elif kind == "orth":
        q, s, b = c["q"], c["s"], c["b"]
        P = torch.zeros(q, s, dtype=torch.float64, device=DEV)
        P.fill_diagonal_(1.0)
        x["P"] = _reflect(P, _units(g, 16, q)) if s else P
        # columns of norms from 1 to 1e-3 with a component in the basis
        x["Y"] = _randn(g, q, b) * torch.logspace(0, -3, b, dtype=torch.float64, device=DEV)
        if s:
            x["Y"] += x["P"] @ _randn(g, s, b)
    elif kind == "small_svd":
        # the block bidiagonal matrix of one Lanczos cycle on a decaying spectrum
        n, b = c["n"], c["b"]
        sig = _decay(4 * n)[:, None]
        P, Pb = _lanczos(lambda X: sig * X, lambda X: sig * X, _randn(g, 4 * n, b), n // b)
        i = torch.arange(n, device=DEV) // b
        x["B"] = (Pb.t() @ (sig * P)) * ((i[:, None] == i) | (i[:, None] == i + 1))
    elif kind in ("spmm", "transpose"):
        f32 = c.get("f32", False)
        x["csr"] = _sparse(g, c["m"], c["n"], c["law"], c["nnz"], torch.float32 if f32 else torch.float64)
        if kind == "spmm":
            x["X"] = _randn(g, c["n"], c["w"], dtype=x["csr"][2].dtype)
    elif kind == "project":
        x["P"] = _randn(g, c["q"], c["s"], dtype=torch.float32)
        x["X"] = _randn(g, c["q"] if c["trans"] else c["s"], c["b"], dtype=torch.float32)
    else:
        x["A"] = _dense(g, c["m"], c["n"], _decay(min(c["m"], c["n"])))
        x["X"] = _randn(g, c["n"], c["w"], dtype=torch.float32)
    return x


def _lanczos(mul, tmul, start, r):
    """Orthonormal bases (right, left) of r blocks of the block Lanczos process."""
    Pb, P = torch.linalg.qr(start)[0], None
    L = Pb
    for i in range(r):
        W = tmul(L)
        for _ in range(2 if P is not None else 0):
            W = W - P @ (P.t() @ W)
        R = torch.linalg.qr(W)[0]
        P = R if P is None else torch.cat([P, R], 1)
        if i + 1 < r:
            W = mul(R)
            for _ in range(2):
                W = W - Pb @ (Pb.t() @ W)
            L = torch.linalg.qr(W)[0]
            Pb = torch.cat([Pb, L], 1)
    return P, Pb


# ---- what the harness calls --------------------------------------------------------------
def prepare(case, seed):
    """What a program holds before the call: the matrix and blocks on the GPU (and, for
    mm_split, the pieces of A laid out once)."""
    c = dict(case)
    x = _inputs(c, seed)
    if "csr" in x:
        x["M"] = tsvd.CsrMatrix(*x["csr"][:3], (c["m"], c["n"]))
        del x["csr"]
    elif c["kind"] == "mm_split":
        x["M"] = tsvd.bf16x3_split(x.pop("A"))
    elif "A" in x:
        x["M"] = x.pop("A")
    if c["kind"] == "lanczos_tol":
        x = {"M": x["M"]}
    x["c"] = c
    return x


def run(state):
    c, kind = state["c"], state["c"]["kind"]
    if kind == "lanczos":
        r = tsvd.blanczos(state["M"], c["k"], c["b"], c["r"], max_restarts=0, start_block=state["start"])
        return r.sigma, r.U, r.V
    if kind == "lanczos_tol":
        r = tsvd.blanczos(state["M"], c["k"], c["b"], c["r"])
        return r.sigma, r.U, r.V
    if kind == "rsvd":
        r = tsvd.rsvd(state["M"], c["k"], c["p"], c["q"], start_block=state["start"])
        return r.sigma, r.U, r.V
    if kind == "backward":
        return tsvd.svd_backward(state["M"], state["s"], state["U"], state["V"], state["sb"], state["Ub"])[0]
    if kind == "orth":
        return tsvd.cgs_cqr2(state["Y"], state["P"])[:3]
    if kind == "small_svd":
        nv = c["nv"]  # the other right vectors are not defined, the other left ones have no fixed sign
        U, s, V, _ = tsvd.small_svd(state["B"], nv)
        return U[:, :nv], s, V[:, :nv]
    if kind == "spmm":
        return tsvd.spmm(state["M"], state["X"])
    if kind == "transpose":
        t = tsvd.csr_transpose(state["M"])
        return t.row_ptr, t.col_idx, t.val
    if kind == "project":
        return tsvd.dense_mm(state["P"], state["X"], trans=c["trans"])
    return tsvd.mm_bf16x6(state["M"], state["X"])


def _nnz(c):
    return c["m"] * c["d"] if c.get("d") else c["m"] * c["n"]


def work(case):
    c, kind = case, case["kind"]
    if kind in ("lanczos", "lanczos_tol", "rsvd"):
        m, n, k, nnz = c["m"], c["n"], c["k"], _nnz(dict(case, d=case.get("d", 0)))
        a_bytes = nnz * (12 if c.get("d") else 8)
        if kind == "rsvd":
            w, t = k + c["p"], c["q"] + 1
            flops = t * (4 * nnz * w + 8 * (m + n) * w * w) + 2 * (m + n) * w * k
            start = min(m, n) * w
        else:
            b, r = c["b"], c["r"]
            s = b * r
            flops = 4 * nnz * s + (m + n) * (8 * b * b * r * (r - 1) // 2 + 8 * b * s) + 2 * (m + n) * s * k
            start = max(m, n) * b
        return {"bytes": a_bytes + 8 * (start + (m + n + 1) * k), "flops": flops}
    if kind == "backward":
        m, n, k, nnz = c["m"], c["n"], c["k"], _nnz(c)
        # 50 iterations of the complement solves: two products with A, one projection
        return {"bytes": nnz * 20 + 8 * k * (2 * m + n), "flops": 50 * (4 * nnz * k + 4 * m * k * k) + 4 * nnz * k}
    if kind == "orth":
        q, s, b = c["q"], c["s"], c["b"]
        return {"bytes": 8 * (q * s + 2 * q * b + s * b + b * b), "flops": 8 * q * s * b + 8 * q * b * b}
    if kind == "small_svd":
        n = c["n"]
        return {"bytes": 8 * n * (n + 2 * c["nv"] + 1), "flops": 12 * n * n * n}
    if kind == "spmm":
        e = 4 if c["f32"] else 8
        return {"bytes": c["nnz"] * (4 + e) + 4 * c["m"] + e * c["w"] * (c["m"] + c["n"]), "flops": 2 * c["nnz"] * c["w"]}
    if kind == "transpose":
        return {"bytes": 24 * c["nnz"] + 4 * (c["m"] + c["n"]), "flops": 0}
    if kind == "project":
        q, s, b = c["q"], c["s"], c["b"]
        return {"bytes": 4 * (q * s + q * b + s * b), "flops": 2 * q * s * b}
    m, n, w = c["m"], c["n"], c["w"]
    return {"bytes": 6 * m * n + 4 * w * (m + n), "flops": 2 * m * n * w}


# ---- the same results in 64 bits, with torch -----------------------------------------------
def _signed(U, s, V, k, by_u=False):
    """The sign convention: the largest entry of each vector of the shorter side is positive."""
    U, V = U[:, :k], V[:, :k]
    W = U if by_u else V
    sgn = torch.sign(W.gather(0, W.abs().argmax(0, keepdim=True)))
    return s[:k], U * sgn, V * sgn


def _svd(B):
    u, s, vt = np.linalg.svd(B.cpu().numpy())
    return tuple(torch.from_numpy(np.ascontiguousarray(t)).to(DEV) for t in (u, s, vt.T))


def _complement_cg(mul, s2, Q, rhs, iters=400):
    """Columns x_j of (s_j^2 I - G) x_j = (I - Q Q^T) rhs_j on the complement of span(Q)."""
    def proj(Z):
        return Z - Q @ (Q.t() @ Z)
    r = proj(rhs)
    x, p, rr = torch.zeros_like(r), r.clone(), (r * r).sum(0)
    stop = rr * 1e-28
    for _ in range(iters):
        if bool((rr <= stop).all()):
            break
        ap = proj(p * s2 - mul(p))
        a = torch.where(rr > stop, rr / (p * ap).sum(0), torch.zeros_like(rr))
        x, r = x + a * p, r - a * ap
        new = (r * r).sum(0)
        p = r + p * torch.where(rr > stop, new / rr, torch.zeros_like(rr))
        rr = new
    return proj(x)


def exact(case, seed):
    c, kind = case, case["kind"]
    x = _inputs(c, seed)
    if kind in ("lanczos", "rsvd"):
        op = _Op(x, c["m"], c["n"])
        a, at, swap = (op.a, op.at, False) if c["m"] >= c["n"] else (op.at, op.a, True)
        if kind == "lanczos":
            P, Pb = _lanczos(lambda X: a @ X, lambda X: at @ X, x["start"], c["r"])
            u, s, v = _svd(Pb.t() @ (a @ P))
        else:
            P = x["start"]
            for _ in range(c["q"] + 1):
                Pb = torch.linalg.qr(a @ P)[0]
                P = torch.linalg.qr(at @ Pb)[0]
            u, s, v = _svd((at @ Pb).t() @ P)
        U, V = Pb @ u[:, : c["k"]], P @ v[:, : c["k"]]
        return _signed(V, s, U, c["k"], by_u=True) if swap else _signed(U, s, V, c["k"])
    if kind == "lanczos_tol":
        return _signed(x["U"], x["s"], x["V"], c["k"])
    if kind == "backward":
        op = _Op(x, c["m"], c["n"])
        s, U, V, Ub = x["s"], x["U"], x["V"], x["Ub"]
        J, d = U.t() @ Ub, s[None, :] ** 2 - s[:, None] ** 2
        F = torch.where(d != 0, 1 / d, torch.zeros_like(d))
        C = (F * (J - J.t())) * s + torch.diag(x["sb"])
        Y = _complement_cg(lambda Z: op.a @ (op.at @ Z), s * s, U, Ub)
        rows, ci = x["csr"][3], x["csr"][1].long()
        return ((U @ C + Y * s)[rows] * V[ci]).sum(1) + (U[rows] * (op.at @ Y)[ci]).sum(1)
    if kind == "orth":
        Y, P = x["Y"], x["P"]
        H = P.t() @ Y
        W = Y - P @ H
        D = P.t() @ W
        Q, R = torch.linalg.qr(W - P @ D)
        sg = torch.sign(torch.diagonal(R))
        return Q * sg, H + D, R * sg[:, None]
    if kind == "small_svd":
        u, s, v = _svd(x["B"])
        _, U, V = _signed(u, s, v, c["nv"])
        return U, s, V
    if kind == "spmm":
        rp, ci, va, _ = x["csr"]
        return torch.sparse_csr_tensor(rp, ci, va.double(), size=(c["m"], c["n"])) @ x["X"].double()
    if kind == "transpose":
        rp, ci, va, rows = x["csr"]
        order = torch.argsort(ci.long() * c["m"] + rows)
        t = _csr(ci.long()[order], rows[order], va[order], c["n"])
        return t
    if kind == "project":
        P = x["P"].double()
        return (P.t() if c["trans"] else P) @ x["X"].double()
    return x["A"] @ x["X"].double()
