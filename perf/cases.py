"""Cases that stand for what a program does with this package.

Seven kinds of work, each through the public Python entry points:

  step       secular_batched on device tensors: a batch of rank-one eigenproblems diag(d) + z z^T
  host       secular_batched_host: the same from pinned host buffers and back
  apply      apply_rank1: Qhat^T X and Qhat Y for the factors of such a batch
  step_grad  SecularEig forward and backward (adjoint of the batched step)
  eig        HSSMatrix.eig: eigenvalues and structured eigenvectors of a symmetric HSS matrix
  func       EigFactor.apply_function: f(A) X (the structured Q applied both ways)
  train      HSSEig forward and backward: gradients of a loss with respect to the generators

The outputs of a whole eigendecomposition are those that the matrix determines (eigenvalues, f(A) X, the
gradient of v^T f(A) v): single eigenvectors of a nearly degenerate pair are not determined by it.
"""
import math
import random

import numpy as np
import torch

import paper_2108_04209_gb300 as sdc
from paper_2108_04209_gb300 import inputs

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # one small merge front: 16 problems, latency and launches count (the size of the package's smoke test)
        dict(name="step_small", kind="step", nprob=16, mlo=8, mhi=300, clusters=0.1),
        # a tree level of small nodes, all below the FMM threshold
        dict(name="step_direct", kind="step", nprob=2048, mlo=100, mhi=500, clusters=0.1),
        # the benchmark's batch: 4096 problems, sizes 32 to 2048, a tenth of the poles clustered
        dict(name="step_batch", kind="step", nprob=4096, mlo=32, mhi=2048, clusters=0.1),
        # the root merge of a large matrix: one odd-sized problem
        dict(name="step_root", kind="step", nprob=1, mlo=100003, mhi=100003, clusters=0.0),
        # a service that receives its problems on the host
        dict(name="host_batch", kind="host", nprob=777, mlo=32, mhi=2048, clusters=0.1),
        # eigenvector blocks of a batch: 19 columns (an odd count) forth and back
        dict(name="apply_batch", kind="apply", nprob=200, mlo=130, mhi=4001, clusters=0.1, cols=19),
        # gradients through a batch of merges, three columns each
        dict(name="step_grad", kind="step_grad", nprob=300, mlo=33, mhi=700, cols=3),
        # a small matrix (the package's n = 512 configuration)
        dict(name="eig_512", kind="eig", n=512, leaf=32, rank=4, clustered=False),
        # the clustered n = 16384 configuration: deflation at every level
        dict(name="eig_clustered", kind="eig", n=16384, leaf=64, rank=8, clustered=True),
        # the headline matrix: n = 131072, leaves of 128, rank 10
        dict(name="eig_large", kind="eig", n=131072, leaf=128, rank=10, clustered=False),
        # exp(-A/s) X on a block of 64 columns, the factor in hand
        dict(name="func_32768", kind="func", n=32768, leaf=128, rank=10, cols=64),
        # a training step with the adjoint configuration's leaves and rank; at half its n = 8192, where the
        # gradient's terms 1 / (eigenvalue gap) leave it determined to about 1e-11
        dict(name="train_4096", kind="train", n=4096, leaf=64, rank=6, cols=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "host", "apply", "step_grad", "eig", "eig", "func", "train"])
    if kind in ("step", "host"):
        mhi = _log_int(rng, 24, 120000)
        cap = 4000000 // (mhi if mhi > 2048 else mhi // 2 + 1)
        nprob = max(1, min(5000, _log_int(rng, 1, max(2, cap))))
        mlo = mhi if nprob == 1 else max(1, _log_int(rng, max(1, mhi // 60), mhi))
        return dict(kind=kind, nprob=nprob, mlo=mlo, mhi=mhi, clusters=rng.choice([0.0, 0.1, 0.1, 0.3]))
    if kind == "apply":
        mhi = _log_int(rng, 40, 6000)
        return dict(kind=kind, nprob=max(1, _log_int(rng, 1, 400000 // mhi)), mlo=max(1, mhi // 30), mhi=mhi,
                    clusters=rng.choice([0.0, 0.1]), cols=rng.randint(1, 40))
    if kind == "step_grad":
        mhi = _log_int(rng, 40, 1200)
        return dict(kind=kind, nprob=max(1, _log_int(rng, 1, 120000 // mhi)), mlo=max(2, mhi // 20), mhi=mhi,
                    cols=rng.randint(1, 8))
    lev = rng.randint(1, 9 if kind == "eig" else 7)
    leaf = rng.randint(17, 128)
    rank = rng.randint(1, 12)
    if kind == "eig":
        return dict(kind=kind, n=leaf << lev, leaf=leaf, rank=rank, clustered=rng.random() < 0.3)
    if kind == "func":
        return dict(kind=kind, n=leaf << lev, leaf=leaf, rank=rank, cols=rng.randint(1, 80))
    lev, rank = min(lev, 5), min(rank, 6)
    return dict(kind=kind, n=leaf << lev, leaf=leaf, rank=rank, cols=rng.randint(1, 2))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _offsets(case):
    """Problem sizes, a property of the case (uniform in [mlo, mhi])."""
    r = random.Random("%d %d %d" % (case["nprob"], case["mlo"], case["mhi"]))
    return np.concatenate([[0], np.cumsum([r.randint(case["mlo"], case["mhi"]) for _ in range(case["nprob"])])])


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _poles(off, clusters, g):
    """Sorted uniform poles per problem; a share of the runs of 8 consecutive ones within 1e-10 of each other."""
    total = int(off[-1])
    sizes = torch.as_tensor(np.diff(off), device=DEV)
    pid = torch.repeat_interleave(torch.arange(len(off) - 1, device=DEV), sizes)
    start = torch.as_tensor(off[:-1], device=DEV)[pid]

    def in_order(v):
        i = torch.argsort(v)
        return v[i[torch.argsort(pid[i], stable=True)]]

    d = in_order(torch.rand(total, dtype=F64, device=DEV, generator=g))
    if clusters > 0:
        run = (torch.arange(total, device=DEV) - start) // 8
        head = start + run * 8
        hit = torch.rand(total, dtype=F64, device=DEV, generator=g)[head] < clusters
        near = d[head] + 1e-10 * torch.rand(total, dtype=F64, device=DEV, generator=g)
        d = in_order(torch.where(hit, near, d))
    return d, pid


def _orthonormal(x):
    return torch.linalg.qr(x).Q


def _hss(case, seed):
    """Generators of a random symmetric HSS matrix, packed for HSSMatrix, and by node for the plain products."""
    g = _gen(seed)
    n, m, r = case["n"], case["leaf"], case["rank"]
    t = inputs.perfect_tree(n, m, r)
    nl, nn = n // m, int(t.nnodes)

    def normal(*s):
        return torch.randn(*s, dtype=F64, device=DEV, generator=g)

    if case.get("clustered"):
        # leaf spectra of fourfold clusters (width 1e-12), eigenvectors tilted slightly into the coupling space
        full = _orthonormal(normal(nl, m, m))
        U = full[:, :, :r].contiguous()
        mu = normal(nl, (m - r + 3) // 4).repeat_interleave(4, 1)[:, :m - r]
        mu = mu + 1e-12 * torch.rand(nl, m - r, dtype=F64, device=DEV, generator=g)
        S = 1e-5 * normal(nl, m, m)
        V = full @ torch.linalg.matrix_exp(S - S.mT)
        D = (V * torch.cat([normal(nl, r), mu], 1)[:, None, :]) @ V.mT
    else:
        D = normal(nl, m, m)
        U = _orthonormal(normal(nl, m, r)) if m >= r else normal(nl, m, r) / math.sqrt(r)
    D = 0.5 * (D + D.mT)
    Q = _orthonormal(normal(nn, 2 * r, r))
    B = normal(nn, r, r) * torch.pow(2.0, -torch.arange(r, dtype=F64, device=DEV))
    R = torch.zeros(nn, r, r, dtype=F64, device=DEV)
    inner = [i for i in range(nn) if t.lchild[i] >= 0 and i != t.root]
    if inner:
        k = torch.as_tensor(inner, device=DEV)
        R[torch.as_tensor(t.lchild[inner].astype(np.int64), device=DEV)] = Q[k, :r]
        R[torch.as_tensor(t.rchild[inner].astype(np.int64), device=DEV)] = Q[k, r:]
    return t, D, U, R, B


def _packed(D, U, R, B):
    """Column-major blocks back to back, the layout of HSSMatrix's tensors."""
    return tuple(x.mT.contiguous().reshape(-1) for x in (D, U, R, B))


def _scale(case):
    """The s of f(A) = exp(-A/s): about the spectral radius of the random leaves."""
    return math.sqrt(2.0 * case["leaf"]) + 4.0


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=dict(case))
    if kind in ("step", "host", "apply", "step_grad"):
        off = _offsets(case)
        total = int(off[-1])
        g = _gen(seed)
        d, pid = _poles(off, case.get("clusters", 0.0), g)
        z = torch.randn(total, dtype=F64, device=DEV, generator=g)
        offs = torch.as_tensor(off, dtype=torch.int64, device=DEV)
        s["opts"] = sdc.default_opts(tau=1e-12)
        if kind == "host":
            s["offs"] = torch.as_tensor(off, dtype=torch.int64).pin_memory()
            s["d"], s["z"] = d.cpu().pin_memory(), z.cpu().pin_memory()
            s["out"] = {k: torch.empty(total, dtype=torch.int32 if k == "org" else F64, pin_memory=True)
                        for k in ("lam", "eta", "org", "vhat", "bnorm")}
            s["out"]["status"] = torch.zeros(1, dtype=torch.int32, pin_memory=True)
            return s
        s["offs"], s["d"], s["z"] = offs, d, z
        if kind == "step":
            # a program that solves batch after batch keeps its output buffers, without the per-root diagnostics
            out = sdc.alloc_rank1_out(case["nprob"], total, d.device, sweeps=False)
            s["out"] = {k: v.zero_() for k, v in out.items() if v is not None and k != "fmm"}
        elif kind == "apply":
            s["fact"] = sdc.secular_batched(offs, d, z, 1.0, s["opts"])
            s["X"] = torch.randn(case["cols"], total, dtype=F64, device=DEV, generator=g).t()
        else:
            size = torch.as_tensor(np.diff(off), device=DEV).to(F64)
            s["z"] = (z / torch.sqrt(size)[pid]).requires_grad_()
            s["d"] = d.requires_grad_()
            s["X"] = torch.randn(case["cols"], total, dtype=F64, device=DEV, generator=g).t().requires_grad_()
        return s
    t, D, U, R, B = _hss(case, seed)
    packed = _packed(D, U, R, B)
    if kind == "train":
        s["tree"] = t
        s["gen"] = [x.requires_grad_() for x in packed]
        s["v"] = torch.randn(case["n"], case["cols"], dtype=F64, device=DEV, generator=_gen(seed + 1)).requires_grad_()
        return s
    s["H"] = sdc.HSSMatrix(t, tensors=packed)
    if kind == "func":
        s["lam"], s["F"] = s["H"].eig()
        s["X"] = torch.randn(case["cols"], case["n"], dtype=F64, device=DEV, generator=_gen(seed + 1)).t()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        return sdc.secular_batched(s["offs"], s["d"], s["z"], 1.0, s["opts"], out=s["out"], check=False)
    if kind == "host":
        return sdc.secular_batched_host(s["offs"], s["d"], s["z"], 1.0, s["opts"], out=s["out"])
    if kind == "apply":
        Y = sdc.apply_rank1(s["offs"], s["fact"], s["X"], trans=True)
        return [Y, sdc.apply_rank1(s["offs"], s["fact"], s["X"], trans=False)]
    if kind == "step_grad":
        lam, Y = sdc.SecularEig.apply(s["offs"], s["d"], s["z"], s["X"], 1.0, 1e-12)
        loss = (torch.exp(-lam)[:, None] * Y * Y).sum()
        return [lam.detach(), loss.detach(), *torch.autograd.grad(loss, (s["d"], s["z"], s["X"]))]
    if kind == "eig":
        lam, s["F"] = s["H"].eig()
        return lam
    if kind == "func":
        return s["F"].apply_function(torch.exp(-s["lam"] / _scale(case)), s["X"])
    lam, Y = sdc.HSSEig.apply(s["tree"], *s["gen"], s["v"], None)
    loss = (torch.exp(-lam / _scale(case))[:, None] * Y * Y).sum()
    return [lam.detach(), loss.detach(), *torch.autograd.grad(loss, (*s["gen"], s["v"]))]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# operations per kept root by fast summation: five sweeps of 64 neighbours (7 each) and a far field (250),
# then zhat and b (11 per neighbour); a problem of m roots needs no more than m neighbours
def _root_flops(m):
    near = np.minimum(m, 64.0)
    return 5 * (7 * near + np.where(m > 256, 250, 0)) + 11 * near


def _hss_steps(case):
    """(rows, problem size) of every rank-one step of the tree: each level runs rank steps over all n rows."""
    lev, m = int(round(math.log2(case["n"] // case["leaf"]))), case["leaf"]
    return [(case["n"], m << (k + 1)) for k in range(lev) for _ in range(case["rank"])]


def work(case):
    kind = case["kind"]
    if kind in ("step", "host", "apply", "step_grad"):
        size = np.diff(_offsets(case)).astype(np.float64)
        total, c = float(size.sum()), case.get("cols", 0)
        solve = float((size * _root_flops(size)).sum())
        use = float((size * np.minimum(size, 64.0)).sum())      # neighbours of all rows
        if kind == "step":
            return {"bytes": total * (16 + 6 * 8 + 3 * 4), "flops": solve}
        if kind == "host":
            return {"bytes": total * (16 + 4 * 8 + 4), "flops": solve}
        if kind == "apply":
            return {"bytes": total * (40 + 12 + 3 * 8 * c), "flops": 2 * use * (3 + 2 * c)}
        return {"bytes": total * (16 + 8 * c + 8 + 16 + 8 * c), "flops": solve + use * (20 + 12 * c)}
    n, m, r = case["n"], case["leaf"], case["rank"]
    nbytes = 8.0 * (n * m + n * r + 4 * r * r * (n // m) + n)
    solve = 4.0 * n * m * m                                      # leaf eigenproblems
    for rows, size in _hss_steps(case):
        solve += rows * (float(_root_flops(float(size))) + min(size, 64) * 2.0 * r)
    per_col = n * m * 2.0 + sum(rows * min(size, 64) * 2.0 for rows, size in _hss_steps(case))
    if kind == "eig":
        return {"bytes": nbytes, "flops": solve}
    if kind == "func":
        c = case["cols"]
        return {"bytes": 8.0 * (2 * n * c + n * m) + 52.0 * n * len(_hss_steps(case)), "flops": 2 * c * per_col}
    return {"bytes": 2 * nbytes, "flops": 3 * solve + 4 * case["cols"] * per_col}


# ---------------------------------------------------------------------------
# the same in plain 64-bit torch
# ---------------------------------------------------------------------------
def _bisect(off, d, z):
    """Eigenvalues of every diag(d) + z z^T by bisection on the gap to the nearer pole, problems of like size together."""
    size = np.diff(off)
    lam = torch.empty(int(off[-1]), dtype=F64, device=DEV)
    order = np.argsort(size)
    at = 0
    while at < len(order):
        end = at + 1
        while end < len(order) and (end + 1 - at) * float(size[order[end]]) ** 2 < 1.5e8:
            end += 1
        group, M = order[at:end], int(size[order[end - 1]])
        at = end
        if M == 0:
            continue
        col = np.arange(M)[None, :]
        ok = torch.as_tensor(col < size[group][:, None], device=DEV)
        idx = torch.as_tensor(np.minimum(off[group][:, None] + col, off[-1] - 1), device=DEV)
        D = torch.where(ok, d[idx], math.inf)
        W = torch.where(ok, z[idx] ** 2, 0.0)
        top = torch.where(ok, D, -math.inf).amax(1, keepdim=True) + W.sum(1, keepdim=True)
        right = torch.cat([D[:, 1:], torch.full_like(D[:, :1], math.inf)], 1)
        right = torch.where(torch.isfinite(right), right, top)
        rows = max(1, int(1.5e8 / (len(group) * M)))
        for a in range(0, M, rows):
            b = min(M, a + rows)
            left, step = torch.where(ok, D, 0.0)[:, a:b], torch.where(ok, right - D, 1.0)[:, a:b]

            def f(org, y):
                gap = (D[:, None, :] - org[:, :, None]) - y[:, :, None]
                return 1.0 + (W[:, None, :] / gap).sum(-1)

            low = f(left, 0.5 * step) >= 0
            org = torch.where(low, left, left + step)
            lo, hi = torch.where(low, 0.0, -0.5 * step), torch.where(low, 0.5 * step, 0.0)
            for _ in range(54):
                mid = 0.5 * (lo + hi)
                neg = f(org, mid) < 0
                lo, hi = torch.where(neg, mid, lo), torch.where(neg, hi, mid)
            lam[idx[:, a:b][ok[:, a:b]]] = (org + 0.5 * (lo + hi))[ok[:, a:b]]
    return lam


def _hss_mv(t, D, U, R, B, x):
    """A x for the HSS matrix of these generators, level by level."""
    nl, m, _ = D.shape
    k = x.shape[1]
    X = x.reshape(nl, m, k)
    kids = {}
    for lev in range(int(t.lmax)):
        ids = sorted((i for i in range(int(t.nnodes)) if t.level[i] == lev), key=lambda i: t.offset[i])
        kids[lev] = (torch.as_tensor([int(t.lchild[i]) for i in ids], device=DEV),
                     torch.as_tensor([int(t.rchild[i]) for i in ids], device=DEV))
    g = U.mT @ X
    up = {}
    for lev in range(int(t.lmax) - 1, -1, -1):
        c1, c2 = kids[lev]
        up[lev] = (g[0::2], g[1::2])
        if lev > 0:
            g = R[c1].mT @ g[0::2] + R[c2].mT @ g[1::2]
    f = None
    for lev in range(int(t.lmax)):
        c1, c2 = kids[lev]
        f1, f2 = B[c1] @ up[lev][1], B[c1].mT @ up[lev][0]
        if lev > 0:
            f1, f2 = f1 + R[c1] @ f, f2 + R[c2] @ f
        f = torch.stack([f1, f2], 1).reshape(-1, f1.shape[1], k)
    y = D @ X
    return (y if f is None else y + U @ f).reshape(-1, k)


def _exp_series(mv, x, s):
    """exp(-A/s) x by its Taylor series (the norm of A/s is about one)."""
    y, t = x, x
    for k in range(1, 40):
        t = mv(t) * (-1.0 / (s * k))
        y = y + t
    return y


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "host"):
        off = _offsets(case)
        if float((np.diff(off).astype(np.float64) ** 2).sum()) > 4e9:
            return None
        g = _gen(seed)
        d, _ = _poles(off, case["clusters"], g)
        lam = _bisect(off, d, torch.randn(int(off[-1]), dtype=F64, device=DEV, generator=g))
        return {"lam": lam}
    if kind == "apply":
        return None                     # the columns of a cluster's eigenvectors depend on what was deflated
    if kind == "step_grad":
        st = prepare(case, seed)
        off = _offsets(case)
        pid = torch.repeat_interleave(torch.arange(case["nprob"], device=DEV), torch.as_tensor(np.diff(off), device=DEV))
        d, z, X = st["d"], st["z"], st["X"]

        def mv(x):
            dot = torch.zeros(case["nprob"], x.shape[1], dtype=F64, device=DEV).index_add(0, pid, z[:, None] * x)
            return d[:, None] * x + z[:, None] * dot[pid]

        loss = (X * _exp_series(mv, X, 1.0)).sum()
        grads = torch.autograd.grad(loss, (d, z, X))
        lam = _bisect(off, d.detach(), z.detach())
        return [lam, loss.detach(), *grads]
    if case["n"] > 8192 and kind == "eig":
        return None
    t, D, U, R, B = _hss(case, seed)
    if kind == "eig":
        A = _hss_mv(t, D, U, R, B, torch.eye(case["n"], dtype=F64, device=DEV))
        return torch.linalg.eigvalsh(0.5 * (A + A.mT))
    s, cols = _scale(case), case["cols"]
    v = torch.randn(cols, case["n"], dtype=F64, device=DEV, generator=_gen(seed + 1)).t() if kind == "func" else \
        torch.randn(case["n"], cols, dtype=F64, device=DEV, generator=_gen(seed + 1))
    if kind == "func":
        return _exp_series(lambda x: _hss_mv(t, D, U, R, B, x), v, s)
    gen = [x.requires_grad_() for x in (D, U, R, B, v)]
    loss = (v * _exp_series(lambda x: _hss_mv(t, D, U, R, B, x), v, s)).sum()
    gD, gU, gR, gB, gv = torch.autograd.grad(loss, gen)
    gD = 0.5 * (gD + gD.mT)
    return [None, loss.detach(), *_packed(gD, gU, gR, gB), gv]
