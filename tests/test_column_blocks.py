"""Blocks of columns through the factors of rank-one steps, Qhat^T X and Qhat X,
at the edges of the kernels' tiles: kept sizes around 16, 32, 64 and the tree's
threshold, 1 to 65 columns (tiles of 8, passes of 64), zero, huge and tiny
columns, an infinite one, and a problem whose poles are too close for the split
positions (FP64 loops).

Reference: the dense Qhat from the step's own outputs times X in FP64.  Each
entry of Qhat is at most one and has a relative error of a few eps on both sides;
the tensor-core sums carry 2^-55 of the largest column value per entry, so a sum
of m products differs by at most (8 eps m) max|x|, far fields (order 22) by 1e-13
of the same scale times sqrt(m)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402
from tests import parity as P  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 15, 16, 17, 31, 33, 63, 64, 65, 129, 511, 513, 2049)


def _step(sizes, close=None):
    rng = np.random.default_rng(3)
    d = [np.sort(rng.uniform(-1, 1, m)) for m in sizes]
    if close is not None:                                   # a gap of 2^-45 of the spread
        d[close][7] = d[close][6] + 2.0 ** -44
    z = [rng.standard_normal(m) / np.sqrt(m) for m in sizes]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    o, dd, zz = (torch.from_numpy(a).cuda() for a in (offs, np.concatenate(d), np.concatenate(z)))
    fact = sdc.secular_batched(o, dd, zz, 1.0, sdc.default_opts(tau=1e-30))
    host = {k: (v.cpu().numpy() if v is not None else None) for k, v in fact.items()}
    Q = [P.dense_qhat(P.gpu_problem(host, offs, p)) for p in range(len(sizes))]
    return offs, o, fact, Q, rng


def _check(offs, o, fact, Q, X, fmm):
    Xg = torch.from_numpy(X).cuda()
    for trans in (True, False):
        Y = sdc.apply_rank1(o, fact, Xg, trans=trans, opts=sdc.default_opts(fmm_min_m=fmm)).cpu().numpy()
        for p, q in enumerate(Q):
            x, y, m = X[offs[p]:offs[p + 1]], Y[offs[p]:offs[p + 1]], len(q)
            ref = (q.T if trans else q) @ x
            tol = (8 * 2.0 ** -52 * m + 1e-13 * np.sqrt(m)) * np.abs(x).max(axis=0)
            assert np.all(np.abs(y - ref) <= tol), (trans, p, m, np.abs(y - ref).max())


@pytest.mark.parametrize("fmm", [-1, 256], ids=["direct", "tree"])
@pytest.mark.parametrize("ncols", [1, 7, 8, 9, 16, 17, 24, 25, 33, 64, 65])
def test_columns_vs_dense(ncols, fmm):
    offs, o, fact, Q, rng = _step(SIZES, close=8)
    X = rng.standard_normal((int(offs[-1]), ncols))
    X[:, ncols // 2] *= 10.0 ** rng.integers(-150, 150)
    if ncols > 2:
        X[:, 0] = 0.0
        X[:, 2] *= 1e-300
    _check(offs, o, fact, Q, X, fmm)


def test_infinite_column_stays_in_its_column():
    offs, o, fact, Q, rng = _step((65, 513))
    X = rng.standard_normal((578, 9))
    X[70, 4] = np.inf
    Xg = torch.from_numpy(X).cuda()
    ok = [c for c in range(9) if c != 4]
    for trans in (True, False):
        Y = sdc.apply_rank1(o, fact, Xg, trans=trans).cpu().numpy()
        assert np.all(np.isfinite(Y[:, ok])) and np.all(np.isfinite(Y[:65, 4]))
        assert not np.any(np.isfinite(Y[65:, 4]))
    _check(offs, o, fact, Q, np.ascontiguousarray(X[:, ok]), -1)
