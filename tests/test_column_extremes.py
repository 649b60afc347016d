"""Blocks of columns through the factors of rank-one steps where a column's
entries or the poles differ by many orders of magnitude: graded columns over a
tight cluster, non-finite entries,
and deflated rows of any value.

Reference and bound: the dense Qhat of the step's own outputs, (8 eps m + 1e-13
sqrt(m)) max|x| per entry (test_column_blocks)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402
from tests import parity as P  # noqa: E402

pytestmark = pytest.mark.gpu


def _factor(d, z, tau):
    """Factor of a batch (lists of poles and weights) and its dense Qhat per problem."""
    offs = np.concatenate([[0], np.cumsum([len(x) for x in d])]).astype(np.int64)
    o, dd, zz = (torch.from_numpy(a).cuda() for a in (offs, np.concatenate(d), np.concatenate(z)))
    fact = sdc.secular_batched(o, dd, zz, 1.0, sdc.default_opts(tau=tau))
    host = {k: (v.cpu().numpy() if v is not None else None) for k, v in fact.items()}
    g = [P.gpu_problem(host, offs, p) for p in range(len(d))]
    return offs, o, fact, g, [P.dense_qhat(x) for x in g]


def _apply(o, fact, X, trans, fmm):
    return sdc.apply_rank1(o, fact, torch.from_numpy(X).cuda(), trans=trans,
                           opts=sdc.default_opts(fmm_min_m=fmm)).cpu().numpy()


def _tol(m, x):
    return (8 * 2.0 ** -52 * m + 1e-13 * np.sqrt(m)) * np.abs(x).max(axis=0)


@pytest.mark.parametrize("fmm", [-1, 256], ids=["direct", "tree"])
@pytest.mark.parametrize("gap", [-40, -36, -30])
def test_graded_columns_over_a_tight_cluster(gap, fmm):
    """512 of 1024 poles a gap of 2^-30 to 2^-40 of the spread apart, boxes of the
    cluster with entries 2^-20 to 2^-45 of the column's largest: their far boxes
    are near in position, so small weights still count."""
    rng = np.random.default_rng(5)
    m = 1024
    d = np.sort(np.concatenate([0.25 + np.arange(512) * 2.0 ** gap, rng.uniform(0.3, 1.0, 511), [1.25]]))
    z = rng.standard_normal(m) / np.sqrt(m)
    offs, o, fact, g, Q = _factor([d], [z], 1e-30)
    assert g[0]["mk"] == m
    X = np.zeros((m, 12))
    for c in range(12):
        X[256:288, c] = 1.0                       # one box of the cluster, another far from it below
        X[384:416, c] = 2.0 ** -(20 + 2.25 * c)
        if c >= 6:
            X[:, c] = np.where(np.arange(m) < 300, X[:, c], 2.0 ** -(10 + 3 * c) * rng.standard_normal(m))
    for trans in (True, False):
        Y = _apply(o, fact, X, trans, fmm)
        ref = (Q[0].T if trans else Q[0]) @ X
        err = np.abs(Y - ref)
        assert np.all(err <= _tol(m, X)), (trans, err.max())


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("ncols", [3, 40])
def test_first_row_stays_in_its_problem(bad, ncols):
    """A NaN or infinity in the block's row 0 reaches the first problem's rows of
    its column only, every row of the others is as without it."""
    rng = np.random.default_rng(6)
    sizes = (33, 1, 2, 40, 700)
    d = [np.sort(rng.uniform(-1, 1, m)) for m in sizes]
    z = [rng.standard_normal(m) / np.sqrt(m) for m in sizes]
    offs, o, fact, g, Q = _factor(d, z, 1e-30)
    X = rng.standard_normal((int(offs[-1]), ncols))
    X[0, 1] = bad
    for fmm in (-1, 256):
        for trans in (True, False):
            Y = _apply(o, fact, X, trans, fmm)
            assert not np.any(np.isfinite(Y[:33, 1]))
            for p in range(1, len(sizes)):
                x, y = X[offs[p]:offs[p + 1]], Y[offs[p]:offs[p + 1]]
                ref = (Q[p].T if trans else Q[p]) @ x
                assert np.all(np.abs(y - ref) <= _tol(sizes[p], x)), (trans, p)


@pytest.mark.parametrize("fmm", [-1, 256], ids=["direct", "tree"])
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e12, 1e300])
def test_deflated_rows_keep_to_themselves(value, fmm):
    """The identity part of the factor: a deflated row passes its entry on unchanged
    and has no part in the kept rows, whose error stays relative to the kept
    entries."""
    rng = np.random.default_rng(7)
    sizes = (40, 900)
    d = [np.sort(rng.uniform(-1, 1, m)) for m in sizes]
    z = [rng.standard_normal(m) / np.sqrt(m) for m in sizes]
    for v in z:
        v[5::11] = 0.0                            # deflated without a rotation: rows 5, 16, ...
    offs, o, fact, g, Q = _factor(d, z, 1e-30)
    n = int(offs[-1])
    X0 = rng.standard_normal((n, 9))
    for trans in (True, False):
        X = X0.copy()
        gone = np.zeros(n, bool)                  # output rows of the deflated slots
        for p, q in enumerate(g):
            assert q["mk"] == sizes[p] - len(range(5, sizes[p], 11))
            slots = np.arange(q["mk"], q["m"])
            merged = np.argsort(q["perm"])[slots]
            X[offs[p] + (q["src"][slots] if trans else merged), 3] = value
            gone[offs[p] + (merged if trans else q["src"][slots])] = True
        Y = _apply(o, fact, X, trans, fmm)
        assert np.array_equal(Y[gone, 3], np.full(gone.sum(), value), equal_nan=True)
        for p, q in enumerate(Q):
            s = slice(int(offs[p]), int(offs[p + 1]))
            ref = (q.T if trans else q) @ X0[s]
            keep = ~gone[s]
            err = np.abs(Y[s] - ref)[keep]
            assert np.all(err <= _tol(sizes[p], X0[s])), (trans, p, err.max())


@pytest.mark.parametrize("fmm", [-1, 256], ids=["direct", "tree"])
def test_non_finite_column_leaves_the_others(fmm):
    """Columns beside one with a NaN or an infinity are those of the block without
    it to rounding: both sides sum the same terms (near, or the same nodes), each
    with 4 eps |C_ij| |x_i|, rows of Qhat have norm one, so 16 eps sqrt(m) max|x|
    covers both; an infinite entry gives signed infinities."""
    rng = np.random.default_rng(8)
    m = 1537
    d, z = np.sort(rng.uniform(-1, 1, m)), rng.standard_normal(m) / np.sqrt(m)
    offs, o, fact, g, Q = _factor([d], [z], 1e-30)
    X = rng.standard_normal((m, 9))
    ok = [c for c in range(9) if c != 4]
    for trans in (True, False):
        ref = _apply(o, fact, X, trans, fmm)
        Qt = Q[0].T if trans else Q[0]
        for bad in (np.nan, np.inf):
            Z = X.copy()
            Z[70, 4] = bad
            Y = _apply(o, fact, Z, trans, fmm)
            err = np.abs(Y - ref)[:, ok].max()
            assert err <= 16 * 2.0 ** -52 * np.sqrt(m) * np.abs(X).max(), (trans, bad, err)
            if fmm < 0 and bad == np.inf:
                assert np.array_equal(Y[:, 4], np.sign(Qt[:, 70]) * np.inf)
            else:
                assert not np.any(np.isfinite(Y[:, 4]))
