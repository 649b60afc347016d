"""Adjoint of the rank-one step at the edges of its tiles: kept sizes around the
32 targets and 32 sources of a tile and the 256 of a pass, 1 to 17 columns (one or
two sum pairs per warp, passes of 8), several problems at once, a degenerate pair.

Reference: reverse mode through torch.linalg.eigh of diag(d) + z z^T in FP64, for a
loss that the signs of eigenvectors leave alone.  Poles are at least 1/2 apart, so
the factors 1/(lambda_k - lambda_l)^2 stay of order one and both sides carry a few
hundred eps of the largest gradient entry per pole: 1e-11 of it is asked."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402

pytestmark = pytest.mark.gpu


def _loss(lam, Y, c):
    return (torch.exp(-lam / c)[:, None] * Y * Y).sum()


@pytest.mark.parametrize("sizes", [(1, 2, 31, 32, 33), (255, 257), (64, 1, 300)], ids=str)
@pytest.mark.parametrize("ncols", [1, 2, 4, 5, 8, 9, 17])
def test_adjoint_vs_eigh(sizes, ncols):
    rng = np.random.default_rng(ncols + sum(sizes))
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d = np.concatenate([np.arange(m) + rng.uniform(0, 0.5, m) for m in sizes])
    z = np.concatenate([rng.choice([-1, 1], m) * rng.uniform(0.3, 1, m) for m in sizes])
    X = rng.standard_normal((int(offs[-1]), ncols))
    o = torch.from_numpy(offs).cuda()
    g = [torch.from_numpy(a).cuda().requires_grad_() for a in (d, z, X)]
    lam, Y = sdc.SecularEig.apply(o, *g, 1.0, 1e-14)
    c = float(max(sizes))
    got = [t.cpu() for t in torch.autograd.grad(_loss(lam, Y, c), g)]
    for p in range(len(sizes)):
        s = slice(int(offs[p]), int(offs[p + 1]))
        r = [torch.from_numpy(a[s]).requires_grad_() for a in (d, z, X)]
        w, Q = torch.linalg.eigh(torch.diag(r[0]) + torch.outer(r[1], r[1]))
        ref = torch.autograd.grad(_loss(w, Q.T @ r[2], c), r)
        for a, b in zip(got, ref):
            assert (a[s] - b).abs().max() <= 1e-11 * b.abs().max(), (p, sizes[p])


def test_degenerate_pair_stays_finite():
    """Two poles a rounding apart with one weight negligible: the pair counts as one
    eigenspace (no coupling), the rest is unaffected."""
    m = 70
    d = np.arange(m, dtype=np.float64)
    d[41] = np.nextafter(d[40], 1e9)
    z = np.full(m, 0.5)
    z[41] = 1e-9
    g = [torch.from_numpy(a).cuda().requires_grad_() for a in (d, z, np.ones((m, 3)))]
    lam, Y = sdc.SecularEig.apply(torch.tensor([0, m], device="cuda"), *g, 1.0, 1e-14)
    for t in torch.autograd.grad(_loss(lam, Y, 70.0), g):
        assert torch.isfinite(t).all()
