"""Weights whose squares reach the end of the exponent range: the step returns (the
roots of subnormal squares keep their guess), and every gap of a normal square is the
one-pole value z_k^2 / (1 + sum_{j != k} z_j^2 / (d_j - d_k)) that a weight far below
its neighbours' distances gives (relative 1e-9: terms of second order are below 1e-60
here, the sum has a few hundred eps)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmm", [-1, 256], ids=["direct", "tree"])
@pytest.mark.parametrize("m", [31, 64, 129])
def test_tiny_squares(m, fmm):
    rng = np.random.default_rng(m)
    d = np.sort(rng.uniform(-1, 1, m))
    z = rng.standard_normal(m) * 10.0 ** rng.uniform(-160, 0, m)
    o, dd, zz = (torch.from_numpy(a).cuda() for a in (np.array([0, m]), d, z))
    out = sdc.secular_batched(o, dd, zz, 1.0, sdc.default_opts(tau=1e-300, fmm_min_m=fmm), check=False)
    assert int(out["status"][0]) == 0 and int(out["mk"][0]) == m
    eta, org, w = out["eta"].cpu().numpy(), out["org"].cpu().numpy(), z * z
    k = np.array([i for i in range(m - 1) if 1e-290 < w[i] < 1e-40])
    rest = np.array([1 + sum(w[j] / (d[j] - d[i]) for j in range(m) if j != i) for i in k])
    k, rest = k[rest > 1e-3], rest[rest > 1e-3]   # a negative rest: the root lies left of its pole
    assert len(k) > m // 4 and np.array_equal(org[k], k)
    assert np.all(np.abs(eta[k] - w[k] / rest) <= 1e-9 * w[k] / rest)
