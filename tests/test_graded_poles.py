"""Trees over poles that the integer box intervals do not resolve: graded over
many orders of magnitude, most of them below 2^-60 of the spread.  The near lists
stay short (directly summed terms against those of uniform poles), and roots, zhat
and b keep the oracle's bounds."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402
from paper_2108_04209_gb300 import _lib, inputs  # noqa: E402
from tests import parity as P  # noqa: E402
from tests.test_gpu_secular import run_batch  # noqa: E402

pytestmark = pytest.mark.gpu


def _poles(m, kind, rng):
    if kind == "uniform":
        return np.sort(rng.uniform(0, 1, m))
    if kind == "graded":
        return np.sort(10.0 ** rng.uniform(-25, 0, m))
    # graded towards 0 from both sides
    return np.sort(np.concatenate([10.0 ** rng.uniform(-20, 0, m // 2), -10.0 ** rng.uniform(-20, 0, m - m // 2)]))


def _terms(d, z, tau):
    """Directly summed terms per root of the tree's secular sweeps."""
    L = _lib.lib()
    o = torch.tensor([0, len(d)]).cuda()
    dd, zz = torch.from_numpy(d).cuda(), torch.from_numpy(z).cuda()
    L.superdc_profile_reset()
    L.superdc_profile_enable(1)
    try:
        out = sdc.secular_batched(o, dd, zz, 1.0, sdc.default_opts(tau=tau))
    finally:
        L.superdc_profile_enable(0)
    n = ctypes.c_int64(0)
    L.superdc_profile_counter(b"fmm_secular_terms", ctypes.byref(n))
    L.superdc_profile_reset()
    assert int(out["fmm"][0]) == 1 and int(out["mk"][0]) == len(d)
    return n.value / len(d)


@pytest.mark.parametrize("kind,m", [("graded", 6000), ("graded", 20000), ("both_ends", 20000)])
def test_near_lists_stay_short(kind, m):
    """At most four times the terms of uniform poles (graded boxes see more
    neighbours, and their roots take more sweeps)."""
    rng = np.random.default_rng(4)
    z = rng.standard_normal(m)
    u = _terms(_poles(m, "uniform", rng), z, 1e-40)
    g = _terms(_poles(m, kind, rng), z, 1e-40)
    assert g <= 4 * u, (g, u)


@pytest.mark.parametrize("kind", ["graded", "both_ends"])
@pytest.mark.parametrize("m", [513, 1500, 2049])
def test_parity_with_the_oracle(kind, m):
    rng = np.random.default_rng(m)
    d = _poles(m, kind, rng)
    z = rng.standard_normal(m)
    tau = 1e-14
    b = inputs.SecularBatch(np.array([0, m], np.int64), d, z, 1.0)
    out = run_batch(b, tau)
    P.compare_problem(P.gpu_problem(out, b.offsets, 0), d, z, tau, mode=0)
