"""Deflation at the edges of its warp segments: sizes around 32 entries of a warp,
128 of the one-warp kernel and multiples of the CTA's segments, chains of rotations
across segments, almost everything deflated and nothing, few problems (1024
threads) and many (512).  Decisions, rotations and layout are those of the oracle's
sequential scan bit for bit."""
import numpy as np
import pytest

pytest.importorskip("torch")

from oracle import rank1 as orank  # noqa: E402
from paper_2108_04209_gb300 import inputs  # noqa: E402
from tests import parity as P  # noqa: E402
from tests.test_gpu_secular import run_batch  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 31, 32, 33, 63, 65, 127, 128, 129, 255, 257, 511, 513, 1023, 1025, 2049, 3333)


def _problem(m, kind, rng):
    d, z = np.sort(rng.uniform(-1, 1, m)), rng.standard_normal(m)
    if kind == "chains":                         # runs of equal poles of every length up to 70
        i = 0
        while i < m:
            n = int(rng.integers(1, 71))
            d[i:i + n] = d[i]
            i += n
    elif kind == "one_chain":
        d[:] = 0.25
    elif kind == "tiny_z":
        z[rng.random(m) < 0.95] *= 1e-20
    elif kind == "mixed":
        z[rng.random(m) < 0.3] = 0.0
        s = rng.random(m) < 0.5
        d[1:][s[1:]] = d[:-1][s[1:]] + 1e-14
    return np.sort(d), z


@pytest.mark.parametrize("kind", ["none", "chains", "one_chain", "tiny_z", "mixed"])
@pytest.mark.parametrize("many", [False, True], ids=["few", "many"])
def test_deflation_matches_sequential_scan(kind, many):
    rng = np.random.default_rng(len(kind) + many)
    sizes = [int(m) for m in rng.choice(SIZES[:13], 200)] if many else list(SIZES)
    probs = [_problem(m, kind, rng) for m in sizes]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    b = inputs.SecularBatch(offs, np.concatenate([p[0] for p in probs]), np.concatenate([p[1] for p in probs]), 1.0)
    tau = 1e-10
    out = run_batch(b, tau)
    for p in range(b.nprob) if not many else range(0, b.nprob, 5):
        d, z = b.problem(p)
        f = orank.rank1_step(d, z, tau)
        P.check_deflation(P.gpu_problem(out, b.offsets, p), f)
