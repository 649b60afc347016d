"""Order of the deflated slots where rotations move values far: a weight just
above tau next to one of order one takes its pole's place across every negligible
entry between them.  Layout against the oracle's sequential scan bit for bit, at
sizes around the kernel's warps, exchange phases and merge runs; and the time of
one value moved across a whole large problem."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rank1 as orank  # noqa: E402
import paper_2108_04209_gb300 as sdc  # noqa: E402
from paper_2108_04209_gb300 import inputs  # noqa: E402
from tests import parity as P  # noqa: E402
from tests.test_gpu_secular import run_batch  # noqa: E402

pytestmark = pytest.mark.gpu

TAU = 1e-10
SIZES = (3, 31, 33, 35, 64, 66, 127, 129, 131, 257, 1025, 2050, 4099)


def _problem(m, kind, rng):
    d = np.sort(rng.uniform(0, 0.4, m))
    z = np.zeros(m)
    if kind == "one":                              # the first value to the far end
        z[0], z[-1] = 1.0, 1.5 * TAU
    elif kind == "pairs":                          # values moved by every distance
        i = 0
        while i + 2 < m:
            n = int(rng.integers(2, 200))
            z[i], z[min(i + n, m) - 1] = 1.0, 1.5 * TAU
            i += n
    elif kind == "chain":                          # one long chain through negligible entries
        z[rng.random(m) < 0.3] = 1.2 * TAU
        z[0] = 1.0
    else:                                          # weights of every size, both zeros among the poles
        z = rng.choice([0.0, 1.0, 1.2 * TAU, 3 * TAU, 1e-6, -1.0], m, p=[0.6, 0.05, 0.2, 0.1, 0.03, 0.02])
        d[rng.random(m) < 0.2] = 0.0
        d = np.sort(d)
        d[(d == 0) & (rng.random(m) < 0.5)] = -0.0
    return d, z


@pytest.mark.parametrize("kind", ["one", "pairs", "chain", "any"])
@pytest.mark.parametrize("many", [False, True], ids=["few", "many"])
def test_order_matches_sequential_scan(kind, many):
    rng = np.random.default_rng(3 * len(kind) + many)
    sizes = [int(m) for m in rng.choice(SIZES[:11], 200)] if many else list(SIZES)
    probs = [_problem(m, kind, rng) for m in sizes]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    b = inputs.SecularBatch(offs, np.concatenate([p[0] for p in probs]), np.concatenate([p[1] for p in probs]), 1.0)
    out = run_batch(b, TAU)
    for p in range(b.nprob) if not many else range(0, b.nprob, 5):
        d, z = b.problem(p)
        P.check_deflation(P.gpu_problem(out, b.offsets, p), orank.rank1_step(d, z, TAU))


def test_far_value_costs_no_pass_per_entry():
    """One value moved across 30000 entries takes a few times the step without it
    (a pass over the slots per entry took a hundred)."""
    n = 30000
    o = torch.tensor([0, n]).cuda()
    d = torch.linspace(0, 0.4, n, dtype=torch.float64).cuda()
    t = []
    for last in (0.0, 1.5 * TAU):
        z = torch.zeros(n, dtype=torch.float64)
        z[0], z[-1] = 1.0, last
        z = z.cuda()
        out = sdc.alloc_rank1_out(1, n, d.device)
        best = np.inf
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sdc.secular_batched(o, d, z, 1.0, sdc.default_opts(tau=TAU), out=out, check=False)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        t.append(best)
    assert t[1] <= 4 * t[0] + 1.0, t
