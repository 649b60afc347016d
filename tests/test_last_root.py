"""The last root of a large problem, right of every pole, whose sums run over the
tree's node weights: its gap against quadruple precision.

The weights carry 1.6e-15 to 1.9e-15 (rms, whatever the level), the FP64 sums over
the boxes and the last step a few eps more: 1e-14 is about three of both together.
(Weights that lose as much on every level again gave 1.3e-14 to 1.9e-14 here.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402
from paper_2108_04209_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,seed", [(60001, 1), (60001, 2), (60001, 3), (100003, 4)])
def test_last_gap_vs_quadruple(m, seed):
    L = np.longdouble
    if np.finfo(L).nmant < 100:
        pytest.skip("long double is not quadruple precision here")
    b = inputs.secular_batch(1, m, m, seed=seed, cluster_frac=0)
    o, d, z = (torch.from_numpy(a).cuda() for a in (b.offsets, b.d, b.z))
    out = sdc.secular_batched(o, d, z, 1.0, sdc.default_opts(tau=1e-12))
    k = int(out["mk"][0]) - 1
    dk, zk = (out[q].cpu().numpy()[:k + 1].astype(L) for q in ("dk", "zk"))
    eta, org = L(float(out["eta"][k])), int(out["org"][k])
    t = (dk - dk[org]) - eta
    f, fp = 1 + np.sum(zk * zk / t), np.sum(zk * zk / t / t)
    assert abs(f / fp / eta) <= 1e-14
