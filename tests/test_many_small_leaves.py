"""Leaves below 96 rows in such number that the lane-per-leaf QL takes them (six
per SM), and just fewer: residual and orthogonality on probes, both at the bound
of the large eigendecompositions' tests (1e-12 sqrt(n))."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402
from paper_2108_04209_gb300 import inputs  # noqa: E402
from oracle import dense  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf", [(17408, 17), (8704, 17), (31744, 31)])
def test_residual_and_orthogonality(n, leaf):
    h = inputs.hss_random(n, leaf, 2, seed=leaf)
    H = sdc.HSSMatrix(h)
    lam, F = H.eig(sdc.default_opts(tau=1e-10))
    X = inputs.normal_block(n, 3, seed=1)
    QX = F.apply_Q(torch.from_numpy(X).cuda())
    QLX = F.apply_Q(lam[:, None] * torch.from_numpy(X).cuda()).cpu().numpy()
    back = F.apply_Q(QX, trans=True).cpu().numpy()
    an = lam.abs().max().item()
    assert np.all(np.diff(lam.cpu().numpy()) >= 0)
    assert np.linalg.norm(dense.hss_matvec(h, QX.cpu().numpy()) - QLX) <= 1e-12 * np.sqrt(n) * an * np.linalg.norm(X)
    assert np.linalg.norm(back - X) <= 1e-12 * np.sqrt(n) * np.linalg.norm(X)
