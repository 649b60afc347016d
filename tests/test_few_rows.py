"""The FMM threshold of eigendecompositions and factor applications with few
rows: the default leaves problems of 512 to 1535 kept entries to the direct
kernels, an explicit threshold still sends them through the tree.  Both
directions, ragged column counts, against the other path on the same factor
(bounds of the tests that compare the two paths, 1e-12 of the block's scale
times sqrt(n), and 1e-10 ||A|| for eigenvalues)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402
from paper_2108_04209_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(511, 512, 513, 40), (1535, 1536, 700), (2048, 1, 0, 1025)], ids=str)
def test_apply_default_vs_tree(sizes):
    rng = np.random.default_rng(sum(sizes))
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d = np.concatenate([np.sort(rng.uniform(-1, 1, m)) for m in sizes])
    z = np.concatenate([rng.standard_normal(m) / np.sqrt(max(m, 1)) for m in sizes])
    o, dd, zz = (torch.from_numpy(a).cuda() for a in (offs, d, z))
    fact = sdc.secular_batched(o, dd, zz, 1.0, sdc.default_opts(tau=1e-12))
    X = torch.from_numpy(rng.standard_normal((int(offs[-1]), 9))).cuda()
    tol = 1e-12 * X.abs().max().item() * np.sqrt(offs[-1])
    for trans in (True, False):
        Y = sdc.apply_rank1(o, fact, X, trans=trans)
        for fm in (512, -1):
            Z = sdc.apply_rank1(o, fact, X, trans=trans, opts=sdc.default_opts(fmm_min_m=fm))
            assert (Y - Z).abs().max().item() <= tol, (trans, fm)


@pytest.mark.parametrize("n,leaf", [(512, 32), (2048, 64), (3008, 47)])
def test_eig_default_vs_tree(n, leaf):
    h = inputs.hss_random(n, leaf, 4, seed=n)
    H = sdc.HSSMatrix(h)
    X = torch.from_numpy(inputs.normal_block(n, 17, seed=3)).cuda()
    lam, F = H.eig(sdc.default_opts(tau=1e-10))
    ref, G = H.eig(sdc.default_opts(tau=1e-10, fmm_min_m=512))
    assert F.get(0, 0, "fmm")[0] == (1 if n >= 1536 else 0) and G.get(0, 0, "fmm")[0] == 1
    an = ref.abs().max().item()
    assert (lam - ref).abs().max().item() <= 1e-10 * an
    tol = 1e-12 * X.abs().max().item() * np.sqrt(n)
    for f, l in ((F, lam), (G, ref)):
        Y = f.apply_Q(f.apply_Q(X, trans=True))
        assert (Y - X).abs().max().item() <= tol
