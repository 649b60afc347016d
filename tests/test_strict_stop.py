"""Stopping constants far below the default: the roots converge within the default
max_iter in about as many sweeps as FP64 sums take (mean 6.7 to 6.9 for these
batches; 8 allowed), through the direct kernels and the tree."""
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402
from paper_2108_04209_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmm", [-1, 256], ids=["direct", "tree"])
@pytest.mark.parametrize("stop_c", [1e-2, 1e-4, 1e-8, 1e-300])
def test_converges_within_the_default_sweeps(stop_c, fmm):
    b = inputs.secular_batch(10, 1000, 3000, seed=3)
    o, d, z = (torch.from_numpy(a).cuda() for a in (b.offsets, b.d, b.z))
    out = sdc.secular_batched(o, d, z, 1.0, sdc.default_opts(tau=1e-12, stop_c=stop_c, fmm_min_m=fmm))
    s = out["sweeps"]
    assert s[s > 0].double().mean().item() <= 8
