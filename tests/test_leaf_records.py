"""The rotation records of many small leaves: where they do not fit, the plan takes
the kernel that does without them instead of failing, with the same eigenvalues
(bound of the tests that compare two paths, 1e-10 ||A||)."""
import pytest

torch = pytest.importorskip("torch")

import paper_2108_04209_gb300 as sdc  # noqa: E402
from paper_2108_04209_gb300 import _lib, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture
def alloc_limit():
    yield _lib.lib().superdc_debug_alloc_limit
    _lib.lib().superdc_debug_alloc_limit(0)


@pytest.mark.parametrize("leaf", [17, 40])
def test_plan_without_room_for_the_records(alloc_limit, leaf):
    n = 1024 * leaf                                # six leaves per SM and more
    H = sdc.HSSMatrix(inputs.hss_random(n, leaf, 2, seed=leaf))
    ref, F = H.eig()
    torch.cuda.synchronize()
    assert alloc_limit(24 * leaf * n) == 0         # half of the records, 48 leaf bytes a row
    lam, G = H.eig()
    torch.cuda.synchronize()
    assert alloc_limit(0) == 0
    assert (lam - ref).abs().max().item() <= 1e-10 * ref.abs().max().item()
