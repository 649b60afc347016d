"""The checked build's guards on the permutation rows of the column kernels: a row
of the neighbouring problem in src or pinv (in range of the block, so that even an
unguarded read stays inside it) latches the index bit, for every column kernel that
reads it; the intact factor latches nothing.  In a child process with the checked
library."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import os
import numpy as np
import torch
import paper_2108_04209_gb300 as sdc
from paper_2108_04209_gb300 import _lib

assert os.path.basename(_lib.lib()._name) == "libsuperdc_check.so"
rng = np.random.default_rng(1)
for close in (False, True):                          # the split kernels, the FP64 loops
    sizes = (700, 900)
    d = [np.sort(rng.uniform(0, 1, m)) for m in sizes]
    if close:
        for x in d:
            x[300] = x[299] + 2.0 ** -45
    z = [rng.standard_normal(m) / 30 for m in sizes]
    offs = torch.tensor([0, 700, 1600]).cuda()
    fact = sdc.secular_batched(offs, torch.from_numpy(np.concatenate(d)).cuda(),
                               torch.from_numpy(np.concatenate(z)).cuda(), 1.0, sdc.default_opts(tau=1e-17))
    X = torch.from_numpy(rng.standard_normal((1600, 5))).cuda()
    for fmm in (-1, 256):
        for slot in (-1, 0, 17, 350, 699):           # -1: intact
            for trans in (True, False):
                f = {k: (v.clone() if v is not None else None) for k, v in fact.items()}
                if slot >= 0:
                    f["src"][slot] = 800             # a row of the second problem
                f["status"].zero_()
                sdc.apply_rank1(offs, f, X, trans=trans, opts=sdc.default_opts(fmm_min_m=fmm))
                got = int(f["status"].item())
                assert got == (0 if slot < 0 else _lib.DEV_INDEX), (close, fmm, slot, trans, got)
print("GUARDS_OK", flush=True)
"""


def test_foreign_rows_are_latched():
    env = dict(os.environ)
    env["SUPERDC_CHECKED"] = "1"
    env["PYTHONPATH"] = ROOT + (os.pathsep + env["PYTHONPATH"] if env.get("PYTHONPATH") else "")
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0 and "GUARDS_OK" in r.stdout, (r.stdout[-3000:], r.stderr[-3000:])
