"""The FP32-split secular sweep (csrc/split.cuh): its arithmetic on the host
against quadruple precision, and the GPU evaluators that use it against the
oracle where it can go wrong (chunk and box edges, poles too close for the
fixed-point parts, spreads and weights out of scale, tiny gaps and weights)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2108_04209_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_04209_gb300", "csrc")

HARNESS = r"""
#include "split.cuh"
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>
typedef __float128 Q;
static Q qabs(Q v) { return v < 0 ? -v : v; }
int main(int argc, char **argv)
{
    const int m = atoi(argv[1]), mode = atoi(argv[2]);
    double worst = 0, worst_low = 0;
    for (int rep = 0; rep < 20; rep++) {
        std::vector<double> d(m), w(m);
        for (auto &x : d) x = drand48();
        if (mode == 1) for (int i = 0; i + 8 < m; i += 24) for (int j = 1; j < 8; j++) d[i + j] = d[i] + 1e-10 * (j + 0.5 * drand48()) / 8;
        if (mode == 2) for (auto &x : d) x = 60 * x - 30;
        if (mode == 3) for (auto &x : d) x = 1e6 + x;
        std::sort(d.begin(), d.end());
        double W = 0;
        for (auto &x : w) { const double z = 2 * drand48() - 1; x = z * z * (drand48() < 0.2 ? 1e-14 : 1.0); W += x; }
        const FfScale s = ff_scale(d[0], d[m - 1], W);
        bool ok = s.ok;
        for (int j = 0; j + 1 < m; j++) ok = ok && ff_gap_ok(d[j], d[j + 1], s.kk);
        if (!ok) { rep--; continue; }
        std::vector<ff_f4> sd(m);
        std::vector<ff_f2> sw(m);
        for (int j = 0; j < m; j++) { sd[j] = ff_pole(d[j], s); sw[j] = ff_weight(w[j], s.kw); }
        for (int k = 0; k + 1 < m; k++) {
            const int K = drand48() < 0.5 ? k : k + 1;
            double y = 0.5 * (d[k + 1] - d[k]) * (drand48() < 0.5 ? drand48() : 1e-9 * drand48());
            if (K != k) y = -y;
            FfAcc A = {};
            const int lo = k / 32 * 32, hi = std::min(lo + 31, m - 2);
            ff_sweep(sd.data(), sw.data(), 0, m, 0, k, lo, hi, ff_point(d[K], y, s), A);
            Q ex = 0, ab = 0, ps = 0, dp = 0, dh = 0;
            for (int j = 0; j < m; j++) {
                if (j == k || j == k + 1) continue;
                const Q t = ((Q)d[j] - (Q)d[K]) - (Q)y, a = (Q)w[j] / t;
                ex += a; ab += qabs(a);
                if (j <= k) { ps += a; dp += a / t; } else dh += a / t;
            }
            if (ab == 0) continue;
            const double c1 = ff_pow2(s.kk + s.kw), c2 = ff_pow2(2 * s.kk + s.kw);
            worst = std::max(worst, (double)(qabs(((Q)A.s + (Q)A.sl) * (Q)c1 - ex) / ab));
            worst_low = std::max(worst_low, (double)(qabs((Q)A.psi * (Q)c1 - ps) / ab));
            worst_low = std::max(worst_low, (double)(qabs((Q)A.dpsi * (Q)c2 - dp) / (dp + dh)));
            worst_low = std::max(worst_low, (double)(qabs((Q)A.dphi * (Q)c2 - dh) / (dp + dh)));
        }
    }
    printf("%.3e %.3e\n", worst, worst_low);
    return 0;
}
"""


HARNESS2 = r"""
#include "split.cuh"
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>
typedef __float128 Q;
static Q qabs(Q v) { return v < 0 ? -v : v; }
int main(int argc, char **argv)
{
    const int m = atoi(argv[1]), clustered = atoi(argv[2]);
    double wb = 0, wz = 0, w2 = 0, wl = 0;
    for (int rep = 0; rep < 10; rep++) {
        std::vector<double> d(m), v(m), eta(m);
        std::vector<int> K(m);
        for (auto &x : d) x = 20 * drand48() - 10;
        if (clustered) for (int i = 0; i + 8 < m; i += 24) for (int j = 1; j < 8; j++) d[i + j] = d[i] + 1e-9 * (j + 0.5 * drand48()) / 8;
        std::sort(d.begin(), d.end());
        const FfScale s = ff_scale(d[0], d[m - 1], 1.0);
        bool ok = s.ok;
        for (int j = 0; j + 1 < m; j++) ok = ok && ff_gap_ok(d[j], d[j + 1], s.kk);
        if (!ok) { rep--; continue; }
        std::vector<ff_f4> D(m), V(m);
        std::vector<ff_w4> Dw(m), Lw(m);
        for (int j = 0; j < m; j++) {
            v[j] = (2 * drand48() - 1) * (drand48() < 0.2 ? 1e-7 : 1.0);
            const ff_t3 t = ff_split3(v[j]);
            V[j] = {t.a, t.b, t.c, 0.0f};
            D[j] = ff_pole(d[j], s);
            Dw[j] = ff_words4(ff_fixed(d[j], s.kk) - s.ref);
            if (j == m - 1) break;
            K[j] = drand48() < 0.5 ? j : j + 1;
            eta[j] = 0.5 * (d[j + 1] - d[j]) * (drand48() < 0.5 ? drand48() : 1e-9 * drand48());
            if (K[j] != j) eta[j] = -eta[j];
            Lw[j] = ff_words4(ff_fixed(d[K[j]], s.kk) + ff_fixed(eta[j], s.kk) - s.ref);
        }
        for (int j = 0; j + 1 < m; j++) {
            ff_t3 S = {};
            ff_sqr_sweep(D.data(), V.data(), m, 0, K[j], ff_point(d[K[j]], eta[j], s), S);
            Q ex = 0;
            for (int i = 0; i < m; i++) {
                if (i == K[j]) continue;
                const Q t = (((Q)d[i] - (Q)d[K[j]]) - (Q)eta[j]) * (Q)ff_pow2(s.kk);
                ex += (Q)v[i] * v[i] / t / t;
            }
            wb = std::max(wb, (double)qabs(((Q)S.a + (Q)S.b + (Q)S.c - ex) / ex));
        }
        for (int i = 0; i < m; i++) {
            FfProd n = {1ull << 63, 0}, e = n;
            const ff_u96 di = {Dw[i].lo, Dw[i].mid, Dw[i].hi};
            ff_prod_sweep(Dw.data(), Lw.data(), m - 1, 0, i, di, n, e);
            Q ex = 1;
            for (int j = 0; j + 1 < m; j++)
                if (j != i && j != i - 1) ex *= qabs((((Q)d[K[j]] - (Q)d[i]) + (Q)eta[j]) / ((Q)d[j] - (Q)d[i]));
            Q got = (Q)n.m / (Q)e.m;
            for (int k = n.e - e.e; k > 0; k--) got *= 2;
            for (int k = n.e - e.e; k < 0; k++) got /= 2;
            wz = std::max(wz, (double)qabs(got / ex - 1));
        }
        for (int i = 0; i + 1 < m; i++) {
            const ff_f2 w = ff_weight(v[i] * v[i], 0);
            float p, pl;
            ff_term2(D[i + 1], w, D[i], p, pl);
            const Q t = ((Q)d[i + 1] - (Q)d[i]) * (Q)ff_pow2(s.kk), ex = (Q)v[i] * v[i] / t / t;
            if ((double)ex > 1e-20) w2 = std::max(w2, (double)qabs(((Q)p + (Q)pl) / ex - 1));
        }
    }
    ff_logtab tab[128];
    for (int i = 0; i < 128; i++) {
        tab[i].c = ff_logc(i);
        const double l = -log((double)tab[i].c);
        tab[i].h = (float)l;
        tab[i].l = (float)(l - tab[i].h);
    }
    for (int i = 0; i < 20000; i++) {
        const double x = ldexp(0.5 + drand48(), (int)(12 * drand48()) - 6);
        const float t = (float)x, tl = (float)(x - t);
        float y, yl;
        ff_log(t, tl, 0, tab, y, yl);
        wl = std::max(wl, fabs(((double)y - log(x)) + (double)yl));
    }
    printf("%.3e %.3e %.3e %.3e\n", wb, wz, w2, wl);
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness2(tmp_path_factory):
    return _build(tmp_path_factory, HARNESS2)


@pytest.mark.parametrize("clustered", [0, 1])
@pytest.mark.parametrize("m", [2, 3, 9, 130])
def test_split_b_zhat_log_against_quadruple_precision(harness2, m, clustered):
    """Sums of squares and products with FP64's accuracy or better: the last bit
    of a position is 2^-94 of the spread, so at half the smallest accepted gap
    (2^-41) a difference is known to 2^-52, and each square doubles it: 2^-50; a
    product of m ratios adds at most 2 m 2^-54.  One-term
    1/(d - x)^2: 2^-44.  log: 2^-44 absolute for exponents up to 6."""
    out = subprocess.run([harness2, str(m), str(clustered)], capture_output=True, text=True, check=True).stdout.split()
    wb, wz, w2, wl = map(float, out)
    assert wb <= 2.0 ** -50
    assert wz <= 2 * m * 2.0 ** -54
    assert w2 <= 2.0 ** -44
    assert wl <= 2.0 ** -44


def _build(tmp_path_factory, text):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ missing")
    tmp = tmp_path_factory.mktemp("split")
    (tmp / "h.cpp").write_text(text)
    exe = str(tmp / "h")
    r = subprocess.run([gxx, "-O1", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, str(tmp / "h.cpp"), "-o", exe],
                       capture_output=True, text=True)
    if "__float128" in r.stderr:
        pytest.skip("no quadruple precision on this machine")
    assert r.returncode == 0, r.stderr[-2000:]
    return exe


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    return _build(tmp_path_factory, HARNESS)


@pytest.mark.parametrize("mode", [0, 1, 2, 3], ids=["uniform", "clustered", "wide", "offset"])
@pytest.mark.parametrize("m", [2, 3, 31, 33, 129, 700])
def test_split_sum_against_quadruple_precision(harness, m, mode):
    """Relative to the sum of the terms' magnitudes: at most 2^-43.5 (per term
    2^-47 from t, 2^-46 from the reciprocal and product, 2^-49 sqrt(m) from the
    additions, a factor of four for the worst of all roots); the single-precision
    sums at most m 2^-23."""
    if mode == 3 and m > 129:
        pytest.skip("poles at 1e6 + U[0,1] are closer than the accepted gap")
    out = subprocess.run([harness, str(m), str(mode)], capture_output=True, text=True, check=True).stdout.split()
    assert float(out[0]) <= 2.0 ** -43.5
    assert float(out[1]) <= max(4, m) * 2.0 ** -23


def _problems():
    rng = np.random.default_rng(17)
    n01 = rng.standard_normal
    probs = []
    for m in (2, 3, 33, 34, 65, 1023, 1024, 1025, 2050):          # windows of 32 roots, chunks of 1024 poles
        probs.append((np.sort(rng.uniform(-30, 30, m)), n01(m)))
    d = np.sort(rng.uniform(0, 1, 400))
    d[200] = d[199] + 3e-15                                         # closer than 2^-41 of the spread
    probs.append((np.sort(d), n01(400) * 1e-2))
    probs.append((np.geomspace(1e-10, 1e20, 400), n01(400)))         # graded: FP64 sweep
    z = n01(500)
    z[7] = 1e7                                                      # the last root far to the right
    probs.append((np.sort(rng.uniform(0, 1, 500)), z))
    z = n01(600)
    z[::3] *= 1e-9                                                  # gaps of 1e-20
    probs.append((np.sort(rng.uniform(-1, 1, 600)), z))
    probs.append((np.sort(1e5 + rng.uniform(0, 1, 200)), n01(200)))   # (the far field works on plain positions)
    offs = np.concatenate([[0], np.cumsum([len(p[0]) for p in probs])]).astype(np.int64)
    return inputs.SecularBatch(offs, np.concatenate([p[0] for p in probs]), np.concatenate([p[1] for p in probs]), 1.0)


@pytest.mark.gpu
@pytest.mark.parametrize("fmm", [-1, 256], ids=["direct", "fmm"])
@pytest.mark.parametrize("sched", [1, 2], ids=["whole", "pole_split"])
def test_split_sweep_vs_oracle(fmm, sched):
    pytest.importorskip("torch")
    from tests import parity as P
    from tests.test_gpu_secular import run_batch
    b = _problems()
    tau = 1e-120                                                    # nothing deflates
    out = run_batch(b, tau, fmm_min_m=fmm, sched=sched)
    assert out["status"][0] == 0
    for p in range(b.nprob):
        d, z = b.problem(p)
        P.compare_problem(P.gpu_problem(out, b.offsets, p), d, z, tau, mode=0)
