"""Split sums of many blocks (csrc/split.cuh) on the host: the error that the direct
sweep over 4000 poles leaves in a root's gap, against quadruple precision and
beside the FP64 form that it replaces (one Newton step from a truncated
single-precision reciprocal, terms of each side added up in order): the median over
400 roots is no larger."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_04209_gb300", "csrc")

HARNESS = r"""
#include "split.cuh"
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
typedef __float128 Q;
static double med(std::vector<double> v) { std::sort(v.begin(), v.end()); return v[v.size() / 2]; }
int main()
{
    const int m = 4000;
    std::mt19937_64 g(1);
    std::normal_distribution<double> N;
    std::uniform_real_distribution<double> U;
    std::vector<double> d(m), w(m), es, ed;
    for (auto &x : d) x = U(g);
    std::sort(d.begin(), d.end());
    double W = 0;
    for (auto &x : w) { const double z = N(g); x = z * z; W += x; }
    const FfScale s = ff_scale(d[0], d[m - 1], W);
    std::vector<ff_f4> sd(m);
    std::vector<ff_f2> sw(m);
    for (int j = 0; j < m; j++) { sd[j] = ff_pole(d[j], s); sw[j] = ff_weight(w[j], s.kw); }
    for (int rep = 0; rep < 400; rep++) {
        const int k = (int)(g() % (m - 1));
        long double lo = 0, hi = (long double)d[k + 1] - d[k];
        const long double D = hi;
        for (int i = 0; i < 70; i++) {
            const long double y = (lo + hi) / 2;
            long double f = 1;
            for (int j = 0; j < m; j++) f += w[j] / (((long double)d[j] - d[k]) - y);
            (f < 0 ? lo : hi) = y;
        }
        const int K = lo < D / 2 ? k : k + 1;
        const double y = (double)(K == k ? lo : lo - D);
        FfAcc A = {};
        const int k0 = k / 32 * 32, k1 = std::min(k0 + 31, m - 2);
        for (int c = 0; c < m; c += 1024) {
            const int cn = std::min(1024, m - c);
            ff_sweep(&sd[c], &sw[c], 0, cn, c, k, k0, k1, ff_point(d[K], y, s), A);
        }
        Q near = 0, all = 0, fp = 0;
        double psi = 0, phi = 0;
        for (int j = 0; j < m; j++) {
            const Q t = ((Q)d[j] - (Q)d[K]) - (Q)y, a = (Q)w[j] / t;
            all += a;
            fp += a / t;
            if (j != k && j != k + 1) near += a;
            const double td = (d[j] - d[K]) - y;
            int e;
            const float mf = (float)(std::floor(std::frexp(std::fabs(td), &e) * 16777216.0) / 16777216.0);
            double r = std::copysign(std::ldexp((double)(1.0f / mf), -e), td);
            r = std::fma(r, std::fma(-td, r, 1.0), r);
            (j <= k ? psi : phi) += w[j] * r;
        }
        const double den = std::fabs((double)(fp * (Q)y));
        es.push_back(std::fabs((double)(((Q)A.s + (Q)A.sl) * (Q)ff_pow2(s.kk + s.kw) - near)) / den);
        ed.push_back(std::fabs((double)((Q)(psi + phi) - all)) / den);
    }
    printf("%.3e %.3e\n", med(es), med(ed));
    return 0;
}
"""


def test_long_sweep_no_worse_than_fp64(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ is missing")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    r = subprocess.run([gxx, "-O2", "-ffp-contract=off", "-std=gnu++17", "-I", CSRC, str(src), "-o", str(exe),
                        "-lquadmath"], capture_output=True, text=True)
    if r.returncode != 0 and "quadmath" in r.stderr:
        pytest.skip("no quadruple precision library")
    assert r.returncode == 0, r.stderr[-2000:]
    split, fp64 = (float(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert 0 < split <= fp64, (split, fp64)
