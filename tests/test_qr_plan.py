"""The TSQR trees of TT-rounding (csrc/qr_plan.h) never need more than their buffers hold.  The last QR's buffers are
laid out for kc n2 rows, before its rank r1 <= kc is known; every tree that some r1 then asks for is compared with what
was laid out: R factors, taus and X blocks of every level, and the number of levels.  Host arithmetic, compiled alone.
Then, on the GPU, sums that lose one rank where such a tree has more chunks than the one for kc n2 rows."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import test_gpu_tt_trees as T

W = T.W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2405_12301_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include <map>
#include "qr_plan.h"
using namespace wg;
// elements that lie between a buffer and the next one handed out
static std::vector<size_t> starts;
static size_t room(const double *p, size_t end)
{
    const size_t o = (size_t)p;
    auto it = std::upper_bound(starts.begin(), starts.end(), o);
    return ((it == starts.end() ? end : *it) - o) / sizeof(double);
}
int main()
{
    long long plans = 0, over = 0;
    auto check = [&](long long most, int k, int spc, int g, int n2, int kc) {
        QRPlan q;
        Bump bp;
        bp.base = (char *)4096;
        qr_take(bp, q, most, k, spc, g, k);
        starts.clear();
        for (auto &l : q.buf) {
            starts.push_back((size_t)l.tau);
            starts.push_back((size_t)l.R);
            if (l.X) starts.push_back((size_t)l.X);
        }
        std::sort(starts.begin(), starts.end());
        const size_t end = 4096 + bp.off;
        for (int r = 1; r <= kc; ++r) {
            qr_plan(q, (long long)r * n2, k, spc, g);
            ++plans;
            bool bad = q.L.size() > q.buf.size();
            for (size_t l = 0; l < q.L.size() && !bad; ++l) {
                const QRPlan::Level &v = q.L[l];
                bad = (size_t)v.C * v.sub * k > room(q.buf[l].tau, end) || (size_t)v.C * k * k > room(q.buf[l].R, end) ||
                      (l > 0 && (size_t)q.L[l - 1].C * k * k > room(q.buf[l].X, end)) || (l > 0 && v.m != (long long)q.L[l - 1].C * k);
            }
            bad = bad || !qr_bind(q, nullptr);
            if (bad && ++over <= 5)
                printf("k %d, %d sub-blocks, groups of %d: laid out for %d x %d rows, too small for %d x %d\n", k, spc, g, kc, n2, r, n2);
        }
    };
    {  // a plan beyond its buffers is told apart
        QRPlan q;
        Bump bp;
        qr_take(bp, q, 640, 32, 2, 2, 32);
        qr_plan(q, 640 + 64, 32, 2, 2);
        over += qr_bind(q, nullptr);
    }
    const int ks[] = {1, 2, 3, 4, 5, 8, 12, 16, 24, 31, 32, 33, 40, 57, 64, 65, 90, 96};
    const int kcs[] = {1, 2, 3, 7, 16, 31, 32, 33, 54, 55, 64, 72, 73, 94, 95, 96};
    for (int k : ks)
        for (int kc : kcs)
            for (int spc : {2, 3, 5, 16})
                for (int g : {2, 4})
                    for (int n2 = 1; n2 <= 1024; n2 += n2 < 160 ? 1 : n2 < 400 ? 7 : 41) check((long long)kc * n2, k, spc, g, n2, kc);
    for (int n2 : {4096, 65537, (1 << 20) - 1, 1 << 20}) check(96ll * n2, 96, 16, 2, n2, 96);
    printf("%lld plans, %lld beyond their buffers\n", plans, over);
    return over != 0;
}
"""


def test_no_tree_outgrows_its_buffers(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(MAIN)
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("n,ranks", [((64, 70, 40), [(28, 16), (27, 16)]),               # 60 chunks; 57 for all 55 ranks
                                     ((128, 44, 40), [(32, 11), (32, 11), (31, 10)])])   # 65 for 94 ranks, 62 for 95
def test_sum_that_loses_one_rank(W, n, ranks):
    rng = np.random.default_rng(n[0])
    terms = [(1.0, T.tt(rng, n, r, 1.0)) for r in ranks]
    terms[1][1][0][:, 0, 0] = terms[0][1][0][:, 0, 0]  # two of the sum's first-core columns are the same
    (G, _), = T.check(W, [terms], 1e-12)
    assert G[0].shape[2] == sum(r[0] for r in ranks) - 1
