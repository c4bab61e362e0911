"""The two steps of the persistent engine's partition (`csrc/persist_plan.h`),
compiled with g++: the split's slot ranges are those of the whole partition, and
the remote entries counted without the lists are the lists', on random consensus
structures and part counts in any order of the subsystems; lists built on
several threads (many slots) are those of a plain pass over the parts.

On the GPU: a request that does not fit in double precision falls back to the
automatic CTA count, with its iterates."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_09410_gb300", "csrc")

DRIVER = r"""
#include "persist_plan.h"
#include <cstdio>
#include <random>
using namespace opf;
static bool plain_lists(int P, const PersistParts &t, const std::vector<int> &soff, const std::vector<int> &segp,
                        const std::vector<int> &pk) {
    const int L = (int)pk.size();
    std::vector<int> part(L), at(L), rem, out(L, -1), seg(L), r0{0}, l0{0};
    std::vector<unsigned short> list;
    for (int q = 0, j = 0; q < P; ++q)
        for (int i = t.s0[q]; i < t.s0[q + 1]; ++i)
            for (int k = soff[t.sub[i]]; k < soff[t.sub[i] + 1]; ++k, ++j) {
                if (t.slot[j] != k) return false;
                part[pk[k]] = q;
                at[pk[k]] = j - t.k0[q];
            }
    for (int q = 0; q < P; ++q) {
        const int nk = t.k0[q + 1] - t.k0[q];
        std::vector<std::vector<int>> lists;
        std::vector<int> number(L, -1);
        for (int j = t.k0[q]; j < t.k0[q + 1]; ++j) {
            const int c0 = segp[t.slot[j]] >> 8, cnt = segp[t.slot[j]] & 255;
            seg[j] = 1;
            if (cnt == 1) continue;
            if (number[c0] < 0) {
                number[c0] = (int)lists.size();
                std::vector<int> e;
                for (int c = c0; c < c0 + cnt; ++c) {
                    if (part[c] == q) { e.push_back(at[c]); continue; }
                    e.push_back(nk + (int)rem.size() - r0[q]);
                    rem.push_back(c);
                    out[t.k0[part[c]] + at[c]] = c;
                }
                while (e.size() % 8) e.push_back(-1);
                for (size_t i = 0; i < e.size(); i += 8) lists.emplace_back(e.begin() + i, e.begin() + i + 8);
            }
            seg[j] = (number[c0] << 8) | cnt;
        }
        r0.push_back((int)rem.size());
        for (const auto &e : lists)
            for (int v : e) list.push_back((unsigned short)(v < 0 ? nk + r0[q + 1] - r0[q] : v));
        l0.push_back((int)(list.size() / 8));
    }
    return rem == t.rem && out == t.out && seg == t.seg && r0 == t.r0 && l0 == t.l0 && list == t.list;
}
int main() {
    std::mt19937 rng(5);
    for (int seed = 0; seed < 404; ++seed) {
        const bool many = seed >= 400;           // 36,000 and 66,000 slots: several threads
        const int S = many ? 6000 + 5000 * (seed & 1) : 1 + rng() % 60, G = many ? 20000 : 1 + rng() % 90,
                  P = many ? 1 + 60 * (seed - 400) : 1 + rng() % 20;
        std::vector<int> soff{0}, gk;
        for (int d = 0; d < S; ++d) {
            const int n = std::min<int>(G, 1 + rng() % 12);
            std::vector<int> g;
            if (many) {                          // neighbours share most globals
                for (int i = 0; i < n; ++i) g.push_back((d * 3 + 17 * i + (int)(rng() % 3 ? 0 : rng() % G)) % G);
                std::sort(g.begin(), g.end());
                g.erase(std::unique(g.begin(), g.end()), g.end());
            } else {
                g.resize(G);
                std::iota(g.begin(), g.end(), 0);
                std::shuffle(g.begin(), g.end(), rng);
                g.resize(n);
            }
            gk.insert(gk.end(), g.begin(), g.end());
            soff.push_back((int)gk.size());
        }
        const int L = (int)gk.size();
        std::vector<int> gstart(G + 1, 0), pk(L), segp(L), order(S);
        for (int g : gk) ++gstart[g + 1];
        for (int g = 0; g < G; ++g) gstart[g + 1] += gstart[g];
        std::vector<int> fill(gstart.begin(), gstart.end() - 1);
        for (int k = 0; k < L; ++k) {
            pk[k] = fill[gk[k]]++;
            segp[k] = (gstart[gk[k]] << 8) | (gstart[gk[k] + 1] - gstart[gk[k]]);
        }
        std::iota(order.begin(), order.end(), 0);
        if (seed & 1) std::shuffle(order.begin(), order.end(), rng);
        std::vector<double> cost(S);
        for (double &c : cost) c = 1.0 + rng() % 50;
        const PersistParts split = persist_split(P, S, order, cost, soff);
        const PersistParts all = persist_parts(P, S, order, cost, soff, segp, pk);
        if (split.s0 != all.s0 || split.k0 != all.k0 || split.sub != all.sub || all.k0[P] != L ||
            persist_remote(P, split, soff, segp) != (long long)all.rem.size() ||
            (P <= 200 && !plain_lists(P, all, soff, segp, pk))) {
            std::printf("FAIL seed %d\n", seed);
            return 1;
        }
    }
    std::printf("ok\n");
    return 0;
}
"""


def test_split_and_count(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-Wall", "-I", CSRC, str(tmp_path / "driver.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.rstrip().endswith("ok"), out.stdout


@pytest.mark.gpu
def test_unfit_request_keeps_the_automatic_plan():
    from paper_2310_09410_gb300 import opf, synth

    feeder = synth.make_feeder(1000, 690, 83, depth_max=60, p_single=0.7, seed=11)

    def solved(s, **how):
        s.reset()
        s.solve(eps_rel=0.0, max_iter=300, check_every=50, precision=opf.PREC_FP64, **how)
        return s.locals() + s.solution()

    with opf.Solver.from_feeder(feeder) as s:
        s.precompute()
        want = solved(s)
        for ctas in (2, 4, 64, 1, 0):            # 64 fits, in another order of the test's sums only
            got = solved(s, engine=opf.ENGINE_PERSISTENT, cluster=ctas)
            for a, b in zip(got, want):
                if ctas == 64:
                    assert np.allclose(a, b, rtol=1e-9, atol=1e-9)
                else:
                    assert np.array_equal(a, b)
