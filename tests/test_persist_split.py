"""The two steps of the persistent engine's partition (`csrc/persist_plan.h`),
compiled with g++: the split's slot ranges are those of the whole partition, and
the remote entries counted without the lists are the lists', on random consensus
structures and part counts in any order of the subsystems.

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
int main() {
    std::mt19937 rng(5);
    for (int seed = 0; seed < 400; ++seed) {
        const int S = 1 + rng() % 60, G = 1 + rng() % 90, P = 1 + rng() % 20;
        std::vector<int> soff{0}, gk;
        for (int d = 0; d < S; ++d) {
            std::vector<int> g(G);
            std::iota(g.begin(), g.end(), 0);
            std::shuffle(g.begin(), g.end(), rng);
            const int n = std::min<int>(G, 1 + rng() % 12);
            gk.insert(gk.end(), g.begin(), g.begin() + n);
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
            persist_remote(P, split, soff, segp) != (long long)all.rem.size()) {
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
