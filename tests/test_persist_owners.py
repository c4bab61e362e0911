"""Owner form of the persistent grid engine.

On the CPU (`csrc/persist_plan.h`, compiled with g++): on random consensus
structures and part counts every subsystem and slot in exactly one part, a
part's globals its slots' distinct ones, every slot's index naming its global,
the owners' ranges covering every global once with their copies counted.

On the GPU, on instances whose globals have many copies (the automatic choice):
FP32 iterates are the cluster engine's bit for bit (the same sums in the same
order; an instance that the warp engine holds stays with the one-cluster form,
whose iterates are that engine's), FP64 iterates the oracle's after 100 iterations to 1e-10 (the bound of
the other engines), and a wait that can never end gives OPF_E_TIMEOUT."""
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
#include <set>
using namespace opf;
static int fail(const char *what, int seed) { std::printf("FAIL %s seed %d\n", what, seed); return 1; }
int main() {
    std::mt19937 rng(11);
    for (int seed = 0; seed < 400; ++seed) {
        const int G = 1 + (int)(rng() % 60), S = 1 + (int)(rng() % 40), P = 1 + (int)(rng() % S);
        std::vector<int> soff(S + 1, 0), gk;
        std::vector<double> cost(S);
        for (int d = 0; d < S; ++d) {
            const int n = 1 + (int)(rng() % 9);
            for (int r = 0; r < n; ++r) gk.push_back((int)(rng() % G));
            soff[d + 1] = (int)gk.size();
            cost[d] = n;
        }
        for (int g = 0; g < G; ++g) {                       // every global has a copy
            bool any = false;
            for (int x : gk) any = any || x == g;
            if (!any) { gk.push_back(g); soff[S] = (int)gk.size(); }
        }
        const int L = (int)gk.size();
        std::vector<int> gstart(G + 1, 0), pk(L), segp(L);
        for (int g : gk) ++gstart[g + 1];
        for (int i = 0; i < G; ++i) gstart[i + 1] += gstart[i];
        std::vector<int> fill(gstart.begin(), gstart.end() - 1);
        for (int k = 0; k < L; ++k) pk[k] = fill[gk[k]]++;
        for (int k = 0; k < L; ++k) segp[k] = (gstart[gk[k]] << 8) | (gstart[gk[k] + 1] - gstart[gk[k]]);
        const PersistOwners o = persist_owners(P, S, G, cost, soff, segp, pk, gk, gstart);
        const PersistParts &t = o.parts;
        std::set<int> subs(t.sub.begin(), t.sub.end());
        if ((int)t.sub.size() != S || (int)subs.size() != S || t.s0[P] != S || t.k0[P] != L) return fail("subsystems", seed);
        std::set<int> slots;
        for (int p = 0; p < P; ++p) {
            std::set<int> used, listed(t.rem.begin() + t.r0[p], t.rem.begin() + t.r0[p + 1]);
            int j = t.k0[p];
            for (int i = t.s0[p]; i < t.s0[p + 1]; ++i)
                for (int k = soff[t.sub[i]]; k < soff[t.sub[i] + 1]; ++k, ++j) {
                    slots.insert(k);
                    used.insert(gk[k]);
                    if (t.slot[j] != k || t.out[j] != pk[k]) return fail("slot", seed);
                    if (t.rem[t.r0[p] + (t.seg[j] >> 8)] != gk[k] || (t.seg[j] & 255) != (segp[k] & 255)) return fail("global", seed);
                }
            if (j != t.k0[p + 1] || used != listed || (int)listed.size() != t.r0[p + 1] - t.r0[p]) return fail("list", seed);
        }
        if ((int)slots.size() != L) return fail("slots", seed);
        if (o.g0[0] != 0 || o.g0[P] != G) return fail("owners", seed);
        for (int p = 0; p < P; ++p)
            if (o.g0[p + 1] < o.g0[p] || o.g0[p + 1] - o.g0[p] > o.most_globals ||
                gstart[o.g0[p + 1]] - gstart[o.g0[p]] > o.most_copies) return fail("owner range", seed);
    }
    std::puts("ok");
    return 0;
}
"""


def test_owner_partition(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "driver.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-Wall", "-I", CSRC, str(src), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout


# (globals, blocks, widest block); the first one fits the warp engine
SHAPES = [(60, 90, 60), (300, 240, 100), (900, 240, 100), (2000, 500, 80), (150, 12, 120)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
def test_owner_form_equals_cluster_engine(shape):
    from paper_2310_09410_gb300 import opf, synth

    g = synth.random_generic(71, n_global=shape[0], n_sub=shape[1], max_n=shape[2], p_free=0.3)

    def iterates(engine):
        with opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"]) as s:
            s.precompute()
            s.solve(rho=10.0, eps_rel=0.0, max_iter=700, check_every=50, precision=opf.PREC_FP32, engine=engine)
            return s.locals() + s.solution()

    try:
        want = iterates(opf.ENGINE_WARP)
    except opf.OPFError as e:
        assert e.code == opf.OPF_E_CAPACITY
        want = iterates(opf.ENGINE_CLUSTER)
    for a, b in zip(iterates(opf.ENGINE_AUTO), want):
        assert np.array_equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
def test_owner_form_matches_oracle(shape):
    from oracle import admm as oracle_admm, lindist
    from paper_2310_09410_gb300 import opf, synth

    g = synth.random_generic(72, n_global=shape[0], n_sub=shape[1], max_n=shape[2], p_free=0.3)
    ref = oracle_admm.admm(lindist.from_generic(g), rho=10.0, max_iter=100, check_every=0)
    with opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"]) as s:
        s.precompute()
        s.solve(rho=10.0, eps_rel=0.0, max_iter=100, check_every=20, precision=opf.PREC_FP64)
        xs, lam = s.locals()
        x, _ = s.solution()
    for got, want in ((xs, ref.xs), (lam, ref.lam), (x, ref.x)):
        assert np.max(np.abs(got - want)) <= 1e-10 * max(1.0, float(np.abs(want).max()))


@pytest.mark.gpu
def test_owner_form_bounded_wait():
    from paper_2310_09410_gb300 import opf, synth

    g = synth.random_generic(73, n_global=300, n_sub=240, max_n=100, p_free=0.3)
    with opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"]) as s:
        s.precompute()
        for precision in (opf.PREC_FP64, opf.PREC_FP32):
            with pytest.raises(opf.OPFError) as e:
                s.solve(rho=10.0, eps_rel=0.0, max_iter=100, check_every=50, precision=precision,
                        flags=opf.SOLVE_TEST_BARRIER_TIMEOUT)
            assert e.value.code == opf.OPF_E_TIMEOUT
            s.reset()
            s.solve(rho=10.0, eps_rel=0.0, max_iter=100, check_every=50, precision=precision)
            assert s.residuals()["iters"] == 100
