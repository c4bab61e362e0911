"""Partition of the persistent grid engine (`csrc/persist_plan.h`), compiled
with g++ and checked on the CPU: on random consensus structures and part
counts (one part, more parts than subsystems), every subsystem and slot in
exactly one part and in decreasing size there, every global's copy list
reading exactly its copies in copy order through the part's own slots and its
remote entries (padded with the zero's index), the exported slots exactly those
another part reads, and an export's destinations exactly its readers' entries.
A planted wrong list entry fails it.

On the GPU: the engine's two forms (one slot per thread; several, where a
part has more than 512 slots) on consensus instances with wide, rank-deficient
and free blocks, against the oracle's iterates after 100 iterations (1e-10 in
FP64; 1e-4 in FP32, the bounds of the other engines)."""
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
static int fail(const char *what, int seed) { std::printf("FAIL %s seed %d\n", what, seed); return 1; }

static int check_dests(const PersistParts &t, int P, const std::vector<int> &uslot, int seed) {
    const PersistDests d = persist_dests(P, t, uslot);
    size_t n = 0;
    for (int p = 0; p < P; ++p)
        for (int j = t.k0[p]; j < t.k0[p + 1]; ++j) {
            const int o = d.d0[p] + (d.dseg[j] >> 8), cnt = d.dseg[j] & 255;
            if (o + cnt > d.d0[p + 1] || (cnt > 0) != (t.out[j] >= 0)) return fail("destination range", seed);
            for (int i = o; i < o + cnt; ++i, ++n) {
                const int r = d.dst[i] >> 16, e = d.dst[i] & 0xffff;
                if (r == p || t.r0[r] + e >= t.r0[r + 1] || uslot[t.rem[t.r0[r] + e]] != t.slot[j])
                    return fail("destination", seed);
            }
        }
    return n == t.rem.size() && d.ok ? 0 : fail("destination count", seed);
}

static int check(const PersistParts &t, int P, int S, const std::vector<int> &soff, const std::vector<int> &gk,
                 const std::vector<int> &pk, const std::vector<int> &gstart, const std::vector<int> &uslot, int seed) {
    const int L = (int)gk.size();
    std::vector<int> seen_s(S, 0), part(L, -1);
    if (t.s0[0] != 0 || t.s0[P] != S || t.k0[P] != L) return fail("ranges", seed);
    for (int p = 0; p < P; ++p) {
        int j = t.k0[p];
        for (int i = t.s0[p]; i < t.s0[p + 1]; ++i) {
            const int d = t.sub[i];
            if (seen_s[d]++) return fail("subsystem twice", seed);
            if (i > t.s0[p] && soff[t.sub[i - 1] + 1] - soff[t.sub[i - 1]] < soff[d + 1] - soff[d])
                return fail("sizes not decreasing", seed);
            for (int k = soff[d]; k < soff[d + 1]; ++k, ++j) {
                if (t.slot[j] != k) return fail("slot order", seed);
                part[k] = p;
            }
        }
        if (j != t.k0[p + 1]) return fail("slot range", seed);
    }
    std::vector<int> read(L, 0);
    for (int p = 0; p < P; ++p) {
        const int nk = t.k0[p + 1] - t.k0[p], nr = t.r0[p + 1] - t.r0[p], nl = t.l0[p + 1] - t.l0[p];
        for (int i = t.r0[p]; i < t.r0[p + 1]; ++i) read[uslot[t.rem[i]]] = 1;
        for (int j = t.k0[p]; j < t.k0[p + 1]; ++j) {
            const int k = t.slot[j], g = gk[k], cnt = gstart[g + 1] - gstart[g];
            if ((t.seg[j] & 255) != cnt) return fail("copies", seed);
            if (cnt == 1) continue;
            const int o = t.seg[j] >> 8;
            if (o < 0 || 8 * o + cnt > 8 * nl) return fail("list range", seed);
            for (int q = cnt; q % 8; ++q)
                if (t.list[8 * (t.l0[p] + o) + q] != nk + nr) return fail("list padding", seed);
            for (int q = 0; q < cnt; ++q) {
                const int e = t.list[8 * (t.l0[p] + o) + q];
                if (e < 0 || e >= nk + nr) return fail("list entry range", seed);
                const int c = e < nk ? pk[t.slot[t.k0[p] + e]] : t.rem[t.r0[p] + e - nk];
                if (c != gstart[g] + q) return fail("list entry", seed);
                if (e >= nk && part[uslot[c]] == p) return fail("own copy read as remote", seed);
            }
        }
    }
    for (int j = 0; j < L; ++j) {
        const int k = t.slot[j];
        if (t.out[j] != (read[k] ? pk[k] : -1)) return fail("exports", seed);
    }
    return 0;
}

int main() {
    std::mt19937 rng(77);
    for (int seed = 0; seed < 1500; ++seed) {
        const int S = 1 + (int)(rng() % 60), G = 2 + (int)(rng() % 90);
        std::vector<std::vector<int>> subs(S);
        for (auto &s : subs) {
            const int n = 1 + (int)(rng() % std::min(G, 12));
            std::vector<char> in(G, 0);
            while ((int)s.size() < n) {
                const int g = (int)(rng() % G);
                if (!in[g]) { in[g] = 1; s.push_back(g); }
            }
        }
        std::stable_sort(subs.begin(), subs.end(), [](auto &a, auto &b) { return a.size() > b.size(); });
        std::vector<int> soff(1, 0), gk, start(S);
        std::vector<double> cost;
        for (auto &s : subs) {
            gk.insert(gk.end(), s.begin(), s.end());
            soff.push_back((int)gk.size());
            cost.push_back(1.0 + (double)(s.size() * s.size()));
        }
        std::iota(start.begin(), start.end(), 0);
        std::shuffle(start.begin(), start.end(), rng);
        const int L = (int)gk.size();
        std::vector<int> gstart(G + 1, 0), pk(L), uslot(L);
        for (int g : gk) ++gstart[g + 1];
        for (int i = 0; i < G; ++i) gstart[i + 1] += gstart[i];
        std::vector<int> fill(gstart.begin(), gstart.end() - 1);
        for (int k = 0; k < L; ++k) { pk[k] = fill[gk[k]]++; uslot[pk[k]] = k; }
        std::vector<int> segp(L);
        for (int k = 0; k < L; ++k) segp[k] = (gstart[gk[k]] << 8) | (gstart[gk[k] + 1] - gstart[gk[k]]);
        std::vector<int> order = persist_order(S, soff, segp, pk, start);
        if ((int)order.size() != S) return fail("order", seed);
        const int P = seed % 5 == 0 ? 1 : 1 + (int)(rng() % (S + 5));
        PersistParts t = persist_parts(P, S, order, cost, soff, segp, pk);
        if (!t.ok || check(t, P, S, soff, gk, pk, gstart, uslot, seed)) return 1;
        if (check_dests(t, P, uslot, seed)) return 1;
        if (seed == 7 && t.list.size() > 1) {
            PersistParts bad = t;
            bad.list[0] ^= 1;
            std::printf("planted: ");
            if (!check(bad, P, S, soff, gk, pk, gstart, uslot, seed)) { std::printf("not caught\n"); return 1; }
        }
    }
    std::printf("ok\n");
    return 0;
}
"""


def test_partition_invariants(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "driver.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "driver"
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-Wall", "-I", CSRC, str(src), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.rstrip().endswith("ok"), out.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("ctas", [1, 2, 7, 40, 200])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_engine_forms_match_oracle(ctas, precision):
    from oracle import admm as oracle_admm, lindist
    from paper_2310_09410_gb300 import opf, synth

    g = synth.random_generic(31, n_global=150, n_sub=60, max_n=40, p_free=0.3)
    ref = oracle_admm.admm(lindist.from_generic(g), rho=10.0, max_iter=100, check_every=0)
    with opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"]) as s:
        s.precompute()
        s.solve(rho=10.0, eps_rel=0.0, max_iter=100, check_every=20, engine=opf.ENGINE_PERSISTENT, cluster=ctas,
                precision=opf.PREC_FP64 if precision == "fp64" else opf.PREC_FP32)
        xs, lam = s.locals()
        x, _ = s.solution()
    for got, want in ((xs, ref.xs), (lam, ref.lam), (x, ref.x)):
        scale = max(1.0, float(np.abs(want).max()))
        assert np.max(np.abs(got - want)) <= (1e-10 if precision == "fp64" else 1e-4) * scale


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_kept_plans_serve_new_loads(precision):
    """Tables, plans and solve graphs kept over opf_precompute: a handle given
    new loads twice returns what a fresh handle of those loads returns."""
    from paper_2310_09410_gb300 import opf, synth

    base = synth.preset_feeder("123", 2001)
    prec = opf.PREC_FP64 if precision == "fp64" else opf.PREC_MIXED

    def solved(s):
        s.precompute()
        s.solve(eps_rel=0.0, max_iter=1500, check_every=50, precision=prec)
        return s.solution()

    with opf.Solver.from_feeder(base) as s:
        solved(s)
        for seed in (7200, 7201):
            f = synth.load_scenario(base, seed)
            s.set_loads(f["load_a"], f["load_b"])
            x, obj = solved(s)
            with opf.Solver.from_feeder(f) as fresh:
                y, want = solved(fresh)
            assert np.array_equal(x, y) and obj == want


def one_cluster_instances():
    from paper_2310_09410_gb300 import opf, synth

    out = [lambda n=n, s=s: opf.Solver.from_feeder(synth.preset_feeder(n, s))
           for n, s in (("13", 1001), ("34", 5034), ("123", 2001))]
    out.append(lambda: opf.Solver.from_feeder(synth.make_feeder(2, 1, 1, seed=3)))
    # blocks up to 63 slots (two warps in the warp engine, odd halves), rank-deficient, free variables
    for seed, n, subs, widest in ((41, 90, 20, 63), (42, 40, 3, 39), (43, 200, 150, 9)):
        g = synth.random_generic(seed, n_global=n, n_sub=subs, max_n=widest, p_free=0.3)
        out.append(lambda g=g: opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"]))
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("case", range(7))
def test_one_cluster_form_equals_warp_engine(case):
    """FP32 iterates of the one-cluster form (the automatic choice at these
    sizes) are the warp engine's bit for bit."""
    from paper_2310_09410_gb300 import opf

    got = []
    for engine in (opf.ENGINE_AUTO, opf.ENGINE_WARP):
        with one_cluster_instances()[case]() as s:
            s.precompute()
            s.solve(eps_rel=0.0, max_iter=700, check_every=50, precision=opf.PREC_FP32, engine=engine)
            got.append(s.locals() + s.solution())
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.gpu
def test_one_cluster_bounded_wait():
    """A wait that can never end (the test hook) gives OPF_E_TIMEOUT, and the
    handle iterates afterwards."""
    from paper_2310_09410_gb300 import opf, synth

    with opf.Solver.from_feeder(synth.preset_feeder("13", 1001)) as s:
        s.precompute()
        for precision in (opf.PREC_FP64, opf.PREC_FP32):
            with pytest.raises(opf.OPFError) as e:
                s.solve(eps_rel=0.0, max_iter=100, check_every=50, precision=precision,
                        flags=opf.SOLVE_TEST_BARRIER_TIMEOUT)
            assert e.value.code == opf.OPF_E_TIMEOUT
            s.reset()
            s.solve(eps_rel=0.0, max_iter=100, check_every=50, precision=precision)
            assert s.residuals()["iters"] == 100
