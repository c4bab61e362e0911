"""Handles solving side by side, a thread and a stream each: every form of the
automatic choice (one cluster, local grid, owner form, several slots per
thread), alone and together with others of its own and of other forms; the
results are those of the handle alone, bit for bit."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def instances():
    from paper_2310_09410_gb300 import opf, synth

    def generic(seed, n, blocks, widest):
        g = synth.random_generic(seed, n_global=n, n_sub=blocks, max_n=widest, p_free=0.2)
        return opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"])

    return [lambda: opf.Solver.from_feeder(synth.preset_feeder("34", 5034)),
            lambda: opf.Solver.from_feeder(synth.preset_feeder("123", 2001)),
            lambda: opf.Solver.from_feeder(synth.make_feeder(450, 310, 37, depth_max=30, p_single=0.4, seed=9)),
            lambda: generic(17, 900, 240, 100),
            lambda: generic(18, 500, 300, 60)]


@pytest.mark.parametrize("precision", ["fp32", "fp64", "mixed"])
def test_results_of_handles_in_threads(precision):
    from paper_2310_09410_gb300 import opf

    prec = {"fp32": opf.PREC_FP32, "fp64": opf.PREC_FP64, "mixed": opf.PREC_MIXED}[precision]
    solvers = [make() for make in instances() for _ in range(2)]
    for s in solvers:
        s.precompute()

    def solved(s):
        s.reset()
        s.solve(eps_rel=0.0, max_iter=1500, check_every=50, precision=prec)
        return s.locals() + s.solution()

    want = [solved(s) for s in solvers]
    for turn in range(3):
        got = [None] * len(solvers)

        def work(i):
            got[i] = solved(solvers[i])

        threads = [threading.Thread(target=work, args=(i,)) for i in range(len(solvers))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for g, w in zip(got, want):
            assert g is not None
            for a, b in zip(g, w):
                assert np.array_equal(a, b)
    for s in solvers:
        s.close()
