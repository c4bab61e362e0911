"""Handles, batches and served models of different sizes in turn.  A kernel's
limit of dynamic shared memory belongs to the kernel, and plans are kept: a
smaller instance that plans the same kernel must not take the limit away from a
larger one that solves again.  Every repeated solve returns the first one's
results bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def feeder(buses):
    from paper_2310_09410_gb300 import synth

    return synth.preset_feeder(str(buses), {13: 1001, 34: 5034, 123: 2001}[buses])


def consensus(n, blocks, widest):
    from paper_2310_09410_gb300 import opf, synth

    g = synth.random_generic(7, n_global=n, n_sub=blocks, max_n=widest, p_free=0.2)
    return opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"])


def handle(kind, size):
    from paper_2310_09410_gb300 import opf, synth

    if kind == "feeder":
        return opf.Solver.from_feeder(feeder(size))
    if kind == "grown":
        return opf.Solver.from_feeder(synth.make_feeder(size, int(0.69 * size), size // 12, depth_max=30, seed=5))
    return consensus(*size)


# form of the automatic choice (or the engine asked for), a larger and a smaller instance
PAIRS = [("feeder", 34, 13, 0), ("feeder", 123, 13, 0), ("grown", 1000, 300, 0), ("consensus", (900, 240, 100), (300, 160, 70), 0),
         ("feeder", 123, 13, 3), ("feeder", 123, 13, 2), ("feeder", 123, 13, 4)]


@pytest.mark.parametrize("kind,large,small,engine", PAIRS)
@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
def test_handles_in_turn(kind, large, small, engine, precision):
    from paper_2310_09410_gb300 import opf

    prec = {"fp64": opf.PREC_FP64, "fp32": opf.PREC_FP32, "mixed": opf.PREC_MIXED}[precision]

    def solved(s, rho):
        s.precompute()
        s.solve(rho=rho, eps_rel=0.0, max_iter=150, check_every=50, precision=prec, engine=engine)
        return s.locals() + s.solution()

    with handle(kind, large) as a, handle(kind, small) as b:
        first = [solved(s, rho) for rho in (100.0, 60.0) for s in (a, b)]
        again = [solved(s, rho) for rho in (100.0, 60.0) for s in (a, b)]
    for x, y in zip(first, again):
        for p, q in zip(x, y):
            assert np.array_equal(p, q)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("k_inst,warps", [(4, 8), (2, 16), (0, 0)])
def test_batches_in_turn(precision, k_inst, warps):
    from paper_2310_09410_gb300 import opf

    prec = opf.PREC_FP64 if precision == "fp64" else opf.PREC_FP32

    def solved(b, rho):
        b.set_start(None, None)
        b.solve(rho=rho, eps_rel=0.0, max_iter=100, check_every=50, precision=prec)
        return b.solution()

    with opf.Solver.from_feeder(feeder(123)) as sa, opf.Solver.from_feeder(feeder(13)) as sb:
        sa.precompute()
        sb.precompute()
        with opf.Batch(sa, 5) as a, opf.Batch(sb, 5) as b:
            if k_inst:
                a.set_shape(prec, k_inst, warps)
                b.set_shape(prec, k_inst, warps)
            loads = {}
            for batch, f in ((a, feeder(123)), (b, feeder(13))):
                loads[batch] = [np.stack([f[k] * (0.8 + 0.05 * j) for j in range(5)]) for k in ("load_a", "load_b")]

            def one(batch, rho):
                batch.set_loads(0, *loads[batch])
                return solved(batch, rho)

            first = [one(x, rho) for rho in (100.0, 60.0) for x in (a, b)]
            again = [one(x, rho) for rho in (100.0, 60.0) for x in (a, b)]
    if k_inst:                       # (the automatic shape is a measurement's: its own rounding)
        for x, y in zip(first, again):
            for p, q in zip(x, y):
                assert np.array_equal(p, q)


def test_served_models_largest_first():
    from paper_2310_09410_gb300 import opf, synth

    solvers = [opf.Solver.from_feeder(feeder(n)) for n in (123, 34, 13)]
    with opf.Server(eps_rel=0.0, max_iter=400, check_every=50, keep_solutions=True) as srv:
        models = []
        for s in solvers:
            s.precompute()
            models.append(srv.add_model([s], 4))
            srv.set_model_shape(models[-1], 2, 16)
        for turn in range(2):                    # every model plans in the first
            for k, n in enumerate((123, 34, 13)):
                g = synth.load_scenario(feeder(n), 60 + k)
                srv.submit(models[k], g["load_a"], g["load_b"], 10 * turn + k)
                left = 1
                while left:
                    srv.step()
                    left -= len(srv.poll())
        got = [[srv.take_solution(10 * turn + k, models[k]) for k in range(3)] for turn in range(2)]
    for x, y in zip(*got):
        assert np.array_equal(x, y)
    for s in solvers:
        s.close()
