"""Single solves on streams of SM partitions: every engine that the automatic
choice takes at its size has to fit the partition (a partition holds no cluster
of more than 8 CTAs), in both precisions; iterates after 100 iterations against
the oracle (1e-10 in FP64, 1e-4 in FP32) and mixed solves that converge.  A
request for an engine that does not fit is refused, not launched."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def feeder(buses):
    from paper_2310_09410_gb300 import synth

    if buses == 200:
        return synth.make_feeder(200, 138, 16, depth_max=30, p_single=0.4, seed=9)
    return synth.preset_feeder(str(buses), {13: 1001, 34: 5034, 123: 2001}[buses])


@pytest.mark.parametrize("n_sm", [8, 32])
@pytest.mark.parametrize("buses", [13, 34, 123, 200])
def test_automatic_engines_fit_the_partition(n_sm, buses):
    from oracle import admm as oracle_admm, lindist
    from paper_2310_09410_gb300 import opf

    f = feeder(buses)
    ref = oracle_admm.admm(oracle_admm.Prepared(lindist.build(f)), rho=100.0, max_iter=100, check_every=0)
    part = opf.SMPartition(n_sm)
    try:
        with opf.Solver.from_feeder(f, stream=part.stream) as s:
            s.precompute()
            for precision, tol in ((opf.PREC_FP64, 1e-10), (opf.PREC_FP32, 1e-4)):
                s.reset()
                s.solve(eps_rel=0.0, max_iter=100, check_every=50, precision=precision, flags=opf.SOLVE_HOST_LOOP)
                for got, want in zip(s.locals(), (ref.xs, ref.lam)):
                    assert np.max(np.abs(got - want)) <= tol * max(1.0, float(np.abs(want).max()))
            s.reset()
            assert s.solve(eps_rel=1e-4, eps_abs_pres=1e9, max_iter=200000, precision=opf.PREC_MIXED,
                           flags=opf.SOLVE_HOST_LOOP)
    finally:
        part.close()


@pytest.mark.parametrize("engine,cluster", [(2, 16), (3, 12)])
def test_unfit_cluster_is_refused(engine, cluster):
    from paper_2310_09410_gb300 import opf

    part = opf.SMPartition(32)
    try:
        with opf.Solver.from_feeder(feeder(123), stream=part.stream) as s:
            s.precompute()
            for precision in (opf.PREC_FP64, opf.PREC_FP32):
                with pytest.raises(opf.OPFError) as e:
                    s.solve(eps_rel=0.0, max_iter=100, check_every=50, precision=precision, engine=engine,
                            cluster=cluster, flags=opf.SOLVE_HOST_LOOP)
                assert e.value.code == opf.OPF_E_CAPACITY
    finally:
        part.close()
