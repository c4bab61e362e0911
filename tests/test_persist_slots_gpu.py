"""The persistent engine's FP32 form for parts of several slots per thread: its
iterates are those of the form with one slot per thread bit for bit, whatever
the CTA count (2 to 4 CTAs, 1 to 3 of the smaller instance: several slots; 16
and more: one), with the tests on
odd and even iterations and a last test off the period."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def instances():
    from paper_2310_09410_gb300 import opf, synth

    yield lambda: opf.Solver.from_feeder(synth.preset_feeder("123", 2001))
    # wide blocks, 20 copies per global
    g = synth.random_generic(61, n_global=80, n_sub=110, max_n=30, p_free=0.3)
    yield lambda: opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"])


@pytest.mark.parametrize("case", [0, 1])
@pytest.mark.parametrize("iters,check_every", [(2, 2), (350, 50), (1234, 6)])
def test_forms_agree_bit_for_bit(case, iters, check_every):
    from paper_2310_09410_gb300 import opf

    got = []
    with list(instances())[case]() as s:
        s.precompute()
        for ctas in (16, 40) + ((2, 3, 4) if case == 0 else (1, 2, 3)):
            s.reset()
            s.solve(eps_rel=0.0, max_iter=iters, check_every=check_every, precision=opf.PREC_FP32,
                    engine=opf.ENGINE_PERSISTENT, cluster=ctas)
            got.append(s.locals() + s.solution()[:1])
    for other in got[1:]:
        for a, b in zip(other, got[0]):
            assert np.array_equal(a, b)


def test_bounded_wait():
    """A barrier that never completes (the test hook) ends with OPF_E_TIMEOUT, and the handle solves afterwards."""
    from paper_2310_09410_gb300 import opf

    with next(instances())() as s:
        s.precompute()
        how = dict(eps_rel=0.0, max_iter=100, check_every=50, precision=opf.PREC_FP32, engine=opf.ENGINE_PERSISTENT,
                   cluster=2)
        with pytest.raises(opf.OPFError) as e:
            s.solve(flags=opf.SOLVE_TEST_BARRIER_TIMEOUT, **how)
        assert e.value.code == opf.OPF_E_TIMEOUT
        s.reset()
        s.solve(**how)
        assert s.residuals()["iters"] == 100
