"""Asking for one instance per CTA in FP32 stays refused, and the error says why."""
import pytest

pytestmark = pytest.mark.gpu


def test_refusal_names_its_reason():
    from paper_2310_09410_gb300 import opf, synth

    with opf.Solver.from_feeder(synth.preset_feeder("13", 1001)) as s:
        s.precompute()
        with opf.Batch(s, 2) as b:
            b.set_shape(opf.PREC_FP32, 1, 16)
            with pytest.raises(opf.OPFError, match="library's own choice"):
                b.solve(eps_rel=0.0, max_iter=50, check_every=50, precision=opf.PREC_FP32)
            b.set_shape(opf.PREC_FP32, 0, 0)     # and the automatic choice still runs
            b.solve(eps_rel=0.0, max_iter=50, check_every=50, precision=opf.PREC_FP32)
