"""The FP32 batch shape the library picks by itself, at batch sizes on both sides
of its rule (one instance per CTA while every CTA has an SM, then two, four,
eight, or half of that) and over task widths: iterates of the first and last
instance against the oracle, to the tolerance of the other FP32 batch tests
(1e-4 after 100 iterations; the shapes differ in the order of FP32 sums only).
One instance per CTA stays refused as a requested shape."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,seed", [("13", 1001), ("34", 5034), ("123", 2001)])
@pytest.mark.parametrize("n", [1, 2, 40, 170, 330])
def test_automatic_shape_tracks_oracle(name, seed, n):
    import torch

    from oracle import lindist
    from paper_2310_09410_gb300 import opf, synth
    from test_batch_gpu import load_arrays, oracle_iterates, rel_err, scenarios

    f = synth.preset_feeder(name, seed)
    fs = scenarios(f, [4100 + j for j in range(n)])
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    want = next((k for k in (1, 2, 4) if -(-n // k) <= n_sm), 8)
    with opf.Solver.from_feeder(f) as s:
        s.precompute()
        with opf.Batch(s, n) as b:
            b.set_loads(0, *load_arrays(fs))
            b.solve(eps_rel=0.0, max_iter=100, check_every=50, precision=opf.PREC_FP32)
            assert np.all(b.status()["iters"] == 100)
            assert b.shape(opf.PREC_FP32)["k_inst"] in (want, max(1, want // 2))
            for j in {0, n - 1}:
                ref = oracle_iterates(lindist.build(fs[j]), 100)
                xs, lam = b.locals(j)
                assert rel_err(xs, ref.xs) <= 1e-4
                assert rel_err(lam, ref.lam) <= 1e-4


def test_one_instance_per_cta_is_not_a_shape():
    from paper_2310_09410_gb300 import opf, synth

    with opf.Solver.from_feeder(synth.preset_feeder("13", 1001)) as s:
        s.precompute()
        with opf.Batch(s, 2) as b:
            b.set_shape(opf.PREC_FP32, 1, 16)
            with pytest.raises(opf.OPFError):
                b.solve(eps_rel=0.0, max_iter=50, check_every=50, precision=opf.PREC_FP32)
