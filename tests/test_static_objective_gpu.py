"""The objective of opf_global_update_static with finite inputs, at the sizes of
each launch form (one block, one cluster, a grid, more globals than threads; on
a partition of 8 SMs too), several calls
in a row on one stream with other inputs and nothing waited for between, so that
a sum taken too early or from an earlier call's partial sums shows.  Reference:
numpy; the objective adds in another order (n 2^-53 of the sum of magnitudes)
and its x are within 4e-16 relative."""
import numpy as np
import pytest

from paper_2310_09410_gb300 import opf

pytestmark = pytest.mark.gpu

SIZES = [1, 31, 33, 256, 257, 511, 512, 513, 1024, 4095, 4096, 4097, 8192, 8193, 20000, 63405, 8 * 152 * 256,
         8 * 152 * 256 + 1, 700001]


def check(n, stream):
    torch = pytest.importorskip("torch")
    calls = []
    for k in range(4):
        rng = np.random.default_rng([n, k])
        seg = np.concatenate([[0], np.cumsum(rng.integers(1, 4, n))]).astype(np.int32)
        u = (1.0 + 20.0 * k) * rng.normal(size=seg[-1])
        c = rng.normal(size=n) + k
        lb = np.where(rng.random(n) < 0.5, -np.inf, -rng.random(n))
        ub = np.where(rng.random(n) < 0.5, np.inf, rng.random(n))
        cnt = np.diff(seg)
        sigma = u[seg[:-1]].copy()
        for q in (1, 2):
            more = cnt > q
            sigma[more] += u[seg[:-1][more] + q]
        terms = c * np.clip((sigma - c) / (100.0 * cnt), lb, ub)
        dev = [torch.from_numpy(a).cuda() for a in (seg, u, c, lb, ub)]
        calls.append((dev, torch.empty(n, dtype=torch.float64, device="cuda"),
                      torch.full((1,), float("nan"), dtype=torch.float64, device="cuda"), terms))
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream().cuda_stream if stream is None else stream
    for dev, x, obj, _ in calls:
        opf.global_update_static(n, *(t.data_ptr() for t in dev), 100.0, x.data_ptr(), obj.data_ptr(), stream)
    torch.cuda.synchronize()
    for dev, x, obj, terms in calls:
        assert abs(float(obj[0]) - terms.sum()) <= (n * 2.0 ** -53 + 8e-16) * np.abs(terms).sum()


@pytest.mark.parametrize("n", SIZES)
def test_objective_of_calls_in_a_row(n):
    check(n, None)


@pytest.mark.parametrize("n", [256, 257, 4096, 4097])
def test_on_a_small_partition(n):
    part = opf.SMPartition(8)
    try:
        check(n, part.stream)
    finally:
        part.close()
