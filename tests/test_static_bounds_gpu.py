"""opf_global_update_static with bounds that are NaN, of either sign: such a
bound bounds nothing, the other one still does.  Sizes of each launch form.
Reference: the comparisons in numpy; the quotient within one unit in the last
place of the division's (4e-16 relative)."""
import numpy as np
import pytest

from paper_2310_09410_gb300 import opf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 512, 513, 4097, 20000])
def test_nan_bounds_bound_nothing(n):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(40 + n)
    seg = np.concatenate([[0], np.cumsum(rng.integers(1, 4, n))]).astype(np.int32)
    u = 50.0 * rng.normal(size=seg[-1])
    u[rng.random(len(u)) < 0.02] = np.inf
    c = rng.normal(size=n)
    kinds = np.array([np.nan, -np.nan, 0.25, np.inf])
    assert np.signbit(kinds[1]) and np.isnan(kinds[1])
    lb, ub = -kinds[rng.integers(0, 4, n)], kinds[rng.integers(0, 4, n)]
    x = (np.add.reduceat(u, seg[:-1]) - c) / (100.0 * np.diff(seg))
    with np.errstate(invalid="ignore"):
        want = np.where(x < lb, lb, x)
        want = np.where(want > ub, ub, want)
    dev = [torch.from_numpy(a).cuda() for a in (seg, u, c, lb, ub)]
    got = torch.empty(n, dtype=torch.float64, device="cuda")
    obj = torch.empty(1, dtype=torch.float64, device="cuda")
    opf.global_update_static(n, *(t.data_ptr() for t in dev), 100.0, got.data_ptr(), obj.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
    got = got.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    fine = np.isfinite(want)
    # (reduceat adds in pairs: two more roundings of the sum of magnitudes)
    slack = 4e-16 * np.abs(want) + 4 * 2.0 ** -53 * np.add.reduceat(np.abs(np.where(np.isinf(u), 0, u)), seg[:-1]) / 100.0
    assert np.all(np.abs(got[fine] - want[fine]) <= slack[fine])
