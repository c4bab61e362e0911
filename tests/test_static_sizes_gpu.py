"""opf_global_update_static at the sizes where its launches change (one warp,
one block, two kernels, more globals than threads) and on values at the edges
of its forms: copy counts past the reciprocal table, infinite bounds, infinite
and NaN u, signed zeros, a rho whose reciprocal overflows.  Reference: the same
formula in numpy (sequential sums, a division).  The quotient is within one
unit in the last place of the division's: 4e-16 relative; the objective adds
in another order: n 2^-53 of the sum of magnitudes."""
import numpy as np
import pytest

from paper_2310_09410_gb300 import opf

pytestmark = pytest.mark.gpu


def reference(seg, u, c, lb, ub, rho):
    cnt = np.diff(seg)
    sigma = u[seg[:-1]].copy()
    for k in range(1, int(cnt.max())):
        more = cnt > k
        sigma[more] += u[seg[:-1][more] + k]
    x = (sigma - c) / (rho * cnt)
    x = np.where(x < lb, lb, x)
    return np.where(x > ub, ub, x)


@pytest.mark.parametrize("n", [1, 31, 33, 512, 513, 4097, 8 * 152 * 256 + 1])
@pytest.mark.parametrize("rho", [100.0, 0.37, 1e-310])
def test_sizes_and_edges(n, rho):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    cnt = rng.integers(1, 4, n)
    cnt[rng.random(n) < 0.05] = rng.integers(14, 40)
    seg = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int32)
    u = rng.normal(size=seg[-1]) * 10.0 ** rng.integers(-6, 6, seg[-1])
    odd = rng.random(len(u)) < 0.01
    u[odd] = rng.choice([np.inf, -np.inf, np.nan, 0.0, -0.0], int(odd.sum()))
    c = np.where(rng.random(n) < 0.3, rng.normal(size=n), 0.0)
    lb = np.where(rng.random(n) < 0.5, -np.inf, -rng.random(n))
    ub = np.where(rng.random(n) < 0.5, np.inf, rng.random(n))
    with np.errstate(all="ignore"):
        want = reference(seg, u, c, lb, ub, rho)
    dev = [torch.from_numpy(a).cuda() for a in (seg, u, c, lb, ub)]
    x = torch.empty(n, dtype=torch.float64, device="cuda")
    obj = torch.empty(1, dtype=torch.float64, device="cuda")
    opf.global_update_static(n, *(t.data_ptr() for t in dev), rho, x.data_ptr(), obj.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
    got = x.cpu().numpy()
    fine = np.isfinite(want)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[~fine & ~np.isnan(want)], want[~fine & ~np.isnan(want)])
    assert np.all(np.abs(got[fine] - want[fine]) <= 4e-16 * np.abs(want[fine]))
    if fine.all():
        terms = c * want
        assert abs(float(obj.cpu()[0]) - terms.sum()) <= (n * 2.0 ** -53 + 4e-16) * np.abs(terms).sum()
