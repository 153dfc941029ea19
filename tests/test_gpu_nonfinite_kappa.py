"""A coefficient that is not finite makes its element's contributions NaN also
where the element's values are zero (0 x NaN, 0 x Inf), in every precision, on
every kernel path and in the coarse solvers: a fixed-point element whose corners
are all zero must not be skipped there."""
import numpy as np
import pytest

from gpu_common import dev, host, jf, kernel_path, torch

pytestmark = pytest.mark.gpu

BAD = [np.nan, np.inf, -np.inf]


def _neighbours(n, where):
    """Interior nodes of the elements `where` (z, y, x)."""
    m = np.zeros((n + 1,) * 3, bool)
    for z, y, x in where:
        m[z:z + 2, y:y + 2, x:x + 2] = True
    inner = np.zeros_like(m)
    inner[1:-1, 1:-1, 1:-1] = True
    return m & inner


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n", [4, 18, 33])
def test_zero_element(n, dtype, bad, monkeypatch):
    kernel_path(monkeypatch, "default")
    rng = np.random.default_rng(n)
    kap = np.exp(rng.normal(size=(n,) * 3))
    where = [(0, 0, 0), (1, 2, 3), (n - 1, n // 2, 1)]
    for e in where:
        kap[e] = bad
    p = jf().Problem("ndk3d", n, 1, kappa=dev(kap))
    want = _neighbours(n, where)
    u = torch.zeros((n + 1,) * 3, dtype=dtype, device="cuda")
    F = host(p.residual(u))
    assert np.array_equal(np.isnan(F), want)
    w = dev(rng.normal(size=F.shape), dtype)
    assert np.array_equal(np.isnan(host(p.vjp(w, u))), want)  # zero direction
    assert np.array_equal(np.isnan(host(p.vjp(u, w))), want)  # zero u


# node (3, 3, 3) of 5^3 nodes carries b; the coefficient of element (0, 0, 0),
# none of whose nodes b reaches in one action, is not finite.  A solver whose
# product holds a NaN cannot return a finite, nonzero solution.
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("method", ["GMRES", "CGQN"])
def test_coarse_solvers_zero_element(method, dtype, bad):
    n0 = 4
    o = jf().default_options(coarse_maxit=1, coarse_method=getattr(jf(), "COARSE_" + method),
                             pc_dtype=jf().F32 if dtype == "f32" else jf().F64)
    kap = torch.ones((2 * n0,) * 3, dtype=torch.float64, device="cuda")
    p = jf().Problem("ndk3d", 2 * n0, 2, kappa=kap, options=o)
    p.mg_setup(torch.zeros(p.shape(), dtype=torch.float64, device="cuda"), 0)
    b = torch.zeros((n0 + 1,) * 3, dtype=torch.float32 if dtype == "f32" else torch.float64, device="cuda")
    b[3, 3, 3] = 1.0
    s = host(p.coarse_solve(b))
    assert np.all(np.isfinite(s)) and np.any(s)
    kap[0, 0, 0] = bad  # (element (0, 0, 0) of the coarse grid has the mean of 8)
    p.set_kappa(kap)
    s = host(p.coarse_solve(b))
    assert not np.all(np.isfinite(s)) or not np.any(s)
