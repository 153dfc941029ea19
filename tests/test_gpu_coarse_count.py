"""nF[0] counts every product the coarse GMRES forms.  It learns of a column's
residual one product late, so a solve that the tolerance stops forms, and counts,
one product more than the columns it uses; one that the iteration limit stops does
not."""
import pytest

from gpu_common import jf, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,levels", [("bratu2d", 16, 2), ("nd3d", 8, 2)])
def test_product_after_the_last_column_is_counted(kind, n, levels):
    def solve(maxit):
        # every coarse solve meets this tolerance with its first column
        o = jf().default_options(coarse_tol=0.999, coarse_maxit=maxit, rtol_newton=1e-6)
        p = jf().Problem(kind, n, levels, lam=2.0, options=o)
        u = torch.zeros(p.shape(), dtype=torch.float64, device="cuda")
        return u, p.solve(u)

    ua, a = solve(1)
    ub, b = solve(0)
    assert torch.equal(ua, ub) and a["linear_its"] == b["linear_its"]
    # one coarse solve per FGMRES iteration: 1 product each by the limit, 2 by the tolerance
    assert b["nF"][0] - a["nF"][0] == a["linear_its"]
    assert b["nJv"][0] - a["nJv"][0] == a["linear_its"]
