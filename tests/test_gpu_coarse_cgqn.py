"""The coarse CG with L-BFGS in a thread-block cluster, in both precisions, 2D and
3D, on both sides of 64 entries (one CTA, several), with entry counts that are no
multiple of the CTA count, first call (pairs collected) and second (pairs used),
against the assembled Jacobian.

u is constant, so that the 3D Jacobians, (1 + u^2) times a weighted Laplacian,
are symmetric; lambda is below the first eigenvalue, so that Bratu's is positive
definite too.  Tolerances: as for the coarse GMRES (test_gpu_coarse_gmres.py), an
FD action differs from J by at most 1e-7 (FP64) or 6e-4 (FP32) of ||J|| ||v||, and
the condition numbers are below 100."""
import numpy as np
import pytest

from gpu_common import dev, host, jf, torch
from oracle import fem, transfer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pc", ["f64", "f32"])
@pytest.mark.parametrize("kind,n0", [("nd3d", 2), ("nd3d", 3), ("ndk3d", 3), ("nd3d", 4), ("ndk3d", 4), ("ndk3d", 5),
                                     ("nd3d", 6), ("nd3d", 9), ("bratu2d", 3), ("bratu2d", 7), ("bratu2d", 8),
                                     ("bratu2d", 13)])
def test_solves(kind, n0, pc):
    d = fem.dim_of(kind)
    rng = np.random.default_rng(n0)
    kap = np.exp(0.25 * rng.normal(size=(2 * n0,) * 3)) if kind == "ndk3d" else None
    f32 = pc == "f32"
    o = jf().default_options(pc_dtype=jf().F32 if f32 else jf().F64, eps_mode_pc=jf().EPS_FP32 if f32 else jf().EPS_PAPER,
                             coarse_method=jf().COARSE_CGQN, coarse_tol=1e-2 if f32 else 1e-7)
    p = jf().Problem(kind, 2 * n0, 2, lam=3.0, kappa=None if kap is None else dev(kap), options=o)
    u = np.full((2 * n0 + 1,) * d, 0.5)
    p.mg_setup(dev(u), 0)
    x0 = transfer.project(u)
    k0 = None if kap is None else kap.reshape(n0, 2, n0, 2, n0, 2).mean(axis=(1, 3, 5))
    J = fem.assemble_jacobian(kind, x0, lam=3.0, kappa=k0)
    J = J.toarray() if hasattr(J, "toarray") else np.asarray(J)
    edge = fem.boundary_mask((n0 + 1,) * d)
    ids = np.flatnonzero(~edge.ravel())
    if J.shape[0] == edge.size:
        J = J[np.ix_(ids, ids)]
    for call in range(2):
        b = np.zeros(edge.shape)
        b.ravel()[ids] = rng.normal(size=ids.size)
        bd = dev(b, torch.float32 if f32 else torch.float64)
        s = host(p.coarse_solve(bd))
        assert np.all(s[edge] == 0)
        r = J @ s.ravel()[ids].astype(float) - b.ravel()[ids]
        assert np.linalg.norm(r) <= (0.06 if f32 else 1e-5) * np.linalg.norm(b), call
