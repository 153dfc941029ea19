"""The one-CTA coarse GMRES at the edges of its thread mapping: one unknown, less
and more unknowns than a dot product's lanes, both lane counts, more unknowns
than threads, basis in shared and in global memory, stops by tolerance and by
the iteration limit, against the assembled Jacobian.

Tolerances: the FD action differs from J by at most 1e-7 (FP64; step 1.5e-8) or
6e-4 (FP32) of ||J|| ||v||, and these Jacobians' condition numbers are below 100
(FP64: n0 <= 31, FP32: n0 <= 8)."""
import numpy as np
import pytest

from gpu_common import dev, host, jf
from oracle import fem, transfer

pytestmark = pytest.mark.gpu


def _case(kind, n0, pc="f64", **kw):
    d = fem.dim_of(kind)
    rng = np.random.default_rng(n0)
    kap = np.exp(0.5 * rng.normal(size=(2 * n0,) * 3)) if kind == "ndk3d" else None
    o = jf().default_options(pc_dtype=jf().F32 if pc == "f32" else jf().F64,
                             eps_mode_pc=jf().EPS_FP32 if pc == "f32" else jf().EPS_PAPER, **kw)
    p = jf().Problem(kind, 2 * n0, 2, lam=3.0, kappa=None if kap is None else dev(kap), options=o)
    u = 0.5 * rng.uniform(-1, 1, size=(2 * n0 + 1,) * d)
    b = np.zeros((n0 + 1,) * d)
    inner = (slice(1, -1),) * d
    u[fem.boundary_mask(u.shape)] = 0.0
    b[inner] = rng.normal(size=b[inner].shape)
    p.mg_setup(dev(u), 0)
    x0 = transfer.project(u)
    k0 = None if kap is None else kap.reshape(n0, 2, n0, 2, n0, 2).mean(axis=(1, 3, 5))
    J = fem.assemble_jacobian(kind, x0, lam=3.0, kappa=k0)
    J = J.toarray() if hasattr(J, "toarray") else np.asarray(J)
    ids = np.flatnonzero(~fem.boundary_mask(b.shape).ravel())
    if J.shape[0] == b.size:
        J = J[np.ix_(ids, ids)]
    import torch
    s = host(p.coarse_solve(dev(b, torch.float32 if pc == "f32" else torch.float64)))
    assert np.all(s[fem.boundary_mask(b.shape)] == 0)
    return J, b.ravel()[ids], s.ravel()[ids].astype(float)


@pytest.mark.parametrize("kind,n0", [("nd3d", 2), ("nd3d", 3), ("ndk3d", 4), ("nd3d", 6), ("nd3d", 9), ("bratu2d", 2),
                                     ("bratu2d", 3), ("bratu2d", 8), ("bratu2d", 12), ("bratu2d", 13), ("bratu2d", 31)])
def test_solves(kind, n0):
    J, b, s = _case(kind, n0)
    assert np.linalg.norm(J @ s - b) <= 1e-5 * np.linalg.norm(b)


@pytest.mark.parametrize("kind,n0", [("nd3d", 2), ("nd3d", 4), ("ndk3d", 5), ("bratu2d", 3), ("bratu2d", 8)])
def test_solves_fp32(kind, n0):
    J, b, s = _case(kind, n0, "f32")
    assert np.linalg.norm(J @ s - b) <= 0.06 * np.linalg.norm(b)


@pytest.mark.parametrize("kind,n0", [("nd3d", 4), ("bratu2d", 8), ("bratu2d", 13)])
def test_stops_at_the_tolerance(kind, n0):
    J, b, s = _case(kind, n0, coarse_tol=1e-2)
    r = np.linalg.norm(J @ s - b) / np.linalg.norm(b)
    assert 1e-6 <= r <= 1e-2 + 1e-5


@pytest.mark.parametrize("kind,n0", [("nd3d", 4), ("bratu2d", 8), ("bratu2d", 13)])
@pytest.mark.parametrize("m", [1, 2, 5])
def test_iteration_limit_gives_the_least_residual(kind, n0, m):
    J, b, s = _case(kind, n0, coarse_maxit=m)
    K = [b]
    for _ in range(m):
        K.append(J @ (K[-1] / np.linalg.norm(K[-1])))
    AK = np.array([J @ k for k in K[:m]]).T
    y = np.linalg.lstsq(AK / np.linalg.norm(AK, axis=0), b, rcond=None)[0]
    least = np.linalg.norm(AK / np.linalg.norm(AK, axis=0) @ y - b)
    assert abs(np.linalg.norm(J @ s - b) - least) <= 1e-5 * np.linalg.norm(b)
