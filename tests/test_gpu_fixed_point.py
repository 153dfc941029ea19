"""The FP64 fixed-point kernel of the 3D diffusion problems (the default FP64
path) against the FP64-pipe kernels ("ep" path) where it can go wrong: tile and
run edges, values it leaves to FP64, aliased outputs.  Both evaluate the same
sums of element integrals: each is within c 2^-53 of the sum of the magnitudes
of an element's terms, c = 64 covering its ~45 roundings, which is what the
tolerance takes from the "ep" result of |w| (the diffusion terms of a node sum
to at most 8 x 16 times the largest corner value's share)."""
import numpy as np
import pytest

from gpu_common import dev, host, jf, kernel_path, torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _pair(monkeypatch, kind, n, **kw):
    kernel_path(monkeypatch, "ep")
    q = jf().Problem(kind, n, 1, **kw)
    kernel_path(monkeypatch, "default")
    return jf().Problem(kind, n, 1, **kw), q


def _kappa(n, seed=3):
    return torch.as_tensor(np.exp(np.random.default_rng(seed).normal(size=(n, n, n))))


def _tol(u, kap, n):
    """64 roundings of the largest terms: 8 elements, stiffness entries up to
    h/3 each way (8 corners), coefficient kappa (1 + max u^2)."""
    m = np.max(np.abs(u[np.isfinite(u)]))
    return 64 * EPS * 8 * 8 / (3.0 * n) * m * (1 + m * m) * (1.0 if kap is None else float(kap.abs().max()))


# one tile and one plane a CTA (2, 3), several tiles with a ragged last one, runs that end inside a tile
@pytest.mark.parametrize("kind", ["nd3d", "ndk3d"])
@pytest.mark.parametrize("n", [2, 3, 7, 18, 31, 33, 50, 65, 129])
def test_matches_fp64_pipe(kind, n, monkeypatch):
    kap = _kappa(n) if kind == "ndk3d" else None
    p, q = _pair(monkeypatch, kind, n, kappa=kap)
    rng = np.random.default_rng(n)
    u, v = rng.normal(size=(2, n + 1, n + 1, n + 1))
    ud, vd = dev(u), dev(v)
    F, G = p.residual(ud), q.residual(ud)
    tol = _tol(u, kap, n)
    assert np.max(np.abs(host(F) - host(G))) <= tol
    eps = 1e-4
    J, K = p.jvp(ud, G, vd, eps=eps), q.jvp(ud, G, vd, eps=eps)
    assert np.max(np.abs(host(J) - host(K))) <= 2 * tol / eps


@pytest.mark.parametrize("what", ["nan", "inf", "overflow", "huge", "tiny", "zero", "mixed", "kappa"])
def test_values_left_to_fp64(what, monkeypatch):
    n = 33
    rng = np.random.default_rng(5)
    u = rng.normal(size=(n + 1,) * 3)
    kap = None
    if what in ("nan", "inf"):
        u[9, 20, 31] = u[17, 3, 3] = np.nan if what == "nan" else -np.inf
    elif what == "overflow":
        u[5, 5, 5] = 1e200
    elif what == "huge":
        u *= 1e30
    elif what == "tiny":
        u *= 1e-130
    elif what == "zero":
        u[:, :20] = 0
    elif what == "mixed":
        u[::3] *= 1e40
        u[1::3] *= 1e-110
    else:
        kap = _kappa(n)
        kap[3, 4, 5], kap[9], kap[20, :, 7] = 0.0, -kap[9], 1e-120
    p, q = _pair(monkeypatch, "nd3d" if kap is None else "ndk3d", n, kappa=kap)
    F, G = host(p.residual(dev(u))), host(q.residual(dev(u)))
    assert np.array_equal(np.isnan(F), np.isnan(G)) and np.array_equal(np.isinf(F), np.isinf(G))
    fine = np.isfinite(G)
    if what == "zero":
        load = host(q.residual(dev(np.zeros_like(u))))
        assert np.array_equal(F[2:-2, 2:18, 2:-2], load[2:-2, 2:18, 2:-2])
    # node by node: the terms a node's 8 elements can hold
    M = np.abs(np.where(np.isfinite(u), u, 0))
    for ax in range(3):
        P = np.pad(M, [(1, 1) if a == ax else (0, 0) for a in range(3)])
        M = np.maximum(np.maximum(np.take(P, range(n + 1), ax), np.take(P, range(2, n + 3), ax)), M)
    M = np.minimum(M, 1e90)
    k = 1.0 if kap is None else float(kap.abs().max())
    tol = 64 * EPS * (64 / (3.0 * n) * M * (1 + M * M) * k + np.abs(np.where(fine, G, 0)))
    assert np.all(np.abs(F - G)[fine] <= tol[fine])


def test_output_may_be_an_input(monkeypatch):
    n = 40
    p, q = _pair(monkeypatch, "nd3d", n)
    rng = np.random.default_rng(8)
    u, v = dev(rng.normal(size=(n + 1,) * 3)), dev(rng.normal(size=(n + 1,) * 3))
    F = q.residual(u)
    J = q.jvp(u, F, v, eps=1e-4)
    w = u.clone()
    p.residual(w, out=w)
    assert torch.equal(w, F)  # the same kernels run
    w = v.clone()
    p.jvp(u, F, w, eps=1e-4, out=w)
    assert torch.equal(w, J)
