"""The FP64 fixed-point kernel of the 3D diffusion problems (the default FP64
path) against the FP64-pipe kernels ("ep" path) where it can go wrong: tile and
run edges, values it leaves to FP64, aliased outputs.  Both evaluate the same
sums of element integrals: each is within c 2^-53 of the sum of the magnitudes
of an element's terms, c = 64 covering its ~45 roundings, which is what the
tolerance takes from the "ep" result of |w| (the diffusion terms of a node sum
to at most 8 x 16 times the largest corner value's share)."""
import functools

import numpy as np
import pytest

from gpu_common import dev, host, jf, kernel_path, torch
from oracle import fem

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


# ---- 2D: strips of 30 node columns, a warp each ---------------------------
# Tolerance as above for the gradient part (stiffness entries up to 2/3, 4
# elements of 4 corners; minimal surface: coefficient at most 1) plus the
# source's lambda h^2 max exp(u).


@functools.lru_cache(maxsize=None)
def _case2d(kind, n, what):
    rng = np.random.default_rng(n)
    u = rng.uniform(-0.9, 0.9, size=(n + 1, n + 1)) / (n if kind == "minsurf2d" else 1)
    if what in ("nan", "inf"):
        u[n // 2, 1] = u[1, n // 3] = np.nan if what == "nan" else np.inf
    elif what == "range":  # Bratu: |u| to 30; minimal surface: slopes to 1e4
        u *= 33.0 if kind == "bratu2d" else 1e4
    elif what == "tiny":
        u *= 1e-130
    elif what == "zero":
        u[: n // 2 + 1] = 0
    with np.errstate(all="ignore"):
        return u, fem.residual(kind, u, 5.0, None, None)


def _tol2d(kind, u, n):
    m = np.max(np.abs(u[np.isfinite(u)]))
    return 64 * EPS * (16 * 2 / 3 * m + (5.0 / n ** 2 * np.exp(m) if kind == "bratu2d" else 0.0))


# one strip and part of a warp (2, 29..32), several strips, ragged rows
@pytest.mark.parametrize("kind,n,what",
                         [(k, n, "plain") for k in ("bratu2d", "minsurf2d") for n in (2, 3, 29, 30, 31, 32, 61, 95, 250)] +
                         [(k, 48, w) for k in ("bratu2d", "minsurf2d") for w in ("nan", "inf", "range", "tiny", "zero")])
def test_2d_matches_oracle(kind, n, what):
    u, G = _case2d(kind, n, what)
    p = jf().Problem(kind, n, 1, lam=5.0)
    F = host(p.residual(dev(u)))
    fine = np.isfinite(G)
    assert np.array_equal(fine, np.isfinite(F))
    tol = _tol2d(kind, u, n)
    assert np.max(np.abs(F - G)[fine]) <= tol
    if what == "plain":
        v = np.random.default_rng(n + 1).normal(size=u.shape) * (0.1 / n if kind == "minsurf2d" else 1.0)
        eps = 1e-4
        inner = np.zeros_like(u)
        inner[1:-1, 1:-1] = 1
        K = (fem.residual(kind, u + eps * v * inner, 5.0, None, None) - G) / eps
        J = host(p.jvp(dev(u), dev(G), dev(v), eps=eps))
        assert np.max(np.abs(J - K)) <= 2 * tol / eps


@pytest.mark.parametrize("lam", [0.0, -3.0, 1e-120])
def test_2d_bratu_lambda(lam):
    n = 40
    u, _ = _case2d("bratu2d", n, "plain")
    F = host(jf().Problem("bratu2d", n, 1, lam=lam).residual(dev(u)))
    G = fem.residual("bratu2d", u, lam, None, None)
    assert np.max(np.abs(F - G)) <= _tol2d("bratu2d", u, n)
