"""The FP64 fixed-point vector-Jacobian product (the default FP64 path without
the coefficient's derivative) against the FP64-pipe kernels ("ep" path): tile and
run edges, values it leaves to FP64, aliased outputs.

Tolerance: 64 roundings of the largest terms of a node, as in
test_gpu_fixed_point.py, with the source term 2 u (grad u . grad w) phi of up to
twice the flux term's size."""
import numpy as np
import pytest

from gpu_common import dev, host, jf, kernel_path, torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _pair(monkeypatch, n, kap=None):
    kind = "nd3d" if kap is None else "ndk3d"
    kernel_path(monkeypatch, "ep")
    q = jf().Problem(kind, n, 1, kappa=kap)
    kernel_path(monkeypatch, "default")
    return jf().Problem(kind, n, 1, kappa=kap), q


def _kappa(n):
    return torch.as_tensor(np.exp(np.random.default_rng(3).normal(size=(n, n, n))))


def _near_max(a):
    """Largest magnitude among a node and its neighbours."""
    M = np.abs(np.where(np.isfinite(a), a, 0))
    for ax in range(3):
        P = np.pad(M, [(1, 1) if k == ax else (0, 0) for k in range(3)])
        m = a.shape[ax]
        M = np.maximum(np.maximum(np.take(P, range(m), ax), np.take(P, range(2, m + 2), ax)), M)
    return M


def _tol(u, w, k, n):
    M = np.minimum(_near_max(u), 1e90)
    return 3 * 64 * EPS * 64 / (3.0 * n) * _near_max(w) * (1 + M * M) * k


@pytest.mark.parametrize("kind", ["nd3d", "ndk3d"])
@pytest.mark.parametrize("n", [2, 3, 7, 18, 31, 33, 50, 65, 129])
def test_matches_fp64_pipe(kind, n, monkeypatch):
    kap = _kappa(n) if kind == "ndk3d" else None
    p, q = _pair(monkeypatch, n, kap)
    u, w = np.random.default_rng(n).normal(size=(2, n + 1, n + 1, n + 1))
    A, B = host(p.vjp(dev(u), dev(w))), host(q.vjp(dev(u), dev(w)))
    assert np.all(np.abs(A - B) <= _tol(u, w, 1.0 if kap is None else float(kap.max()), n))
    assert torch.equal(p.vjp(dev(u), dev(w)), p.vjp(dev(u), dev(w)))


@pytest.mark.parametrize("what", ["nan", "inf", "direction nan", "direction inf", "huge", "tiny", "zero", "kappa"])
def test_values_left_to_fp64(what, monkeypatch):
    n = 33
    u, w = np.random.default_rng(5).normal(size=(2,) + (n + 1,) * 3)
    kap = None
    if what in ("nan", "inf"):
        u[9, 20, 31] = u[17, 3, 3] = np.nan if what == "nan" else -np.inf
        w[8:11, 19:22] = 0  # (0 x NaN)
    elif what.startswith("direction"):
        w[9, 20, 31] = np.nan if what.endswith("nan") else np.inf
    elif what == "huge":
        u[:, 4] *= 1e30
        w[5, 5, 5] = 1e100
    elif what == "tiny":
        u[:20] *= 1e-130
        w[:, 20:] *= 1e-110
    elif what == "zero":
        u[:, :20] = 0
        w[10:25] = 0
    else:
        kap = _kappa(n)
        kap[3, 4, 5], kap[9], kap[20, :, 7] = 0.0, -kap[9], 1e-120
    p, q = _pair(monkeypatch, n, kap)
    A, B = host(p.vjp(dev(u), dev(w))), host(q.vjp(dev(u), dev(w)))
    assert np.array_equal(np.isnan(A), np.isnan(B)) and np.array_equal(np.isinf(A), np.isinf(B))
    fine = np.isfinite(B)
    tol = _tol(u, w, 1.0 if kap is None else float(kap.abs().max()), n)
    assert np.all(np.abs(A - B)[fine] <= tol[fine])


def test_output_may_be_the_direction(monkeypatch):
    n = 40
    p, q = _pair(monkeypatch, n)
    u, w = (dev(a) for a in np.random.default_rng(8).normal(size=(2,) + (n + 1,) * 3))
    want = q.vjp(u, w)
    p.vjp(u, w, out=w)
    assert torch.equal(w, want)  # the same kernels run


def test_coefficient_derivative_keeps_its_kernels(monkeypatch):
    n = 20
    p, q = _pair(monkeypatch, n, _kappa(n))
    u, w = (dev(a) for a in np.random.default_rng(9).normal(size=(2,) + (n + 1,) * 3))
    for a, b in zip(p.vjp(u, w, dkappa=True), q.vjp(u, w, dkappa=True)):
        assert torch.equal(a, b)
