"""The FP32 z-marching kernel of the 3D diffusion problems (the default FP32 path
from n = 17 on) against the FP64 evaluation of the same FP32 inputs, at the
edges of its tiles: one tile, ragged last tiles, an odd and an even number of
element rows, runs that end inside a tile.

Tolerance: 64 roundings of the largest terms of a node, as in
test_gpu_fixed_point.py with 2^-24; the vector-Jacobian product's second term
2 u (grad u . grad w) phi adds twice the flux term's size."""
import numpy as np
import pytest

from gpu_common import dev, host, jf, kernel_path, torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


@pytest.mark.parametrize("kind", ["nd3d", "ndk3d"])
@pytest.mark.parametrize("n", [17, 18, 19, 31, 33, 50, 65, 96, 129])
def test_matches_fp64(kind, n, monkeypatch):
    kernel_path(monkeypatch, "default")
    rng = np.random.default_rng(n)
    kap = torch.as_tensor(np.exp(rng.normal(size=(n, n, n))).astype(np.float32).astype(np.float64)) if kind == "ndk3d" else None
    p = jf().Problem(kind, n, 1, kappa=kap)
    u, v = rng.normal(size=(2, n + 1, n + 1, n + 1)).astype(np.float32)
    ud, vd = dev(u), dev(v)
    u64, v64 = ud.double(), vd.double()
    m, k = float(np.abs(u).max()), 1.0 if kap is None else float(kap.max())
    tol = 64 * EPS * 64 / (3.0 * n) * m * (1 + m * m) * k
    F = host(p.residual(ud))
    assert np.max(np.abs(F - host(p.residual(u64)))) <= tol
    edge = np.ones(F.shape, bool)
    edge[1:-1, 1:-1, 1:-1] = False
    assert np.all(F[edge] == 0)
    eps = 0.25
    J = host(p.jvp(ud, p.residual(ud), vd, eps=eps))
    K = host(p.jvp(u64, p.residual(u64), v64, eps=eps))
    w = m + eps * float(np.abs(v).max())
    assert np.max(np.abs(J - K)) <= 2 * 64 * EPS * 64 / (3.0 * n) * w * (1 + w * w) * k / eps
    mv = float(np.abs(v).max())
    tol = 3 * 64 * EPS * 64 / (3.0 * n) * mv * (1 + m * m) * k
    assert np.max(np.abs(host(p.vjp(ud, vd)) - host(p.vjp(u64, v64)))) <= tol
    assert torch.equal(p.residual(ud), p.residual(ud))


def test_nan_reaches_its_neighbours(monkeypatch):
    kernel_path(monkeypatch, "default")
    n = 33
    u = np.random.default_rng(1).normal(size=(n + 1,) * 3).astype(np.float32)
    u[9, 16, 20] = np.nan
    F = host(jf().Problem("nd3d", n, 1).residual(dev(u)))
    want = np.zeros(F.shape, bool)
    want[8:11, 15:18, 19:22] = True
    assert np.array_equal(np.isnan(F), want)
