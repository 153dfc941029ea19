"""The FP32 strip kernels of the 2D problems (30 node columns a warp) against the
FP64 evaluation of the same FP32 inputs, at the edges of strips and warps.

Tolerance: 64 roundings of the largest terms, as for the FP64 strips in
test_gpu_fixed_point.py with 2^-24."""
import numpy as np
import pytest

from gpu_common import dev, host, jf, torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


@pytest.mark.parametrize("kind", ["bratu2d", "minsurf2d"])
@pytest.mark.parametrize("n", [2, 3, 29, 30, 31, 32, 61, 95, 250])
def test_matches_fp64(kind, n):
    rng = np.random.default_rng(n)
    scale = 1.0 / n if kind == "minsurf2d" else 1.0
    u, v = (scale * rng.uniform(-0.9, 0.9, size=(2, n + 1, n + 1))).astype(np.float32)
    p = jf().Problem(kind, n, 1, lam=5.0)
    ud, vd = dev(u), dev(v)
    u64, v64 = ud.double(), vd.double()

    def tol(m):
        return 64 * EPS * (16 * 2 / 3 * m + (5.0 / n ** 2 * np.exp(m) if kind == "bratu2d" else 0.0))

    m = float(np.abs(u).max())
    F = host(p.residual(ud))
    assert np.max(np.abs(F - host(p.residual(u64)))) <= tol(m)
    edge = np.ones(F.shape, bool)
    edge[1:-1, 1:-1] = False
    assert np.all(F[edge] == 0)
    eps = 0.25
    J = host(p.jvp(ud, p.residual(ud), vd, eps=eps))
    K = host(p.jvp(u64, p.residual(u64), v64, eps=eps))
    assert np.max(np.abs(J - K)) <= 2 * tol(m + eps * float(np.abs(v).max())) / eps
    assert torch.equal(p.residual(ud), p.residual(ud))


@pytest.mark.parametrize("kind", ["bratu2d", "minsurf2d"])
@pytest.mark.parametrize("x", [1, 29, 30, 31, 59, 60, 61, 94])
def test_nan_reaches_its_neighbours(kind, x):
    n = 95
    u = np.random.default_rng(1).uniform(-0.5, 0.5, size=(n + 1, n + 1)).astype(np.float32) / n
    u[40, x] = np.nan
    F = host(jf().Problem(kind, n, 1, lam=5.0).residual(dev(u)))
    want = np.zeros(F.shape, bool)
    want[39:42, x - 1:x + 2] = True
    want[[0, -1]] = want[:, [0, -1]] = False
    assert np.array_equal(np.isnan(F), want)
