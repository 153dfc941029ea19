"""The FD step K / ||v|| from a reduction's last block: scaling v by 2^k scales
the step by 2^-k, so J v / 2^k keeps its value over the whole exponent range of
||v||^2, for one block and for many; a ||v||^2 of zero or beyond the range gives
a zero action.

Tolerance: the difference of two residuals a step apart, 64 roundings of the
largest terms of a node each (as in test_gpu_fixed_point.py), over the step; the
step itself is right to 2^-50."""
import numpy as np
import pytest

from gpu_common import dev, host, jf, torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.mark.parametrize("kind,n", [("bratu2d", 3), ("bratu2d", 31), ("bratu2d", 300), ("nd3d", 4), ("nd3d", 16),
                                    ("nd3d", 33), ("nd3d", 70)])
def test_scaled_direction(kind, n):
    d = 2 if kind == "bratu2d" else 3
    rng = np.random.default_rng(n)
    u, v = rng.normal(size=(2,) + (n + 1,) * d)
    inner = (slice(1, -1),) * d
    p = jf().Problem(kind, n, 1, lam=2.0)
    ud = dev(u)
    Fu = p.residual(ud)
    N = (n - 1) ** d
    nrm = np.linalg.norm(v[inner])
    eps = 2.0 ** -26 * (N + np.abs(u[inner]).sum()) / (N * nrm)
    m = np.abs(u).max() + eps * np.abs(v).max()
    size = 8 * m + 2.0 * np.exp(m) / n ** 2 if d == 2 else 64 / (3.0 * n) * m * (1 + m * m)
    base = host(p.jvp(ud, Fu, dev(v)))
    ref = host(p.jvp(ud, Fu, dev(v), eps=float(eps)))
    tol = 2 * 2 * 64 * EPS * size / eps + 2.0 ** -40 * np.abs(ref).max()
    assert np.max(np.abs(base - ref)) <= tol
    for k in (-500, -333, -1, 1, 250, 490):
        J = host(p.jvp(ud, Fu, dev(np.ldexp(v, k))))
        assert np.max(np.abs(np.ldexp(J, -k) - ref)) <= tol, k
    for k in (-700, 600):
        assert not torch.any(p.jvp(ud, Fu, dev(np.ldexp(v, k)))), k
