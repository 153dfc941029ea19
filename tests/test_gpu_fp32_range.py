"""Range of the FP32 path.

Norms: an FP32 vector's norm is summed in FP64 beyond a row, so scaling the
vector by 2^k, with every row's FP32 sum of squares finite and normal, scales the
norm exactly, the FD step by 2^-k exactly, and leaves u + eps v and so the action's
bits as they are, also where the sum over all rows exceeds FP32's range.

Elements: the 3D diffusion terms are formed without a common factor, so F(u) is
right wherever its largest terms, u^3 times the corners' stiffness, are in FP32's
range.  Tolerance: 64 roundings of those terms, as in test_gpu_fp32_tiles.py."""
import numpy as np
import pytest

from gpu_common import dev, host, jf, kernel_path, torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


# squares of N(0, 1) 2^60 stay below 2^125; 29791 and 65025 of them exceed 2^128
@pytest.mark.parametrize("kind,n", [("nd3d", 32), ("bratu2d", 256)])
@pytest.mark.parametrize("k", [-40, 60])
def test_action_of_a_scaled_direction(kind, n, k, monkeypatch):
    kernel_path(monkeypatch, "default")
    d = 2 if kind == "bratu2d" else 3
    rng = np.random.default_rng(n)
    u, v = rng.normal(size=(2,) + (n + 1,) * d).astype(np.float32)
    p = jf().Problem(kind, n, 1, lam=2.0)
    ud = dev(u)
    Fu = p.residual(ud)
    base = p.jvp(ud, Fu, dev(v), eps_mode=jf().EPS_FP32)
    assert torch.any(base != 0)
    J = p.jvp(ud, Fu, dev(np.ldexp(v, k)), eps_mode=jf().EPS_FP32)
    assert torch.equal(torch.ldexp(J, torch.tensor(-k, device="cuda")), base)


# the start of a Chebyshev sweep from zero, d = b / theta: b is scaled so that the
# squares of d sum to about 2^131, of which a warp's share is 2^11 times smaller
def test_sweep_of_a_scaled_right_hand_side(monkeypatch):
    kernel_path(monkeypatch, "default")
    n = 128
    o = jf().default_options(pc_dtype=jf().F32, eps_mode_pc=jf().EPS_FP32, cheb_degree=2)
    p = jf().Problem("nd3d", n, 6, options=o)
    rng = np.random.default_rng(1)
    u, b = 0.1 * rng.normal(size=(2,) + (n + 1,) * 3)
    b[[0, -1]] = b[:, [0, -1]] = b[:, :, [0, -1]] = 0
    p.mg_setup(dev(u), 0)
    theta = 0.5 * (o.cheb_lo + o.cheb_hi) * p.level_info(5)["lambda_max"]
    k = int(np.floor((131 - np.log2(np.sum((b / theta) ** 2))) / 2))
    b = b.astype(np.float32)
    s = [p.smooth(dev(np.ldexp(b, e)), torch.zeros(p.shape(), device="cuda"), s_is_zero=True) for e in (0, k)]
    assert torch.any(s[0] != 0)
    assert torch.equal(torch.ldexp(s[1], torch.tensor(-k, device="cuda")), s[0])


@pytest.mark.parametrize("kind", ["nd3d", "ndk3d"])
@pytest.mark.parametrize("n", [17, 40])
def test_large_values(kind, n, monkeypatch):
    kernel_path(monkeypatch, "default")
    rng = np.random.default_rng(n)
    m = 2.0 ** 40  # u^3 = 2^120
    u = (m * rng.uniform(-1, 1, size=(n + 1,) * 3)).astype(np.float32)
    kap = torch.ones((n,) * 3, dtype=torch.float64) if kind == "ndk3d" else None
    p = jf().Problem(kind, n, 1, kappa=kap)
    F, G = host(p.residual(dev(u))), host(p.residual(dev(u.astype(np.float64))))
    assert np.all(np.isfinite(F))
    assert np.max(np.abs(F - G)) <= 64 * EPS * 64 / (3.0 * n) * m * (1 + m * m)
