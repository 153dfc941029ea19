"""The range of levels that run in one thread-block cluster (JFNK_EP3D_CLUSTER_*)
is a choice about those levels only: the others keep the kernels they have by
default, bit for bit."""
import numpy as np
import pytest

from gpu_common import dev, jf, kernel_path, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("env,n,same", [
    ({"JFNK_EP3D_CLUSTER_MAX_N": "0"}, 33, True),    # no cluster at all
    ({"JFNK_EP3D_CLUSTER_MAX_N": "0"}, 20, True),
    ({"JFNK_EP3D_CLUSTER_MIN_N": "12"}, 33, True),   # clusters for 12 to 16
    ({"JFNK_EP3D_CLUSTER_MAX_N": "20"}, 33, True),   # clusters for 16 to 20
    ({"JFNK_EP3D_CLUSTER_MAX_N": "20"}, 20, False),
])
def test_cluster_range_is_about_its_levels(env, n, same, monkeypatch):
    kernel_path(monkeypatch, "default")
    u = dev(np.random.default_rng(n).normal(size=(n + 1,) * 3), torch.float32)
    want = jf().Problem("nd3d", n, 1).residual(u)
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    got = jf().Problem("nd3d", n, 1).residual(u)
    assert torch.equal(got, want) == same
