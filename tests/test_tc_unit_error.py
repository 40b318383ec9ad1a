"""Error of the tensor-core far field on a tree large enough for its longest work units, for smooth vectors:
sums of one sign, whose FP32 accumulation rounds the same way at every step."""
import numpy as np
import pytest

from paper_1812_10722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _smooth(c, B, seed):
    rng = np.random.default_rng(seed)
    cols = []
    for _ in range(2 * B):
        k, ph, a = 1.5 * rng.normal(size=3), rng.uniform(0, 2 * np.pi), rng.normal(size=2)
        cols.append((1.0 + 0.5 * np.cos(c @ k + ph)) * complex(*a))
    return np.stack([np.concatenate([cols[2 * j], cols[2 * j + 1] / 5]) for j in range(B)])


# bounds: the errors of TF32 parts in units of 32 boxes and 2048 sources, measured on these inputs (M2P,
# P2P, and both on the tensor cores)
@pytest.mark.parametrize("B,bounds", [(32, (4.74e-6, 1.59e-6, 6.13e-6)), (64, (4.73e-6, 2.06e-6, 6.57e-6))])
def test_smooth_vectors_on_long_units(B, bounds):
    from paper_1812_10722_gb300 import lspr
    v, t = I.icosphere(6, 10.0)   # 81920 panels
    x = _smooth(v[t].mean(1) / 10.0, B, 3)
    s = np.full(B, I.drude_eps(380.0) / I.EPS_WATER)
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        ctx.tree_build(0.4, 7, 512)
        ref = ctx.matvec(x, s, "tree_ff")
        err = []
        for mask in (1, 2, 3):
            ctx.set_tensor_cores(mask)
            y = ctx.matvec(x, s, "tree_fp32")
            err.append(np.linalg.norm(y - ref) / np.linalg.norm(ref))
        assert ctx.device_errors() == 0
    assert all(e <= b for e, b in zip(err, bounds)), err
