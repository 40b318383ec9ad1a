"""Near-singular search on a mesh of very different panel sizes: the cells (sized by the largest panel)
then hold more small panels than a warp takes at a time, in targets and in candidates."""
import numpy as np
import pytest

from paper_1812_10722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sub,R", [(1, 1.0), (2, 1.0), (3, 0.5)])
def test_mixed_sizes_match_the_oracle(oracle, sub, R):
    from paper_1812_10722_gb300 import lspr
    vb, tb = I.icosphere(0, 10.0)          # 20 large panels
    vs, ts = I.icosphere(sub, R)           # small ones near one vertex of them
    vs = vs + vb[0] * 1.15
    v, t = np.concatenate([vb, vs]), np.concatenate([tb, ts + len(vb)]).astype(np.int32)
    x = I.random_complex(2 * len(t), seed=3)
    s = I.drude_eps(380.0) / I.EPS_WATER
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        assert ctx.info()["n_near"] - len(t) == oracle.near_pairs(v, t)[0]
        y = ctx.matvec(x, s, "direct_fp64")
    yo = oracle.matvec(v, t, x, s)
    # 1e-6: the bound of the direct FP64 product (the semi-analytical self integral at 9 nodes)
    assert np.linalg.norm(y - yo) < 1e-6 * np.linalg.norm(yo)
