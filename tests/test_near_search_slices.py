"""Near-singular search where many panels share a cell (cells are sized by the largest panel over the
threshold): every slice of a cell is searched, and none of them by a warp alone for the whole cell."""
import time

import numpy as np
import pytest

from paper_1812_10722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _near_pairs(v, t, thr):
    p = v[t]
    c = p.mean(1)
    L = np.sqrt(np.linalg.norm(np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), axis=1))
    d = np.linalg.norm(c[:, None] - c[None], axis=2)
    np.fill_diagonal(d, np.inf)
    return int(np.count_nonzero(L[None] / d >= thr))


@pytest.mark.parametrize("thr", [0.011, 0.037, 0.083, 0.19, 0.41])
@pytest.mark.parametrize("sub", [0, 1, 2, 3])
def test_pairs_of_crowded_cells(sub, thr):
    # from all panels in one cell (20 to 1280) to a few per cell
    from paper_1812_10722_gb300 import lspr
    v, t = I.icosphere(sub, 10.0)
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t, threshold=thr)
        assert ctx.info()["n_near"] - len(t) == _near_pairs(v, t, thr)


def test_mixed_panel_sizes_take_no_serial_search():
    # 20 large panels beside 5120 small ones, which share a few cells: 1.5 ms, 4.6 with a warp per panel and
    # 224 with a warp per cell
    from paper_1812_10722_gb300 import lspr
    vb, tb = I.icosphere(0, 10.0)
    vs, ts = I.icosphere(4, 1.0)
    v = np.concatenate([vb, vs + vb[0] * 1.15])
    t = np.concatenate([tb, ts + len(vb)]).astype(np.int32)
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        dt = []
        for _ in range(5):
            t0 = time.perf_counter()
            ctx.mesh_upload(v, t)
            dt.append(time.perf_counter() - t0)
    assert sorted(dt)[2] < 0.03
