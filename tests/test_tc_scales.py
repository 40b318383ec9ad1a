"""Scales of the tensor-core far field's FP16 operands: inputs of any magnitude, right-hand sides of
very different ones, meshes of any size on a recorded graph, and the TF32 parts that very different
P2P distances fall back to."""
import numpy as np
import pytest

from paper_1812_10722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lspr():
    from paper_1812_10722_gb300 import lspr as L
    return L


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("B,mask", [(5, 1), (26, 3), (40, 3), (70, 3)])
def test_magnitudes_of_the_right_hand_sides(lspr, B, mask):
    # column j carries the factor c_j; every product is linear, so y_j = c_j y(x_j).  FP32 products of
    # the two scalings differ by their roundings: 3e-5, the bound of the tensor-core product
    v, t = I.icosphere(3, 10.0)
    x = I.random_complex(2 * len(t), seed=B, batch=B)
    s = np.full(B, I.drude_eps(380.0) / I.EPS_WATER)
    c = 10.0 ** np.linspace(-25, 20, B)
    c[1] = 0.0
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        ctx.tree_build(0.5, 6, 40)
        ctx.set_tensor_cores(mask)
        y1 = ctx.matvec(x, s, "tree_fp32")
        yc = ctx.matvec(x * c[:, None], s, "tree_fp32")
        xn = x.copy()
        xn[2, 7] = np.nan
        yn = ctx.matvec(xn, s, "tree_fp32")
        ref = ctx.matvec(x, s, "tree_ff")
    assert np.all(yc[1] == 0.0)
    for j in range(B):
        assert _rel(y1[j], ref[j]) < 3e-5
        if j != 1:
            assert _rel(yc[j] / c[j], y1[j]) < 3e-5, (j, c[j])
        if j == 2:
            assert not np.all(np.isfinite(yn[j]))
        else:
            assert _rel(yn[j], y1[j]) < 3e-5, j


@pytest.mark.parametrize("B", [24, 33, 64])
@pytest.mark.parametrize("gap", [1.0, 5e-4])
def test_p2p_distances_choose_the_parts(lspr, B, gap):
    # a copy of panel 0 moved along its normal: its nodes lie `gap` from that panel's centroid, so 5e-4 nm
    # makes the ratio of P2P distances larger than 4096 (TF32 parts) and 1 nm does not (FP16).  The panel
    # sits at the origin, where FP32 coordinates resolve the gap.  Both against the FP32 pipe's P2P on the
    # same FP32 coordinates, at the bound of the tensor-core product.
    v, t = I.icosphere(3, 10.0)
    v = v - v[t[0]].mean(0)
    p = v[t[0]]
    n = np.cross(p[1] - p[0], p[2] - p[0])
    v = np.concatenate([v, p + gap * n / np.linalg.norm(n)])
    t = np.concatenate([t, [[len(v) - 3, len(v) - 2, len(v) - 1]]]).astype(np.int32)
    x = I.random_complex(2 * len(t), seed=B, batch=B)
    s = np.full(B, I.drude_eps(380.0) / I.EPS_WATER)
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        ctx.tree_build(0.5, 6, 500)
        ref = ctx.matvec(x, s, "tree_fp32")
        ctx.set_tensor_cores(3)
        y = ctx.matvec(x, s, "tree_fp32")
        assert ctx.device_errors() == 0
    for j in range(B):
        assert _rel(y[j], ref[j]) < 3e-5


def test_recorded_graph_follows_the_mesh_size(lspr):
    # the same mesh in other units has the same sizes everywhere: the graph recorded for the first must
    # not serve the second with the first's scales
    lam = I.wavelengths(360, 400, 26)
    ep = I.drude_eps(lam)
    kw = dict(tol=1e-6, mode="tree_fp32", refine=True, maxiter=2000)
    meshes = [I.icosphere(3, R) for R in (10.0, 160.0, 0.3)]
    with lspr.Context(0) as ctx:
        ctx.set_tensor_cores(3)
        sig = []
        for v, t in meshes + meshes[:1]:
            ctx.mesh_upload(v, t)
            ctx.tree_build(0.5, 6, 40)
            sig.append(ctx.solve(ep, I.EPS_WATER, lam, **kw).sigma_ext)
        assert ctx.device_errors() == 0
    for q, R in enumerate((10.0, 160.0, 0.3, 10.0)):   # sigma scales with R^3 in the quasistatic limit
        assert np.allclose(sig[q] * (10.0 / R) ** 3, sig[0], rtol=1e-4)


@pytest.mark.parametrize("B", [1, 3])
def test_vectors_from_another_stream(lspr, B):
    torch = pytest.importorskip("torch")
    v, t = I.icosphere(3, 10.0)
    s = np.full(B, I.drude_eps(380.0) / I.EPS_WATER)
    x = torch.as_tensor(I.random_complex(2 * len(t), seed=4, batch=B), device="cuda")
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        want = ctx.matvec(x, s, "direct_fp64")
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            big = torch.ones(1 << 27, device="cuda")
            for _ in range(20):
                big = big * 1.0000001
            xs = x * (big[0] * 0 + 1)      # ready only after the work queued before it
            got = ctx.matvec(xs, s, "direct_fp64")
        torch.cuda.synchronize()
    assert torch.allclose(got, want, rtol=1e-12, atol=0)
