"""Tensor-core far field of right-hand sides with a zero layer, zero or tiny ones, on boxes smaller than
one length unit (their scale lengths enter the operands to the power of the order)."""
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


def _batch(n, B, seed, tiny):
    """Columns with phi = 0, dphi = 0, both, a tiny factor on all or on one layer, and ordinary ones."""
    x = I.random_complex(2 * n, seed=seed, batch=B)
    x[0, :n] = 0.0
    x[1, n:] = 0.0
    if B > 2:
        x[2] = 0.0
        x[3] *= tiny
        x[4, n:] *= tiny
        x[5, :n] *= tiny
    return x


# scale lengths 1/16 and 1/4 (R = 0.3, 1), below 1e-4 (R = 1e-3), and 1/4 to 1 (20480 panels, R = 10);
# parts of, one and two units of right-hand sides; M2P alone and with the P2P.  The tiny factors leave the
# FP32 moments (weight times radius to the order) normal or nearly so
@pytest.mark.parametrize("B,mask", [(2, 1), (16, 1), (26, 3), (64, 3)])
@pytest.mark.parametrize("sub,R,P,ncrit,tiny", [(3, 1.0, 8, 40, 1e-25), (3, 0.3, 4, 40, 1e-25), (3, 0.3, 7, 40, 1e-25),
                                                (3, 1e-3, 6, 40, 1e-3), (5, 10.0, 5, 256, 1e-25)])
def test_zero_and_tiny_layers(lspr, sub, R, P, ncrit, tiny, B, mask):
    # against the float-float operator at the bound of the tensor-core product
    v, t = I.icosphere(sub, R)
    x = _batch(len(t), B, B + P, tiny)
    s = np.full(B, I.drude_eps(380.0) / I.EPS_WATER)
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        ctx.tree_build(0.5, P, ncrit)
        ctx.set_tensor_cores(mask)
        y = ctx.matvec(x, s, "tree_fp32")
        ref = ctx.matvec(x, s, "tree_ff")
        assert ctx.device_errors() == 0
    assert np.all(np.isfinite(y))
    for j in range(B):
        if np.any(x[j]):
            assert _rel(y[j], ref[j]) < 3e-5, j
        else:
            assert np.all(y[j] == 0.0)


def test_unrefined_solve_with_an_index_matched_wavelength(lspr):
    # eps_in = eps_out: b = 0, x = 0, and the explicit residual after the others' cycle is A 0 = 0
    v, t = I.icosphere(4, 3.0)
    lam = I.wavelengths(370, 390, 3)
    ep = np.asarray(I.drude_eps(lam))
    kw = dict(tol=1e-4, mode="tree_fp32", maxiter=2000)
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        ctx.tree_build(0.5, 6, 100)
        ref = ctx.solve(ep, I.EPS_WATER, lam, **kw)
        ep[1] = I.EPS_WATER
        got = ctx.solve(ep, I.EPS_WATER, lam, **kw)
    assert got.sigma_ext[1] == 0.0
    # two solves to 1e-4 of the same systems
    assert np.allclose(got.sigma_ext[[0, 2]], ref.sigma_ext[[0, 2]], rtol=1e-2)
