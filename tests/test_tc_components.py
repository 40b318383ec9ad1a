"""Tensor-core far field of vectors whose real and imaginary parts differ much in size.  With a real ratio
of permittivities the two are separate real products, and each keeps the bound of the product."""
import numpy as np
import pytest

from paper_1812_10722_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", [1e-9, 1e-18])
@pytest.mark.parametrize("B,mask", [(2, 1), (16, 1), (20, 1), (26, 3), (33, 3), (64, 3)])
def test_small_real_or_imaginary_parts(B, mask, small):
    from paper_1812_10722_gb300 import lspr
    v, t = I.icosphere(4, 10.0)
    n2 = 2 * len(t)
    x = I.random_complex(n2, seed=B, batch=B)
    x.imag[::2] *= small          # even columns: small imaginary parts, odd ones: small real parts
    x.real[1::2] *= small
    x.imag[0, n2 // 2:] /= small  # column 0: in phi only
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        ctx.tree_build(0.5, 6, 60)
        ctx.set_tensor_cores(mask)
        y = ctx.matvec(x, np.full(B, 1.7), "tree_fp32")
        ref = ctx.matvec(x, np.full(B, 1.7), "tree_ff")
        assert ctx.device_errors() == 0
    for j in range(B):
        for a, b in ((y[j].real, ref[j].real), (y[j].imag, ref[j].imag)):
            assert np.linalg.norm(a - b) < 3e-5 * np.linalg.norm(b), j


# right-hand sides beyond one block column of the scaling kernels (512), and channel sets of two surfaces
@pytest.mark.parametrize("B,mask,two", [(520, 1, False), (520, 3, False), (5, 1, True), (20, 3, True), (270, 3, True)])
def test_small_parts_of_many_sets(B, mask, two):
    from paper_1812_10722_gb300 import lspr
    v, t = I.icosphere(3, 10.0)
    surf = None
    if two:
        surf = np.repeat(np.arange(2, dtype=np.int32), len(t))
        v, t = np.concatenate([v, 0.5 * v + [0.0, 0.0, 16.0]]), np.concatenate([t, t + len(v)]).astype(np.int32)
    x = I.random_complex(2 * len(t), seed=B, batch=B)
    x.imag[::2] *= 1e-9
    x.real[1::2] *= 1e-9
    s = np.tile([1.7, 0.6], (B, 1)) if two else np.full(B, 1.7)
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t, surf_id=surf)
        ctx.tree_build(0.5, 6, 60)
        ctx.set_tensor_cores(mask)
        y = ctx.matvec(x, s, "tree_fp32")
        ref = ctx.matvec(x, s, "tree_ff")
        assert ctx.device_errors() == 0
    for j in range(B):
        for a, b in ((y[j].real, ref[j].real), (y[j].imag, ref[j].imag)):
            assert np.linalg.norm(a - b) < 3e-5 * np.linalg.norm(b), j
