"""The line path of the preconditioner (k_sobolev_x.cu, k_sobolev_yz.cu): every size whose tiles
have a remainder or whose transform has its own radices and that no other test runs, on a random
gradient against the operator in its eigenbasis (FP64 DCT-II); and the z-planes without an active
vertex, which the forward passes skip.

Tolerance: check_close's 1e-6 of max|result| plus 1e-5 relative.  Six length-n transforms of FP32
butterflies add O(log2 n) * 6e-8 of the level's norm each; the operator only shrinks (its
eigenvalues lie in (0, 1]), and a white gradient of unit variance gives outputs of order one, so
the sum stays near 3e-7 of the norm, below 1e-6 of the largest of millions of values."""
import numpy as np
import pytest

from oracle import pdg_oracle as O
from paper_2509_18097_gb300 import synth
from tests import gpu_helpers as H
from tests.test_gpu_precondition import ctx_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 12, 18, 36, 54, 72, 81, 108, 144, 243, 256])
def test_random_gradient_matches_eigenbasis(n):
    from paper_2509_18097_gb300 import binding as B

    lam = 0.84375
    g = np.random.Generator(np.random.PCG64(n)).standard_normal((n**3, 3)).astype(np.float32)
    ctx = ctx_for(B, n, lam0=lam)
    try:
        out = B.pdg_precondition(ctx, 0, g, np.empty_like(g))
    finally:
        B.pdg_destroy(ctx)
    ref = O.sobolev_precondition_spectral(g.reshape(n, n, n, 3).astype(np.float64), lam).reshape(-1, 3)
    H.check_close(f"n={n}", out, ref)


@pytest.mark.parametrize("n,before", [(36, 2.640e-7), (108, 3.193e-7), (162, 3.353e-7), (216, 3.481e-7)])
def test_error_no_larger_than_before_the_register_transforms(n, before):
    """Relative RMS error against FP64 of a white gradient; `before`: that of the Stockham transforms in
    shared memory, which the register transforms replaced, on the same input."""
    from paper_2509_18097_gb300 import binding as B

    g = np.random.Generator(np.random.PCG64(1000 + n)).standard_normal((n**3, 3)).astype(np.float32)
    ctx = ctx_for(B, n, lam0=0.25)
    try:
        out = B.pdg_precondition(ctx, 0, g, np.empty_like(g))
    finally:
        B.pdg_destroy(ctx)
    ref = O.sobolev_precondition_spectral(g.reshape(n, n, n, 3).astype(np.float64), 0.25).reshape(-1, 3)
    assert np.sqrt(((out - ref) ** 2).mean() / (ref**2).mean()) <= before


@pytest.mark.parametrize("lam", [1e20, 1e38])
@pytest.mark.parametrize("n", [6, 27, 96])
def test_largest_lambdas_leave_the_mean(n, lam):
    """Any finite lambda is accepted.  The operator then keeps the constant mode alone (the next factor,
    (1 + lambda mu)^-2, is below 1e-34), whatever the intermediate products overflow to.  Tolerance as
    above: the gradient's mean is 1, its deviation 0.1, so the result is as large as the terms."""
    from paper_2509_18097_gb300 import binding as B

    r = np.random.Generator(np.random.PCG64(n))
    g = (1.0 + 0.1 * r.standard_normal((n**3, 3))).astype(np.float32)
    ctx = ctx_for(B, n, lam0=lam)
    try:
        out = B.pdg_precondition(ctx, 0, g, np.empty_like(g))
    finally:
        B.pdg_destroy(ctx)
    assert np.isfinite(out).all()
    H.check_close(f"n={n} lambda={lam}", out, np.broadcast_to(g.astype(np.float64).mean(0), out.shape))


@pytest.mark.parametrize("res", [(27, 54), (48, 81)])
def test_planes_without_active_vertices(res):
    """A frame whose points lie in a thin slab after one that filled the domain: what the first
    frame left in the skipped planes must not reach the second (bitwise a new context's)."""
    from paper_2509_18097_gb300 import binding as B

    r = np.random.Generator(np.random.PCG64(3))
    v, _, e = synth.icosphere(2)
    flat = lambda p: (p * np.array([1.0, 1.0, 0.05]) + np.array([0.0, 0.0, 0.4])).astype(np.float32)  # noqa: E731
    wide, slab = synth.sphere_points(r, 700).astype(np.float32) * 1.3, flat(synth.sphere_points(r, 600))
    out = []
    for first in (wide, slab):
        ctx = B.pdg_create(B.pdg_config_default(res=res), flat(v), e, first, max_pts=700)
        try:
            B.pdg_set_debug(ctx, True)
            if first is wide:  # its end makes the slab the source cloud; the template stays in place
                B.pdg_begin_frame(ctx, wide)
                B.pdg_step(ctx, 1)
                for l, n in enumerate(res):
                    B.pdg_write_theta(ctx, l, np.zeros((n**3, 3), np.float32))
                B.pdg_end_frame(ctx)
                B.pdg_fit_frame(ctx, slab, 0)
            B.pdg_begin_frame(ctx, slab)
            B.pdg_step(ctx, 1)
            out.append([B.pdg_read(ctx, B.BUF_PGRAD, l, np.empty((n**3, 3), np.float32)) for l, n in enumerate(res)])
        finally:
            B.pdg_destroy(ctx)
    for a, b in zip(*out):
        assert np.abs(a).max() > 0
        assert np.array_equal(a, b)
