"""The template-mesh solves in one launch (k_mesh.cu, k_mesh_solve): one, two and four vertices per
thread, a mesh too large for it (a launch per iteration), vertices with more neighbours than a
thread holds and with none.  One iteration each, every stage against the oracle on the GPU's own
input, at the tolerances of test_gpu_mesh.py (two Chebyshev solves to 1e-7, their FP32 recurrences
within 1.1e-6 of max|result|)."""
import numpy as np
import pytest

from paper_2509_18097_gb300 import synth
from tests import test_gpu_mesh as M

pytestmark = pytest.mark.gpu


def cloud(n=2000):
    r = np.random.Generator(np.random.PCG64(5))
    return (synth.torus_points(r, n) * 1.02).astype(np.float32)


# one thread block takes 512 vertices times those per thread, on at most 152 SMs
@pytest.mark.parametrize("nu,nv", [(27, 19), (396, 198), (560, 280), (800, 400)])
def test_torus(nu, nv):
    v, _, e = synth.torus_mesh(nu, nv)
    M.check_one_step(v, e, cloud())


def test_hub_and_isolated_vertices():
    r = np.random.Generator(np.random.PCG64(6))
    v = synth.torus_points(r, 60).astype(np.float32)
    e = np.stack([np.zeros(40, np.int32), np.arange(1, 41, dtype=np.int32)], 1)  # vertices 41..59 have no edge
    M.check_one_step(v, e, cloud(300))


def test_wait_that_runs_out_is_a_status_and_leaves_the_template():
    """40 blocks meet at 270 barriers an iteration; with one look each, the first to arrive gives up."""
    from paper_2509_18097_gb300 import binding as B

    v, _, e = synth.torus_mesh(200, 100)
    p0 = cloud()
    X = lambda c: B.pdg_get_vertices(c, np.empty((len(v), 3), np.float32))  # noqa: E731
    ctx, fresh = M.make_ctx(B, v, e, p0), M.make_ctx(B, v, e, p0)
    try:
        before = X(ctx)
        B.pdg_debug_mesh_wait(ctx, 1)
        with pytest.raises(B.PdgError) as ei:
            B.pdg_fit_mesh(ctx, p0, 3)
        assert ei.value.status == B.ERR_TIMEOUT
        assert np.array_equal(X(ctx), before)
        with pytest.raises(B.PdgError) as ei:
            B.pdg_read(ctx, B.BUF_MESH_PGRAD, 0, np.empty((len(v), 3), np.float32))
        assert ei.value.status == B.ERR_STATE
        B.pdg_debug_mesh_wait(ctx, 0)  # and the context works as before
        a, b = B.pdg_fit_mesh(ctx, p0, 3), B.pdg_fit_mesh(fresh, p0, 3)
        assert a.loss_total == b.loss_total
        assert np.array_equal(X(ctx), X(fresh))
        assert not np.array_equal(X(ctx), before)
    finally:
        B.pdg_destroy(ctx)
        B.pdg_destroy(fresh)


def star(degree):
    r = np.random.Generator(np.random.PCG64(7))
    v = synth.torus_points(r, degree + 1).astype(np.float32)
    return v, np.stack([np.zeros(degree, np.int32), np.arange(1, degree + 1, dtype=np.int32)], 1)


@pytest.mark.parametrize("degree", [4096, 4097])
def test_vertex_with_thousands_of_edges(degree):
    """Either side of the line beyond which a vertex's edges take longer than the others should wait.
    The hub's FP32 sum of its edges rounds by sqrt(degree) 6e-8 = 4e-6 of itself, a part of the result's
    scale after the solve: inside check_one_step's 1e-5."""
    v, e = star(degree)
    M.check_one_step(v, e, cloud(500), lam=0.01)


def test_no_wait_beside_a_vertex_with_thousands_of_edges():
    from paper_2509_18097_gb300 import binding as B

    v, e = star(4097)
    ctx = M.make_ctx(B, v, e, cloud(500))
    try:
        B.pdg_debug_mesh_wait(ctx, 1)  # any wait would run out
        assert B.pdg_fit_mesh(ctx, cloud(500), 1, 0.01).status == B.OK
    finally:
        B.pdg_destroy(ctx)


def test_refused_cooperative_launch_takes_the_other_form(monkeypatch):
    """The first iteration refused, and each of a fit's: against the oracle and, over several
    iterations, within Adam's steps of the one-launch fit (both solve to 1e-7; the sign of a gradient
    component within rounding of zero may differ, 2 lr a step)."""
    from paper_2509_18097_gb300 import binding as B

    make = M.make_ctx

    def refusing(*args, **kw):
        ctx = make(*args, **kw)
        B.pdg_debug_mesh_refuse(ctx, 1)
        return ctx

    v, _, e = synth.torus_mesh(60, 30)
    with monkeypatch.context() as m:
        m.setattr(M, "make_ctx", refusing)
        M.check_one_step(v, e, cloud())
    got = []
    for n in (0, 2, 5):
        ctx = make(B, v, e, cloud())
        try:
            B.pdg_debug_mesh_refuse(ctx, n)
            st = B.pdg_fit_mesh(ctx, cloud(), 5)
            got.append((st.cd_mesh, B.pdg_get_vertices(ctx, np.empty((len(v), 3), np.float32))))
        finally:
            B.pdg_destroy(ctx)
    for loss, x in got[1:]:
        assert abs(loss - got[0][0]) <= 1e-5 * got[0][0]
        assert np.abs(x - got[0][1]).max() <= 5 * 2 * M.LR
