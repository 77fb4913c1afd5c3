"""Device buffers that the library's kernels use in place against the copying routes (host memory, a
buffer off its 4-byte boundary): the same bits, since only the way in and out differs."""
import numpy as np
import pytest

from tests.test_gpu_parity import small_sphere
from tests.test_gpu_precondition import ctx_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 32, 48, 81])
def test_precondition_in_place_matches_host_buffers(n):
    import torch

    from paper_2509_18097_gb300 import binding as B

    g = np.random.Generator(np.random.PCG64(n)).standard_normal((n**3, 3)).astype(np.float32)
    ctx = ctx_for(B, n, lam0=0.7)
    try:
        ref = B.pdg_precondition(ctx, 0, g, np.empty_like(g))
        gd = torch.from_numpy(g).cuda()
        out = B.pdg_precondition(ctx, 0, gd, torch.full_like(gd, float("nan")))
        assert np.array_equal(out.cpu().numpy(), ref)
        assert np.array_equal(gd.cpu().numpy(), g)  # the input is only read
        B.pdg_precondition(ctx, 0, gd, gd)  # out may be g
        assert np.array_equal(gd.cpu().numpy(), ref)
    finally:
        B.pdg_destroy(ctx)


@pytest.mark.parametrize("res", [(1, 4, 16), (6, 27)])
def test_read_into_device_and_unaligned_buffers(res):
    import torch

    from paper_2509_18097_gb300 import binding as B

    w = small_sphere(seed=71, n_src=300, n_tgt=321, res=res)
    ctx = B.pdg_create(B.pdg_config_default(res=res), w.template, w.edges, w.source, max_pts=321)
    try:
        B.pdg_begin_frame(ctx, w.target)
        B.pdg_step(ctx, 2)
        rows = len(w.template) + len(w.source)
        for which, level, k in [(B.BUF_Y, 0, rows), (B.BUF_POINT_GRAD, 0, rows)] + [
                (b, l, n**3) for l, n in enumerate(res) for b in (B.BUF_THETA, B.BUF_GRAD)]:
            host = B.pdg_read(ctx, which, level, np.empty((k, 3), np.float32))
            dev = B.pdg_read(ctx, which, level, torch.empty((k, 3), device="cuda"))
            raw = torch.empty(12 * k + 1, dtype=torch.uint8, device="cuda")[1:]
            B.pdg_read(ctx, which, level, raw)
            assert np.array_equal(dev.cpu().numpy(), host)
            assert np.array_equal(raw.cpu().numpy().view(np.float32).reshape(k, 3), host)
    finally:
        B.pdg_destroy(ctx)


def test_grid_loss_same_on_host_and_device_grids():
    import torch

    from paper_2509_18097_gb300 import binding as B
    from paper_2509_18097_gb300.autograd import grid_loss

    w = small_sphere(seed=72, n_src=500, n_tgt=400)
    ctx = B.pdg_create(B.pdg_config_default(res=w.res), w.template, w.edges, w.source, max_pts=500)
    got = []
    try:
        B.pdg_begin_frame(ctx, w.target)
        for dev in ("cpu", "cuda"):
            th = [torch.tensor(t, device=dev, requires_grad=True) for t in w.thetas]
            loss = grid_loss(ctx, th)
            (2.0 * loss).backward()
            assert loss.device.type == dev and loss.dtype == torch.float64
            got.append([loss.item()] + [t.grad.cpu().numpy() for t in th])
    finally:
        B.pdg_destroy(ctx)
    assert got[0][0] == got[1][0]
    for a, b in zip(got[0][1:], got[1][1:]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("dev", ["cpu", "cuda"])
def test_grid_loss_may_be_changed_in_place(dev):
    import torch

    from paper_2509_18097_gb300 import binding as B
    from paper_2509_18097_gb300.autograd import grid_loss

    w = small_sphere(seed=73, n_src=300, n_tgt=200)
    ctx = B.pdg_create(B.pdg_config_default(res=w.res), w.template, w.edges, w.source, max_pts=300)
    try:
        B.pdg_begin_frame(ctx, w.target)
        th = [torch.tensor(t, device=dev, requires_grad=True) for t in w.thetas]
        grid_loss(ctx, th).backward()
        plain = [t.grad.clone() for t in th]
        for t in th:
            t.grad = None
        loss = grid_loss(ctx, th)
        before = loss.item()
        loss *= 2.0
        loss += sum((t.double() ** 2).sum() for t in th)
        loss.backward()
        assert loss.item() == 2.0 * before + sum((t.detach().double() ** 2).sum() for t in th).item()
        for t, g in zip(th, plain):  # the regulariser's part is 2 theta; both sums in FP32
            d = (t.grad - (2.0 * g + 2.0 * t.detach())).abs().max()
            assert d <= 2.0**-22 * (2.0 * g.abs().max() + 2.0 * t.detach().abs().max())
    finally:
        B.pdg_destroy(ctx)
