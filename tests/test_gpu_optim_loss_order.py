"""The optimiser's, the loss's and the allocation-free depth sort's kernels at
the edges of their tiles, vector groups and block-size switch."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 1024, 4097])
@pytest.mark.parametrize("offset", [0, 1])
def test_adam_step_groups_and_rests(gs3, n, offset):
    """16-byte aligned arrays go four elements at a time, the rest and unaligned arrays one by one."""
    import torch
    from paper_2410_11419_gb300 import _native as N
    g = torch.Generator().manual_seed(10 * n + offset)
    host = [torch.randn(n + offset + 3, generator=g) for _ in range(3)] + [torch.rand(n + offset + 3, generator=g)]
    p, grad, m, v = (x.cuda() for x in host)
    view = [x[offset:offset + n] for x in (p, grad, m, v)]
    lr, b1, b2, eps, step, lo = 1e-2, 0.9, 0.999, 1e-15, 7, -0.5
    N.gs3_adam_step(*view, lr, b1, b2, eps, step, lo, torch.cuda.current_stream().cuda_stream)
    f1, f2, f3 = (float(np.float32(x)) for x in (b1, b2, lr))
    p0, g0, m0, v0 = (x.double().numpy()[offset:offset + n] for x in host)
    m1 = f1 * m0 + (1 - f1) * g0
    v1 = f2 * v0 + (1 - f2) * g0 * g0
    d = f3 * (m1 / (1 - f1 ** step)) / (np.sqrt(v1 / (1 - f2 ** step)) + eps)
    p1 = np.maximum(lo, p0 - d)
    # FP32 roundings (2^-24 each): two per moment on terms that may cancel, and
    # about eight in the step, whose moments carry theirs
    u = 2.0 ** -24
    em, ev = 2 * u * (np.abs(f1 * m0) + np.abs((1 - f1) * g0)), 3 * u * v1
    ed = np.abs(d) * (8 * u + ev / (2 * v1)) + em * np.abs(d / np.where(m1 == 0, 1, m1))
    for x, want, tol in ((m, m1, em), (v, v1, ev), (p, p1, ed + 2 * u * np.abs(p0))):
        x = x.cpu().double().numpy()
        assert np.all(np.abs(x[offset:offset + n] - want) <= tol + 1e-30)
    for x, h in zip((p, m, v), (host[0], host[2], host[3])):  # nothing outside the range changes
        keep = np.r_[0:offset, offset + n:n + offset + 3]
        assert np.array_equal(x.cpu().numpy()[keep], h.numpy()[keep])


@pytest.mark.parametrize("w,h", [(1, 1), (5, 70), (31, 33), (32, 32), (33, 31), (64, 96), (101, 7)])
def test_loss_tile_edges(gs3, oracle, w, h):
    """Images around the 32-pixel tiles and smaller than the 11-pixel window, against the FP64 loss."""
    import torch
    from oracle import torch_ref as TR
    from paper_2410_11419_gb300 import render as R
    g = torch.Generator().manual_seed(w * 1000 + h)
    img, tgt = torch.rand((h, w, 3), generator=g), torch.rand((h, w, 3), generator=g)
    loss, dimg = R.loss_l1_dssim(img.cuda(), tgt.cuda())
    want, L = TR.image_grad_of_loss(img.numpy(), tgt.numpy())
    # the window sums carry 22 FP32 roundings each; the variance differences
    # (squares minus squared means, at least C2 = 9e-4 below sums of about 1)
    # amplify them by up to about 1e3
    tol = 1e3 * 22 * 2.0 ** -24
    assert abs(float(loss) - L) <= tol
    assert np.abs(dimg.cpu().numpy() - want).max() <= tol * max(1e-12, np.abs(want).max())


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 5000, 524288, 524289])
def test_depth_order_block_sizes(gs3, n):
    """1024 keys per block up to 512 blocks, 2048 past that; ties keep their order."""
    import torch
    from paper_2410_11419_gb300 import _native as N
    host = np.random.default_rng(n).integers(0, 1 << 18, n, dtype=np.uint32) * np.uint32(9973)
    out = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    N.gs3_depth_order_static(torch.from_numpy(host.view(np.int32)).cuda(), n, out,
                             torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(out.cpu().numpy(), np.argsort(host, kind="stable"))
