"""Depth orders of up to 4096 keys, which one block sorts, around its rounds of
512 keys, and the first size past it; ties keep their order, keys use all 32 bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 511, 512, 513, 1536, 1537, 4095, 4096, 4097])
@pytest.mark.parametrize("kind", ["wide", "ties", "same", "falling"])
def test_small_sorts(gs3, n, kind):
    import torch
    from paper_2410_11419_gb300 import _native as N
    g = np.random.default_rng(n)
    host = {"wide": lambda: g.integers(0, 1 << 32, n, dtype=np.uint32),
            "ties": lambda: g.integers(0, 7, n, dtype=np.uint32) * np.uint32(0x10010011),
            "same": lambda: np.full(n, 0x3F800000, np.uint32),
            "falling": lambda: np.arange(n, 0, -1, dtype=np.uint32) * np.uint32(1 << 19)}[kind]()
    out = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    N.gs3_depth_order_static(torch.from_numpy(host.view(np.int32)).cuda(), n, out,
                             torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(out.cpu().numpy(), np.argsort(host, kind="stable"))
