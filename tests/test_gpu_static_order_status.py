"""The allocation-free depth sort reports a bounded wait that ran out."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("after", [100, 5000, 600000])
def test_timeout_is_reported_and_cleared(gs3, after):
    """The self-test's first pass waits for words that no block writes; the next call, of one block
    or of several, clears the status and sorts."""
    import torch
    from paper_2410_11419_gb300 import _native as N
    stream = torch.cuda.current_stream().cuda_stream
    assert N.gs3_selftest_depth_order_timeout(20000) == N.GS3_ERR_TIMEOUT
    assert N.gs3_depth_order_static_status(stream) == N.GS3_ERR_TIMEOUT
    host = np.random.default_rng(after).integers(0, 1 << 20, after, dtype=np.uint32)
    out = torch.full((after,), -1, dtype=torch.int32, device="cuda")
    N.gs3_depth_order_static(torch.from_numpy(host.view(np.int32)).cuda(), after, out, stream)
    assert N.gs3_depth_order_static_status(stream) == N.GS3_OK
    assert np.array_equal(out.cpu().numpy(), np.argsort(host, kind="stable"))
