"""A caller that captures its own CUDA graph warms a solve up first.  Right-hand-side counts share
buffers per bucket (the next power of two), so a count of a warmed bucket must not allocate: in a
capture an allocation is an error.  The replayed solve gives what the launched one gives, to the
order of FP32 sums.
"""

import pytest

from test_gpu_mm import Blocks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm,nrhs", [(17, 32), (33, 60), (65, 120)])
def test_capture_of_a_larger_count_in_a_warm_bucket(warm, nrhs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B = Blocks(nrhs, 1.0)
    A = B.operator()
    opts = dict(n_terms=2, n_levels=1, refine=True, graph=False)
    b, _ = B.vectors(nrhs)
    bt = torch.from_numpy(b).cuda()
    want, got = torch.empty_like(bt), torch.zeros_like(bt)
    A.solve(bt[:warm].contiguous(), torch.empty_like(bt[:warm]), **opts)
    torch.cuda.synchronize()
    held = A.info().device_bytes
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        g.capture_begin()
        A.solve(bt, got, stream=s, **opts)
        g.capture_end()
    assert A.info().device_bytes == held
    g.replay()
    torch.cuda.synchronize()
    A.solve(bt, want, **opts)
    A.sync_status()
    assert (got - want).abs().max() <= 1e-5 * want.abs().max()
    A.close()
