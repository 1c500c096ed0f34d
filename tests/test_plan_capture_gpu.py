"""A plan's launch recorded into the caller's graph, in every configuration."""
import pytest

from paper_1412_6862_gb300 import hd
from tests.test_batch_gpu import check_batch, make_batch

pytestmark = pytest.mark.gpu

PACKETS = 150


@pytest.fixture(scope="module")
def batch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_6862_gb300 import build
    build.build()
    hd.lib()
    return make_batch(PACKETS, seed=91, max_cw=30_000)


# with and without a launch before the capture (which resolves the configuration, or records its graph)
@pytest.mark.parametrize("first", [False, True])
@pytest.mark.parametrize("variant", range(10))
def test_captured_and_replayed(batch, variant, first):
    import torch
    pkts, exp = batch
    plan = hd.Plan(pkts)
    plan.select(variant)
    err = torch.full((PACKETS,), 77, dtype=torch.int64, device="cuda")
    if first:
        plan.launch(err)
        torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        plan.launch(err, cuda_stream=stream)
    for _ in range(2):
        for p in pkts:
            p[1].fill_(-1)
        err.fill_(77)
        graph.replay()
        torch.cuda.synchronize()
        check_batch(pkts, exp, err)
    for p in pkts:
        p[1].fill_(-1)
    plan.launch(err)  # not captured again
    torch.cuda.synchronize()
    check_batch(pkts, exp, err)
    plan.close()
    assert hd.hd_device_status() == 0
