"""Launches of one plan on several streams: they share the plan's claim counters,
so each has to begin behind the one before, whatever stream that was on."""
import pytest

from paper_1412_6862_gb300 import hd
from tests.test_batch_gpu import check_batch, make_batch

pytestmark = pytest.mark.gpu

PACKETS = 200


@pytest.fixture(scope="module")
def batch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_6862_gb300 import build
    build.build()
    hd.lib()
    return make_batch(PACKETS, seed=77, max_cw=60_000)


# every configuration: the single-kernel ones are launched directly, the others as a graph
@pytest.mark.parametrize("variant", range(10))
def test_two_streams_without_waiting(batch, variant):
    import torch
    pkts, exp = batch
    plan = hd.Plan(pkts)
    if variant >= plan.info()["num_variants"]:
        pytest.skip("no such configuration")
    plan.select(variant)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    errs = [torch.full((PACKETS,), 77, dtype=torch.int64, device="cuda") for _ in range(7)]
    for p in pkts:
        p[1].fill_(-1)
    torch.cuda.synchronize()
    for i in range(24):  # the last seven launches' counts are looked at, each in its own array
        plan.launch(errs[i % len(errs)], cuda_stream=streams[i % 2])
    torch.cuda.synchronize()
    for err in errs:
        check_batch(pkts, exp, err)
    # one array of counts for both streams, three streams, one of them new at each turn
    for i in range(12):
        plan.launch(errs[0], cuda_stream=streams[i % 2] if i % 3 else torch.cuda.Stream())
    torch.cuda.synchronize()
    check_batch(pkts, exp, errs[0])
    plan.close()
    assert hd.hd_device_status() == 0
