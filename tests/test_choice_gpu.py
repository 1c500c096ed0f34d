"""The configurations that a plan and the host pipeline choose by themselves,
against the oracle: plans of one packet up to one round of tiles and more, with
and without n = 15; one large stream through the host pipeline in one call."""
import numpy as np
import pytest

from paper_1412_6862_gb300 import hd
from tests import gpu_cases as gc
from tests.test_batch_gpu import check_batch, make_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_6862_gb300 import build
    build.build()
    hd.lib()


# tiles on both sides of 2048 and 8192, where the choice changes
@pytest.mark.parametrize("lengths", [(3, 7, 31, 63, 127, 255), (7, 15, 63)])
@pytest.mark.parametrize("packets,max_cw", [(1, 40), (2, 5000), (40, 3000), (300, 20_000), (250, 90_000)])
def test_plan_default(packets, max_cw, lengths):
    import torch
    pkts, exp = make_batch(packets, seed=packets + len(lengths), max_cw=max_cw, lengths=lengths)
    plan = hd.Plan(pkts)
    err = torch.full((packets,), 77, dtype=torch.int64, device="cuda")
    for _ in range(2):
        for p in pkts:
            p[1].fill_(-1)
        plan.launch(err)
        torch.cuda.synchronize()
        check_batch(pkts, exp, err)
    plan.close()
    assert hd.hd_device_status() == 0


# one chunk just below and above 24 MB of copies (cut into four pieces), ragged, pinned and pageable
@pytest.mark.parametrize("N", [1_550_003, 1_572_864, 1_700_003])
@pytest.mark.parametrize("pinned", [True, False])
def test_host_one_large_stream(N, pinned):
    import torch
    n, k = 63, 57
    stream, _, _ = gc.received_stream(n, N, seed=N, p1=0.1, p2=0.01)
    exp_out, exp_syn, exp_err = gc.expected(stream, n, N, hd.SYN_U8)
    src = torch.from_numpy(stream.view(np.int32).copy())
    out, sy = torch.zeros(hd.words_for(N * k), dtype=torch.int32), torch.zeros(N, dtype=torch.uint8)
    if pinned:
        src, out, sy = src.pin_memory(), out.pin_memory(), sy.pin_memory()
    _, _, e = hd.decode_host(src, n, N, syn_type=hd.SYN_U8, out=out, syndromes=sy)
    assert np.array_equal(out.numpy().view(np.uint32)[:exp_out.size], exp_out)
    assert np.array_equal(sy.numpy()[:N], exp_syn) and e == exp_err
