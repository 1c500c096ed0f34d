"""What a plan resolves on its first launch holds for as long as it is true: not
past a missing decode table, not under another cap on the CTAs."""
import subprocess
import sys

import pytest

from paper_1412_6862_gb300 import hd
from tests.captured import Captured
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
    yield
    hd.hd_set_max_ctas(0)


def first_launch_captured(variant: int) -> None:
    """In a process of its own: the decode tables do not exist yet."""
    import torch
    hd.lib()
    pkts, exp = make_batch(60, seed=5)
    plan = hd.Plan(pkts)
    plan.select(variant)
    err = torch.full((60,), 77, dtype=torch.int64, device="cuda")
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        plan.launch(err, cuda_stream=stream)
    graph.replay()  # decodes without the tables
    torch.cuda.synchronize()
    check_batch(pkts, exp, err)
    counts = []
    for _ in range(2):
        for p in pkts:
            p[1].fill_(-1)
        before = hd.hd_launch_count()
        plan.launch(err)
        counts.append(hd.hd_launch_count() - before)
        torch.cuda.synchronize()
        check_batch(pkts, exp, err)
    # the first launch outside the capture fills the tables that the configuration reads
    tables = bin(plan.info()["table_lookup"]).count("1")
    assert counts == [2 + tables, 2], counts


@pytest.mark.parametrize("variant", [0, 7])  # the n = 7 table; both
def test_tables_missing_at_a_captured_first_launch(variant):
    code = f"from tests.test_plan_geometry_gpu import first_launch_captured as f; f({variant})"
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("variant", [0, 4])
def test_cap_set_after_the_first_launch(variant):
    import torch
    pkts, exp = make_batch(60, seed=6)
    plan = hd.Plan(pkts)
    plan.select(variant)
    err = torch.full((60,), 77, dtype=torch.int64, device="cuda")
    plan.launch(err)
    whole = Captured(lambda s: plan.launch(err, cuda_stream=s))
    hd.hd_set_max_ctas(3)
    capped = Captured(lambda s: plan.launch(err, cuda_stream=s))
    err.fill_(77)
    plan.launch(err)
    torch.cuda.synchronize()
    check_batch(pkts, exp, err)
    hd.hd_set_max_ctas(0)
    again = Captured(lambda s: plan.launch(err, cuda_stream=s))
    assert max(whole.kernels) > 3 and max(capped.kernels) == 3
    assert again.kernels == whole.kernels
    plan.close()
