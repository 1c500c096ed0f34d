"""hd_decode_streams: which streams share a branch.  The depth of a captured call
is the clear of the counters and the decodes of its longest branch."""
import pytest

from paper_1412_6862_gb300 import hd
from tests import gpu_cases as gc
from tests.captured import Captured

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_6862_gb300 import build
    build.build()
    hd.lib()


def _run(specs):
    """Decode the streams (n, codewords) in one call against the oracle; the captured call."""
    import torch
    made, rows = [], []
    for i, (n, N) in enumerate(specs):
        stream, _, _ = gc.received_stream(n, N, seed=i + N)
        d_in, k = gc.to_device(stream), hd.code_params(n)[1]
        out = torch.full((hd.words_for(N * k),), -1, dtype=torch.int32, device="cuda")
        syn = torch.full((N,), 0x5A, dtype=torch.uint8, device="cuda")
        err = torch.full((1,), 77, dtype=torch.int64, device="cuda")
        made.append((d_in, out, syn, err, stream))
        rows.append((d_in.data_ptr(), n, N, out.data_ptr(), syn.data_ptr(), hd.SYN_U8, err.data_ptr()))
    jobs = hd.stream_jobs(rows)

    def call(s):
        hd.check(hd.hd_decode_streams(jobs, len(specs), s.cuda_stream), "hd_decode_streams")

    call(torch.cuda.current_stream())
    torch.cuda.synchronize()
    for (n, N), (d_in, out, syn, err, stream) in zip(specs, made):
        gc.assert_same((out, syn, err), gc.expected(stream, n, N, hd.SYN_U8), n, N, hd.SYN_U8)
    return Captured(call)


def test_large_streams_each_have_a_branch():
    # 15.3 Mbit that the lanes decode, and 13.5 to 14.7 Mbit of short codewords that they do not
    c = _run([(255, 60_000), (7, 2_100_000), (15, 900_000), (7, 2_000_000)])
    assert c.depth == 2 and len(c.kernels) == 5


def test_pinned_short_stream_has_a_branch():
    hd.hd_variant_select(63, hd.SYN_U8, 0)
    try:
        c = _run([(63, 60_000), (31, 20_000), (31, 20_001)])
    finally:
        hd.hd_variant_select(63, hd.SYN_U8, -1)
    assert c.depth <= 3 and len(c.kernels) == 4


def test_short_streams_side_by_side_when_captured():
    # the caller's stream and eight branches: ten streams, the last one behind another
    specs = [((7, 15, 31, 63)[i % 4], 20_000 - i) for i in range(10)]
    c = _run(specs[:9])
    assert c.depth == 2 and len(c.kernels) == 10
    assert _run(specs).depth == 3
