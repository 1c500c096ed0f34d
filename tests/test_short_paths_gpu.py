"""Where the shortened-code decoder changes its path, against the oracle: every
word count of the one-segment-per-lane kernel and its edges (lengths around
multiples of 32, the last lane length 959 and the first tiled one 960), streams
of one CTA (which overwrites the counters itself), of a few tiles and of uneven
tiles, with and without counters and syndromes."""
import numpy as np
import pytest

import oracle
from paper_1412_6862_gb300 import hd
from tests.test_short_gpu import _check, _received
from tests import gpu_cases as gc

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


@pytest.mark.parametrize("words", range(1, 31))
def test_lane_lengths(words):
    for n in (32 * words - 1, 32 * words, 32 * words + 5):
        if n < 960:
            for N in (1, 33, 2051):
                _check(n, N, hd.SYN_U16, seed=n + N)
    _check(max(3, 32 * words - 17), 999, hd.SYN_NONE, seed=words)


@pytest.mark.parametrize("cap", [0, 1, 2])
@pytest.mark.parametrize("n,N", [(16, 70_001), (255, 9001), (544, 9001), (959, 5003), (960, 5003), (1023, 13),
                                 (1078, 9001), (3212, 12), (3212, 13), (3212, 3649), (8013, 4001), (16384, 601),
                                 (32767, 301)])
def test_stream_lengths(n, N, cap):
    hd.hd_set_max_ctas(cap)
    try:
        _check(n, N, hd.SYN_U16, seed=n + N)
    finally:
        hd.hd_set_max_ctas(0)


# the edges of the tiles: all codewords in one CTA or one tile per warp of every SM (24 | 25,
# 3648 | 3649 codewords), more than one round, the last table in shared memory and the first in
# global memory (18,600 | 18,700), lanes and tiles of a large stream (768), two codewords per stage there or one (28,544 | 28,545)
@pytest.mark.parametrize("n,N", [(961, 24), (1023, 25), (1024, 3648), (1100, 40_001), (1500, 160_001), (2047, 3649),
                                 (2048, 7300), (4095, 7297), (4096, 20_011), (12_000, 3649), (18_600, 3649),
                                 (768, 349_520), (768, 349_527), (959, 280_001),
                                 (1023, 70_001), (1536, 50_001), (2048, 40_001), (8191, 9001),
                                 (18_600, 4001), (18_700, 4001), (28_544, 5003), (28_545, 5003), (32_767, 4865)])
def test_tile_shapes(n, N):
    _check(n, N, hd.SYN_U16, seed=n + N)


@pytest.mark.parametrize("n", [40, 300, 2000])
def test_one_cta_without_counters(n):
    import torch
    N = 9
    rx, _, _ = _received(n, N, seed=n)
    eo, es, ee, ed = oracle.decode_short(rx, n, N, oracle.SYN_U16, threads=1)
    d = gc.to_device(rx, pad_words=4)
    out = torch.full((eo.size + 4,), -1, dtype=torch.int32, device="cuda")
    det = torch.full((1,), 77, dtype=torch.int64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    assert hd.hd_decode_short(d.data_ptr(), n * N, n, N, out.data_ptr(), None, hd.SYN_NONE, None, det.data_ptr(),
                              st) == hd.HD_OK
    torch.cuda.synchronize()
    assert np.array_equal(gc.host_u32(out)[:eo.size], eo) and int(det.item()) == ed
    out.fill_(-1)
    assert hd.hd_decode_short(d.data_ptr(), n * N, n, N, out.data_ptr(), None, hd.SYN_NONE, None, None, st) == hd.HD_OK
    torch.cuda.synchronize()
    assert np.array_equal(gc.host_u32(out)[:eo.size], eo)
