"""The full-length and SECDED encoders on the GPU against the oracle, bit by
bit, at the edges of their paths: a lane's fields and a tile's 32 codewords,
the largest stream encoded one codeword per lane, the streaming kernel with a
ragged tail, and (with a cap on the CTAs) every warp's ring wrapping."""
import numpy as np
import pytest

import oracle
from paper_1412_6862_gb300 import hd, synth
from tests import gpu_cases as gc

pytestmark = pytest.mark.gpu

ALL_N = [3, 7, 15, 31, 63, 127, 255]


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


def _check(n, N, secded, cap=0):
    import torch
    m, k = hd.code_params(n)
    L = n + (1 if secded else 0)
    data = synth.random_words(n + N, N * k)
    want = gc.oracle_encode_parallel(oracle.encode_secded if secded else oracle.encode, data, n, N, k, L)
    out = torch.full((hd.words_for(N * L) + 8,), -1, dtype=torch.int32, device="cuda")
    dirty = data.copy()
    if (N * k) % 32:  # pad bits past the last message are not part of it
        dirty[-1] |= np.uint32((0xFFFFFFFF << ((N * k) % 32)) & 0xFFFFFFFF)
    hd.hd_set_max_ctas(cap)
    (hd.encode_secded if secded else hd.encode)(gc.to_device(dirty), n, N, out=out)
    torch.cuda.synchronize()
    hd.hd_set_max_ctas(0)
    got = gc.host_u32(out)
    bad = np.nonzero(got[:want.size] != want)[0]
    assert bad.size == 0, f"n={n} N={N} secded={secded}: {bad.size} words differ, first {bad[:4]}"
    assert (got[want.size:] == 0xFFFFFFFF).all()  # nothing past the stream is written
    assert hd.hd_device_status() == 0


@pytest.mark.parametrize("secded", [False, True])
@pytest.mark.parametrize("n", ALL_N)
def test_lane_path_edges(n, secded):
    for N in (1, 2, 5, 31, 32, 33, 1023, 1025, 40_009):
        _check(n, N, secded)


@pytest.mark.parametrize("cap", [0, 6])
@pytest.mark.parametrize("n", ALL_N)
def test_streaming_path_and_tail(n, cap):
    for N in (116_736, 194_560, 311_296, 311_297, 327_680 + 1021):  # the lane path's last sizes, chunks with a tail
        _check(n, N, False, cap)


# Segments of any length: below a word (a stream word holds several), at the
# words' and the checksum positions' edges, the paper's lengths and the longest;
# counts from one segment to several tiles per warp.
@pytest.mark.parametrize("n,N", [
    (3, 1), (3, 700_001), (4, 33), (7, 100_003), (16, 200_001), (30, 99_999), (31, 4097), (32, 4097), (33, 150_001),
    (62, 5), (63, 9999), (64, 9999), (65, 120_007), (95, 3001), (96, 3001), (128, 70_001), (129, 2), (544, 60_001),
    (1023, 777), (1024, 777), (1025, 20_011), (3212, 15_013), (8013, 3001), (16383, 7), (16384, 500), (16415, 501),
    (32752, 3), (32767, 1), (32767, 1201)])
@pytest.mark.parametrize("cap", [0, 3])
def test_encode_short_paths(n, N, cap):
    import torch
    r, k = hd.hd_short_params(n)
    data = synth.random_words(n * 3 + N, N * k)
    want = gc.oracle_encode_parallel(oracle.encode_short, data, n, N, k, n)
    if (N * k) % 32:
        data = data.copy()
        data[-1] |= np.uint32((0xFFFFFFFF << ((N * k) % 32)) & 0xFFFFFFFF)
    out = torch.full((hd.words_for(N * n) + 8,), -1, dtype=torch.int32, device="cuda")
    hd.hd_set_max_ctas(cap)
    hd.encode_short(gc.to_device(data), n, N, out=out)
    torch.cuda.synchronize()
    hd.hd_set_max_ctas(0)
    got = gc.host_u32(out)
    bad = np.nonzero(got[:want.size] != want)[0]
    assert bad.size == 0, f"n={n} N={N}: {bad.size} words differ, first {bad[:4]}"
    assert (got[want.size:] == 0xFFFFFFFF).all()
