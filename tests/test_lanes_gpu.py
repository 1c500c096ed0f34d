"""Where a decode changes its path, against the oracle: one CTA that writes the
counts itself (up to 1024 codewords), one codeword per lane (up to one tile per
resident warp) and whole chunks with the ragged tail in the same launch, plain
and SECDED, every n and syndrome type.  The counters start dirty, so a path
that neither clears nor overwrites them fails."""
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


def _plain(n, N, syn, cap):
    import torch
    m, k = hd.code_params(n)
    rx, _, _ = gc.received_stream(n, N, seed=n + N, p1=0.2, p2=0.02)
    exp = gc.expected(rx, n, N, syn)
    out = torch.full((hd.words_for(N * k) + 8,), -1, dtype=torch.int32, device="cuda")
    sy = None if syn == hd.SYN_NONE else torch.full((N + 16,), 0x55, device="cuda",
                                                    dtype=torch.uint8 if syn == hd.SYN_U8 else torch.int16)
    err = torch.full((1,), 999, dtype=torch.int64, device="cuda")
    hd.hd_set_max_ctas(cap)
    hd.decode(gc.to_device(rx), n, N, syn, out=out, syndromes=sy, err_count=err)
    torch.cuda.synchronize()
    hd.hd_set_max_ctas(0)
    gc.assert_same((out, sy, err), exp, n, N, syn)
    assert (gc.host_u32(out)[hd.words_for(N * k):] == 0xFFFFFFFF).all()
    if sy is not None:
        assert (sy.cpu().numpy()[N:] == 0x55).all()


def _secded(n, N, syn, cap):
    import torch
    m, k = hd.code_params(n)
    rx = oracle.encode_secded(synth.random_words(N, N * k), n, N)
    synth.apply_errors(rx, synth.error_events(N + n, n + 1, N, p1=0.2, p2=0.05))
    eo, es, ee, ed = oracle.decode_secded(rx, n, N, syn if syn != hd.SYN_NONE else oracle.SYN_U16, threads=8)
    out = torch.full((hd.words_for(N * k) + 8,), -1, dtype=torch.int32, device="cuda")
    sy = None if syn == hd.SYN_NONE else torch.full((N + 16,), 0x55, device="cuda",
                                                    dtype=torch.uint8 if syn == hd.SYN_U8 else torch.int16)
    cnt = torch.full((2,), 777, dtype=torch.int64, device="cuda")
    hd.hd_set_max_ctas(cap)
    hd.decode_secded(gc.to_device(rx), n, N, syn, out=out, syndromes=sy, counts=cnt)
    torch.cuda.synchronize()
    hd.hd_set_max_ctas(0)
    nw = hd.words_for(N * k)
    got = gc.host_u32(out)
    assert np.array_equal(got[:nw], eo[:nw]), (n, N)
    assert (got[nw:] == 0xFFFFFFFF).all()
    if sy is not None:
        s = sy.cpu().numpy()
        assert np.array_equal(s[:N].view(es.dtype) if syn == hd.SYN_U16 else s[:N], es[:N].astype(
            np.uint16 if syn == hd.SYN_U16 else np.uint8)), (n, N)
        assert (s[N:] == 0x55).all()
    assert cnt.cpu().numpy().tolist() == [ee, ed]


@pytest.mark.parametrize("secded", [False, True])
@pytest.mark.parametrize("n", ALL_N)
def test_path_boundaries(n, secded):
    run = _secded if secded else _plain
    for syn in (hd.SYN_NONE, hd.SYN_U8, hd.SYN_U16):
        if secded and syn == hd.SYN_U8 and n == 255:
            continue
        for N, cap in ((1, 0), (32, 0), (481, 0), (1024, 0), (1025, 0), (311_296, 0), (311_297 + 1021, 0),
                       (7 * 1024 + 991, 2)):
            run(n, N, syn, cap)
    assert hd.hd_device_status() == 0


def test_counts_may_be_null():
    """One CTA's direct counts with the pointers left out."""
    import torch
    st = torch.cuda.current_stream().cuda_stream
    rx, _, _ = gc.received_stream(63, 300, seed=1)
    d, out = gc.to_device(rx), torch.zeros(600, dtype=torch.int32, device="cuda")
    assert hd.hd_decode(d.data_ptr(), 63 * 300, 63, 300, out.data_ptr(), None, hd.SYN_NONE, None, st) == hd.HD_OK
    det = torch.full((1,), 5, dtype=torch.int64, device="cuda")
    assert hd.hd_decode_secded(d.data_ptr(), 64 * 200, 63, 200, out.data_ptr(), None, hd.SYN_NONE, None,
                               det.data_ptr(), st) == hd.HD_OK
    torch.cuda.synchronize()
    es = oracle.decode_secded(rx, 63, 200, oracle.SYN_U16, threads=1)
    assert int(det.item()) == es[3]
