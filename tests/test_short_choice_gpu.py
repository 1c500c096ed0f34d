"""hd_short_autotune(): the configuration it returns is the one that decodes the
length afterwards, at any size."""
import pytest

from paper_1412_6862_gb300 import hd
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
    yield
    hd.hd_short_variant_select(-1)


def _recorded(n, N):
    """The kernels of one decode, recorded but not run."""
    import torch
    r, k = hd.hd_short_params(n)
    d_in = torch.zeros(hd.words_for(N * n) + 4, dtype=torch.int32, device="cuda")
    out = torch.empty(hd.words_for(N * k) + 4, dtype=torch.int32, device="cuda")

    hd.decode_short(d_in, n, 1, hd.SYN_NONE)  # builds the length's table, which a capture refuses

    def call(s):
        hd.check(hd.hd_decode_short(d_in.data_ptr(), n * N, n, N, out.data_ptr(), None, hd.SYN_NONE, None, None,
                                    s.cuda_stream), "hd_decode_short")

    return Captured(call)


# lengths whose lanes win, by a quarter or more; one near the line; longer ones
@pytest.mark.parametrize("n", [100, 300, 400, 700, 959, 961, 2679])
def test_the_returned_configuration_is_the_kept_one(n):
    N = 50_000
    v = hd.hd_short_autotune(n, N, 3)
    tuned = _recorded(n, N)
    hd.hd_short_variant_select(v)
    pinned = _recorded(n, N)
    hd.hd_short_variant_select(-1)
    assert tuned.functions == pinned.functions and tuned.kernels == pinned.kernels


def test_the_choice_holds_at_any_size():
    n = 800
    lanes = hd.hd_short_variant_count() - 1
    hd.hd_short_variant_select(lanes)
    want = _recorded(n, 100).functions
    hd.hd_short_variant_select(-1)
    assert hd.hd_short_autotune(n, 25, 20) == lanes  # 20,000 bits: the tiles take a third longer
    assert _recorded(n, 25).functions == want
    assert _recorded(n, (1 << 28) // n + 1).functions == want  # tiles, had it not been tuned


def test_lanes_pinned_for_a_length_they_do_not_decode():
    built_in = _recorded(2001, 5000)
    hd.hd_short_variant_select(hd.hd_short_variant_count() - 1)
    pinned = _recorded(2001, 5000)
    hd.hd_short_variant_select(-1)
    assert pinned.functions == built_in.functions and pinned.kernels == built_in.kernels
