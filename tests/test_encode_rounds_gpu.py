"""The SECDED encoder when its warps take several groups each (a cap on the CTAs),
against the oracle: streams that end on a round, on a group, and inside one."""
import pytest

from paper_1412_6862_gb300 import hd
from tests.test_encode_gpu import _check

pytestmark = pytest.mark.gpu

# codewords a warp takes per step
GROUP = {3: 2048, 7: 1024, 15: 512, 31: 256, 63: 128, 127: 64, 255: 64}


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


@pytest.mark.parametrize("cap", [1, 2])
@pytest.mark.parametrize("n", sorted(GROUP))
def test_secded_several_groups_a_warp(n, cap):
    rounds = 8 * cap * GROUP[n]  # eight warps per CTA
    for N in (3 * rounds, 3 * rounds + GROUP[n], 4 * rounds - 1, 5 * rounds + 3 * GROUP[n] + 17):
        _check(n, N, True, cap)
