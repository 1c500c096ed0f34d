"""The configuration a plan takes by itself: by its tiles, its bytes and the share
of the code lengths among them, on both sides of each line.  The plans are not
launched (every configuration's results are compared elsewhere)."""
import pytest

from paper_1412_6862_gb300 import hd

pytestmark = pytest.mark.gpu

THREE, TWO, FOUR_WARPS, TABLE12, TABLE14, GROUPS = 0, 1, 4, 6, 7, 9
MBIT = 1 << 20


# (n: packets of 1 Mbit of codewords), syndrome type, the choice
@pytest.mark.parametrize("packets,syn,want", [
    ({63: 30}, 1, FOUR_WARPS), ({63: 100}, 1, TWO), ({63: 500}, 1, TWO), ({63: 1000}, 1, THREE),
    ({31: 1000}, 2, THREE), ({127: 1000}, 0, THREE), ({31: 300, 63: 300, 127: 300}, 1, THREE),
    ({255: 1500}, 1, TWO), ({7: 1200}, 1, THREE), ({7: 1200}, 2, TWO), ({7: 1000}, 0, TWO),
    ({7: 600, 63: 600}, 0, THREE),
    ({15: 60}, 1, TABLE12), ({15: 300}, 1, TABLE14), ({15: 1200}, 1, TABLE14), ({15: 400, 63: 800}, 1, TABLE14),
    ({7: 120, 15: 120, 31: 120, 63: 120, 127: 120, 255: 120}, 1, TABLE14),
    ({7: 240, 15: 240, 31: 240, 63: 240, 127: 240, 255: 240}, 1, THREE),
    ({15: 60, 63: 600, 127: 600}, 1, THREE), ({15: 100, 255: 1000}, 1, TWO), ({15: 30, 255: 300}, 1, TWO),
    ({3: 100}, 1, TWO), ({3: 40, 63: 1000}, 1, TWO), ({3: 10, 63: 1000}, 1, THREE),
    # about 512 MB with n = 127
    ({127: 2000}, 1, THREE), ({127: 2100}, 1, GROUPS), ({63: 1100, 127: 1100}, 1, GROUPS), ({63: 2100}, 1, THREE),
    # more than 768 MB
    ({63: 3500}, 1, GROUPS), ({255: 3600}, 1, GROUPS), ({7: 2500}, 1, THREE), ({7: 2000}, 2, TWO),
    ({7: 1500, 63: 1500}, 1, THREE), ({7: 1500, 15: 1500}, 1, GROUPS),
    ({7: 600, 15: 600, 31: 600, 63: 600, 127: 600, 255: 600}, 1, GROUPS),
])
def test_choice(packets, syn, want):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_6862_gb300 import build
    build.build()
    hd.lib()
    buf = torch.empty(4, dtype=torch.int32, device="cuda").data_ptr()
    rows = [(buf, buf, buf if syn else None, MBIT // n, n, syn) for n, count in packets.items() for _ in range(count)]
    plan = hd.hd_plan_create(hd.packet_table(rows), len(rows))
    try:
        assert hd.hd_plan_get_info(plan)["variant"] == want, hd.hd_plan_get_info(plan)
    finally:
        hd.hd_plan_destroy(plan)
