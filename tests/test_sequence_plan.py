"""How a batched sequence is cut up and which form of it runs, as the library decides it on the host (148 SMs, no device needed).  The times
quoted were measured on a B200 for 35 timesteps."""
import pytest

from paper_1802_00150_b200 import amq

SMS = 148


def plan(cell, I, H, kw, ka, batch, form=-1):
    return amq.selftest_sequence_plan(cell == "gru", I, H, kw, ka, batch, SMS, form)


@pytest.mark.parametrize("cell,I,H,kw,batch", [("lstm", 2000, 2000, 2, 200), ("gru", 1500, 1500, 2, 200), ("lstm", 1200, 1600, 2, 256)])
def test_two_teams_quantize_at_up_to_three_bits_only(cell, I, H, kw, batch):
    """Vectors of 2049 to 4096 elements, several per CTA: two teams of eight warps, sixteen elements a thread, are faster up to three bits (1370
    against 1418 us for the first problem) and spill at four (2660 against 2153 us)."""
    for ka in (1, 2, 3, 4):
        _, (ctas, block, warps), _ = plan(cell, I, H, kw, ka, batch, amq.FORM_STREAMING)
        assert block > ctas
        assert warps == (16 if ka == 4 else 8)
