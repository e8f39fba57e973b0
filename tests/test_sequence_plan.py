"""How a batched sequence is cut up, which form of it and which product runs, as the library decides it on the host (148 SMs, no device
needed).  The times quoted were measured on a B200, of sequences for 35 timesteps."""
import os
import shutil

import pytest

from paper_1802_00150_b200 import build

if not (os.path.exists(build.LIB) and os.path.exists(build.BINDING)):
    if shutil.which("nvcc") is None:
        pytest.skip("library not built and nvcc not available", allow_module_level=True)
    build.build()

from paper_1802_00150_b200 import amq  # noqa: E402

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


# cell, I, H, bits of the weights and of the activations, sequences; us as a chain of launches, with the weights streamed, with the weights
# in tensor memory (None: the form does not take the problem)
MEASURED = [
    ("gru", 1900, 1900, 2, 3, 256, 15675, 1376, 7292),
    ("lstm", 1920, 1920, 2, 2, 64, 591, 610, 1286),
    ("gru", 256, 1536, 3, 3, 128, 830, 671, 3368),
    ("lstm", 128, 1600, 3, 3, 200, 1700, 1007, 5192),
    ("lstm", 128, 1600, 3, 3, 32, 747, 509, 1106),
    ("lstm", 1024, 1024, 3, 3, 256, 1293, 865, 995),
    ("lstm", 1024, 1024, 2, 2, 1024, 1830, 1810, 1791),
    ("lstm", 1024, 1024, 3, 3, 64, 509, 519, 420),
    ("gru", 2048, 2048, 2, 3, 256, 1692, 1420, None),
    ("gru", 300, 650, 3, 2, 20, 1606, 381, 241),
    ("lstm", 300, 300, 2, 2, 64, 403, 331, 254),
    ("gru", 217, 1556, 3, 2, 159, 7313, 702, 2637),
    ("gru", 1664, 1984, 2, 4, 215, 2579, 2250, 8060),
    ("gru", 79, 1408, 4, 4, 258, 21150, 1401, 3408),
    ("lstm", 312, 1792, 4, 3, 48, 945, 700, None),
    ("lstm", 1024, 1024, 4, 4, 64, 606, 686, 625),
    ("lstm", 1536, 1536, 2, 2, 2, 454, 419, 313),
    ("gru", 1024, 1024, 2, 3, 4096, 6976, 7280, 10847),
    ("lstm", 1024, 1024, 2, 2, 4096, 5670, 6614, 7403),
    ("lstm", 300, 300, 2, 2, 4096, 2063, 3181, 1788),
    ("lstm", 2048, 2048, 2, 2, 2048, 6819, 7265, None),
    ("lstm", 960, 1344, 4, 4, 5706, 30394, None, None),
    ("gru", 100, 313, 4, 2, 4606, 30310, 3418, 2793),
]


@pytest.mark.parametrize("cell,I,H,kw,ka,batch,chain,streaming,resident", MEASURED)
def test_the_form_taken_is_the_fastest_measured_one_or_close_to_it(cell, I, H, kw, ka, batch, chain, streaming, resident):
    """Many passes of few vectors over weights in tensor memory cost several times what streaming them does; thousands of sequences go
    fastest as a chain.  Estimates that differ by a few percent may choose wrongly, by no more than that."""
    times = {amq.FORM_CHAIN: chain, amq.FORM_STREAMING: streaming, amq.FORM_RESIDENT: resident}
    form, split, clocks = plan(cell, I, H, kw, ka, batch)
    assert times[form] is not None and times[form] <= 1.06 * min(t for t in times.values() if t is not None)
    # (35 timesteps at 1965 MHz and up to 25 us around them; the worst of the fits is 31 % off)
    assert abs(clocks * 35 / 1965 + 25 - times[form]) <= 0.32 * times[form] + 25
    for f in (amq.FORM_STREAMING, amq.FORM_RESIDENT):
        if times[f] is None:
            with pytest.raises(amq.AmqError):
                plan(cell, I, H, kw, ka, batch, f)


def test_a_split_covers_the_problem_and_the_counters_cover_the_split():
    """Over sizes of every kind: the blocks cover the batch, the CTAs fit the device at once (they wait for one another), the counters in the
    workspace (64 words per eight vectors) cover the blocks, and forcing the form that was chosen gives the same split."""
    import random
    rng = random.Random(5)
    for _ in range(400):
        gru, I, H, batch = rng.random() < 0.5, rng.randint(1, 2048), rng.randint(1, 2048), int(2 ** rng.uniform(1, 13))
        kw, ka, sms = rng.randint(1, 4), rng.randint(1, 4), rng.choice([148, 148, 132, 20, 1])
        form, split, clocks = amq.selftest_sequence_plan(gru, I, H, kw, ka, batch, sms)
        if form == amq.FORM_CHAIN:
            continue
        ctas, block, warps = split
        blocks = -(-batch // block)
        assert blocks * ctas <= sms and blocks <= -(-batch // 8) and warps in (4, 8, 16) and clocks > 0
        assert amq.selftest_sequence_plan(gru, I, H, kw, ka, batch, sms, form)[1:] == (split, clocks)


@pytest.mark.parametrize("m,n,kw,ka,batch,streaming,resident", [
    (4096, 2048, 3, 3, 64, 11.0, 14.9),
    (6144, 4096, 2, 3, 256, 37.4, 37.5),
    (32768, 1024, 3, 2, 512, 109.3, 60.1),
    (9999, 650, 2, 2, 600, 33.3, 29.2),
    (4096, 1024, 2, 2, 64, 8.3, 11.0),
    (4096, 2048, 2, 2, 64, 9.8, 12.6),
    (62364, 320, 3, 3, 3, 33.4, 14.9),
    (61767, 1536, 3, 4, 815, 756.3, 334.6),
    (42773, 192, 3, 4, 753, 364.7, 135.8),
    (4275, 2096, 2, 3, 157, 12.9, 21.2),
    (666, 128, 3, 2, 18, 6.7, 9.5),
    (16078, 128, 4, 4, 469, 116.3, 48.1),
    (768, 2752, 4, 2, 13, 8.7, 16.9),
    (551, 7487, 4, 2, 15, 14.9, 27.1),
    (1813, 7744, 4, 3, 26, 16.9, 29.2),
])
def test_the_product_taken_is_the_faster_measured_one_or_close_to_it(m, n, kw, ka, batch, streaming, resident):
    """Times in us of the tensor-core product with both operands streamed and with resident activations."""
    form, clocks = amq.selftest_product_plan(m, n, kw, ka, batch, SMS)
    times = {amq.PRODUCT_STREAMING: streaming, amq.PRODUCT_RESIDENT: resident}
    assert times[form] <= 1.06 * min(streaming, resident)
    for c, t in zip(clocks, (streaming, resident)):
        assert abs(c / 1965 - t) <= 0.21 * t                # (the worst of the fits)
