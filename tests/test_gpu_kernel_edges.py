"""The kernels that take over whole calls (resident-operand product, batched sequences in one launch, decoding in one launch, the
bulk quantizer, the output softmax), each at the sizes where its tiling can go wrong, against the CPU oracle or against the
call-by-call form that the oracle pins."""
import numpy as np
import pytest
import torch

import oracle
import parity
from paper_1802_00150_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amq():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    from paper_1802_00150_b200 import amq as binding
    return binding


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(torch.float32).cuda()


def cdev(c):
    return torch.from_numpy(np.ascontiguousarray(c).view(np.int32)).cuda()


def quantized(shape, std, k, seed, stream):
    return oracle.quantize_rows(synth.normal(shape, std, seed, stream).astype(np.float64), k, 2)


@pytest.mark.parametrize("m,n,kw,ka,batch,offset", [
    (1, 1, 1, 1, 16, 0),                # one row, one column
    (127, 255, 2, 2, 31, 0),            # one short of the row tile, of a slot of 256 positions, of a block of vectors
    (129, 257, 3, 3, 33, 1),            # one past each of them, output rows off every 16-byte boundary
    (130, 8448, 1, 4, 17, 0),           # the longest rows the operand is kept for
    (130, 8449, 1, 1, 17, 0),           # one more: the streaming kernel
    (4000, 512, 4, 1, 2, 3),            # the smallest batch, many rows
    (300, 1000, 4, 4, 97, 2),
])
def test_product_at_the_edges_of_its_tiles(amq, m, n, kw, ka, batch, offset):
    Wc, Wa = quantized((m, n), 0.03, kw, 200 + m, 1)
    Xc, Xb = quantized((batch, n), 1.0, ka, 200 + m, 2)
    bias = synth.normal((m,), 0.1, 200 + m, 3)
    out = torch.full((batch, m + offset + 2), 7.0, device="cuda")
    amq.binary_gemm(cdev(Wc), dev(Wa), cdev(Xc), dev(Xb), n, bias=dev(bias), y=out[:, offset:offset + m])
    ref = oracle.binary_gemm(Wc, Wa, Xc, Xb, n, bias.astype(np.float64))
    assert np.abs(out[:, offset:offset + m].cpu().numpy() - ref).max() <= 1e-5 * (np.abs(ref).max() + 1)
    assert torch.all(out[:, :offset] == 7.0) and torch.all(out[:, offset + m:] == 7.0)      # nothing written beside the rows
    assert amq.device_status() == 0


@pytest.mark.parametrize("m,n,kw,ka,batch,offset", [
    (1, 1, 1, 1, 16, 0), (127, 255, 2, 2, 31, 0), (129, 257, 3, 3, 33, 1), (130, 8448, 1, 4, 17, 0), (4000, 512, 4, 1, 2, 3),
    (300, 1000, 4, 4, 97, 2), (128, 256, 1, 2, 64, 0), (43, 1024, 3, 2, 128, 0), (20000, 130, 2, 2, 129, 0),
])
def test_both_tensor_core_products_at_the_edges_of_their_tiles(amq, m, n, kw, ka, batch, offset):
    """The sizes above and those where the streaming form's tiles end, on either kernel, whichever the library takes.  Tolerance: k_w k_a
    products of exact integers and fp32 coefficients, summed in fp32."""
    Wc, Wa = quantized((m, n), 0.03, kw, 210 + m, 1)
    Xc, Xb = quantized((batch, n), 1.0, ka, 210 + m, 2)
    bias = synth.normal((m,), 0.1, 210 + m, 3)
    ref = oracle.binary_gemm(Wc, Wa, Xc, Xb, n, bias.astype(np.float64))
    for form in (amq.PRODUCT_STREAMING, amq.PRODUCT_RESIDENT):
        out = torch.full((batch, m + offset + 2), 7.0, device="cuda")
        amq.selftest_binary_gemm(cdev(Wc), dev(Wa), cdev(Xc), dev(Xb), n, form, bias=dev(bias), y=out[:, offset:offset + m])
        assert np.abs(out[:, offset:offset + m].cpu().numpy() - ref).max() <= 1e-5 * (np.abs(ref).max() + 1), form
        assert torch.all(out[:, :offset] == 7.0) and torch.all(out[:, offset + m:] == 7.0)
    assert amq.device_status() == 0


@pytest.mark.parametrize("cell,I,H,kw,ka,batch", [
    ("lstm", 1, 1, 1, 1, 2),            # the smallest
    ("lstm", 255, 33, 3, 2, 9),         # one short of a slot, one unit past a tile of 32, one vector past a block of 8
    ("lstm", 300, 640, 2, 3, 33),
    ("gru", 257, 129, 2, 2, 31),        # the column split one past a slot, one unit past a tile of 128
    ("gru", 512, 256, 4, 4, 65),        # the split on a slot
    ("gru", 2100, 2050, 1, 2, 5),       # rows of more than 4096 positions
    ("lstm", 70, 1200, 4, 4, 70),       # two tiles of plane-rows, several passes over the vectors
    ("lstm", 1030, 500, 3, 2, 130),
    ("gru", 1700, 1900, 1, 2, 3),       # fifteen slots: nearly all of tensor memory
    ("lstm", 4000, 200, 2, 2, 17),      # weights that do not stay in tensor memory
])
def test_batched_sequence_at_the_edges_of_its_tiles(amq, cell, I, H, kw, ka, batch):
    """Three timesteps in one call equal three calls of one timestep bit for bit; the first is held against the oracle."""
    steps, n, gates = 3, I + H, 4 if cell == "lstm" else 3
    Wc, Wa = quantized((gates * H, n), 0.05, kw, 300 + H, 1)
    bias = synth.normal((4 * H,), 0.1, 300 + H, 2)
    xs = synth.uniform((steps, batch, I), -1, 1, 301, 1)
    h0, c0 = synth.uniform((batch, H), -1, 1, 301, 2), synth.uniform((batch, H), -1, 1, 301, 3)
    ws = amq.new_workspace(I, H, batch, ka)
    args = (cdev(Wc), dev(Wa), dev(bias), I, H)
    x, h, c = dev(xs), dev(h0), dev(c0)
    if cell == "lstm":
        seq, last, c_last = amq.lstm_sequence(*args, x, h, c, ka, 2, ws, want_h_seq=True)
        ref, c_ref = oracle.lstm_step(Wc, Wa, bias, I, H, xs[0], h0, c0, ka, 2)
    else:
        seq, last = amq.gru_sequence(*args, x, h, ka, 2, ws, want_h_seq=True)
        ref = oracle.gru_step(Wc, Wa, bias, I, H, xs[0], h0, ka, 2)
    _, beta = oracle.quantize_rows(np.concatenate([xs[0], h0], axis=1).astype(np.float64), ka, 2)
    assert np.abs(seq[0].cpu().numpy() - ref).max() <= 3.0 * parity.output_tolerance(Wa, beta, n).max() + 1e-6
    for t in range(steps):
        if cell == "lstm":
            _, h, c = amq.lstm_sequence(*args, x[t:t + 1], h, c, ka, 2, ws)
        else:
            _, h = amq.gru_sequence(*args, x[t:t + 1], h, ka, 2, ws)
        assert torch.equal(h, seq[t]), t
    assert torch.equal(h, last) and (cell == "gru" or torch.equal(c, c_last))
    assert amq.workspace_status(ws) == 0


@pytest.mark.parametrize("V,I,H,ke,kw,ks,ka,steps", [
    (1, 1, 1, 1, 1, 1, 1, 1),           # one word, one unit
    (149, 33, 147, 1, 2, 4, 2, 5),      # SMs without units, one word more than SMs
    (3001, 96, 149, 2, 3, 2, 1, 9),     # an odd number of units per SM, three row planes
    (5000, 1000, 257, 4, 4, 1, 4, 7),   # three 128-bit chunks of the state
    (40000, 64, 2048, 3, 1, 3, 3, 4),   # the widest state, output rows that do not all fit a SM
])
def test_decoding_in_one_launch_equals_the_chain_of_kernels(amq, V, I, H, ke, kw, ks, ka, steps):
    """Asked for log-probabilities the call runs kernel by kernel (held against the oracle elsewhere), without them in one launch:
    the same tokens and the same state bit for bit, called again as well (no word of the first call may be taken for a new one)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(V)
    q = lambda shape, std, k: amq.quantize(torch.randn(shape, device="cuda", generator=g) * std, k, 2)
    We, Wi, Wh, Ws = q((V, I), 1.0, ke), q((4 * H, I), 0.2, kw), q((4 * H, H), 0.1, kw), q((V, H), 0.2, ks)
    bias, bias_s = torch.randn((4 * H,), device="cuda", generator=g) * 0.1, torch.randn((V,), device="cuda", generator=g) * 0.1
    ws = amq.new_decode_workspace(V, I, H, ke, ka)
    runs = []
    for logp in (torch.empty((steps, V), device="cuda"), None, None):
        tokens = torch.full((steps + 1,), V // 2, dtype=torch.int32, device="cuda")
        h, c = torch.full((1, H), 0.25, device="cuda"), torch.zeros((1, H), device="cuda")
        amq.lm_greedy_decode(*We, *Wi, *Wh, bias, *Ws, bias_s, I, H, ka, 2, tokens, h, c, ws, logp=logp)
        runs.append((tokens, h, c))
    for r in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(r, runs[0]))
    assert amq.device_status() == 0


@pytest.mark.parametrize("rows,n,ld,skip", [(3, 2, 5, 3), (5, 2047, 2049, 1), (5, 2049, 2051, 2), (4, 10239, 10241, 3), (3, 10241, 10243, 1),
                                            (2, 49151, 49157, 1), (2, 49153, 49153, 3)])
def test_log_softmax_of_rows_off_the_16_byte_boundary(amq, rows, n, ld, skip):
    z = synth.normal((rows, n), 3.0, 400 + n, 1)
    z[0, 0] = z[0].max() + 1.0                                     # the maximum before the first boundary
    z[-1, n - 1] = z[-1].max() + 2.0
    flat = torch.full((rows * ld + 8,), float("nan"), device="cuda")
    wide = flat[skip:skip + rows * ld].view(rows, ld)
    wide[:, :n] = dev(z)
    logp, arg = amq.log_softmax_argmax(wide[:, :n])
    ref, rarg = oracle.log_softmax_argmax(z.astype(np.float64))
    assert np.abs(logp.cpu().numpy() - ref).max() <= 2e-5
    assert np.array_equal(arg.cpu().numpy(), rarg)


@pytest.mark.parametrize("n", [2048, 4096, 5120, 6144, 8192, 10240, 16384, 20480, 24576, 32768, 40960, 49152])
@pytest.mark.parametrize("past", [0, 1])
def test_log_softmax_at_the_edges_of_its_sizes(amq, n, past):
    """Every length at which another CTA size takes over, and one more; the first row starts on a 16-byte boundary, the next do not where the
    length is odd.  Tolerance: fp32 sum of up to 49153 exponentials, its logarithm and one subtraction (logits within +-17)."""
    n += past
    z = synth.normal((3, n), 3.0, 450 + n, 1)
    z[1, n - 1] = z[1].max() + 1.0
    logp, arg = amq.log_softmax_argmax(dev(z))
    ref, rarg = oracle.log_softmax_argmax(z.astype(np.float64))
    assert np.abs(logp.cpu().numpy() - ref).max() <= 2e-5
    assert np.array_equal(arg.cpu().numpy(), rarg)


@pytest.mark.parametrize("rows,n,k", [(2100, 1023, 3), (2100, 1024, 4), (2100, 65, 4), (1100, 513, 2), (3, 2049, 4)])
def test_quantizer_with_levels_out_of_order(amq, rows, n, k):
    """Rows whose refitted coefficients come out negative or not in decreasing order (two clusters and a constant part), so that the
    levels have to be sorted before the tree decisions; T = 4 cycles, edges of the warp and CTA ownership."""
    x = synth.normal((rows, n), 1.0, 500 + n, 1)
    u = synth.uniform01(rows * n, 500 + n, 2).reshape(rows, n)
    x = np.where(u < 0.5, 1.0 + 0.01 * x, np.where(u < 0.55, -3.0 + 0.2 * x, 0.02 * x)).astype(np.float32)
    codes, coeffs = amq.quantize(dev(x), k, 4)
    b = parity.unpack_rows(codes.cpu().numpy(), n)
    assert parity.pad_bits_zero(codes.cpu().numpy(), n)
    coeffs = coeffs.cpu().numpy().astype(np.float64)
    for r in range(0, rows, max(1, rows // 24)):
        oa, ob = oracle.quantize(x[r].astype(np.float64), k, 4)
        got = ((x[r] - coeffs[r] @ b[r]) ** 2).sum()
        want = ((x[r] - oa @ ob) ** 2).sum()
        assert abs(got - want) <= 1e-3 * max(want, 1e-6 * (x[r].astype(np.float64) ** 2).sum()), r


@pytest.mark.parametrize("n,k", [(1, 2), (7, 3), (9, 4), (31, 2), (33, 3), (255, 3), (256, 4), (257, 2), (258, 4), (1000, 3), (1023, 2), (1024, 4), (1024, 1)])
def test_bulk_quantization_at_the_edges_of_a_warps_rows(amq, n, k):
    """A warp per row: eight or thirty-two elements a thread, its last threads partly or wholly past the end; rows of ties (all of one
    magnitude, whole numbers) beside random ones."""
    x = synth.normal((1025, n), 0.05, 77 + n, k)
    x[3] = 0.25
    x[4] = -0.5
    x[5] = np.round(x[5] * 40)
    x[6] = 0.0

    def gpu(v, kk, T):
        codes, coeffs = amq.quantize(dev(v), kk, T)
        rows = np.r_[0:40, 1024]                    # (the oracle is slow)
        return codes.cpu().numpy().view(np.uint32)[rows], coeffs.cpu().numpy()[rows]

    rows = np.r_[0:40, 1024]
    random = [i for i, r in enumerate(rows) if r not in (3, 4, 5, 6)]
    parity.compare_quantizer(x[rows][random], k, 2, lambda v, kk, T: tuple(a[random] for a in gpu(x, kk, T)))
    # ties: several codes are correct, what they reconstruct is not free
    codes, coeffs = gpu(x, k, 2)
    bits = parity.unpack_rows(codes, n)
    for r in (3, 4, 6):
        assert np.abs(oracle.reconstruct(coeffs[r].astype(np.float64), bits[r]) - x[r]).max() <= 1e-6 * np.abs(x[r]).max()
    as_close_as_the_oracle(x[5:6], coeffs[5:6], bits[5:6], k)


def as_close_as_the_oracle(x, coeffs, bits, k):
    """Squared residuals of the rows within 1e-3 of the oracle's (its objective's bound for rows that took another side of a tie)."""
    for r in range(len(x)):
        oa, ob = oracle.quantize(x[r].astype(np.float64), k, 2)
        got = ((x[r] - coeffs[r].astype(np.float64) @ bits[r]) ** 2).sum()
        want = ((x[r] - oa @ ob) ** 2).sum()
        assert abs(got - want) <= 1e-3 * max(want, 1e-6 * (x[r].astype(np.float64) ** 2).sum()), r


@pytest.mark.parametrize("k", [2, 3, 4])
@pytest.mark.parametrize("n", [64, 300, 1000])
def test_rows_of_few_values(amq, n, k):
    """Levels that tie or nearly tie: rows of two to four distinct values (coefficients of equal magnitude, coefficients that vanish), whole
    numbers, values of very different size; by a warp per row and by a CTA per row."""
    sets = [(1, -1), (2, 0, -2), (1, 3, -1, -3), (0.25, -0.5), (1, 2, 3), (-1, 0, 1, 2), (4, 2, 1), (1e6, 1, -1), (3, -3, 1), (0.1, -0.1, 0.3)]
    pick = synth.uniform((1025, n), 0.0, 1.0, 700 + n, 1)
    x = np.empty((1025, n), np.float32)
    for r in range(1025):
        s = np.array(sets[r % len(sets)], np.float32)
        x[r] = s[np.minimum((pick[r] * len(s)).astype(int), len(s) - 1)]
    x[20:40] = np.round(synth.normal((20, n), 4.0, 700 + n, 2))
    for rows in (1025, 40):
        residual = []
        for T in (0, 1, 2):
            codes, coeffs = amq.quantize(dev(x[:rows]), k, T)
            bits, a = parity.unpack_rows(codes[:40].cpu().numpy().view(np.uint32), n), coeffs[:40].cpu().numpy().astype(np.float64)
            residual.append(np.array([((x[r] - a[r] @ bits[r]) ** 2).sum() for r in range(40)]))
        as_close_as_the_oracle(x[:20], a[:20], bits[:20], k)
        # Whole numbers meet midpoints exactly, an element there may go either way, and the cycles then lead to other fixed points (one row of
        # 60 at four bits ended further than 1e-3 from the oracle's).  What holds whichever way it goes: the greedy start's residual, of which
        # a tie (a residue of zero, either sign) changes nothing, and that no cycle raises it; 1e-5 of the row for fp32 coefficients.
        size = (x[:40].astype(np.float64) ** 2).sum(axis=1)
        for r in range(20, 40):
            oa, ob = oracle.quantize(x[r].astype(np.float64), k, 0)
            want = ((x[r] - oa @ ob) ** 2).sum()
            assert abs(residual[0][r] - want) <= 1e-3 * max(want, 1e-6 * size[r]), r
        assert (residual[1] <= residual[0] + 1e-5 * size).all() and (residual[2] <= residual[1] + 1e-5 * size).all()


@pytest.mark.parametrize("n,small", [(1, 1.0), (9, 0.1), (257, 0.02), (1025, 0.3), (2048, 0.1), (2049, 0.5)])
def test_three_bits_whose_levels_do_not_ascend(amq, n, small):
    """Vectors of large and of small elements, as [x ; h] is: the coefficients then come in any order of size, the smallest of them often
    below the difference of the others."""
    x = synth.normal((48, n), 1.0, 400 + n, 1)
    x[:, n // 2:] *= small
    x[24:, ::3] += 3.0

    def gpu(v, k, T):
        codes, coeffs = amq.quantize(dev(v), k, T)
        return codes.cpu().numpy().view(np.uint32), coeffs.cpu().numpy()

    parity.compare_quantizer(x, 3, 2, gpu)
    a = np.abs(gpu(x, 3, 1)[1])                     # (what the last cycle's table is made of, but for one refit)
    if n > 9:
        assert (a[:, 0] < a[:, 1] + a[:, 2]).any() or (np.argsort(-a, axis=1) != np.arange(3)).any()


@pytest.mark.parametrize("n,kw,ka", [
    (13 * 128 - 5, 2, 2),               # four chunks of 128 bits for the first lane of a row's segment only
    (16 * 128, 2, 3), (17 * 128, 2, 1),  # for all, and one left over
    (6 * 128, 3, 2), (7 * 128, 3, 2),   # none, the first
    (31 * 128 + 1, 4, 4),               # several groups and a remainder
    (25 * 128, 1, 2),
])
def test_one_sequence_lstm_at_the_edges_of_its_groups_of_chunks(amq, n, kw, ka):
    """Bit counts through full adders, sixteen words at a time, and word by word for what is left.  Tolerance: that of a step's state (three
    times the product's 1e-3 of the largest possible pre-activation), on the device's own weight codes."""
    H, I = 40, n - 40
    Wc, Wa = quantized((4 * H, n), 0.03, kw, 500 + n, 1)
    x, h, c = synth.normal((1, I), 1.0, 500 + n, 2), synth.uniform((1, H), -1, 1, 500 + n, 3), synth.uniform((1, H), -1, 1, 500 + n, 4)
    bias = synth.normal((4 * H,), 0.1, 500 + n, 5)
    got = amq.lstm_step(cdev(Wc), dev(Wa), dev(bias), I, H, dev(x), dev(h), dev(c), ka, 2, amq.new_workspace(I, H, 1, ka))
    want = oracle.lstm_step(Wc, Wa, bias.astype(np.float64), I, H, x, h, c, ka, 2)
    _, beta = oracle.quantize_rows(np.concatenate([x, h], axis=1).astype(np.float64), ka, 2)
    tol = 3e-3 * np.abs(Wa).sum(axis=1).max() * np.abs(beta).sum()
    for g, w in zip(got, want):
        assert np.abs(g.cpu().numpy() - w).max() <= tol


@pytest.mark.parametrize("cell,I,H,batch", [
    ("lstm", 96, 40, 1), ("gru", 128, 64, 1), ("lstm", 700, 900, 1),                # one sequence: teams of four and eight warps, sixteen elements a thread
    ("lstm", 96, 40, 9), ("gru", 260, 252, 20), ("lstm", 500, 900, 33),             # the three forms of a batch
])
def test_steps_on_vectors_whose_levels_tie(amq, cell, I, H, batch):
    """[x ; h] of as many +-1 as +-3: coefficients (2, 1, 0) at three bits, levels that tie in pairs, a table that is sorted inside the recurrent
    kernels too, and an exact reconstruction whichever of a pair is taken, so that the step is the textbook one on [x ; h] itself.  Tolerance: the
    pre-activations are sums of n terms of up to 3 |w| in fp32, some 1e-6 of their absolute sum; gates have slopes up to 1, c up to 3."""
    n, gates = I + H, 4 if cell == "lstm" else 3
    Wc, Wa = quantized((gates * H, n), 0.05, 2, 900 + n, 1)
    W = np.einsum("rk,rkn->rn", Wa, parity.unpack_rows(Wc, n).astype(np.float64))
    bias = synth.normal((4 * H,), 0.1, 900 + n, 2)
    z = np.empty((batch, n))
    for b in range(batch):
        order = np.argsort(synth.uniform((n,), 0, 1, 900 + n, 10 + b))
        z[b, order] = np.tile([1.0, -1.0, 3.0, -3.0], n // 4)
    x, h = dev(z[None, :, :I]), dev(z[:, I:])
    c = synth.uniform((batch, H), -1, 1, 900 + n, 3)
    sig = lambda v: 1.0 / (1.0 + np.exp(-v))
    if cell == "lstm":
        i, f, o, g = (z @ W.T + bias).reshape(batch, 4, H).transpose(1, 0, 2)
        c_ref = sig(f) * c + sig(i) * np.tanh(g)
        want = (sig(o) * np.tanh(c_ref), c_ref)
    else:
        pre, b4 = (z @ W.T).reshape(batch, 3, H), bias.reshape(4, H)
        nx, nh = z[:, :I] @ W[2 * H:, :I].T, z[:, I:] @ W[2 * H:, I:].T
        r, u = sig(pre[:, 0] + b4[0]), sig(pre[:, 1] + b4[1])
        want = ((1 - u) * np.tanh(nx + b4[2] + r * (nh + b4[3])) + u * z[:, I:],)
    tol = 4e-6 * 3 * (np.abs(z) @ np.abs(W).T).max() + 1e-5
    Wd = (cdev(Wc), dev(Wa), dev(bias), I, H)
    ws = amq.new_workspace(I, H, batch, 3)
    results = []
    if batch == 1:
        results.append(amq.lstm_step(*Wd, x[0], h, dev(c), 3, 2, ws) if cell == "lstm" else (amq.gru_step(*Wd, x[0], h, 3, 2, ws),))
    else:
        for form in (0, 1, 2):
            results.append(amq.selftest_batched_sequence(*Wd, x, h, dev(c) if cell == "lstm" else None, 3, 2, ws, form)[1:])
    assert amq.workspace_status(ws) == 0
    for got in results:
        for g, w in zip(got, want):
            assert np.abs(g.cpu().numpy() - w).max() <= tol
