"""The give-up path of bounded device-side waits, exercised without hurting the GPU: a status word written from
the host, and the kernels whose CTAs wait for one another (batch-1 and batched sequences, decoding) run with waits that are made to
run out (a smaller bound on the same bounded polls, or the ordinary one, for tags and counts nobody publishes).  Nothing here faults, traps or spins
without a limit."""
import numpy as np
import pytest
import torch

from paper_1802_00150_b200 import synth

pytestmark = pytest.mark.gpu

TIMEOUT = -6


@pytest.fixture(scope="module")
def amq():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    from paper_1802_00150_b200 import amq as binding
    return binding


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def small_model(amq, I, H, k_w=2, seed=80):
    W = synth.normal((4 * H, I + H), 0.08, seed, 1)
    return amq.quantize(dev(W), k_w, 2)


def test_status_word_written_from_the_host_is_reported_and_cleared_by_the_next_call(amq):
    I, H, ka = 64, 48, 2
    Wcodes, Walpha = small_model(amq, I, H)
    for batch in (1, 5):                       # the batch-1 kernel and a batched one-launch kernel
        ws = amq.new_workspace(I, H, batch, ka)
        assert amq.workspace_status(ws) == 0
        ws[:4] = torch.tensor([1, 0, 0, 0], dtype=torch.uint8, device="cuda")
        assert amq.workspace_status(ws) == TIMEOUT
        assert amq.status_string(TIMEOUT) != ""
        x = dev(synth.uniform((batch, I), -1, 1, 81, 1))
        h = dev(synth.uniform((batch, H), -1, 1, 81, 2))
        c = dev(synth.uniform((batch, H), -1, 1, 81, 3))
        amq.lstm_step(Wcodes, Walpha, None, I, H, x, h, c, ka, 2, ws)
        assert amq.workspace_status(ws) == 0
    for form in (amq.FORM_CHAIN, amq.FORM_STREAMING, amq.FORM_RESIDENT):        # every form of the last, batched call
        ws[:4] = torch.tensor([1, 0, 0, 0], dtype=torch.uint8, device="cuda")
        assert amq.workspace_status(ws) == TIMEOUT
        amq.selftest_batched_sequence(Wcodes, Walpha, None, I, H, x[None], h, c, ka, 2, ws, form)
        assert amq.workspace_status(ws) == 0


@pytest.mark.parametrize("I,H,steps,limit", [(64, 48, 4, 64), (256, 300, 6, 200), (1024, 1024, 35, 1000)])
def test_waits_that_run_out_set_the_status_and_leave_the_context_usable(amq, I, H, steps, limit):
    ka = 2
    Wcodes, Walpha = small_model(amq, I, H)
    xs = dev(synth.normal((steps, 1, I), 1.0, 82, 1))
    h0 = torch.zeros((1, H), device="cuda")
    c0 = torch.zeros((1, H), device="cuda")
    ws = amq.new_workspace(I, H, 1, ka)
    want = amq.lstm_sequence(Wcodes, Walpha, None, I, H, xs, h0, c0, ka, 2, amq.new_workspace(I, H, 1, ka), want_h_seq=True)
    h_last, c_last = amq.selftest_sequence_give_up(Wcodes, Walpha, None, I, H, xs, h0, c0, ka, 2, ws, limit)
    assert amq.workspace_status(ws) == TIMEOUT          # every CTA gave up in step 1 and said so
    assert torch.all(h_last == 0) and torch.all(c_last == 0)      # outputs untouched
    # the same workspace, the same stream, the next call: status cleared, results as from a fresh workspace
    got = amq.lstm_sequence(Wcodes, Walpha, None, I, H, xs, h0, c0, ka, 2, ws, want_h_seq=True)
    assert amq.workspace_status(ws) == 0
    for g, w in zip(got, want):
        assert torch.equal(g, w)


@pytest.mark.parametrize("late", [1, 2])
@pytest.mark.parametrize("form,cell,I,H,batch,kw,ka", [
    (2, "lstm", 64, 48, 9, 2, 2),           # one block of vectors, more CTAs than quantize
    (2, "gru", 300, 650, 150, 3, 2),       # several vectors per CTA
    (2, "lstm", 1024, 1024, 64, 3, 3),
    (1, "lstm", 64, 200, 40, 2, 2),         # several blocks
    (1, "gru", 2048, 2048, 256, 2, 3),
])
def test_batched_waits_that_run_out_set_the_status_and_leave_the_context_usable(amq, form, cell, I, H, batch, kw, ka, late):
    """late 1: nobody sees enough quantized vectors in step 0; late 2: nobody sees enough finished products in step 1."""
    steps, gru = 3, cell == "gru"
    Wcodes, Walpha = amq.quantize(dev(synth.normal(((3 if gru else 4) * H, I + H), 0.08, 85, 1)), kw, 2)
    xs = dev(synth.normal((steps, batch, I), 1.0, 85, 2))
    h0, c0 = dev(synth.uniform((batch, H), -1, 1, 85, 3)), None if gru else dev(synth.uniform((batch, H), -1, 1, 85, 4))
    args = (Wcodes, Walpha, None, I, H, xs, h0, c0, ka, 2)
    ws = amq.new_workspace(I, H, batch, ka)
    want = amq.selftest_batched_sequence(*args, amq.new_workspace(I, H, batch, ka), form)
    h_seq, h_last, c_last = amq.selftest_batched_sequence(*args, ws, form, late=late)
    assert amq.workspace_status(ws) == TIMEOUT
    assert torch.all(h_last == 0) and (gru or torch.all(c_last == 0))       # outputs untouched
    if late == 2:
        assert torch.equal(h_seq[0], want[0][0])                            # step 0 waits for nothing that is late
    # the same workspace, the same stream, the next call: status cleared, results as from a fresh workspace (the tensor memory is free again)
    got = amq.selftest_batched_sequence(*args, ws, form)
    assert amq.workspace_status(ws) == 0
    assert all(torch.equal(g, w) for g, w in zip(got, want) if w is not None)


@pytest.mark.parametrize("cell,I,H,batch,kw,ka", [
    ("lstm", 64, 48, 9, 2, 2),              # words of h in pairs
    ("gru", 301, 651, 150, 3, 2),           # single words, several vectors per team of warps
    ("lstm", 1024, 1024, 64, 3, 3),
])
def test_states_that_never_come_set_the_status_and_leave_the_context_usable(amq, cell, I, H, batch, kw, ka):
    """late 3 (weights in tensor memory): nobody sees the states of step 0 in step 1."""
    steps, gru, form = 3, cell == "gru", 2
    Wcodes, Walpha = amq.quantize(dev(synth.normal(((3 if gru else 4) * H, I + H), 0.08, 87, 1)), kw, 2)
    xs = dev(synth.normal((steps, batch, I), 1.0, 87, 2))
    h0, c0 = dev(synth.uniform((batch, H), -1, 1, 87, 3)), None if gru else dev(synth.uniform((batch, H), -1, 1, 87, 4))
    args = (Wcodes, Walpha, None, I, H, xs, h0, c0, ka, 2)
    ws = amq.new_workspace(I, H, batch, ka)
    want = amq.selftest_batched_sequence(*args, amq.new_workspace(I, H, batch, ka), form)
    h_seq, h_last, c_last = amq.selftest_batched_sequence(*args, ws, form, late=3)
    assert amq.workspace_status(ws) == TIMEOUT
    assert torch.all(h_last == 0) and (gru or torch.all(c_last == 0))       # outputs untouched
    assert torch.equal(h_seq[0], want[0][0])                                # step 0 needs no state of another CTA
    got = amq.selftest_batched_sequence(*args, ws, form)
    assert amq.workspace_status(ws) == 0
    assert all(torch.equal(g, w) for g, w in zip(got, want) if w is not None)


@pytest.mark.parametrize("cell,I,H,batch,steps,kw,ka", [
    ("lstm", 3, 1, 2, 9, 1, 1),             # one unit
    ("gru", 7, 33, 5, 8, 2, 3),             # odd widths: single words
    ("lstm", 0, 129, 17, 6, 3, 4),          # no inputs at all
    ("lstm", 260, 256, 70, 5, 2, 2),        # a pair of words across x and h never
    ("gru", 129, 127, 300, 4, 2, 2),        # several vectors per team, several passes: states in memory, behind a counter
    ("lstm", 33, 65, 1000, 3, 2, 3), ("gru", 64, 128, 700, 4, 2, 2),
])
def test_states_travel_as_words_at_every_width(amq, cell, I, H, batch, steps, kw, ka):
    """One launch and launches of one step each (which read their state from memory): the same steps, twice on one workspace, by words and, where
    a team quantizes several vectors, without."""
    gru = cell == "gru"
    Wcodes, Walpha = amq.quantize(dev(synth.normal(((3 if gru else 4) * H, I + H), 0.08, 89, 1)), kw, 2)
    ws = amq.new_workspace(I, H, batch, ka)
    for seed in (2, 12):
        xs = dev(synth.normal((steps, batch, I), 1.0, 89, seed)) if I else torch.empty((steps, batch, 0), device="cuda")
        h, c = dev(synth.uniform((batch, H), -1, 1, 89, seed + 1)), None if gru else dev(synth.uniform((batch, H), -1, 1, 89, seed + 2))
        h_seq, h_last, c_last = amq.selftest_batched_sequence(Wcodes, Walpha, None, I, H, xs, h, c, ka, 2, ws, 2)
        assert amq.workspace_status(ws) == 0
        fresh = amq.new_workspace(I, H, batch, ka)
        for t in range(steps):
            one, h, c = amq.selftest_batched_sequence(Wcodes, Walpha, None, I, H, xs[t:t + 1], h, c, ka, 2, fresh, 2)
            assert torch.equal(one[0], h_seq[t])
        assert torch.equal(h, h_last) and (gru or torch.equal(c, c_last))


@pytest.mark.parametrize("cell,I,H,batch,kw,ka", [("lstm", 64, 48, 9, 2, 2), ("gru", 300, 650, 20, 3, 2), ("lstm", 1024, 1024, 64, 3, 3), ("gru", 129, 127, 300, 2, 2)])
def test_words_of_an_earlier_call_are_not_taken_for_this_calls(amq, cell, I, H, batch, kw, ka):
    """A call of two steps leaves words of timestep 1 behind, the ones that the next call on the workspace looks for in its second step: behind
    the count of that call's first products, when they have been overwritten.  Other inputs every time, without a synchronisation in between."""
    gru = cell == "gru"
    Wcodes, Walpha = amq.quantize(dev(synth.normal(((3 if gru else 4) * H, I + H), 0.08, 90, 1)), kw, 2)
    ws = amq.new_workspace(I, H, batch, ka)
    calls = []
    for r, steps in enumerate((2, 2, 5, 2, 3, 2, 2, 4)):
        calls.append((dev(synth.normal((steps, batch, I), 1.0, 91, 3 * r)), dev(synth.uniform((batch, H), -1, 1, 91, 3 * r + 1)),
                      None if gru else dev(synth.uniform((batch, H), -1, 1, 91, 3 * r + 2))))
    run = lambda call, w: amq.selftest_batched_sequence(Wcodes, Walpha, None, I, H, *call, ka, 2, w, 2)
    got = [run(call, ws) for call in calls]
    assert amq.workspace_status(ws) == 0
    for call, g in zip(calls, got):
        fresh = amq.new_workspace(I, H, batch, ka)
        want = run(call, fresh)
        assert amq.workspace_status(fresh) == 0
        assert all(torch.equal(a, b) for a, b in zip(g, want) if a is not None)


@pytest.mark.parametrize("cell,kw,ka,steps", [("lstm", 2, 2, 13), ("lstm", 3, 3, 24), ("gru", 2, 3, 17)])
def test_host_chunks_of_two_steps_do_not_read_each_others_words(amq, cell, kw, ka, steps):
    """From 13 to 24 timesteps the first chunk of a host call is a launch of two steps: it leaves words of timestep 1, which the second chunk's
    launch, on the same counters, looks for as well.  The host call equals the device call bit for bit."""
    I = H = 1024
    batch, gru = 96, cell == "gru"                              # 5 MB and more of inputs: copied in chunks
    assert amq.selftest_sequence_plan(gru, I, H, kw, ka, batch)[0] == 2
    Wcodes, Walpha = amq.quantize(dev(synth.normal(((3 if gru else 4) * H, I + H), 0.05, 92, 1)), kw, 2)
    ws, staging = amq.new_workspace(I, H, batch, ka), amq.new_host_staging(I, H, batch, steps)
    for seed in (2, 12, 22):
        xs = torch.from_numpy(synth.normal((steps, batch, I), 1.0, 92, seed)).pin_memory()
        h0, c0 = (torch.from_numpy(synth.uniform((batch, H), -1, 1, 92, seed + i)).pin_memory() for i in (1, 2))
        h, c, seq = torch.empty_like(h0).pin_memory(), torch.empty_like(c0).pin_memory(), torch.empty((steps, batch, H)).pin_memory()
        if gru:
            amq.gru_sequence_host(Wcodes, Walpha, None, I, H, xs, h0, ka, 2, ws, staging, h, h_seq=seq)
            want = amq.gru_sequence(Wcodes, Walpha, None, I, H, xs.cuda(), h0.cuda(), ka, 2, amq.new_workspace(I, H, batch, ka), want_h_seq=True)
            got = (seq, h)
        else:
            amq.lstm_sequence_host(Wcodes, Walpha, None, I, H, xs, h0, c0, ka, 2, ws, staging, h, c, h_seq=seq)
            want = amq.lstm_sequence(Wcodes, Walpha, None, I, H, xs.cuda(), h0.cuda(), c0.cuda(), ka, 2, amq.new_workspace(I, H, batch, ka), want_h_seq=True)
            got = (seq, h, c)
        assert amq.workspace_status(ws) == 0
        assert all(torch.equal(g, w.cpu()) for g, w in zip(got, want))


@pytest.mark.parametrize("late", [1, 2])
@pytest.mark.parametrize("V,I,H", [(149, 33, 147), (3001, 96, 149), (42000, 1024, 1024)])
def test_decoding_waits_that_run_out_set_the_status_and_leave_the_context_usable(amq, V, I, H, late):
    steps, ka = 4, 2
    q = lambda shape, std, seed: amq.quantize(dev(synth.normal(shape, std, 86, seed)), 2, 2)
    We, Wi, Wh, Ws = q((V, I), 1.0, 1), q((4 * H, I), 0.2, 2), q((4 * H, H), 0.1, 3), q((V, H), 0.2, 4)
    ws = amq.new_decode_workspace(V, I, H, 2, ka)

    def start():
        tokens = torch.full((steps + 1,), -7, dtype=torch.int32, device="cuda")
        tokens[0] = V // 2
        return tokens, torch.full((1, H), 0.25, device="cuda"), torch.zeros((1, H), device="cuda")

    want, got, left = start(), start(), start()
    call = lambda f, r, *more: f(*We, *Wi, *Wh, None, *Ws, None, I, H, ka, 2, *r, ws, *more)
    call(amq.lm_greedy_decode, want)
    assert amq.device_status() == 0
    call(amq.selftest_decode_give_up, left, late)
    assert amq.device_status() == TIMEOUT and amq.device_status() == 0      # (the read clears it)
    assert all(torch.equal(a, b) for a, b in zip(left, start()))            # tokens and state as they were
    call(amq.lm_greedy_decode, got)
    assert amq.device_status() == 0
    assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_give_up_selftest_rejects_what_it_cannot_run(amq):
    I, H, ka = 64, 48, 2
    Wcodes, Walpha = small_model(amq, I, H)
    xs = dev(synth.normal((3, 1, I), 1.0, 83, 1))
    h0 = torch.zeros((1, H), device="cuda")
    ws = amq.new_workspace(I, H, 1, ka)
    for bad_limit in (0, 1 << 20):
        with pytest.raises(amq.AmqError) as e:
            amq.selftest_sequence_give_up(Wcodes, Walpha, None, I, H, xs, h0, h0.clone(), ka, 2, ws, bad_limit)
        assert e.value.status == -1
    h1 = torch.zeros((9, H), device="cuda")
    for form, late, counted, steps in ((0, 1, 0, 3), (1, 3, 0, 3), (2, 1, 5, 3), (2, 2, 0, 1)):
        with pytest.raises(amq.AmqError) as e:
            amq.selftest_batched_sequence(Wcodes, Walpha, None, I, H, torch.zeros((steps, 9, I), device="cuda"), h1, h1.clone(), ka, 2,
                                          amq.new_workspace(I, H, 9, ka), form, counted, late)
        assert e.value.status == -1
    with pytest.raises(amq.AmqError) as e:      # no words: nothing of the kind to look for
        h = torch.zeros((700, H), device="cuda")
        amq.selftest_batched_sequence(Wcodes, Walpha, None, I, H, torch.zeros((3, 700, I), device="cuda"), h, h.clone(), ka, 2,
                                      amq.new_workspace(I, H, 700, ka), 2, 0, 3)
    assert e.value.status == -2
    with pytest.raises(amq.AmqError) as e:      # a single step waits for nothing: refused
        amq.selftest_sequence_give_up(Wcodes, Walpha, None, I, H, xs[:1], h0, h0.clone(), ka, 2, ws, 100)
    assert e.value.status == -1


@pytest.mark.parametrize("form,cell,I,H,batch,kw,ka", [
    (2, "lstm", 64, 48, 9, 2, 2), (2, "gru", 300, 650, 20, 3, 2),      # one block of vectors; more CTAs than quantize
    (1, "lstm", 64, 200, 40, 2, 2), (1, "gru", 300, 650, 70, 1, 3),    # several blocks
])
def test_progress_counters_may_wrap(amq, form, cell, I, H, batch, kw, ka):
    """The counters of a one-launch sequence count CTAs times timesteps: past 2^31 (the sign of an int) and across 2^32 the results stay those
    of a run that starts at zero."""
    steps, gru = 4, cell == "gru"
    Wcodes, Walpha = amq.quantize(dev(synth.normal(((3 if gru else 4) * H, I + H), 0.08, 84, 1)), kw, 2)
    xs = dev(synth.normal((steps, batch, I), 1.0, 84, 2))
    h0, c0 = dev(synth.uniform((batch, H), -1, 1, 84, 3)), None if gru else dev(synth.uniform((batch, H), -1, 1, 84, 4))
    ws = amq.new_workspace(I, H, batch, ka)
    ctas = amq.selftest_sequence_plan(gru, I, H, kw, ka, batch, form=form)[1][0]
    want = amq.selftest_batched_sequence(Wcodes, Walpha, None, I, H, xs, h0, c0, ka, 2, ws, form)
    assert amq.workspace_status(ws) == 0
    for wrap in (31, 32):
        counted = min((1 << wrap) // ctas - 2, (1 << 31) - 1 - steps)      # reached within the four timesteps
        got = amq.selftest_batched_sequence(Wcodes, Walpha, None, I, H, xs, h0, c0, ka, 2, ws, form, counted)
        assert amq.workspace_status(ws) == 0
        assert all(torch.equal(g, w) for g, w in zip(got, want) if w is not None), wrap
