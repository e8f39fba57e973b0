"""Streams and events that a host call keeps for the next one: they do not outlive their context, and several threads may call at once."""
import os
import subprocess
import sys
import threading

import pytest
import torch

from paper_1802_00150_b200 import synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# A process of its own, without torch's allocator (which does not survive a reset): the same host call twice, a device reset, twice again.
AFTER_RESET = r"""
import ctypes, sys
import numpy as np
sys.path.insert(0, ".")
from paper_1802_00150_b200 import synth
lib = ctypes.CDLL("paper_1802_00150_b200/libamq_b200.so")
rt = ctypes.CDLL("libcudart.so.12")                # (already loaded by the library: the same instance)
drv = ctypes.CDLL("libcuda.so.1")
vp, sz, ci = ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int
lib.amq_cell_workspace_bytes.restype = lib.amq_cell_host_staging_bytes.restype = sz
I, H, batch, steps, ka = 1024, 96, 40, 29, 3       # 4.75 MB of inputs: copied in chunks on a kept stream
W = synth.normal((4 * H, I + H), 0.05, 1, 1)
xs = synth.normal((steps, batch, I), 1.0, 1, 2)
h0, c0 = synth.uniform((batch, H), -1, 1, 1, 3), synth.uniform((batch, H), -1, 1, 1, 4)
wpr = 4 * ((I + H + 127) // 128)

def ok(e):
    assert e == 0, e

def device(nbytes, host=None):
    p = vp()
    ok(rt.cudaMalloc(ctypes.byref(p), sz(nbytes)))
    if host is not None:
        ok(rt.cudaMemcpy(p, vp(host.ctypes.data), sz(nbytes), 1))
    return p

def run():
    w, codes, alpha = device(W.nbytes, W), device(4 * H * 2 * wpr * 4), device(4 * H * 2 * 4)
    ok(lib.amq_quantize(w, 4 * H, I + H, I + H, 2, 2, codes, alpha, None))
    wb, sb = lib.amq_cell_workspace_bytes(I, H, batch, ka), lib.amq_cell_host_staging_bytes(I, H, batch, steps)
    ws, st = device(wb), device(sb)
    h, c, seq = np.zeros_like(h0), np.zeros_like(c0), np.zeros((steps, batch, H), np.float32)
    q = lambda a: vp(a.ctypes.data)
    for _ in range(2):
        ok(lib.amq_lstm_sequence_host(codes, alpha, None, I, H, 2, q(xs), steps, q(h0), q(c0), batch, ka, 2, q(seq), q(h), q(c),
                                      ws, sz(wb), st, sz(sb), None))
        ok(lib.amq_workspace_status(ws, None))
    return h, c, seq

def context_id():
    n = ctypes.c_ulonglong()
    ok(drv.cuCtxGetId(None, ctypes.byref(n)))
    return n.value

first, before = run(), context_id()
ok(rt.cudaDeviceReset())
again, after = run(), context_id()
assert before != after, "a reset context has another id"
assert all(np.array_equal(a, b) for a, b in zip(first, again)) and np.abs(first[0]).max() > 0
print("same results")
"""


def test_a_host_call_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", AFTER_RESET], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same results" in r.stdout, r.stdout + r.stderr


def test_host_calls_from_more_threads_than_lanes_are_kept():
    from paper_1802_00150_b200 import amq
    I, H, batch, steps, ka, threads = 1024, 64, 40, 27, 2, 6
    Wc, Wa = amq.quantize(torch.from_numpy(synth.normal((4 * H, I + H), 0.05, 2, 1)).cuda(), 2, 2)
    xs = torch.from_numpy(synth.normal((threads, steps, batch, I), 1.0, 2, 2)).pin_memory()
    h0 = torch.from_numpy(synth.uniform((batch, H), -1, 1, 2, 3)).pin_memory()
    c0 = torch.from_numpy(synth.uniform((batch, H), -1, 1, 2, 4)).pin_memory()
    want = [amq.lstm_sequence(Wc, Wa, None, I, H, xs[k].cuda(), h0.cuda(), c0.cuda(), ka, 2, amq.new_workspace(I, H, batch, ka))[1].cpu()
            for k in range(threads)]
    got = [[] for _ in range(threads)]
    buffers = [(amq.new_workspace(I, H, batch, ka), amq.new_host_staging(I, H, batch, steps), torch.empty((batch, H)).pin_memory(),
                torch.empty((batch, H)).pin_memory(), torch.cuda.Stream()) for _ in range(threads)]
    torch.cuda.synchronize()

    def work(k):
        ws, staging, h, c, stream = buffers[k]
        with torch.cuda.stream(stream):
            for _ in range(5):
                amq.lstm_sequence_host(Wc, Wa, None, I, H, xs[k], h0, c0, ka, 2, ws, staging, h, c)
                got[k].append(h.clone())

    pool = [threading.Thread(target=work, args=(k,)) for k in range(threads)]
    for t in pool:
        t.start()
    for t in pool:
        t.join()
    for k in range(threads):
        assert len(got[k]) == 5 and all(torch.equal(h, want[k]) for h in got[k])
