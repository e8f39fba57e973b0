"""What users of this library have it do, as cases that can be timed and compared: recurrent steps and sequences (one
sequence and many, device and host buffers, stacked and paper form), greedy decoding, the output layer, matrix-vector and
batched products on on-line quantized activations, and row-wise weight quantization.

Sizes are those of the library's own workloads (paper_1802_00150_b200.synth) and of the paper's language models (hidden 300,
1024, vocabularies 10000 and 42000, 30-35 timesteps), plus ragged ones.  Weights are Gaussian with the spread of a trained
recurrent layer, inputs N(0, 1), states inside (-1, 1); a case's inputs follow from the seed alone.
"""
import math

import torch

from paper_1802_00150_b200 import amq

T = 2                       # alternating cycles; the paper uses two throughout


def listed():
    return [
        # one LSTM step of a small language model for a single stream, state kept by the caller: pure latency
        {"name": "lstm_step_300", "op": "step", "cell": "lstm", "I": 300, "H": 300, "batch": 1, "k_w": 2, "k_a": 2},
        # the layer of a larger language model over one sequence
        {"name": "lstm_sequence_1024_b1", "op": "sequence", "cell": "lstm", "I": 1024, "H": 1024, "batch": 1, "steps": 35,
         "k_w": 2, "k_a": 2},
        # the same layer at three bits, serving 64 sequences at once
        {"name": "lstm_sequence_1024_b64", "op": "sequence", "cell": "lstm", "I": 1024, "H": 1024, "batch": 64, "steps": 35,
         "k_w": 3, "k_a": 3},
        # a wide GRU layer over 256 sequences: the largest recurrent problem
        {"name": "gru_sequence_2048_b256", "op": "sequence", "cell": "gru", "I": 2048, "H": 2048, "batch": 256, "steps": 35,
         "k_w": 2, "k_a": 3},
        # a mid-size GRU with ragged widths and a small batch
        {"name": "gru_sequence_650_b20", "op": "sequence", "cell": "gru", "I": 300, "H": 650, "batch": 20, "steps": 30,
         "k_w": 3, "k_a": 2},
        # inputs and results in host memory, copies inside the call
        {"name": "lstm_host_sequence_1024_b64", "op": "host_sequence", "cell": "lstm", "I": 1024, "H": 1024, "batch": 64,
         "steps": 35, "k_w": 2, "k_a": 2},
        # the paper's own cell: rows of a quantized embedding in, only the state quantized on-line
        {"name": "lstm_embedded_1024_b64", "op": "embedded", "vocab": 10000, "I": 1024, "H": 1024, "batch": 64, "steps": 35,
         "k_w": 3, "k_a": 3},
        # greedy decoding of one stream with the 42000-word output layer
        {"name": "decode_42000", "op": "decode", "vocab": 42000, "I": 1024, "H": 1024, "steps": 64, "k_w": 2, "k_a": 2},
        # scoring: output layer and log-probabilities of a batch of states, ragged
        {"name": "score_9999_b600", "op": "score", "vocab": 9999, "H": 650, "batch": 600, "k_w": 2, "k_a": 2},
        # on-line quantization of one vector and its matrix-vector product (Table 6)
        {"name": "gemv_4096", "op": "gemv", "m": 4096, "n": 1024, "k_w": 2, "k_a": 2},
        # offline quantization of a large weight matrix
        {"name": "quantize_32768x1024", "op": "quantize", "rows": 32768, "n": 1024, "k_w": 3},
        # that matrix applied to a batch of activations
        {"name": "project_32768_b512", "op": "project", "m": 32768, "n": 1024, "batch": 512, "k_w": 3, "k_a": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# widths: over the whole range, one in two a multiple of 64 as most models have it, the others whatever comes
def _width(rng, lo, hi):
    v = _log_int(rng, lo, hi)
    return max(lo, v // 64 * 64) if rng.random() < 0.5 else v


def draw(rng):
    ops = ["step", "sequence", "sequence", "sequence", "host_sequence", "embedded", "decode", "score", "gemv", "quantize", "project"]
    most = max(_size(c) for c in listed())
    while True:
        c = {"op": rng.choice(ops), "k_w": rng.choice([2, 2, 3, 3, 4])}
        op = c["op"]
        if op != "quantize":
            c["k_a"] = rng.choice([2, 2, 3, 3, 4])
        if op in ("step", "sequence", "host_sequence"):
            c.update(cell=rng.choice(["lstm", "gru"]), I=_width(rng, 64, 2048), H=_width(rng, 128, 2048))
        if op == "step":
            c.update(batch=rng.choice([1, _log_int(rng, 1, 64)]))
        if op in ("sequence", "host_sequence", "embedded"):
            c.update(batch=rng.choice([1, _log_int(rng, 2, 256), _log_int(rng, 16, 256)]), steps=_log_int(rng, 8, 64))
        if op == "embedded":
            c.update(vocab=_log_int(rng, 2000, 42000), I=_width(rng, 128, 2048), H=_width(rng, 128, 2048))
        if op == "decode":
            c.update(vocab=_log_int(rng, 2000, 42000), I=_width(rng, 128, 2048), H=_width(rng, 128, 2048), steps=_log_int(rng, 16, 128))
        if op == "score":
            c.update(vocab=_log_int(rng, 2000, 42000), H=_width(rng, 128, 2048), batch=_log_int(rng, 16, 2240))
        if op == "gemv":
            c.update(m=_log_int(rng, 512, 42000), n=_width(rng, 128, 2048))
        if op == "quantize":
            c.update(rows=_log_int(rng, 512, 65536), n=_width(rng, 128, 4096))
        if op == "project":
            c.update(m=_log_int(rng, 1024, 65536), n=_width(rng, 128, 4096), batch=_log_int(rng, 2, 1024))
        if _size(c) <= most:
            return c


def _size(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


# ---- what a pass cannot do without ----------------------------------------------------------------------------------


def _packed(rows, n, k):
    return rows * k * ((n + 7) // 8 + 4)            # planes and coefficients


def _quantizer_ops(n, k):
    return 2 * (T + 1) * k * n + 2 * T * k * k * n  # the paper's count for one vector of n elements


def work(case):
    """Every input read once, every output written once; a product counts as the dense one it stands for (2 m n per vector)."""
    op, k_w, k_a = case["op"], case["k_w"], case.get("k_a", 0)
    if op in ("step", "sequence", "host_sequence"):
        I, H, batch, steps, lstm = case["I"], case["H"], case["batch"], case.get("steps", 1), case["cell"] == "lstm"
        m = (4 if lstm else 3) * H
        state = (2 if lstm else 1) * 4 * H * batch
        return {"bytes": _packed(m, I + H, k_w) + 16 * H + 4 * steps * batch * (I + (H if op == "sequence" else 0)) + 2 * state,
                "flops": steps * batch * (2 * m * (I + H) + _quantizer_ops(I + H, k_a))}
    if op == "embedded":
        I, H, batch, steps = case["I"], case["H"], case["batch"], case["steps"]
        rows = steps * batch
        return {"bytes": _packed(min(rows, case["vocab"]), I, k_w) + _packed(4 * H, I, k_w) + _packed(4 * H, H, k_w) + 16 * H
                + 4 * rows * (1 + H) + 16 * H * batch,
                "flops": rows * (8 * H * (I + H) + _quantizer_ops(H, k_a))}
    if op == "decode":
        I, H, vocab, steps = case["I"], case["H"], case["vocab"], case["steps"]
        return {"bytes": _packed(steps, I, k_w) + _packed(4 * H, I, k_w) + _packed(4 * H, H, k_w) + 16 * H + _packed(vocab, H, k_w)
                + 4 * vocab + 16 * H + 4 * steps,
                "flops": steps * (8 * H * (I + H) + 2 * vocab * H + _quantizer_ops(H, k_a))}
    if op == "score":
        H, vocab, batch = case["H"], case["vocab"], case["batch"]
        return {"bytes": 4 * batch * H + _packed(vocab, H, k_w) + 4 * vocab + 4 * batch * (vocab + 1),
                "flops": batch * (2 * vocab * H + _quantizer_ops(H, k_a) + 4 * vocab)}
    if op in ("gemv", "project"):
        m, n, batch = case["m"], case["n"], case.get("batch", 1)
        return {"bytes": 4 * batch * n + _packed(m, n, k_w) + 4 * m + 4 * batch * m, "flops": batch * (2 * m * n + _quantizer_ops(n, k_a))}
    rows, n = case["rows"], case["n"]
    return {"bytes": 4 * rows * n + _packed(rows, n, k_w), "flops": rows * _quantizer_ops(n, k_w)}


def tolerance(case):
    """Quantization is discontinuous: two correct fp32 implementations put the few elements that lie within rounding of a
    threshold on different sides.  One such element of an activation vector moves that vector's outputs by about a percent
    (one step of a 2-4 bit code), and a recurrent layer carries it on; hence the activations' own precision is what bounds
    results behind an on-line quantizer.  The quantizer's coefficients are fp32 sums."""
    if case["op"] == "quantize":
        return {"rel": 1e-4, "max": 2e-2, "differ": 1e-3}
    return {"rel": 1e-2, "max": 0.5, "differ": 1e-2}


# ---- inputs and passes ----------------------------------------------------------------------------------------------


def _weights(gen, rows, n, k):
    """Quantized planes and coefficients of a Gaussian matrix."""
    w = torch.empty((rows, n), device="cuda").normal_(0.0, 1.0 / math.sqrt(n), generator=gen)
    return amq.quantize(w, k, T)


def _normal(gen, *shape, std=1.0):
    return torch.empty(shape, device="cuda").normal_(0.0, std, generator=gen)


def _state(gen, *shape):
    return torch.empty(shape, device="cuda").uniform_(-1.0, 1.0, generator=gen)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    op, k_w = case["op"], case["k_w"]
    s = {"case": case}
    if op in ("step", "sequence", "host_sequence"):
        I, H, batch, steps, lstm = case["I"], case["H"], case["batch"], case.get("steps", 1), case["cell"] == "lstm"
        s["W"] = _weights(gen, (4 if lstm else 3) * H, I + H, k_w)
        s["bias"] = _normal(gen, 4 * H, std=0.1)
        s["x"] = _normal(gen, steps, batch, I)
        s["h"], s["c"] = _state(gen, batch, H), _state(gen, batch, H)
        s["workspace"] = amq.new_workspace(I, H, batch, case["k_a"])
        if op == "step":
            s["x"] = s["x"][0]
        if op == "host_sequence":
            s["staging"] = amq.new_host_staging(I, H, batch, steps)
            for key in ("x", "h", "c"):
                s[key] = s[key].cpu().pin_memory()
            s["h_last"], s["c_last"] = torch.empty_like(s["h"]).pin_memory(), torch.empty_like(s["c"]).pin_memory()
    elif op in ("embedded", "decode"):
        I, H, vocab, steps = case["I"], case["H"], case["vocab"], case["steps"]
        s["We"] = _weights(gen, vocab, I, k_w)
        s["Wi"], s["Wh"] = _weights(gen, 4 * H, I, k_w), _weights(gen, 4 * H, H, k_w)
        s["bias"] = _normal(gen, 4 * H, std=0.1)
        if op == "embedded":
            batch = case["batch"]
            s["tokens"] = torch.randint(vocab, (steps, batch), device="cuda", generator=gen, dtype=torch.int32)
            s["h"], s["c"] = _state(gen, batch, H), _state(gen, batch, H)
            s["workspace"] = amq.new_paper_workspace(H, batch, steps, case["k_a"])
        else:
            s["Ws"], s["bias_s"] = _weights(gen, vocab, H, k_w), _normal(gen, vocab, std=0.1)
            s["tokens"] = torch.zeros(steps + 1, device="cuda", dtype=torch.int32)
            s["tokens"][0] = torch.randint(vocab, (1,), device="cuda", generator=gen, dtype=torch.int32)[0]
            s["h"], s["c"] = _state(gen, H), _state(gen, H)
            s["workspace"] = amq.new_decode_workspace(vocab, I, H, k_w, case["k_a"])
    elif op == "score":
        s["Ws"], s["bias_s"] = _weights(gen, case["vocab"], case["H"], k_w), _normal(gen, case["vocab"], std=0.1)
        s["h"] = _state(gen, case["batch"], case["H"])
    elif op in ("gemv", "project"):
        s["W"], s["bias"] = _weights(gen, case["m"], case["n"], k_w), _normal(gen, case["m"], std=0.1)
        s["x"] = _normal(gen, *((case["n"],) if op == "gemv" else (case["batch"], case["n"])))
    else:
        s["w"] = _normal(gen, case["rows"], case["n"], std=1.0 / math.sqrt(case["n"]))
    return s


def run(s):
    case = s["case"]
    op, k_a = case["op"], case.get("k_a")
    if op == "quantize":
        return amq.quantize(s["w"], case["k_w"], T)
    if op == "gemv":
        return amq.quantized_gemv(*s["W"], s["x"], k_a, T, bias=s["bias"])
    if op == "project":
        codes, beta = amq.quantize(s["x"], k_a, T)
        return amq.binary_gemm(*s["W"], codes, beta, case["n"], bias=s["bias"])
    if op == "score":
        codes, beta = amq.quantize(s["h"], k_a, T)
        return amq.log_softmax_argmax(amq.binary_gemm(*s["Ws"], codes, beta, case["H"], bias=s["bias_s"]))
    I, H = case["I"], case["H"]
    if op == "decode":
        h, c = s["h"].clone(), s["c"].clone()          # the call updates the state in place
        tokens = amq.lm_greedy_decode(*s["We"], *s["Wi"], *s["Wh"], s["bias"], *s["Ws"], s["bias_s"], I, H, k_a, T, s["tokens"],
                                      h, c, s["workspace"])
        return tokens, h, c
    if op == "embedded":
        codes, beta = amq.embedding_rows(*s["We"], I, s["tokens"])
        return amq.lstm_sequence_paper(*s["Wi"], *s["Wh"], s["bias"], I, H, codes, beta, s["h"], s["c"], k_a, T, s["workspace"],
                                       want_h_seq=True)
    lstm, W, bias, ws = case["cell"] == "lstm", s["W"], s["bias"], s["workspace"]
    if op == "step":
        if lstm:
            return amq.lstm_step(*W, bias, I, H, s["x"], s["h"], s["c"], k_a, T, ws)
        return amq.gru_step(*W, bias, I, H, s["x"], s["h"], k_a, T, ws)
    if op == "sequence":
        if lstm:
            return amq.lstm_sequence(*W, bias, I, H, s["x"], s["h"], s["c"], k_a, T, ws, want_h_seq=True)
        return amq.gru_sequence(*W, bias, I, H, s["x"], s["h"], k_a, T, ws, want_h_seq=True)
    if lstm:
        return amq.lstm_sequence_host(*W, bias, I, H, s["x"], s["h"], s["c"], k_a, T, ws, s["staging"], s["h_last"], s["c_last"])
    return amq.gru_sequence_host(*W, bias, I, H, s["x"], s["h"], k_a, T, ws, s["staging"], s["h_last"])
