"""Entry points that are launched as programmatic dependents of whatever the caller's stream holds: what the kernel in front writes (weights
included) is read after it has been written, and what it reads is written after it has been read, without a synchronisation by the
caller; the same inside a CUDA graph, behind nodes that are no kernels and behind another stream."""
import pytest
import torch

from paper_1802_00150_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amq():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    from paper_1802_00150_b200 import amq as binding
    return binding


def dev(a):
    return torch.from_numpy(a).to(torch.float32).cuda()


# rows, columns, vectors, weight and activation bits: products of one and of several waves of tiles, from one row tile on, on both tensor-core
# kernels, and (2 vectors) the CUDA-core kernel
PROBLEMS = [(60, 130, 16, 2, 2), (2000, 300, 64, 2, 2), (5000, 1024, 96, 3, 3), (9999, 650, 200, 2, 2), (20000, 1024, 256, 4, 4), (300, 257, 2, 1, 2)]


# (forms 1 and 2, the tensor-core kernels, start at 16 vectors here)
@pytest.mark.parametrize("m,n,batch,kw,ka,form", [p + (f,) for p in PROBLEMS for f in (None, 1, 2) if f is None or p[2] >= 16])
def test_products_wait_for_the_kernel_in_front(amq, m, n, batch, kw, ka, form):
    """The weights, the activations and the bias change between products that follow one another on the stream, written by this library's
    quantizer and by foreign kernels in turn; every product leaves the bits of one that had the GPU to itself."""
    product = lambda *a, **k: amq.binary_gemm(*a, **k) if form is None else amq.selftest_binary_gemm(*a, form, **k)
    w = [dev(synth.normal((m, n), 0.03, 600 + m, i)) for i in range(2)]
    x = [dev(synth.normal((batch, n), 1.0, 600 + m, 2 + i)) for i in range(2)]
    b = [dev(synth.normal((m,), 0.1, 600 + m, 4 + i)) for i in range(2)]
    W, X = [amq.quantize(v, kw, 2) for v in w], [amq.quantize(v, ka, 2) for v in x]
    alone = {}
    for i in range(2):
        for j in range(2):
            torch.cuda.synchronize()
            alone[i, j] = product(*W[i], *X[j], n, bias=b[j])
            torch.cuda.synchronize()
    codes, alpha, xcodes, beta, bias, y = (torch.empty_like(t) for t in (*W[0], *X[0], b[0], alone[0, 0]))
    rounds, kept = 12, []
    for r in range(rounds):
        i, j = (r // 2) % 2, r % 2
        if r % 3 == 0:                                      # a foreign kernel writes the bias, the weights and the activations, the activations last
            bias.copy_(b[j]); codes.copy_(W[i][0]); alpha.copy_(W[i][1]); xcodes.copy_(X[j][0]); beta.copy_(X[j][1])
        elif r % 3 == 1:                                    # the weights last, by the quantizer
            amq.quantize(x[j], ka, 2, xcodes, beta); bias.copy_(b[j]); amq.quantize(w[i], kw, 2, codes, alpha)
        else:                                               # the activations last, by the quantizer
            bias.copy_(b[j]); amq.quantize(w[i], kw, 2, codes, alpha); amq.quantize(x[j], ka, 2, xcodes, beta)
        product(codes, alpha, xcodes, beta, n, bias=bias, y=y)
        kept.append((i, j, y.clone()))                      # (the next product overwrites what this reads)
    torch.cuda.synchronize()
    assert amq.device_status() == 0
    for i, j, got in kept:
        assert torch.equal(got, alone[i, j])


@pytest.mark.parametrize("rows,n,k", [(64, 700, 3), (1200, 200, 2), (1200, 1000, 3), (40, 5000, 4)])
def test_quantizer_and_softmax_wait_for_the_kernel_in_front(amq, rows, n, k):
    x = [dev(synth.normal((rows, n), 1.0, 620 + n, i)) for i in range(2)]
    want = []
    for v in x:
        torch.cuda.synchronize()
        want.append((*amq.quantize(v, k, 2), *amq.log_softmax_argmax(v)))
        torch.cuda.synchronize()
    buf, kept = torch.empty_like(x[0]), []
    for r in range(12):
        buf.copy_(x[r % 2])
        out = amq.quantize(buf, k, 2) if r < 6 else amq.log_softmax_argmax(buf)
        kept.append((r, out))
    torch.cuda.synchronize()
    for r, out in kept:
        for g, w in zip(out, want[r % 2][:2] if r < 6 else want[r % 2][2:]):
            assert torch.equal(g, w)


@pytest.mark.parametrize("m,n,batch,kw,ka", PROBLEMS)
def test_entry_points_in_a_cuda_graph(amq, m, n, batch, kw, ka):
    """Scoring captured behind a memset, a copy and an event of another stream, replayed on new inputs."""
    W = amq.quantize(dev(synth.normal((m, n), 0.03, 640 + m, 1)), kw, 2)
    xs = [dev(synth.normal((batch, n), 1.0, 640 + m, 2 + i)) for i in range(3)]

    def score(v):
        codes, beta = amq.quantize(v, ka, 2)
        return amq.log_softmax_argmax(amq.binary_gemm(*W, codes, beta, n))

    want = [tuple(t.clone() for t in score(v)) for v in xs]
    static, bias = xs[0].clone(), torch.ones(batch, n, device="cuda")
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        main = torch.cuda.current_stream()
        first = score(static)                               # behind nothing
        other = torch.empty_like(static)
        other.copy_(static)                                 # behind a copy
        second = score(other)
        side.wait_stream(main)
        with torch.cuda.stream(side):
            third_in = static + 0.0
        bias.zero_()
        main.wait_stream(side)                              # behind a join of two streams
        third = score(third_in)
    for i in (1, 2, 0, 1):
        static.copy_(xs[i])
        graph.replay()
        torch.cuda.synchronize()
        for got in (first, second, third):
            assert all(torch.equal(g, w) for g, w in zip(got, want[i]))
    assert amq.device_status() == 0
