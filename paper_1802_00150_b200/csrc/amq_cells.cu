// Quantized LSTM / GRU steps and sequences (Eq. 6; on-line quantization of the activation, Sec. 4): each step is the row
// quantizer on z = [x ; h] followed by the binary product with the gates behind it.  No step returns to the host.  One sequence
// runs in one launch (amq_rnn_persistent.cu), a batch in one launch (amq_rnn_resident.cu, amq_rnn_batched.cu) or as a chain of two
// launches per step on the caller's stream.
#include "amq_common.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>

namespace amq {

namespace {

struct CellCall {
    const uint32_t* Wcodes; const float* Walpha; const float* bias;
    int I, H, k_w, batch, k_a, T;
    bool gru;
};

amq_status validate(const CellCall& c, const void* workspace, size_t workspace_bytes)
{
    if (!c.Wcodes || !c.Walpha || c.I < 0 || c.H < 1 || c.batch < 0) return AMQ_ERR_INVALID_ARG;
    if (!valid_k(c.k_w) || !valid_k(c.k_a) || c.T < 0 || c.I + c.H > AMQ_MAX_N) return AMQ_ERR_UNSUPPORTED;
    if (!aligned16(c.Wcodes)) return AMQ_ERR_ALIGNMENT;
    if (!workspace || workspace_bytes < amq_cell_workspace_bytes(c.I, c.H, c.batch, c.k_a)) return AMQ_ERR_WORKSPACE;
    if (!aligned16(workspace)) return AMQ_ERR_ALIGNMENT;
    return AMQ_OK;
}

bool use_persistent(const CellCall& c)
{
    int grid, upc;
    size_t smem;
    return persistent_supported(c.I, c.H, c.batch, c.k_w, c.k_a, c.gru, &grid, &upc, &smem);
}

amq_status enqueue_persistent(const CellCall& c, const CellWorkspace& ws, const float* x_seq, int steps,
                              const float* h0, const float* c0, float* h_seq, float* h_last, float* c_last,
                              cudaStream_t st, unsigned poll_limit = 0, unsigned tag_bias = 0)
{
    // the caller has cleared the status words and, for more than one step, the exchange words behind them (stale
    // step tags must not match; a single step polls nothing)
    return launch_rnn_persistent(c.Wcodes, c.Walpha, c.bias, c.I, c.H, c.k_w, c.k_a, c.T, c.gru, x_seq, steps,
                                 h0, c0, h_seq, h_last, c_last, ws.hx, ws.status, st, poll_limit, tag_bias);
}

// (inputs come from the preceding kernels of the stream: ordinary loads after the wait, no read-only path)
__global__ void lstm_gates_kernel(const float* pre, const float* addend, const float* c_in, float* h_out, float* c_out, int H)
{
    grid_dependency_wait();
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= H) return;
    float g4[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) g4[g] = __ldcg(pre + g * H + u) + (addend ? __ldcg(addend + g * H + u) : 0.0f);
    const float ig = 1.0f / (1.0f + __expf(-g4[0])), fg = 1.0f / (1.0f + __expf(-g4[1])), og = 1.0f / (1.0f + __expf(-g4[2]));
    const float c = fg * __ldcg(c_in + u) + ig * tanhf(g4[3]);
    c_out[u] = c;
    h_out[u] = og * tanhf(c);
}

BatchedSequence batched_call(const CellCall& c, const CellWorkspace& ws, const float* x_seq, int steps, const float* h0, const float* c0,
                             float* h_seq, float* h_last, float* c_last)
{
    return BatchedSequence{c.Wcodes, c.Walpha, c.bias, c.I, c.H, c.I + c.H, c.k_w, c.k_a, c.T, c.batch, steps, c.gru, x_seq, h0, c0,
                           h_seq, h_last, c_last, {ws.h[0], ws.h[1]}, ws.c, nullptr, ws.zcodes, ws.zbeta, ws.counters, ws.status, 0, 0};
}

// quantize z = [x ; h_in] into the workspace, then product + gates
amq_status enqueue_step(const CellCall& c, const CellWorkspace& ws, const float* x, const float* h_in,
                        const float* c_in, float* h_out, float* c_out, cudaStream_t st)
{
    GemmArgs a{};
    a.Wcodes = c.Wcodes; a.Walpha = c.Walpha; a.m = (c.gru ? 3 : 4) * c.H; a.n = c.I + c.H; a.k_w = c.k_w;
    a.xcodes = ws.zcodes; a.xbeta = ws.zbeta; a.batch = c.batch; a.k_a = c.k_a;
    a.bias = c.bias;
    if (use_persistent(c))      // batch 1: one launch of the weight-stationary kernel, a sequence of one step
        return enqueue_persistent(c, ws, x, 1, h_in, c_in, nullptr, h_out, c_out, st);
    a.epilogue = c.gru ? EPI_GRU : EPI_LSTM;
    a.I = c.I; a.H = c.H; a.h_in = h_in; a.c_in = c_in; a.h_out = h_out; a.c_out = c_out;
    // the quantizer may be scheduled while the product of the previous timestep still runs (it waits for it first
    // thing) when that product runs as a single wave
    amq_status s = launch_quantize(x, c.I, c.I, h_in, c.H, c.H, c.batch, c.k_a, c.T, ws.zcodes, ws.zbeta, st,
                                   gemm_tc_single_wave(a));
    if (s != AMQ_OK) return s;
    a.overlap_with_previous = true;             // the quantizer above is the previous kernel of the stream
    return launch_binary_gemm(a, st);
}

// Inputs that arrive in chunks of timesteps: chunk q holds the steps begin[q] .. begin[q + 1] - 1, complete after ready[q].
constexpr int MAX_CHUNKS = 8;
struct Chunks {
    int count;
    int begin[MAX_CHUNKS + 1];
    cudaEvent_t ready[MAX_CHUNKS + 1];      // (one more, for the start of the copy stream)
};

// Copy stream and events of one host call.  Creating and destroying them cost 100 us a call, so up to LANES of a device wait for the next
// call (of any thread: a lane belongs to one call at a time); a lane more than that is destroyed when its call ends.
//
// Streams and events belong to a context and go with it, so lanes are kept for a device's primary context only, under its id (unique in
// the process: a device reset makes another).  A call that finds lanes of another id forgets them: they went with their context.  In a
// context that the application made with the driver API a call creates and destroys its own.
constexpr int LANES = 4, LANE_DEVICES = 16;
struct CopyLane { int device; unsigned long long context; cudaStream_t stream; cudaEvent_t event[MAX_CHUNKS + 1]; };     // context 0: not kept
struct KeptLanes { unsigned long long context; int count; CopyLane lane[LANES]; };
std::mutex g_lanes_mutex;
KeptLanes g_lanes[LANE_DEVICES];

// Id of the current context when it is the primary context of its device, else (or when the driver does not tell) 0.
unsigned long long primary_context_id()
{
    struct Driver {
        PFN_cuCtxGetCurrent_v4000 current = nullptr;
        PFN_cuCtxGetDevice_v2000 device = nullptr;
        PFN_cuDevicePrimaryCtxGetState_v7000 state = nullptr;
        PFN_cuDevicePrimaryCtxRetain_v7000 retain = nullptr;
        PFN_cuDevicePrimaryCtxRelease_v11000 release = nullptr;
        PFN_cuCtxGetId_v12000 id = nullptr;
        bool all = false;
        Driver()
        {
            auto get = [](const char* name, unsigned version) {
                void* f = nullptr;
                cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
                return cudaGetDriverEntryPointByVersion(name, &f, version, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess ? f : nullptr;
            };
            current = reinterpret_cast<PFN_cuCtxGetCurrent_v4000>(get("cuCtxGetCurrent", 4000));
            device = reinterpret_cast<PFN_cuCtxGetDevice_v2000>(get("cuCtxGetDevice", 2000));
            state = reinterpret_cast<PFN_cuDevicePrimaryCtxGetState_v7000>(get("cuDevicePrimaryCtxGetState", 7000));
            retain = reinterpret_cast<PFN_cuDevicePrimaryCtxRetain_v7000>(get("cuDevicePrimaryCtxRetain", 7000));
            release = reinterpret_cast<PFN_cuDevicePrimaryCtxRelease_v11000>(get("cuDevicePrimaryCtxRelease", 11000));
            id = reinterpret_cast<PFN_cuCtxGetId_v12000>(get("cuCtxGetId", 12000));
            all = current && device && state && retain && release && id;
        }
    };
    static const Driver d;
    CUcontext current = nullptr, primary = nullptr;
    CUdevice device;
    unsigned long long id = 0;
    unsigned flags;
    int active = 0;
    if (!d.all || d.current(&current) != CUDA_SUCCESS || !current || d.device(&device) != CUDA_SUCCESS ||
        d.state(device, &flags, &active) != CUDA_SUCCESS || !active || d.retain(&primary, device) != CUDA_SUCCESS)
        return 0;
    if (primary != current || d.id(current, &id) != CUDA_SUCCESS) id = 0;
    d.release(device);
    return id;
}

void destroy_lane(CopyLane& l)
{
    for (cudaEvent_t& e : l.event) if (e) { cudaEventDestroy(e); e = nullptr; }
    if (l.stream) { cudaStreamDestroy(l.stream); l.stream = nullptr; }
}

cudaError_t take_lane(CopyLane* out)
{
    CopyLane l{};
    cudaError_t e = cudaGetDevice(&l.device);
    if (e != cudaSuccess) return e;
    if (l.device < LANE_DEVICES) l.context = primary_context_id();
    if (l.context) {
        std::lock_guard<std::mutex> lock(g_lanes_mutex);
        KeptLanes& kept = g_lanes[l.device];
        if (kept.context != l.context) { kept.context = l.context; kept.count = 0; }
        if (kept.count > 0) { *out = kept.lane[--kept.count]; return cudaSuccess; }
    }
    e = cudaStreamCreateWithFlags(&l.stream, cudaStreamNonBlocking);
    for (int q = 0; q <= MAX_CHUNKS && e == cudaSuccess; ++q) e = cudaEventCreateWithFlags(&l.event[q], cudaEventDisableTiming);
    *out = l;
    return e;
}

void give_lane(CopyLane& l)
{
    if (l.context) {
        std::lock_guard<std::mutex> lock(g_lanes_mutex);
        KeptLanes& kept = g_lanes[l.device];
        if (kept.context == l.context && kept.count < LANES) { kept.lane[kept.count++] = l; l = CopyLane{}; return; }
    }
    destroy_lane(l);
}

// The counters as they stand after `counted` timesteps (self-test).
amq_status start_counters(const BatchedSequence& s, SequenceForm form, const SequenceShape& shape, int counted, cudaStream_t st)
{
    for (int b = 0; b < shape.blocks; ++b) {
        const int in_block = s.batch - b * shape.block < shape.block ? s.batch - b * shape.block : shape.block;
        const int quantizers = form == SEQ_RESIDENT && in_block < shape.ctas ? in_block : shape.ctas;
        const uint32_t word[2] = {(uint32_t)counted * (uint32_t)quantizers, (uint32_t)counted * (uint32_t)shape.ctas};
        for (int q = 0; q < 2; ++q)
            AMQ_CUDA_TRY(cudaMemcpyAsync(s.counters + (size_t)b * 64 + 32 * q, &word[q], 4, cudaMemcpyHostToDevice, st));
    }
    AMQ_CUDA_TRY(cudaStreamSynchronize(st));            // (the words are on this stack)
    return AMQ_OK;
}

// What the self-test asks for: a form, timesteps the counters start with, waits that run out.
struct Forced { SequenceForm form; int counted, late; };

// `chunks` (may be NULL): the stream waits for a chunk's event before the first kernel that reads it (batched calls only).
amq_status enqueue_sequence(const CellCall& c, const CellWorkspace& ws, const float* x_seq, int steps,
                            const float* h0, const float* c0, float* h_seq, float* h_last, float* c_last,
                            cudaStream_t st, const Chunks* chunks = nullptr, const Forced* forced = nullptr)
{
    const size_t state = (size_t)c.batch * c.H, state_bytes = state * sizeof(float);
    const bool persistent = steps > 0 && use_persistent(c);
    // (the exchange words or the counters lie directly behind the status words: one clear)
    AMQ_CUDA_TRY(cudaMemsetAsync(ws.status, 0, 256 + ((persistent && steps > 1) ? ws.hx_bytes : 0) + ws.counter_bytes, st));
    if (persistent)
        return enqueue_persistent(c, ws, x_seq, steps, h0, c0, h_seq, h_last, c_last, st);
    const BatchedSequence whole = batched_call(c, ws, x_seq, steps, h0, c0, h_seq, h_last, c_last);
    SequenceShape shape{};
    const SequenceForm form = forced ? forced->form : batched_sequence_form(whole, 0, &shape);
    if (forced && form != SEQ_CHAIN && !sequence_shape(whole, form, 0, &shape)) return AMQ_ERR_UNSUPPORTED;
    if (steps > 0 && form != SEQ_CHAIN) {
        if (forced && forced->counted > 0) {
            const amq_status r = start_counters(whole, form, shape, forced->counted, st);
            if (r != AMQ_OK) return r;
        }
        // one launch for all steps, or one per chunk, the state handed on in the caller's h_last / c_last
        for (int q = 0; q < (chunks ? chunks->count : 1); ++q) {
            const int s0 = chunks ? chunks->begin[q] : 0, s1 = chunks ? chunks->begin[q + 1] : steps;
            if (chunks) AMQ_CUDA_TRY(cudaStreamWaitEvent(st, chunks->ready[q], 0));
            BatchedSequence b = batched_call(c, ws, x_seq + (size_t)s0 * c.batch * c.I, s1 - s0, q ? h_last : h0, q ? c_last : c0,
                                             h_seq ? h_seq + (size_t)s0 * state : nullptr, h_last, c_last);
            b.counted = s0; b.launched = q;
            if (forced) { b.counted += forced->counted; b.launched += forced->counted; b.late = forced->late; }
            const amq_status r = launch_batched_sequence(b, form, shape, st);
            if (r != AMQ_OK) return r;
        }
        return AMQ_OK;
    }
    if (!c.gru) AMQ_CUDA_TRY(cudaMemcpyAsync(ws.c, c0, state_bytes, cudaMemcpyDeviceToDevice, st));
    const float* h_prev = h0;
    for (int s = 0; s < steps; ++s) {
        float* h_next = h_seq ? h_seq + (size_t)s * c.batch * c.H : ws.h[s & 1];
        const float* x = x_seq + (size_t)s * c.batch * c.I;
        for (int q = 0; chunks && q < chunks->count; ++q)
            if (s == chunks->begin[q]) AMQ_CUDA_TRY(cudaStreamWaitEvent(st, chunks->ready[q], 0));
        amq_status r = enqueue_step(c, ws, x, h_prev, ws.c, h_next, ws.c, st);
        if (r != AMQ_OK) return r;
        h_prev = h_next;
    }
    AMQ_CUDA_TRY(cudaMemcpyAsync(h_last, h_prev, state_bytes, cudaMemcpyDeviceToDevice, st));
    if (!c.gru) AMQ_CUDA_TRY(cudaMemcpyAsync(c_last, ws.c, state_bytes, cudaMemcpyDeviceToDevice, st));
    return AMQ_OK;
}

amq_status step_entry(const CellCall& c, const CellWorkspace& ws, const float* x, const float* h_in, const float* c_in, float* h_out,
                      float* c_out, cudaStream_t st)
{
    // (one sequence: the kernel clears the status word itself, a clear of its own costs as much host time as the launch)
    if (c.batch == 1 && use_persistent(c)) return enqueue_persistent(c, ws, x, 1, h_in, c_in, nullptr, h_out, c_out, st);
    AMQ_CUDA_TRY(cudaMemsetAsync(ws.status, 0, 256 + ws.counter_bytes, st));
    const BatchedSequence b = batched_call(c, ws, x, 1, h_in, c_in, nullptr, h_out, c_out);
    SequenceShape shape;
    const SequenceForm form = batched_sequence_form(b, 0, &shape);
    if (form != SEQ_CHAIN) return launch_batched_sequence(b, form, shape, st);
    return enqueue_step(c, ws, x, h_in, c_in, h_out, c_out, st);
}

amq_status sequence_entry(const CellCall& c, const float* x_seq, int steps, const float* h0, const float* c0,
                          float* h_seq, float* h_last, float* c_last,
                          void* workspace, size_t workspace_bytes, cudaStream_t st)
{
    amq_status s = validate(c, workspace, workspace_bytes);
    if (s != AMQ_OK) return s;
    if (steps < 0 || !h0 || !h_last || (!c.gru && (!c0 || !c_last)) || (steps > 0 && c.I > 0 && !x_seq))
        return AMQ_ERR_INVALID_ARG;
    if (h_last == h0 || (!c.gru && c_last == c0)) return AMQ_ERR_INVALID_ARG;
    if (c.batch == 0) return AMQ_OK;
    CellWorkspace ws = carve_cell_workspace(workspace, c.I, c.H, c.batch, c.k_a);
    return enqueue_sequence(c, ws, x_seq, steps, h0, c0, h_seq, h_last, c_last, st);
}

struct HostStaging {
    float* x_seq; float* h0; float* c0; float* h_seq; float* h_last; float* c_last;
    size_t bytes;
};

HostStaging carve_staging(void* base, int I, int H, int batch, int steps)
{
    HostStaging s;
    char* p = static_cast<char*>(base);
    size_t off = 0;
    const size_t state = round_up((size_t)batch * H * 4, 256);
    s.x_seq = reinterpret_cast<float*>(p + off);  off += round_up((size_t)steps * batch * I * 4, 256);
    s.h0 = reinterpret_cast<float*>(p + off);     off += state;
    s.c0 = reinterpret_cast<float*>(p + off);     off += state;
    s.h_seq = reinterpret_cast<float*>(p + off);  off += round_up((size_t)steps * batch * H * 4, 256);
    s.h_last = reinterpret_cast<float*>(p + off); off += state;
    s.c_last = reinterpret_cast<float*>(p + off); off += state;
    s.bytes = off;
    return s;
}

amq_status sequence_host_entry(const CellCall& c, const float* x_seq_host, int steps, const float* h0_host,
                               const float* c0_host, float* h_seq_host, float* h_last_host, float* c_last_host,
                               void* workspace, size_t workspace_bytes, void* staging, size_t staging_bytes,
                               cudaStream_t st)
{
    amq_status s = validate(c, workspace, workspace_bytes);
    if (s != AMQ_OK) return s;
    if (steps < 0 || !h0_host || !h_last_host || (!c.gru && (!c0_host || !c_last_host)) ||
        (steps > 0 && c.I > 0 && !x_seq_host))
        return AMQ_ERR_INVALID_ARG;
    if (!staging || staging_bytes < amq_cell_host_staging_bytes(c.I, c.H, c.batch, steps)) return AMQ_ERR_WORKSPACE;
    if (!aligned16(staging)) return AMQ_ERR_ALIGNMENT;
    if (c.batch == 0) return AMQ_OK;
    CellWorkspace ws = carve_cell_workspace(workspace, c.I, c.H, c.batch, c.k_a);
    HostStaging hs = carve_staging(staging, c.I, c.H, c.batch, steps);
    const size_t state_bytes = (size_t)c.batch * c.H * sizeof(float);
    const size_t x_bytes = (size_t)steps * c.batch * c.I * sizeof(float);
    // Large inputs of a batched call travel in chunks of timesteps on a stream of their own, so that the copy of the later
    // timesteps runs beside the kernels of the earlier ones (C4: 73 MB of inputs); the kernels wait for a chunk's event before
    // its first step.  Chunks grow from a twelfth of the sequence by 1.6 to a quarter (a remainder below half a chunk joins the last):
    // nothing runs during the first copy, and every chunk is a launch.
    const bool chunked = x_bytes >= ((size_t)4 << 20) && steps >= 2 && !(steps > 0 && use_persistent(c));
    Chunks chunks{};
    CopyLane lane{};
    // the small copies of the initial state go first: host-to-device copies are served in the order they were submitted,
    // whatever their stream, and the chain's first kernel needs them
    cudaError_t e = cudaMemcpyAsync(hs.h0, h0_host, state_bytes, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !c.gru) e = cudaMemcpyAsync(hs.c0, c0_host, state_bytes, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_fail(e);
    if (chunked) {
        for (int done = 0, size = (steps + 11) / 12; done < steps; ++chunks.count) {
            chunks.begin[chunks.count] = done;
            done = chunks.count == MAX_CHUNKS - 1 || done + size + size / 2 > steps ? steps : done + size;
            chunks.begin[chunks.count + 1] = done;
            size = (size * 8 + 4) / 5;
            if (size > (steps + 3) / 4) size = (steps + 3) / 4;
        }
        e = take_lane(&lane);
        for (int q = 0; q <= MAX_CHUNKS; ++q) chunks.ready[q] = lane.event[q];
        // the copy stream starts after what the caller's stream holds so far (the staging buffer may still be in use there)
        if (e == cudaSuccess) e = cudaEventRecord(chunks.ready[chunks.count], st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(lane.stream, chunks.ready[chunks.count], 0);
        const size_t step_bytes = (size_t)c.batch * c.I * sizeof(float);
        for (int q = 0; q < chunks.count && e == cudaSuccess; ++q) {
            const int s0 = chunks.begin[q], s1 = chunks.begin[q + 1];
            e = cudaMemcpyAsync(reinterpret_cast<char*>(hs.x_seq) + s0 * step_bytes,
                                reinterpret_cast<const char*>(x_seq_host) + s0 * step_bytes, (size_t)(s1 - s0) * step_bytes,
                                cudaMemcpyHostToDevice, lane.stream);
            if (e == cudaSuccess) e = cudaEventRecord(chunks.ready[q], lane.stream);
        }
        if (e != cudaSuccess) { if (lane.stream) cudaStreamSynchronize(lane.stream); destroy_lane(lane); return cuda_fail(e); }
    } else if (x_bytes) {
        AMQ_CUDA_TRY(cudaMemcpyAsync(hs.x_seq, x_seq_host, x_bytes, cudaMemcpyHostToDevice, st));
    }
    s = enqueue_sequence(c, ws, hs.x_seq, steps, hs.h0, hs.c0, h_seq_host ? hs.h_seq : nullptr, hs.h_last, hs.c_last, st,
                         chunked ? &chunks : nullptr);
    // the lane goes back, and its next user may record its events again, once the caller's stream has passed every wait for them
    struct Return {
        CopyLane& lane; cudaStream_t st;
        ~Return() { if (lane.stream) { cudaStreamSynchronize(lane.stream); cudaStreamSynchronize(st); give_lane(lane); } }
    } give_back{lane, st};
    if (s != AMQ_OK) return s;
    if (h_seq_host && steps > 0)
        AMQ_CUDA_TRY(cudaMemcpyAsync(h_seq_host, hs.h_seq, (size_t)steps * state_bytes, cudaMemcpyDeviceToHost, st));
    AMQ_CUDA_TRY(cudaMemcpyAsync(h_last_host, hs.h_last, state_bytes, cudaMemcpyDeviceToHost, st));
    if (!c.gru) AMQ_CUDA_TRY(cudaMemcpyAsync(c_last_host, hs.c_last, state_bytes, cudaMemcpyDeviceToHost, st));
    AMQ_CUDA_TRY(cudaStreamSynchronize(st));
    return AMQ_OK;
}

}  // namespace

amq_status launch_lstm_gates(const float* pre, const float* addend, const float* c_in, float* h_out, float* c_out, int H,
                             cudaStream_t st, bool overlap_with_previous)
{
    AMQ_CUDA_TRY(launch_kernel(lstm_gates_kernel, dim3((unsigned)((H + 255) / 256)), dim3(256), 0, st, overlap_with_previous,
                               pre, addend, c_in, h_out, c_out, H));
    AMQ_LAUNCH_CHECK();
    return AMQ_OK;
}

}  // namespace amq

extern "C" {

size_t amq_cell_workspace_bytes(int I, int H, int batch, int k_a)
{
    if (I < 0 || H < 1 || batch < 0 || !amq::valid_k(k_a)) return 0;
    return amq::carve_cell_workspace(nullptr, I, H, batch, k_a).bytes;
}

size_t amq_cell_host_staging_bytes(int I, int H, int batch, int steps)
{
    if (I < 0 || H < 1 || batch < 0 || steps < 0) return 0;
    return amq::carve_staging(nullptr, I, H, batch, steps).bytes;
}

amq_status amq_lstm_step(const uint32_t* Wcodes, const float* Walpha, const float* bias, int I, int H, int k_w,
                         const float* x, const float* h_in, const float* c_in, int batch, int k_a, int T,
                         float* h_out, float* c_out, void* workspace, size_t workspace_bytes, void* stream)
{
    amq::CellCall c{Wcodes, Walpha, bias, I, H, k_w, batch, k_a, T, false};
    amq_status s = amq::validate(c, workspace, workspace_bytes);
    if (s != AMQ_OK) return s;
    if (!h_in || !c_in || !h_out || !c_out || (I > 0 && !x) || h_out == h_in) return AMQ_ERR_INVALID_ARG;
    if (batch == 0) return AMQ_OK;
    amq::CellWorkspace ws = amq::carve_cell_workspace(workspace, I, H, batch, k_a);
    return amq::step_entry(c, ws, x, h_in, c_in, h_out, c_out, (cudaStream_t)stream);
}

amq_status amq_gru_step(const uint32_t* Wcodes, const float* Walpha, const float* bias, int I, int H, int k_w,
                        const float* x, const float* h_in, int batch, int k_a, int T,
                        float* h_out, void* workspace, size_t workspace_bytes, void* stream)
{
    amq::CellCall c{Wcodes, Walpha, bias, I, H, k_w, batch, k_a, T, true};
    amq_status s = amq::validate(c, workspace, workspace_bytes);
    if (s != AMQ_OK) return s;
    if (!h_in || !h_out || (I > 0 && !x) || h_out == h_in) return AMQ_ERR_INVALID_ARG;
    if (batch == 0) return AMQ_OK;
    amq::CellWorkspace ws = amq::carve_cell_workspace(workspace, I, H, batch, k_a);
    return amq::step_entry(c, ws, x, h_in, nullptr, h_out, nullptr, (cudaStream_t)stream);
}

amq_status amq_lstm_sequence(const uint32_t* Wcodes, const float* Walpha, const float* bias, int I, int H, int k_w,
                             const float* x_seq, int steps, const float* h0, const float* c0,
                             int batch, int k_a, int T, float* h_seq, float* h_last, float* c_last,
                             void* workspace, size_t workspace_bytes, void* stream)
{
    amq::CellCall c{Wcodes, Walpha, bias, I, H, k_w, batch, k_a, T, false};
    return amq::sequence_entry(c, x_seq, steps, h0, c0, h_seq, h_last, c_last, workspace, workspace_bytes,
                               (cudaStream_t)stream);
}

amq_status amq_gru_sequence(const uint32_t* Wcodes, const float* Walpha, const float* bias, int I, int H, int k_w,
                            const float* x_seq, int steps, const float* h0, int batch, int k_a, int T,
                            float* h_seq, float* h_last, void* workspace, size_t workspace_bytes, void* stream)
{
    amq::CellCall c{Wcodes, Walpha, bias, I, H, k_w, batch, k_a, T, true};
    return amq::sequence_entry(c, x_seq, steps, h0, nullptr, h_seq, h_last, nullptr, workspace, workspace_bytes,
                               (cudaStream_t)stream);
}

amq_status amq_lstm_sequence_host(const uint32_t* Wcodes, const float* Walpha, const float* bias,
                                  int I, int H, int k_w, const float* x_seq_host, int steps,
                                  const float* h0_host, const float* c0_host, int batch, int k_a, int T,
                                  float* h_seq_host, float* h_last_host, float* c_last_host,
                                  void* workspace, size_t workspace_bytes, void* staging, size_t staging_bytes,
                                  void* stream)
{
    amq::CellCall c{Wcodes, Walpha, bias, I, H, k_w, batch, k_a, T, false};
    return amq::sequence_host_entry(c, x_seq_host, steps, h0_host, c0_host, h_seq_host, h_last_host, c_last_host,
                                    workspace, workspace_bytes, staging, staging_bytes, (cudaStream_t)stream);
}

amq_status amq_gru_sequence_host(const uint32_t* Wcodes, const float* Walpha, const float* bias,
                                 int I, int H, int k_w, const float* x_seq_host, int steps,
                                 const float* h0_host, int batch, int k_a, int T,
                                 float* h_seq_host, float* h_last_host,
                                 void* workspace, size_t workspace_bytes, void* staging, size_t staging_bytes,
                                 void* stream)
{
    amq::CellCall c{Wcodes, Walpha, bias, I, H, k_w, batch, k_a, T, true};
    return amq::sequence_host_entry(c, x_seq_host, steps, h0_host, nullptr, h_seq_host, h_last_host, nullptr,
                                    workspace, workspace_bytes, staging, staging_bytes, (cudaStream_t)stream);
}

amq_status amq_selftest_sequence_give_up(const uint32_t* Wcodes, const float* Walpha, const float* bias,
                                         int I, int H, int k_w,
                                         const float* x_seq, int steps, const float* h0, const float* c0,
                                         int k_a, int T, float* h_last, float* c_last,
                                         void* workspace, size_t workspace_bytes, unsigned poll_limit, void* stream)
{
    amq::CellCall c{Wcodes, Walpha, bias, I, H, k_w, 1, k_a, T, false};
    amq_status s = amq::validate(c, workspace, workspace_bytes);
    if (s != AMQ_OK) return s;
    if (steps < 2 || !h0 || !c0 || !h_last || !c_last || (I > 0 && !x_seq) || h_last == h0 || c_last == c0)
        return AMQ_ERR_INVALID_ARG;
    if (poll_limit < 1 || poll_limit > 65536) return AMQ_ERR_INVALID_ARG;
    if (!amq::use_persistent(c)) return AMQ_ERR_UNSUPPORTED;
    amq::CellWorkspace ws = amq::carve_cell_workspace(workspace, I, H, 1, k_a);
    AMQ_CUDA_TRY(cudaMemsetAsync(ws.status, 0, 256 + ws.hx_bytes, (cudaStream_t)stream));
    // expected tags are offset by 2^30: the tags the CTAs publish (1 .. steps) never match
    return amq::enqueue_persistent(c, ws, x_seq, steps, h0, c0, nullptr, h_last, c_last, (cudaStream_t)stream,
                                   poll_limit, 1u << 30);
}

amq_status amq_selftest_batched_sequence(const uint32_t* Wcodes, const float* Walpha, const float* bias, int I, int H, int k_w, int gru,
                                         const float* x_seq, int steps, const float* h0, const float* c0, int batch, int k_a, int T,
                                         float* h_seq, float* h_last, float* c_last, void* workspace, size_t workspace_bytes,
                                         int form, int counted, int late, void* stream)
{
    amq::CellCall c{Wcodes, Walpha, bias, I, H, k_w, batch, k_a, T, gru != 0};
    amq_status s = amq::validate(c, workspace, workspace_bytes);
    if (s != AMQ_OK) return s;
    if (steps < 1 || !h0 || !h_last || (!c.gru && (!c0 || !c_last)) || (I > 0 && !x_seq) || h_last == h0 || (!c.gru && c_last == c0))
        return AMQ_ERR_INVALID_ARG;
    if (form < AMQ_FORM_CHAIN || form > AMQ_FORM_RESIDENT || counted < 0 || counted > 0x7fffffff - steps) return AMQ_ERR_INVALID_ARG;
    if (late < 0 || late > 3 || (late > 0 && (form == AMQ_FORM_CHAIN || counted > 0)) || (late >= 2 && steps < 2) ||
        (late == 3 && form != AMQ_FORM_RESIDENT))
        return AMQ_ERR_INVALID_ARG;
    if (batch < 2) return AMQ_ERR_UNSUPPORTED;
    amq::CellWorkspace ws = amq::carve_cell_workspace(workspace, I, H, batch, k_a);
    const amq::Forced forced{(amq::SequenceForm)form, counted, late};
    return amq::enqueue_sequence(c, ws, x_seq, steps, h0, c0, h_seq, h_last, c_last, (cudaStream_t)stream, nullptr, &forced);
}

amq_status amq_selftest_sequence_plan(int gru, int I, int H, int k_w, int k_a, int batch, int sm_count, int* form, int* split, double* clocks)
{
    if (I < 0 || H < 1 || batch < 1 || sm_count < 0 || !form || !split || !clocks || *form < -1 || *form > AMQ_FORM_RESIDENT)
        return AMQ_ERR_INVALID_ARG;
    if (!amq::valid_k(k_w) || !amq::valid_k(k_a) || I + H > AMQ_MAX_N) return AMQ_ERR_UNSUPPORTED;
    amq::BatchedSequence s{};
    s.I = I; s.H = H; s.n = I + H; s.k_w = k_w; s.k_a = k_a; s.T = 2; s.batch = batch; s.steps = 1; s.gru = gru != 0;
    amq::SequenceShape shape{};
    if (*form < 0) *form = amq::batched_sequence_form(s, sm_count, &shape);
    else if (*form != AMQ_FORM_CHAIN && !amq::sequence_shape(s, (amq::SequenceForm)*form, sm_count, &shape)) return AMQ_ERR_UNSUPPORTED;
    if (*form == AMQ_FORM_CHAIN) { shape = amq::SequenceShape{}; shape.clocks = amq::chain_clocks(s, sm_count); }
    split[0] = shape.ctas; split[1] = shape.block; split[2] = shape.warps;
    *clocks = shape.clocks;
    return AMQ_OK;
}

amq_status amq_workspace_status(const void* workspace, void* stream)
{
    if (!workspace) return AMQ_ERR_INVALID_ARG;
    AMQ_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    uint32_t word = 0;
    AMQ_CUDA_TRY(cudaMemcpy(&word, workspace, sizeof(word), cudaMemcpyDeviceToHost));
    return word == 0 ? AMQ_OK : AMQ_ERR_TIMEOUT;
}

}  // extern "C"
