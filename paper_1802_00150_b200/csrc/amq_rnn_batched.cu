// Batched quantized LSTM / GRU sequences (Eq. 6; stacked form of Fig. 3, right): ONE cooperative launch for all timesteps.
//
// The batch is cut into blocks of TB vectors; P CTAs (one per SM) share a block, each with its own blocks of hidden units.  A
// timestep is, in every CTA: quantize this CTA's share of the block's vectors z = [x_t ; h_{t-1}] (Algorithm 2, teams of 8 or 16
// warps), wait for the other P - 1 CTAs' shares, expand the planes of the whole block into shared memory, run the product of the own
// gate rows (amq_resident.cuh) with the gates in the epilogue, wait for the other CTAs' h.  The two waits are counters in the
// workspace, one pair per block of vectors: blocks never wait for one another.
//
// This is the form for weights that do not fit tensor memory, and for those that do where amq_rnn_resident.cu would need many passes of a few
// vectors over them; the two and the chain of launches compete on their estimated time (batched_sequence_form below).
//
// Against a quantizer launch and a product launch per timestep this takes out two launches (some 6 us of host time each on this
// machine, which had become longer than the kernels), the set-up of tensor memory and barriers, and the repeated expansion
// of the activation planes by every tile of weight rows.  What bounds a timestep now: the steps of the weight pipeline (240-300
// clocks per 256 bit positions of 128 plane-rows), the quantizer's chain of reductions, and the two waits (GRU 2048, 256 sequences,
// 2/3 bits, 32 vectors a block, clocks of a timestep: wait for h 1700, quantizer 12100, publish and wait for planes 2800, expansion of the
// activations 4700, weights 37000, last epilogue 5900, publish 1100).
#include "amq_resident.cuh"
#include "amq_sequence.cuh"

namespace amq {

namespace {

constexpr int SEQ_Y_LD = 132;                   // row stride of the staged pre-activations
using R = ResRoles<2, 8, 3>;                     // (640 threads: 96 registers each; the quantizer and the epilogue spill with 64)
constexpr int SEQ_QUANT_WARPS = 16;             // warps that quantize: two teams of 8, or one of 16
constexpr int SEQ_NG = 2;                       // groups of eight vectors per epilogue thread: blocks of up to 32 vectors

struct SeqParams {
    ResProblem p;               // units = H
    const float* bias;
    int H, steps, k_a;
    SeqVectors z;
    const float* x_seq; const float* h0; const float* c0;
    float* h_seq; float* h_last; float* c_last;
    float* h[2]; float* c;
    const float* addend;        // [steps][batch][4H] added before the gates, or null
    uint32_t* counters;         // [blocks][64]: word 0 quantized shares, word 32 finished products
    int planes_word, h_word;    // where a block's CTAs look for them: 0 and 32 (the self-test of the waits: the next word, which stays 0)
    uint32_t* status;
    int counted;                // timesteps in the counters at the start
    int P, unit_blocks, b_bytes;
    int team_warps;             // warps per quantized vector
    int unit_steps;             // pipeline steps of a block of units
};

// shared memory behind the activation operand
struct __align__(16) SeqShared {
    float beta[256];
    float alpha[2][AMQ_MAX_K * 128];
    uint32_t table[RES_TABLE];
    ResSync sync;
};

// The state update of one (unit, vector) from its staged pre-activations `yv` (gate g at yv[32 g]) and biases.
__device__ __forceinline__ void seq_cell(const SeqParams& a, const float* yv, const float (&bias)[4], const float* addend, size_t o,
                                         const float* h_prev, const float* c_prev, float* h_next, float* h_also, float* c_next)
{
    float g4[4], h;
#pragma unroll
    for (int g = 0; g < 4; ++g) g4[g] = yv[32 * g] + bias[g];
    if (a.p.cell == RES_LSTM) {
        if (addend) {
#pragma unroll
            for (int g = 0; g < 4; ++g) g4[g] += __ldcg(addend + (size_t)g * a.H);
        }
        const float ig = seq_logistic(g4[0]), fg = seq_logistic(g4[1]), og = seq_logistic(g4[2]), gg = tanhf(g4[3]);
        const float c = fg * __ldcg(c_prev + o) + ig * gg;
        c_next[o] = c;
        h = og * tanhf(c);
    } else {
        const float rg = seq_logistic(g4[0]), zg = seq_logistic(g4[1]), cand = tanhf(g4[2] + rg * g4[3]);
        h = (1.0f - zg) * cand + zg * __ldcg(h_prev + o);
    }
    h_next[o] = h;
    if (h_also) h_also[o] = h;
}

template <int KA, int EPT>
__global__ void __launch_bounds__(R::THREADS, 1)
rnn_batched_kernel(const __grid_constant__ SeqParams a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const ResProblem& p = a.p;
    // The warp's number in a uniform register leaves one more to the quantizer, which spills otherwise (35 steps of LSTM 1728/1024, 48 sequences,
    // 3-bit weights and activations: 641 us, 602 us so).  At four bits, and at two with sixteen elements a thread, the registers come
    // out the worse for it (2 to 7 % slower).
    constexpr bool UNIFORM = KA != 4 && !(KA == 2 && EPT == 16);
    const int tid = threadIdx.x, warp = UNIFORM ? __shfl_sync(0xffffffffu, tid >> 5, 0) : tid >> 5, lane = tid & 31, H = a.H;
    const int bb = (int)blockIdx.x / a.P, part = (int)blockIdx.x - bb * a.P, b0 = bb * p.TB;
    const int in_block = p.batch - b0 < p.TB ? p.batch - b0 : p.TB;         // vectors of this block
    const int tiles = (a.unit_blocks - part + a.P - 1) / a.P;              // blocks of 32 units
    SeqShared& sh = *reinterpret_cast<SeqShared*>(smem_raw + a.b_bytes);
    float* sY = reinterpret_cast<float*>(&sh + 1);                          // [TB][SEQ_Y_LD] pre-activations of a tile
    QuantScratch<KA, SEQ_QUANT_WARPS>* scratch = reinterpret_cast<QuantScratch<KA, SEQ_QUANT_WARPS>*>(&sh + 1);    // (they are dead then)
    const uint32_t sB = smem_u32(smem_raw);
    uint32_t* counter = a.counters + (size_t)bb * 64;

    res_fill_table(p, sh.table);
    if (tid == 0) res_sync_init<R>(sh.sync);
    if (warp == R::MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&sh.sync.tmem_slot)), "r"((uint32_t)RES_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xffffffffu, sh.sync.tmem_slot, 0);
    if (warp < 4) write_unit_scales(tmem, p.ring * p.N, warp);

    ResIssueState issue{0, 0, 0, 1};                // (apart and from constants: it stays in uniform registers)
    // stage of an expander or accumulator of an epilogue warp, and its parity: the same two registers, the quantizer needs the others
    int at = warp < R::EXP_WARPS ? warp >> 2 : 0;
    uint32_t at_parity = warp < R::EXP_WARPS ? 1u : 0u;
    int quant_parity = 0;
    bool ok = true;

#pragma unroll 1
    for (int t = 0; t < a.steps; ++t) {
        const bool last = t + 1 == a.steps;
        const float* h_prev = t == 0 ? a.h0 : (a.h_seq ? a.h_seq + (size_t)(t - 1) * p.batch * H : a.h[(t - 1) & 1]);

        // ---- 1. this CTA's share of the block's vectors ----
        if (t > 0) {
            if (tid == 0) ok = seq_wait(counter + a.h_word, seq_target(a.counted + t, a.P));
            if (__syncthreads_or(!ok)) { ok = false; break; }
        }
        if (warp < SEQ_QUANT_WARPS) {
            const float* x = a.x_seq + (size_t)t * p.batch * a.z.xn;
            const int teams = a.team_warps == 8 ? 2 : 1, team = teams == 2 ? warp >> 3 : 0;
            const QuantTeam quant{warp - 8 * team, 8 + team, a.team_warps * 32};
#pragma unroll 1
            for (int v = part + team * a.P; v < in_block; v += teams * a.P)
                seq_quantize<KA, EPT, SEQ_QUANT_WARPS>(a.z, x, h_prev, b0 + v, scratch[team], quant, quant_parity);
        }
        __syncthreads();
        if (tid == 0) {
            seq_publish(counter);
            ok = seq_wait(counter + a.planes_word, seq_target(a.counted + t + 1, a.P));
        }
        if (__syncthreads_or(!ok)) { ok = false; break; }

        // ---- 2. the planes of the whole block as the activation operand ----
        if (tid < p.N) {
            const int b = b0 + res_row_vector<KA>(tid), j = res_row_plane<KA>(tid);
            sh.beta[tid] = tid < p.TB * KA && b < p.batch ? __ldcg(a.z.zbeta + (size_t)b * KA + j) : 0.0f;
        }
        res_expand_activations<KA, 2>(p, a.z.zcodes, a.z.row_bytes >> 4, a.z.half_bytes >> 4, b0, sB);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

        // ---- 3. product, gates ----
        if (warp < R::EXP_WARPS) {
            ResFeeder<R, RES_GRU> feed;
            // (steps of earlier timesteps: the groups take turns without a break)
            const uint32_t skip = (uint32_t)(warp >> 2) - (uint32_t)t * (uint32_t)(tiles * a.unit_steps);
            feed.start(p, sh.table, part, a.P, tiles, tid & 127, (int)(skip & (R::GROUPS - 1)));
            ResFeedState state{at, at_parity};
            ok = res_feed(p, sh.sync, sh.table, feed, tmem, state);
            at = state.stage; at_parity = state.parity;
        } else if (warp == R::MMA_WARP) {
            ok = res_issue(p, sh.sync, tiles, tmem, sB, issue);
        } else if (warp < R::MMA_WARP) {
            const int te = tid - 32 * R::EXP_WARPS, quarter = warp & 3, sub = (warp - R::EXP_WARPS) >> 2, rl = quarter * 32 + (lane >> 2);
            float* h_next = last ? a.h_last : (a.h_seq ? a.h_seq + (size_t)t * p.batch * H : a.h[t & 1]);
            float* h_also = last && a.h_seq ? a.h_seq + (size_t)t * p.batch * H : nullptr;
            const float* c_prev = t == 0 ? a.c0 : a.c;
            float* c_next = last ? a.c_last : a.c;
            ResDrainState drain{at, at_parity};
            f32x2 beta[SEQ_NG][KA];
            res_load_beta<R, KA, SEQ_NG>(p, sh.beta, sub, beta);
#pragma unroll 1
            for (int it = 0; it < tiles && ok; ++it) {
                const int ub = part + it * a.P;
                float* sa = sh.alpha[it & 1];
                {
                    const int wr = res_row<RES_GRU>(p, ub, te & 127);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int plane = (te >> 7) + 2 * q;
                        sa[plane * 128 + (te & 127)] = plane < p.k_w && wr >= 0 ? __ldg(p.Walpha + (size_t)wr * p.k_w + plane) : 0.0f;
                    }
                }
                res_epi_bar<R>(false);              // (also: everybody is past the tile before last, whose buffer this is)
                f32x2 y[SEQ_NG][4];
                ok = res_drain_tile<R, KA, SEQ_NG>(p, sh.sync, sa, quarter, sub, tmem, beta, drain, y);
#pragma unroll
                for (int g = 0; g < SEQ_NG; ++g) {
                    const int e = (R::SPLIT * g + sub) * 8 + 2 * (lane & 3);
                    if (e >= p.TB) break;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float y0, y1;
                        unpack2(y[g][i], y0, y1);
                        sY[e * SEQ_Y_LD + rl + 8 * i] = y0;
                        sY[(e + 1) * SEQ_Y_LD + rl + 8 * i] = y1;
                    }
                }
                // lane quarter = gate: lane = unit, one vector per warp
                const int u = ub * 32 + lane;
                float bias[4];
#pragma unroll
                for (int g = 0; g < 4; ++g) bias[g] = (a.bias && u < H) ? __ldg(a.bias + g * H + u) : 0.0f;
                res_epi_bar<R>(false);
                const float* addend = a.addend ? a.addend + ((size_t)t * p.batch + b0) * 4 * H + u : nullptr;
                if (u < H) {
#pragma unroll 1
                    for (int e = te >> 5; e < in_block; e += R::EPI_WARPS)
                        seq_cell(a, sY + e * SEQ_Y_LD + lane, bias, addend ? addend + (size_t)e * 4 * H : nullptr, (size_t)(b0 + e) * H + u,
                                 h_prev, c_prev, h_next, h_also, c_next);
                }
                __syncwarp();                       // (the next tile's values are staged behind the barrier inside its drain)
            }
            at = drain.ring; at_parity = drain.parity;
        }
        if (__syncthreads_or(!ok)) { ok = false; break; }
        if (tid == 0) seq_publish(counter + 32);
    }

    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (!ok) {      // (uniform) give the tensor core time to drain before tensor memory is released
        if (tid == 0) atomicExch(a.status, 1u);
        __nanosleep(1000000);
        __syncthreads();
    }
    if (warp == R::MMA_WARP)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"((uint32_t)RES_TMEM_COLS) : "memory");
}

struct SeqPlan { SeqParams a; int grid; size_t smem; double clocks; };

size_t seq_more_smem(const ResProblem& p)
{
    // the staged pre-activations; the quantizer's scratch uses the same bytes
    constexpr size_t scratch = 2 * sizeof(QuantScratch<4, SEQ_QUANT_WARPS>);
    const size_t y = (size_t)p.TB * SEQ_Y_LD * 4;
    return sizeof(SeqShared) + (y > scratch ? y : scratch);
}

// Estimated clocks of a timestep: quantizer rounds (by activation bits), steps and epilogues of a CTA's blocks of units, expansion of the
// activations, waits.  Fitted to 415 problems (LSTM and GRU, 1 to 4 bits, 2 to 5000 sequences, widths 64 to 2048) on a B200 when the planes lay
// row by row and the epilogue added a constant per operand row, within 6 %
// (standard deviation; 19 % at worst).
double streaming_clocks(const ResProblem& p, int k_a, int P, int unit_blocks, int unit_steps, int team_warps)
{
    const int teams = SEQ_QUANT_WARPS / team_warps, vectors = (p.TB + P - 1) / P, per_cta = (unit_blocks + P - 1) / P;
    const double quantizer = (k_a <= 2 ? 6000.0 : k_a == 3 ? 8000.0 : 16800.0) * (p.n > team_warps * 256 ? 1.3 : 1.0);
    return 6200.0 + (vectors + teams - 1) / teams * quantizer + per_cta * (1.5 * unit_steps * res_slot_clocks(p) + 3000.0 + 14.0 * p.N * p.k_w) +
           11.0 * p.N * p.NS;
}

// `only`: blocks of that many vectors (0: the best)
bool plan(const BatchedSequence& s, int sms, int only, SeqPlan* out)
{
    if (s.batch < 2 || s.H < 1 || s.n > AMQ_MAX_N || (s.gru && s.I < 1)) return false;
    SeqParams a{};
    ResProblem p{};
    p.W = s.Wcodes; p.Walpha = s.Walpha; p.k_w = s.k_w; p.wpr = words_per_row(s.n);
    p.vec32 = p.wpr % 8 == 0 && (reinterpret_cast<uintptr_t>(s.Wcodes) & 31) == 0;
    p.cell = s.gru ? RES_GRU : RES_LSTM; p.units = s.H; p.n = s.n; p.I = s.I; p.batch = s.batch;
    if (s.gru) {
        p.nx = (s.I + 255) / 256; p.xw = s.I / 256;
        p.NS = p.nx + (s.n - 256 * p.xw + 255) / 256;
    } else {
        p.NS = (s.n + 255) / 256;
    }
    // block of vectors with the least estimated time per timestep
    double best = 0.0;
    const int ub = (s.H + 31) / 32, steps = p.k_w * ((p.NS + 1) / 2);
    for (int TB = 8; TB <= 8 * SEQ_NG * R::SPLIT; TB += 8) {
        if (only && TB != only) continue;
        ResProblem q = p;
        q.TB = TB;
        if (!res_set_block<R>(q, TB, s.k_a, seq_more_smem(q))) break;
        const int blocks = (s.batch + TB - 1) / TB;
        if (blocks > sms) continue;
        const int P = ub < sms / blocks ? ub : sms / blocks;
        // Several vectors per CTA: two teams take one each, sixteen elements a thread; their chains of reductions overlap (35 steps of GRU
        // 2048, 256 sequences, 3-bit activations: 1561 us with one team of sixteen warps, 1496 us; 4 to 27 % less over 24 problems with
        // 1 to 3 bits).  Not at four bits, where sixteen elements do not fit the registers (LSTM 2000/2000, 200 sequences: 2153 us
        // against 2660).
        const int team_warps = s.n <= 2048 || (s.n <= 4096 && TB > P && s.k_a <= 3) ? 8 : 16;
        const double t = streaming_clocks(q, s.k_a, P, ub, steps, team_warps);
        if (best == 0.0 || t < best) { best = t; a.p = q; a.P = P; a.unit_blocks = ub; a.unit_steps = steps; a.team_warps = team_warps; }
        if (TB >= s.batch) break;
    }
    if (best == 0.0) return false;
    const int blocks = (s.batch + a.p.TB - 1) / a.p.TB;
    a.b_bytes = a.p.NS * a.p.N * 128;
    a.bias = s.bias; a.H = s.H; a.steps = s.steps; a.k_a = s.k_a;
    a.z = SeqVectors{s.n, a.p.wpr, s.H, s.n - s.H, s.T, s.zcodes, s.zbeta, 16, (size_t)s.batch * s.k_a * 16};      // (pieces of all rows together: neighbouring lanes load neighbouring pieces)
    a.x_seq = s.x_seq; a.h0 = s.h0; a.c0 = s.c0; a.h_seq = s.h_seq; a.h_last = s.h_last; a.c_last = s.c_last;
    a.h[0] = s.h[0]; a.h[1] = s.h[1]; a.c = s.c; a.addend = s.addend;
    a.counters = s.counters; a.counted = s.counted; a.status = s.status;
    a.planes_word = s.late == 1 ? 1 : 0; a.h_word = s.late == 2 ? 33 : 32;
    out->grid = blocks * a.P;
    out->smem = (size_t)a.b_bytes + seq_more_smem(a.p);
    out->a = a;
    out->clocks = best;
    return true;
}

template <int KA>
amq_status launch(const SeqPlan& pl, cudaStream_t st)
{
    auto kernel = pl.a.p.n <= pl.a.team_warps * 256 ? rnn_batched_kernel<KA, 8> : rnn_batched_kernel<KA, 16>;
    AMQ_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem));
    SeqParams args = pl.a;
    void* params[] = {&args};
    AMQ_CUDA_TRY(cudaLaunchCooperativeKernel((void*)kernel, dim3((unsigned)pl.grid), dim3(R::THREADS), params, pl.smem, st));
    __atomic_fetch_add(&g_kernel_launches, 1ull, __ATOMIC_RELAXED);
    return AMQ_OK;
}

}  // namespace

bool streaming_sequence_shape(const BatchedSequence& s, int sms, SequenceShape* out)
{
    SeqPlan pl;
    if (sms < 1) sms = res_sm_count();
    if (!plan(s, sms, 0, &pl)) return false;
    *out = SequenceShape{sms, pl.grid / pl.a.P, pl.a.p.TB, pl.a.P, pl.a.team_warps, pl.clocks};
    return true;
}

amq_status launch_streaming_sequence(const BatchedSequence& s, const SequenceShape& shape, cudaStream_t st)
{
    SeqPlan pl;
    if (!plan(s, shape.sms, shape.block, &pl)) return AMQ_ERR_UNSUPPORTED;
    switch (s.k_a) {
        case 1: return launch<1>(pl, st);
        case 2: return launch<2>(pl, st);
        case 3: return launch<3>(pl, st);
        case 4: return launch<4>(pl, st);
    }
    return AMQ_ERR_UNSUPPORTED;
}

SequenceForm batched_sequence_form(const BatchedSequence& s, int sms, SequenceShape* out)
{
    // The least estimated time.  The weights are worth keeping in tensor memory while the vectors of a block need few passes over them: 35
    // timesteps of LSTM 1024/1024, 64 sequences, 3/3 bits take 400 us resident, 482 streamed; of GRU 1900/1900, 256 sequences, 2/3 bits
    // (52 passes of five vectors) 7268 us resident, 1264 streamed.  Over 122 problems (2 to 5000 sequences) the choice costs 0.3 % on
    // average against the best form of each, 9 % at worst (always the resident form: 19 %, and six times the time at worst).
    if (sms < 1) sms = res_sm_count();
    SequenceShape shape;
    SequenceForm form = SEQ_CHAIN;
    double best = 0.0;
    if (resident_sequence_shape(s, sms, &shape)) { form = SEQ_RESIDENT; best = shape.clocks; *out = shape; }
    if (streaming_sequence_shape(s, sms, &shape) && (best == 0.0 || shape.clocks < best)) { form = SEQ_STREAMING; best = shape.clocks; *out = shape; }
    // From eight tiles of 256 operand rows on the product of the chain fills the machine for longer than its launches take (LSTM 2048/2048,
    // 2048 sequences, 2/2 bits: 6915 us, streamed 7669; GRU 1024/1024, 4096 sequences, 2/3 bits: 6991, streamed 7045, resident 10915);
    // below, none of 69 problems was faster as a chain by more than 0.3 %, and where its product has to run on the CUDA cores it takes up to
    // 12 times as long.
    if (best > 0.0 && (long long)s.batch * s.k_a >= 2048) {
        const double chain = chain_clocks(s, sms);
        if (chain > 0.0 && chain < best) form = SEQ_CHAIN;
    }
    return form;
}

}  // namespace amq
