// Batched quantized LSTM / GRU sequences whose weights stay in TENSOR MEMORY (Eq. 6; Sec. 4): one cooperative launch for all timesteps.
//
// The hidden units are split over all the CTAs of a block of vectors, so that a CTA's share of the plane-rows is a tile or a few of 128
// lanes; expanded to E2M1 nibbles ONCE, they lie in tensor memory (n / 8 columns per tile) for the whole sequence.  A timestep is, in
// every CTA: quantize the own share of the vectors z = [x_t ; h_{t-1}] (Algorithm 2), wait for the other shares, expand the planes
// of all vectors into shared memory slot by slot while the MMAs of the finished slots run, fold the accumulators with the
// coefficients, apply the gates, store h as words that the others' quantizers look for.
//
// Against streaming the packed weights through an expander every timestep (amq_rnn_batched.cu) this takes the weights out of the loop: at
// n = 2048, 1024 units, 64 vectors, 3 bits each the product phase was 16600 of a timestep's 30000 clocks, most of it the expansion
// of 128 plane-rows x 3 per CTA; here the CTAs expand the activations instead, which are fewer.  What bounds a timestep now: the
// quantizer's chain of reductions, the wait for the words of h (an L2 round trip) and for the planes (that, a fence and an atomic), the tensor
// pipe (N / 2 clocks per 64 positions) where N is large.
//
// Plane-rows: lane 4 k_w u + k_w g + i of a tile = plane i of gate g of unit u, as many whole units as fit 128 lanes.  The four "gates" of a GRU
// are r, z and the x and h parts of the candidate: positions that a row does not have (the other part, past n) are zero nibbles,
// which add nothing, so the activation operand needs no masks and no split.
//
// Measured (clocks of a timestep, 64 vectors, 1024 units, n = 2048, 3 bits; 147 CTAs, 368 us for 35 timesteps): words of h and quantizer 7050,
// publish 1650, wait for planes 1500, their loads 1700, expansion 2400, rest of the MMAs 2250, folding 1850, gates 1850.  (374 us and some 200
// clocks more in the quantizer since it asks whether levels tie; with h in memory behind a counter 394 us: wait for h 1150, publish
// 1050 more; streamed weights 482 us.)
//
// More vectors than one accumulator (N <= 256 operand rows) or shared memory holds are taken in passes over the same weights.
#include "amq_sequence.cuh"
#include "amq_tcgen05.cuh"

namespace amq {

namespace {

// Sixteen warps (128 registers a thread: the quantizer and the folding spill with the 96 that a seventeenth leaves); while the others expand
// operand rows the last one issues the MMAs.
constexpr int RS_WARPS = 16, RS_THREADS = 32 * RS_WARPS, RS_MMA_WARP = RS_WARPS - 1, RS_FEEDERS = 32 * RS_MMA_WARP;
constexpr int RS_CHUNKS = 4;                    // (row, slot) pairs per thread and pass: shared memory holds 1800
constexpr int RS_TMEM_COLS = 512, RS_SF_COLS = 16;
constexpr int RS_SMEM_LIMIT = 226 * 1024, RS_SMEM_MIN = 116 * 1024;       // (more than half an SM's: one CTA per SM)

struct RsParams {
    const uint32_t* W; const float* Walpha; const float* bias;
    SeqVectors z;
    int I, k_w, gru, steps, batch;
    const float* x_seq; const float* h0; const float* c0;
    float* h_seq; float* h_last; float* c_last;
    unsigned long long* hx;     // [batch][H]: {h value, timestep}, from CTA to CTA
    float* h[2];                // the states where there are no words and no h_seq
    const float* addend;        // [steps][batch][4H] added before the gates, or null
    uint32_t* counters;         // [blocks][64]: word 0 quantized shares, word 32 finished products
    int planes_word, h_word;    // where a block's CTAs look for them: 0 and 32 (the self-test of the waits: the next word, which stays 0)
    uint32_t tag_bias;          // added to the timestep that is looked for in hx: 0 (self-test: 2^30)
    uint32_t* status;
    int counted, launched;      // timesteps and launches in the counters at the start
    int P, block;               // CTAs and vectors of a block
    int upc, upt, tiles;        // units per CTA, per tile of 128 lanes
    int TB, N, NS;              // vectors and operand rows of a pass, slots of 256 positions
    int b_bytes;
};

struct __align__(16) RsShared {
    float beta[288];                // (a group of eight vectors may reach past the last row)
    uint64_t chunk[RS_CHUNKS], done;
    uint32_t tmem_slot;
};

__device__ __forceinline__ uint32_t rs_upper_bits(int n) { return n >= 32 ? 0u : 0xffffffffu << (n < 0 ? 0 : n); }

// h travels from the CTAs that compute it to those that quantize it as words {value, timestep}: value and "ready" arrive together, with no
// fence in front of a counter and no load behind a wait (the same words as in amq_rnn_persistent.cu).  A reader never meets the words of
// another call: it looks at them first in the second timestep, behind a counter, and a word is overwritten only after every
// CTA of the block has seen the planes made of it.
// The words also keep the planes and coefficients of a timestep from being overwritten too soon, which no counter does: a vector's words are
// stored only after the CTA has consumed all that vector's planes and coefficients (they are in its shared memory, multiplied and folded, by
// the time its gates run), and the quantizer that writes the next ones waits for the words of every unit, so of every CTA of the block
// (each has units).  Planes loaded ahead, or words stored before the fold, would break that: then they need a buffer per parity.
__device__ __forceinline__ unsigned long long rs_load_word(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ ulonglong2 rs_load_words(const unsigned long long* p)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void rs_store_word(unsigned long long* p, float value, uint32_t tag)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" :: "l"(p), "l"(((unsigned long long)tag << 32) | __float_as_uint(value)) : "memory");
}

// This thread's elements of h in z = [x ; h] from the words of timestep `tag`; false when they did not come.
struct RsWords {
    const unsigned long long* words;        // null: h is in memory as it is (the first timestep)
    uint32_t tag;
    unsigned limit;                         // looks at a word before giving up
    template <int EPT>
    __device__ __forceinline__ bool gather(const SeqVectors& a, int vector, int t0, float (&w)[EPT]) const
    {
        const unsigned long long* p = words + (size_t)vector * a.H + (t0 - a.xn);
        const bool pairs = (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
        uint32_t pending = 0;
#pragma unroll
        for (int j = 0; j < EPT; ++j) pending |= (t0 + j >= a.xn && t0 + j < a.n ? 1u : 0u) << j;
#pragma unroll 1
        for (unsigned spins = 0; pending && spins < limit; ++spins) {
            unsigned long long v[EPT];              // (all the loads, then all the looks: one round trip)
            if (pairs && pending == (1u << EPT) - 1u) {
#pragma unroll
                for (int q = 0; q < EPT / 2; ++q) {
                    const ulonglong2 two = rs_load_words(p + 2 * q);
                    v[2 * q] = two.x; v[2 * q + 1] = two.y;
                }
            } else {
#pragma unroll
                for (int j = 0; j < EPT; ++j) v[j] = (pending >> j) & 1u ? rs_load_word(p + j) : 0ull;
            }
#pragma unroll
            for (int j = 0; j < EPT; ++j)
                if (((pending >> j) & 1u) && (uint32_t)(v[j] >> 32) == tag) { w[j] = __uint_as_float((uint32_t)v[j]); pending &= ~(1u << j); }
        }
        return pending == 0;
    }
};

// The CTA's plane-rows -> tensor memory, worker warp = (lane quarter, every fourth slot).  Bit 1 = -1 on both operands.
__device__ __forceinline__ void rs_expand_weights(const RsParams& a, uint32_t a0, int u0, int warp, int lane)
{
    const int r = (warp & 3) * 32 + lane, per_unit = 4 * a.k_w, ul = r / per_unit, g = (r - ul * per_unit) / a.k_w, i = r - ul * per_unit - g * a.k_w;
#pragma unroll 1
    for (int tile = 0; tile < a.tiles; ++tile) {
        const int ut = tile * a.upt + ul, u = u0 + ut;
        const bool live = ul < a.upt && ut < a.upc && u < a.z.H;
        const uint32_t* row = a.W + (live ? ((size_t)((a.gru && g == 3 ? 2 : g) * a.z.H + u) * a.k_w + i) * a.z.wpr : 0);
        const int lo = a.gru && g == 3 ? a.I : 0, hi = !live ? 0 : a.gru && g == 2 ? a.I : a.z.n;
#pragma unroll 1
        for (int h = warp >> 2; h < 2 * a.NS; h += RS_WARPS / 4) {      // 128 positions, 16 columns
            const uint4 v = live && 4 * h < a.z.wpr ? __ldg(reinterpret_cast<const uint4*>(row) + h) : make_uint4(0, 0, 0, 0);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            uint32_t y[16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = 32 * (4 * h + q);
                const uint32_t valid = rs_upper_bits(lo - e) & ~rs_upper_bits(hi - e);
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    y[4 * s + q] = (((w[q] << (3 - s)) & 0x88888888u) | 0x22222222u) & (((valid >> s) & 0x11111111u) * 15u);
            }
            asm volatile(
                "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                :: "r"(a0 + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(tile * a.NS * 32 + 16 * h)), "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]),
                   "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]), "r"(y[8]), "r"(y[9]), "r"(y[10]), "r"(y[11]), "r"(y[12]), "r"(y[13]),
                   "r"(y[14]), "r"(y[15]) : "memory");
        }
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

// One operand row's 256 positions -> 128 bytes (the order inside a slot is that of the weights' columns)
__device__ __forceinline__ void rs_expand_row(uint32_t addr, const uint4& v, int h)
{
    const uint32_t swizzle = (addr >> 3) & 0x70u;   // (row mod 8) * 16
#pragma unroll
    for (int s = 0; s < 4; ++s)
        st_shared_v4(addr + ((uint32_t)((4 * h + s) << 4) ^ swizzle), ((v.x << (3 - s)) & 0x88888888u) | 0x22222222u,
                     ((v.y << (3 - s)) & 0x88888888u) | 0x22222222u, ((v.z << (3 - s)) & 0x88888888u) | 0x22222222u,
                     ((v.w << (3 - s)) & 0x88888888u) | 0x22222222u);
}

// Folded rows of a vector: whole 16-byte pieces, an odd number of them (neighbouring vectors in different banks).
__host__ __device__ inline int rs_folded_stride(int rows) { return (rows >> 2 | 1) << 2; }

// The four gates of a unit from its 4 KW folded plane-rows, planes added in order.
template <int KW>
__device__ __forceinline__ void rs_unit_sums(const float* folded, const float* alpha, float (&g4)[4])
{
    float s[4 * KW], al[4 * KW];
#pragma unroll
    for (int q = 0; q < KW; ++q) {
        const float4 v = reinterpret_cast<const float4*>(folded)[q], w = reinterpret_cast<const float4*>(alpha)[q];
        s[4 * q] = v.x; s[4 * q + 1] = v.y; s[4 * q + 2] = v.z; s[4 * q + 3] = v.w;
        al[4 * q] = w.x; al[4 * q + 1] = w.y; al[4 * q + 2] = w.z; al[4 * q + 3] = w.w;
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        g4[g] = 0.0f;
#pragma unroll
        for (int i = 0; i < KW; ++i) g4[g] = fmaf(al[g * KW + i], s[g * KW + i], g4[g]);
    }
}

// WORDS: h travels as words, otherwise in memory behind a counter (two kernels: the one without the words' code is the smaller).
template <int KA, int NW, bool WORDS>
__global__ void __launch_bounds__(RS_THREADS, 1)
rnn_resident_kernel(const __grid_constant__ RsParams a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // The warp's number in a uniform register where that is the faster code (61 problems timed): at four bits, whose quantizer then spills 12
    // instead of 56 bytes a thread (3 % at teams of four warps), and at two bits with teams of four or eight (1 %); elsewhere it is 1 %
    // slower.
    constexpr bool UNIFORM = KA == 4 || (KA == 2 && NW <= 8);
    const int tid = threadIdx.x, warp = UNIFORM ? __shfl_sync(0xffffffffu, tid >> 5, 0) : tid >> 5, lane = tid & 31, H = a.z.H, k_w = a.k_w;
    const int bb = (int)blockIdx.x / a.P, part = (int)blockIdx.x - bb * a.P, b0 = bb * a.block;
    const int in_block = a.batch - b0 < a.block ? a.batch - b0 : a.block, quantizers = in_block < a.P ? in_block : a.P;
    const int u0 = part * a.upc, units = u0 < H ? (H - u0 < a.upc ? H - u0 : a.upc) : 0;
    const int rows_per_tile = a.upt * 4 * k_w, all_rows = a.upc * 4 * k_w, LD = rs_folded_stride(all_rows);
    RsShared& sh = *reinterpret_cast<RsShared*>(smem_raw + a.b_bytes);
    float* sAlpha = reinterpret_cast<float*>(&sh + 1);              // [all_rows]
    float* sBias = sAlpha + all_rows;                               // [upc][4]
    float* sState = sBias + 4 * a.upc;                              // [block][upc]: c (LSTM) or h (GRU)
    // in the operand's bytes while it is dead: the quantizer's scratch, the folded rows [TB][LD]
    QuantScratch<KA, NW>* scratch = reinterpret_cast<QuantScratch<KA, NW>*>(smem_raw);
    float* sS = reinterpret_cast<float*>(smem_raw);
    const uint32_t sB = smem_u32(smem_raw);
    uint32_t* counter = a.counters + (size_t)bb * 64;

    if (tid == 0) {
#pragma unroll
        for (int q = 0; q < RS_CHUNKS; ++q) mbar_init(smem_u32(&sh.chunk[q]), RS_MMA_WARP);
        mbar_init(smem_u32(&sh.done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == RS_MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&sh.tmem_slot)), "r"((uint32_t)RS_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
#pragma unroll 1
    for (int q = tid; q < all_rows; q += RS_THREADS) {
        const int ul = q / (4 * k_w), g = (q - ul * 4 * k_w) / k_w, i = q - ul * 4 * k_w - g * k_w;
        sAlpha[q] = ul < units ? __ldg(a.Walpha + ((size_t)(a.gru && g == 3 ? 2 : g) * H + u0 + ul) * k_w + i) : 0.0f;
    }
#pragma unroll 1
    for (int q = tid; q < 4 * units; q += RS_THREADS) sBias[q] = a.bias ? __ldg(a.bias + (size_t)(q & 3) * H + u0 + (q >> 2)) : 0.0f;
    const float* state0 = a.gru ? a.h0 : a.c0;
#pragma unroll 1
    for (int q = tid; q < in_block * units; q += RS_THREADS) {
        const int v = q / units, ul = q - v * units;
        sState[v * a.upc + ul] = __ldcg(state0 + (size_t)(b0 + v) * H + u0 + ul);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // All 512 columns start at column 0.  (As a constant the address keeps the operands of the MMAs in uniform registers.)
    constexpr uint32_t tmem = 0;
    const uint32_t sf = tmem + (uint32_t)(a.tiles * a.N), a0 = sf + RS_SF_COLS;
    if (warp < 4) write_unit_scales(tmem, a.tiles * a.N, warp);
    rs_expand_weights(a, a0, u0, warp, lane);      // (made visible to the MMAs by the barriers of the first timestep)

    const QuantTeam quant{warp % NW, 8 + warp / NW, NW * 32};
    int quant_parity = 0;
    uint32_t phase = 0;                             // of the mbarriers: one per pass
    // every CTA takes the slots from another one on: they all read the same planes at the same time
    const int first_slot = part % a.NS;
    int rows_now = 0, slot_0 = 0, row_0 = 0, d_slot = 0, d_row = 0;     // this thread's first (slot, row) of a pass, and the step to the next
    const int v_0 = tid / units, ul_0 = tid - v_0 * units, d_v = RS_THREADS / units, d_ul = RS_THREADS - d_v * units;    // the same of (vector, unit)
    bool ok = sh.tmem_slot == tmem;

#pragma unroll 1
    for (int t = 0; ok && t < a.steps; ++t) {
        const bool last = t + 1 == a.steps;

        // ---- 1. this CTA's share of the block's vectors ----
        if (part < quantizers) {                    // (uniform over the CTA)
            if (WORDS ? t == 1 : t > 0) {           // (words: those of another call are gone)
                if (tid == 0) ok = seq_wait(counter + a.h_word, seq_target(WORDS ? a.launched + 1 : a.counted + t, a.P));
                if (__syncthreads_or(!ok)) { ok = false; break; }
            }
            const float* x = a.x_seq + (size_t)t * a.batch * a.z.xn;
            const float* h_prev = t == 0 || WORDS ? a.h0 : (a.h_seq ? a.h_seq + (size_t)(t - 1) * a.batch * H : a.h[(t - 1) & 1]);
#pragma unroll 1
            for (int v = part + warp / NW * a.P; v < in_block; v += RS_WARPS / NW * a.P) {
                if constexpr (WORDS)
                    ok &= seq_quantize<KA, 8, NW, true>(a.z, x, h_prev, b0 + v, scratch[warp / NW], quant, quant_parity,
                                                  RsWords{t == 0 ? nullptr : a.hx, (uint32_t)t + a.tag_bias, ok ? SEQ_POLL_LIMIT : 1u});
                else
                    seq_quantize<KA, 8, NW, false>(a.z, x, h_prev, b0 + v, scratch[warp / NW], quant, quant_parity);
                // the next timestep's inputs on their way into L2
                const int e = (quant.warp * 32 + lane) * 8;
                if (!last && e < a.z.xn)
                    asm volatile("prefetch.global.L2 [%0];" :: "l"(x + (size_t)(a.batch + b0 + v) * a.z.xn + e));
            }
            if (__syncthreads_or(!ok)) { ok = false; break; }
            if (tid == 0) seq_publish(counter);
        }
        if (tid == 0) ok = seq_wait(counter + a.planes_word, seq_target(a.counted + t + 1, quantizers));
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        if (__syncthreads_or(!ok)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

        float* h_seq = a.h_seq ? a.h_seq + (size_t)t * a.batch * H : nullptr;
#pragma unroll 1
        for (int v0 = 0; v0 < in_block; v0 += a.TB, phase ^= 1u) {
            const int nv = in_block - v0 < a.TB ? in_block - v0 : a.TB, rows = nv * KA;
            if (warp == RS_MMA_WARP) {
                if (v0 > 0) __syncthreads();
                // ---- 2. MMAs of a slot as soon as its operand rows are there ----
                const bool issues = elect_one();
                const uint32_t idesc = (1u << 7) | (1u << 10) | ((uint32_t)(a.N >> 3) << 17) | (1u << 23) | (8u << 24);     // E2M1, E8M0, M 128
                const uint64_t desc = smem_desc(sB);
                const uint32_t lo = (uint32_t)desc, hi = (uint32_t)(desc >> 32);
                int s = 0;
                uint32_t b = lo + (uint32_t)(first_slot * a.N * 8), w = a0 + (uint32_t)(first_slot * 32), wrap = (uint32_t)(a.NS - first_slot);
#pragma unroll 1
                for (int have = 1; s < a.NS && ok; ++have) {
                    ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sh.chunk[have - 1]), phase));
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    // the slots whose rows the chunks so far cover, without a look at anything in between
                    int end = have * RS_FEEDERS / rows;
                    if (end > a.NS) end = a.NS;
#pragma unroll 1
                    for (; s < end; ++s) {
                        if (s == (int)wrap) { b = lo; w = a0; }
                        uint32_t wt = w, acc = tmem;
#pragma unroll 1
                        for (int tile = 0; tile < a.tiles; ++tile) {
                            if (issues) mma_mxf4_stage_ta(acc, wt, b, hi, idesc, s != 0 ? 1u : 0u, sf);
                            wt += (uint32_t)(a.NS * 32); acc += (uint32_t)a.N;
                        }
                        b += (uint32_t)(a.N * 8); w += 32;
                    }
                }
                if (issues && ok) mma_commit(smem_u32(&sh.done));
                __syncwarp();
            } else {
                const size_t row0 = (size_t)(b0 + v0) * KA, half = (size_t)a.batch * KA;
                if (rows != rows_now) {
                    rows_now = rows;
                    slot_0 = tid / rows; row_0 = tid - slot_0 * rows; d_slot = RS_FEEDERS / rows; d_row = RS_FEEDERS - d_slot * rows;
                }
                uint4 lo[RS_CHUNKS], hi[RS_CHUNKS];
                uint32_t addr[RS_CHUNKS];           // 0: no such pair
                int slot = slot_0, row = row_0;
#pragma unroll
                for (int q = 0; q < RS_CHUNKS; ++q) {
                    addr[q] = 0;
                    if (slot < a.NS) {              // (other SMs wrote the planes: not through the read-only path)
                        const int s = slot + first_slot < a.NS ? slot + first_slot : slot + first_slot - a.NS;
                        addr[q] = sB + (uint32_t)((s * a.N + row) * 128);
                        const uint4* src = reinterpret_cast<const uint4*>(a.z.zcodes) + (size_t)(2 * s) * half + row0 + row;
                        lo[q] = __ldcg(src);
                        hi[q] = 8 * s + 4 < a.z.wpr ? __ldcg(src + half) : make_uint4(0, 0, 0, 0);
                    }
                    slot += d_slot; row += d_row;
                    if (row >= rows) { row -= rows; ++slot; }
                }
                if (v0 > 0) __syncthreads();        // the folded rows of the pass before have been read
                if (tid < rows) sh.beta[tid] = __ldcg(a.z.zbeta + row0 + tid);
#pragma unroll
                for (int q = 0; q < RS_CHUNKS; ++q) {
                    if (addr[q]) {
                        rs_expand_row(addr[q], lo[q], 0);
                        rs_expand_row(addr[q], hi[q], 1);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&sh.chunk[q])) : "memory");
                }
            }

            // the first addends of this thread on their way
            float ahead[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (a.addend && v_0 < nv) {
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    ahead[g] = __ldcg(a.addend + (((size_t)t * a.batch + b0 + v0 + v_0) * 4 + g) * H + u0 + ul_0);
            }

            // ---- 3. accumulators: sum over the activation planes of every plane-row ----
            __syncthreads();                        // (the coefficients)
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&sh.done), phase))) ok = false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int r = (warp & 3) * 32 + lane;
#pragma unroll 1
            for (int tile = 0; tile < a.tiles && ok; ++tile) {
                const int in_tile = all_rows - tile * rows_per_tile < rows_per_tile ? all_rows - tile * rows_per_tile : rows_per_tile;
                if ((warp & 3) * 32 >= in_tile) break;          // (uniform over the warp)
                const uint32_t acc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(tile * a.N);
#pragma unroll 1
                for (int g = (warp >> 2) * 8; g < nv; g += RS_WARPS / 4 * 8) {
                    int d[KA][8];
                    float beta[8 * KA];
#pragma unroll
                    for (int q = 0; q < KA; ++q) tmem_ld8(acc + (uint32_t)(g * KA + 8 * q), d[q]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int q = 0; q < KA; ++q)
                        asm volatile("" : "+r"(d[q][0]), "+r"(d[q][1]), "+r"(d[q][2]), "+r"(d[q][3]), "+r"(d[q][4]), "+r"(d[q][5]),
                                          "+r"(d[q][6]), "+r"(d[q][7]));
#pragma unroll
                    for (int q = 0; q < 2 * KA; ++q) {
                        const float4 v = *reinterpret_cast<const float4*>(sh.beta + g * KA + 4 * q);
                        beta[4 * q] = v.x; beta[4 * q + 1] = v.y; beta[4 * q + 2] = v.z; beta[4 * q + 3] = v.w;
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float s = beta[e * KA] * __int_as_float(d[e * KA / 8][e * KA % 8]);
#pragma unroll
                        for (int j = 1; j < KA; ++j)
                            s = fmaf(beta[e * KA + j], __int_as_float(d[(e * KA + j) / 8][(e * KA + j) % 8]), s);
                        if (g + e < nv && r < in_tile) sS[(g + e) * LD + tile * rows_per_tile + r] = s;
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();

            // ---- 4. sum over the weight planes, gates ----
            int v = v_0, ul = ul_0;
#pragma unroll 1
            for (; v < nv && ok; v += d_v, ul += d_ul) {
                if (ul >= units) {
                    ul -= units;
                    if (++v >= nv) break;
                }
                const size_t o = (size_t)(b0 + v0 + v) * H + u0 + ul;
                const float* add = a.addend ? a.addend + ((size_t)t * a.batch + b0 + v0 + v) * 4 * H + u0 + ul : nullptr;
                const float* ss = sS + v * LD + ul * 4 * k_w;
                const float* al = sAlpha + ul * 4 * k_w;
                float* state = sState + (v0 + v) * a.upc + ul;
                float g4[4];
                if (k_w == 1) rs_unit_sums<1>(ss, al, g4);
                else if (k_w == 2) rs_unit_sums<2>(ss, al, g4);
                else if (k_w == 3) rs_unit_sums<3>(ss, al, g4);
                else rs_unit_sums<4>(ss, al, g4);
                const float4 bias = *reinterpret_cast<const float4*>(sBias + 4 * ul);
                g4[0] += bias.x; g4[1] += bias.y; g4[2] += bias.z; g4[3] += bias.w;
                if (add) {
#pragma unroll
                    for (int g = 0; g < 4; ++g) g4[g] += v == v_0 ? ahead[g] : __ldcg(add + (size_t)g * H);
                }
                float h;
                if (!a.gru) {
                    const float ig = seq_logistic(g4[0]), fg = seq_logistic(g4[1]), og = seq_logistic(g4[2]);
                    const float c = fg * *state + ig * tanhf(g4[3]);
                    *state = c;
                    if (last) a.c_last[o] = c;
                    h = og * tanhf(c);
                } else {
                    const float rg = seq_logistic(g4[0]), zg = seq_logistic(g4[1]), cand = tanhf(g4[2] + rg * g4[3]);
                    h = (1.0f - zg) * cand + zg * *state;
                    *state = h;
                }
                if (last) a.h_last[o] = h;
                else if (WORDS) rs_store_word(a.hx + o, h, (uint32_t)t + 1);
                else if (!h_seq) a.h[t & 1][o] = h;
                if (h_seq) h_seq[o] = h;
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        if (__syncthreads_or(!ok)) { ok = false; break; }
        if (tid == 0 && (t == 0 || !WORDS)) seq_publish(counter + 32);
    }

    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (!ok) {      // (uniform) give the tensor core time to drain before tensor memory is released
        if (tid == 0) atomicExch(a.status, 1u);
        __nanosleep(1000000);
        __syncthreads();
    }
    if (warp == RS_MMA_WARP)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(sh.tmem_slot), "r"((uint32_t)RS_TMEM_COLS) : "memory");
}

struct RsPlan { RsParams a; int grid, warps; bool words; size_t smem; double clocks; };

// Estimated clocks of a timestep: quantizer rounds (by activation bits and warps per vector), per pass over the weights the tensor pipe, the
// expansion of the activations, the folding and the gates, and the waits.  Fitted, with h in memory behind a counter, to 383 problems (LSTM and GRU, 1 to 4 bits, 2 to
// 5000 sequences, widths 64 to 2048) on a B200, within 6 % (standard deviation; 17 % at worst).
double resident_clocks(int k_a, int warps, int block, int P, int TB, int N, int NS, int tiles, int upc)
{
    const int teams = RS_WARPS / warps, vectors = (block + P - 1) / P, passes = (block + TB - 1) / TB, rows = TB * k_a;
    const double quantizer = (k_a <= 2 ? 3700.0 : k_a == 3 ? 5900.0 : 10400.0) + (warps == 4 ? 0.0 : warps == 8 ? 900.0 : 2100.0);
    const double mma = 2.0 * NS * tiles * (N > 92 ? N : 92);
    return 5000.0 + (vectors + teams - 1) / teams * quantizer +
           passes * (2000.0 + 1.3 * mma + 1.2 * rows * NS + 16.5 * tiles * rows + 880.0 * ((TB * upc + RS_THREADS - 1) / RS_THREADS));
}

// Block of vectors x vectors per pass with the least estimated time per timestep; false when the weights do not fit tensor memory.  `only`:
// that many blocks (0: the best).
bool plan(const BatchedSequence& s, int sms, int only, RsPlan* out)
{
    if (s.batch < 2 || s.H < 1 || s.n > 4096 || (s.gru && s.I < 1)) return false;
    const int NS = (s.n + 255) / 256, upt = 32 / s.k_w, NW = s.n <= 1024 ? 4 : s.n <= 2048 ? 8 : 16;
    double best = 0.0;
    RsPlan p{};
    for (int blocks = only ? only : 1; blocks <= s.batch && blocks <= sms && !(only && blocks > only); ++blocks) {
        const int block = (s.batch + blocks - 1) / blocks;
        if ((block < 8 && blocks > 1) || (s.batch + block - 1) / block != blocks) continue;
        int P = sms / blocks;
        const int upc = (s.H + P - 1) / P, tiles = (upc + upt - 1) / upt, all_rows = upc * 4 * s.k_w;
        P = (s.H + upc - 1) / upc;
        for (int passes = 1; passes <= 64 && passes <= block; ++passes) {
            const int TB = (block + passes - 1) / passes, N = (TB * s.k_a + 15) / 16 * 16;
            if (N > 256 || tiles * (32 * NS + N) + RS_SF_COLS > RS_TMEM_COLS || TB * s.k_a * NS > RS_CHUNKS * RS_FEEDERS) continue;
            size_t b = (size_t)NS * N * 128;
            const size_t folded = (size_t)TB * rs_folded_stride(all_rows) * 4, scratch = RS_WARPS / NW * sizeof(QuantScratch<4, 16>);
            if (folded > b) b = folded;
            if (scratch > b) b = scratch;
            b = round_up(b, 1024);
            const size_t smem = b + sizeof(RsShared) + ((size_t)all_rows + 4 * upc + (size_t)block * upc) * 4;
            if (smem > (size_t)RS_SMEM_LIMIT) continue;
            // The splits are ranked by the parts that tell them apart: the quantizer's rounds; per pass the slower of expansion and tensor
            // pipe, the folding, the gates.  (Ranked by resident_clocks 18 of 383 problems get another split: the same time on
            // average, 5 % slower to 5 % faster.)
            const int teams = RS_WARPS / NW, vectors = (block + P - 1) / P;
            const double expand = 2.2 * TB * s.k_a * NS, mma = 4.0 * NS * tiles * (N > 92 ? 0.5 * N : 46.0);
            const double fold = 5.0 * tiles * TB * s.k_a, gates = 500.0 * ((TB * upc + RS_THREADS - 1) / RS_THREADS);
            const double t = (vectors + teams - 1) / teams * (s.k_a >= 3 ? 4500.0 : 3500.0) + passes * ((expand > mma ? expand : mma) + fold + gates + 1500.0);
            if (best == 0.0 || t < best) {
                best = t;
                p.clocks = resident_clocks(s.k_a, NW, block, P, TB, N, NS, tiles, upc);
                p.a.P = P; p.a.block = block; p.a.upc = upc; p.a.upt = upt; p.a.tiles = tiles; p.a.TB = TB; p.a.N = N; p.a.NS = NS;
                p.a.b_bytes = (int)b; p.grid = blocks * P; p.warps = NW;
                p.smem = smem > (size_t)RS_SMEM_MIN ? smem : (size_t)RS_SMEM_MIN;
            }
            break;                                  // (more passes of fewer vectors never pay)
        }
    }
    if (best == 0.0) return false;
    RsParams& a = p.a;
    a.W = s.Wcodes; a.Walpha = s.Walpha; a.bias = s.bias;
    a.z = SeqVectors{s.n, words_per_row(s.n), s.H, s.n - s.H, s.T, s.zcodes, s.zbeta, 16, (size_t)s.batch * s.k_a * 16};
    a.I = s.I; a.k_w = s.k_w; a.gru = s.gru; a.steps = s.steps; a.batch = s.batch;
    a.x_seq = s.x_seq; a.h0 = s.h0; a.c0 = s.c0; a.h_seq = s.h_seq; a.h_last = s.h_last; a.c_last = s.c_last;
    // Words where a team of warps quantizes one vector a timestep: the time from a CTA's h to the planes made of it is what counts there.  Where it
    // takes several in turn, twice the bytes and a look at every word count more; a single timestep has no words to look at.  Eight timesteps,
    // words against none: 58 problems of one vector a team 0.94 to 1.01 of the time (LSTM 512/1024, 21 sequences, 3/3 bits 94 us against 97), 51 of
    // 2 to 35 vectors 1.00 to 1.17 (GRU 128/128, 3530 sequences, 2/2 bits 217 us against 187; LSTM 1919/185, 1297 sequences, 2/3 bits 527 against 485).
    const int teams = RS_WARPS / p.warps, vectors = (a.block + a.P - 1) / a.P;
    p.words = s.steps > 1 && vectors <= teams;
    if (s.late == 3 && !p.words) return false;
    a.hx = reinterpret_cast<unsigned long long*>(s.h[0]);       // (the two states, one behind the other)
    a.h[0] = s.h[0]; a.h[1] = s.h[1];
    a.launched = s.launched; a.tag_bias = s.late == 3 ? 1u << 30 : 0u;
    a.addend = s.addend; a.counters = s.counters; a.counted = s.counted; a.status = s.status;
    a.planes_word = s.late == 1 ? 1 : 0; a.h_word = s.late == 2 ? 33 : 32;
    *out = p;
    return true;
}

template <int KA, int NW>
amq_status launch(const RsPlan& pl, cudaStream_t st)
{
    auto kernel = pl.words ? rnn_resident_kernel<KA, NW, true> : rnn_resident_kernel<KA, NW, false>;
    AMQ_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem));
    RsParams args = pl.a;
    void* params[] = {&args};
    AMQ_CUDA_TRY(cudaLaunchCooperativeKernel((void*)kernel, dim3((unsigned)pl.grid), dim3(RS_THREADS), params, pl.smem, st));
    __atomic_fetch_add(&g_kernel_launches, 1ull, __ATOMIC_RELAXED);
    return AMQ_OK;
}

template <int KA>
amq_status launch_warps(const RsPlan& pl, cudaStream_t st)
{
    return pl.warps == 4 ? launch<KA, 4>(pl, st) : pl.warps == 8 ? launch<KA, 8>(pl, st) : launch<KA, 16>(pl, st);
}

}  // namespace

bool resident_sequence_shape(const BatchedSequence& s, int sms, SequenceShape* out)
{
    RsPlan pl;
    int dev = 0;
    if (sms < 1 && (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)) return false;
    if (!plan(s, sms, 0, &pl)) return false;
    *out = SequenceShape{sms, pl.grid / pl.a.P, pl.a.block, pl.a.P, pl.warps, pl.clocks};
    return true;
}

amq_status launch_resident_sequence(const BatchedSequence& s, const SequenceShape& shape, cudaStream_t st)
{
    RsPlan pl;
    if (!plan(s, shape.sms, shape.blocks, &pl)) return AMQ_ERR_UNSUPPORTED;
    switch (s.k_a) {
        case 1: return launch_warps<1>(pl, st);
        case 2: return launch_warps<2>(pl, st);
        case 3: return launch_warps<3>(pl, st);
        case 4: return launch_warps<4>(pl, st);
    }
    return AMQ_ERR_UNSUPPORTED;
}

}  // namespace amq
