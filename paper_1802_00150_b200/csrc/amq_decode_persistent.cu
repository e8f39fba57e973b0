// Greedy decoding of one sequence (Eq. 6, the arg-max token fed back) as ONE cooperative launch for all tokens.
//
// Every CTA (one per SM) owns a few hidden units and a share of the vocabulary; their packed rows stay in shared memory for the whole
// call (vocabulary 42000 x 1024 at 2 bits: 73 KB of output rows and 14 KB of gate rows per SM; output rows that do not fit are
// read from L2 every token).  A token is, in every CTA:
//   the token's embedding row (already quantized) -> W_i x + b for the own units -> gates with the recurrent part kept from before ->
//   publish the own h values; gather all of h, quantize it (every CTA for itself: one exchange instead of a second round);
//   the own rows of the output layer -> the share's maximum -> publish; W_h h_hat of the own units for the next token, which hides the
//   flight of the maxima; gather the maxima -> the next token.
// Both exchanges are tagged words that are polled until the tag of this token arrives (see amq_rnn_persistent.cu): value and "ready"
// travel together.  Every wait is bounded; when one runs out the CTA sets the device status word and leaves.
//
// The arithmetic is that of the kernel-per-step chain (integer dot products, coefficients in the same order, the same gates and the
// same quantizer over the same ownership), so both give the same bits.  The chain took six launches and 21 us per token, most of
// it launch gaps and the start-up of short kernels; what is left is two exchanges among all SMs and the quantizer's reductions.
#include "amq_common.cuh"
#include "amq_quantize_device.cuh"

namespace amq {

namespace {

constexpr int DEC_THREADS = 256, DEC_WARPS = DEC_THREADS / 32, DEC_EPT = 8;
constexpr unsigned DEC_POLL_LIMIT = 1u << 20;
constexpr int DEC_COPIES = PERSISTENT_EXCHANGE_COPIES;      // copies of both exchange areas

struct DecodeArgs {
    const uint4* We; const float* We_alpha; int vocab, I, k_e;
    const uint4* Wi; const float* Wi_alpha; const uint4* Wh; const float* Wh_alpha; const float* bias; int H, k_w;
    const uint4* Ws; const float* Ws_alpha; const float* bias_s;
    int T, steps;
    int32_t* tokens; float* h; float* c;
    unsigned long long* hx; size_t hx_stride;       // [2][copies][stride]: {h value, tag}
    ulonglong2* best;                               // [2][copies][grid]: {logit, tag}, {index, tag}
    const unsigned long long* hx_polled;            // where the CTAs look for them: hx and best (the self-test of the waits: half an area
    const ulonglong2* best_polled;                  // further, where step 0 writes nothing)
    uint32_t* status;
    int CHI, CHH;                                   // 128-bit chunks of a plane of x, of h
    int upc, rpc, resident;                         // hidden units, vocabulary rows per CTA, how many of those rows stay in shared memory
};

__device__ __forceinline__ unsigned long long dec_load(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ ulonglong2 dec_load2(const ulonglong2* p)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void dec_store(unsigned long long* p, uint32_t value, uint32_t tag)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" :: "l"(p), "l"(((unsigned long long)tag << 32) | value) : "memory");
}

__device__ __forceinline__ int dec_popc(const uint4& a, const uint4& b)
{
    return __popc(a.x ^ b.x) + __popc(a.y ^ b.y) + __popc(a.z ^ b.z) + __popc(a.w ^ b.w);
}

// (value, index) maximum; among equal values the smaller index wins
__device__ __forceinline__ void dec_max(float& v, int& i, float ov, int oi)
{
    if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
}
__device__ __forceinline__ void dec_warp_max(float& v, int& i)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        dec_max(v, i, __shfl_xor_sync(0xffffffffu, v, off), __shfl_xor_sync(0xffffffffu, i, off));
}

// One hidden unit's four gate rows times the planes `x`: lane = (row, chunk within a segment of SEG lanes), then lane g < 4 gets gate g:
// sum over planes of alpha_i beta_j D_ij in that order.  Whole warp.
__device__ __forceinline__ float dec_unit(const uint4* rows, const float* alpha, int k_w, const uint4* x, const float* beta, int k_x, int CH, int n)
{
    const int lane = threadIdx.x & 31, R = 4 * k_w, SEG = R <= 4 ? 8 : R <= 8 ? 4 : 2;
    const int row = lane / SEG, chunk = lane - row * SEG;
    int acc[AMQ_MAX_K];
#pragma unroll
    for (int j = 0; j < AMQ_MAX_K; ++j) acc[j] = 0;
    if (row < R) {
        const uint4* w = rows + (size_t)row * CH;
        for (int c = chunk; c < CH; c += SEG) {
            const uint4 v = w[c];
#pragma unroll
            for (int j = 0; j < AMQ_MAX_K; ++j)
                if (j < k_x) acc[j] += dec_popc(v, x[j * CH + c]);
        }
    }
    for (int off = SEG >> 1; off > 0; off >>= 1) {
#pragma unroll
        for (int j = 0; j < AMQ_MAX_K; ++j) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], off);
    }
    float y = 0.0f;
    const int gate = lane & 3;
    for (int i = 0; i < k_w; ++i) {
        const float al = alpha[gate * k_w + i];
#pragma unroll
        for (int j = 0; j < AMQ_MAX_K; ++j) {
            const int d = __shfl_sync(0xffffffffu, acc[j], (gate * k_w + i) * SEG);
            if (j < k_x) y += al * beta[j] * (float)(n - 2 * d);
        }
    }
    return y;
}

template <int KS, int KA>
__global__ void __launch_bounds__(DEC_THREADS, 1)
decode_persistent_kernel(const __grid_constant__ DecodeArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int CHI = a.CHI, CHH = a.CHH, H = a.H, k_w = a.k_w, k_e = a.k_e, R = 4 * k_w;
    const int u0 = (int)blockIdx.x * a.upc, units = u0 < H ? (H - u0 < a.upc ? H - u0 : a.upc) : 0;
    const int r0 = (int)blockIdx.x * a.rpc, rows = r0 < a.vocab ? (a.vocab - r0 < a.rpc ? a.vocab - r0 : a.rpc) : 0;

    uint4* sWi = reinterpret_cast<uint4*>(smem_raw);                // [upc][4 k_w][CHI]
    uint4* sWh = sWi + (size_t)a.upc * R * CHI;                     // [upc][4 k_w][CHH]
    uint4* sX = sWh + (size_t)a.upc * R * CHH;                      // [k_e][CHI]
    uint4* sH = sX + AMQ_MAX_K * CHI;                               // [KA][CHH]
    uint4* sWs = sH + AMQ_MAX_K * CHH;                              // [resident][KS][CHH]
    float* sWsA = reinterpret_cast<float*>(sWs + (size_t)a.resident * KS * CHH);    // [rpc][KS]
    float* sBs = sWsA + (size_t)a.rpc * KS;                         // [rpc]
    float* sIA = sBs + a.rpc;                                       // [upc][4 k_w]
    float* sHA = sIA + a.upc * R;                                   // [upc][4 k_w]
    float* sBias = sHA + a.upc * R;                                 // [upc][4]
    float* sPre = sBias + 4 * a.upc;                                // [upc][4]  W_h h_hat of the next token
    float* sC = sPre + 4 * a.upc;                                   // [upc]
    float* sHn = sC + a.upc;                                        // [upc]
    float* sXb = sHn + a.upc;                                       // [4]
    float* sHb = sXb + 4;                                           // [4]
    float* sMaxV = sHb + 4;                                         // [DEC_WARPS]
    int* sMaxI = reinterpret_cast<int*>(sMaxV + DEC_WARPS);         // [DEC_WARPS]
    QuantScratch<KA, DEC_WARPS>* scratch = reinterpret_cast<QuantScratch<KA, DEC_WARPS>*>(
        (reinterpret_cast<uintptr_t>(sMaxI + DEC_WARPS) + 15) & ~uintptr_t(15));

    // ---- resident rows and coefficients: plane-row (unit, gate, i) of W_i, W_h; the first `resident` rows of the output share ----
    for (int q = tid; q < units * R * CHI; q += DEC_THREADS) {
        const int pr = q / CHI, ul = pr / R, gi = pr - ul * R, gate = gi / k_w, i = gi - gate * k_w;
        sWi[q] = __ldg(a.Wi + (((size_t)gate * H + u0 + ul) * k_w + i) * CHI + (q - pr * CHI));
    }
    for (int q = tid; q < units * R * CHH; q += DEC_THREADS) {
        const int pr = q / CHH, ul = pr / R, gi = pr - ul * R, gate = gi / k_w, i = gi - gate * k_w;
        sWh[q] = __ldg(a.Wh + (((size_t)gate * H + u0 + ul) * k_w + i) * CHH + (q - pr * CHH));
    }
    for (int q = tid; q < units * R; q += DEC_THREADS) {
        const int ul = q / R, gi = q - ul * R, gate = gi / k_w, i = gi - gate * k_w;
        sIA[q] = __ldg(a.Wi_alpha + ((size_t)gate * H + u0 + ul) * k_w + i);
        sHA[q] = __ldg(a.Wh_alpha + ((size_t)gate * H + u0 + ul) * k_w + i);
    }
    for (int q = tid; q < 4 * units; q += DEC_THREADS) sBias[q] = a.bias ? __ldg(a.bias + (size_t)(q & 3) * H + u0 + (q >> 2)) : 0.0f;
    for (int q = tid; q < units; q += DEC_THREADS) { sC[q] = a.c[u0 + q]; sHn[q] = a.h[u0 + q]; }
    const int res_rows = rows < a.resident ? rows : a.resident;
    for (int q = tid; q < res_rows * KS * CHH; q += DEC_THREADS) sWs[q] = __ldg(a.Ws + (size_t)r0 * KS * CHH + q);
    for (int q = tid; q < rows * KS; q += DEC_THREADS) sWsA[q] = __ldg(a.Ws_alpha + (size_t)r0 * KS + q);
    for (int q = tid; q < rows; q += DEC_THREADS) sBs[q] = a.bias_s ? __ldg(a.bias_s + r0 + q) : 0.0f;
    for (int q = tid; q < KA * CHH * 4; q += DEC_THREADS) reinterpret_cast<uint32_t*>(sH)[q] = 0u;      // plane words no thread owns
    quant_scratch_init(*scratch);
    __syncthreads();

    const int e0 = tid * DEC_EPT, my_copy = (int)(blockIdx.x % (unsigned)DEC_COPIES);
    uint32_t valid = 0;
#pragma unroll
    for (int j = 0; j < DEC_EPT; ++j) valid |= (e0 + j < H ? 1u : 0u) << j;
    // output rows: SEG lanes per row, one 128-bit chunk of every plane per lane
    const int SEG = CHH <= 2 ? 2 : CHH <= 4 ? 4 : CHH <= 8 ? 8 : 16, sub = lane & (SEG - 1), per_warp = 32 / SEG;
    const bool has = sub < CHH;
    int parity = 0, gave_up = 0;
    int token = __ldcg(a.tokens);

    for (int t = -1; t < a.steps; ++t) {
        // ---- 1. the new state of the own units (t = -1: the start state only gets quantized) ----
        if (t >= 0) {
            token = token < 0 ? 0 : (token >= a.vocab ? a.vocab - 1 : token);      // out-of-range ids are clamped, never dereferenced
            for (int q = tid; q < k_e * CHI; q += DEC_THREADS) sX[q] = __ldg(a.We + (size_t)token * k_e * CHI + q);
            if (tid < k_e) sXb[tid] = __ldg(a.We_alpha + (size_t)token * k_e + tid);
            __syncthreads();
            for (int ul = warp; ul < units; ul += DEC_WARPS) {
                const int gate = lane & 3;
                const float proj = dec_unit(sWi + (size_t)ul * R * CHI, sIA + ul * R, k_w, sX, sXb, k_e, CHI, a.I) + sBias[4 * ul + gate];
                const float g = sPre[4 * ul + gate] + proj;
                float g4[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) g4[q] = __shfl_sync(0xffffffffu, g, q);
                const float ig = 1.0f / (1.0f + __expf(-g4[0])), fg = 1.0f / (1.0f + __expf(-g4[1])), og = 1.0f / (1.0f + __expf(-g4[2]));
                const float c = fg * sC[ul] + ig * tanhf(g4[3]);
                const float h = og * tanhf(c);
                if (lane < DEC_COPIES)
                    dec_store(a.hx + ((size_t)(t & 1) * DEC_COPIES + lane) * a.hx_stride + u0 + ul, __float_as_uint(h), (uint32_t)(t + 1));
                __syncwarp();
                if (lane == 0) { sC[ul] = c; sHn[ul] = h; }
            }
        }

        // ---- 2. all of h, quantized; its planes for the output layer and for the recurrent product of the next token ----
        float w[DEC_EPT];
        uint32_t pending = t >= 0 ? valid : 0u;
#pragma unroll
        for (int j = 0; j < DEC_EPT; ++j) w[j] = (t < 0 && (valid >> j) & 1u) ? __ldcg(a.h + e0 + j) : 0.0f;
        const unsigned long long* hx = a.hx_polled + ((size_t)(t & 1) * DEC_COPIES + my_copy) * a.hx_stride;
        for (unsigned spins = 0; pending && spins < DEC_POLL_LIMIT; ++spins) {
            unsigned long long v[DEC_EPT];
#pragma unroll
            for (int j = 0; j < DEC_EPT; ++j) v[j] = (pending >> j) & 1u ? dec_load(hx + e0 + j) : 0ull;
#pragma unroll
            for (int j = 0; j < DEC_EPT; ++j)
                if (((pending >> j) & 1u) && (uint32_t)(v[j] >> 32) == (uint32_t)(t + 1)) {
                    w[j] = __uint_as_float((uint32_t)v[j]);
                    pending &= ~(1u << j);
                }
        }
        gave_up |= pending != 0;
        float beta[KA];
        uint32_t bits[KA];
        quantize_group<KA, DEC_EPT, DEC_WARPS>(w, valid, H, quant_padding_consecutive(H, DEC_EPT), a.T, beta, bits, *scratch, &gave_up, &parity);
        if (gave_up) break;                         // (uniform: the quantizer's first barrier has taken the vote)
        if (e0 < CHH * 128) {
#pragma unroll
            for (int j = 0; j < KA; ++j) reinterpret_cast<uint8_t*>(sH + j * CHH)[tid] = (uint8_t)bits[j];
        }
        if (tid == 0) {
#pragma unroll
            for (int j = 0; j < KA; ++j) sHb[j] = beta[j];
        }
        __syncthreads();

        // ---- 3. the own rows of the output layer, their maximum ----
        if (t >= 0) {
            uint4 xr[KA];
#pragma unroll
            for (int j = 0; j < KA; ++j) xr[j] = has ? sH[j * CHH + sub] : make_uint4(0, 0, 0, 0);
            float mv = -INFINITY;
            int mi = 0x7fffffff;
            auto load = [&](int r, uint4 (&v)[KS]) {        // (two loads, not one through a pointer to either: that would be a generic load)
                const size_t at = (size_t)r * KS * CHH + sub;
#pragma unroll
                for (int i = 0; i < KS; ++i) v[i] = make_uint4(0, 0, 0, 0);
                if (has && r < res_rows) {
#pragma unroll
                    for (int i = 0; i < KS; ++i) v[i] = sWs[at + i * CHH];
                } else if (has && r < rows) {
#pragma unroll
                    for (int i = 0; i < KS; ++i) v[i] = __ldg(a.Ws + (size_t)r0 * KS * CHH + at + i * CHH);
                }
            };
            // Two rows per lane segment at a time, so that one's shuffles run beside the other's bit counts (284 rows of two planes per SM:
            // 7200 clocks of a token before, 6600 now; the bit counts alone need 2300).
            constexpr int PAIRS = (KS * KA + 1) / 2;
            const int stride = DEC_WARPS * per_warp;
            for (int r = warp * per_warp + lane / SEG; r - lane / SEG < rows; r += 2 * stride) {
                uint4 v[2][KS];
                load(r, v[0]);
                load(r + stride, v[1]);
                // counts of differing bits: at most 2048, two to a register
                uint32_t d[2][PAIRS];
#pragma unroll
                for (int p = 0; p < 2; ++p)
#pragma unroll
                    for (int q = 0; q < PAIRS; ++q) {
                        d[p][q] = (uint32_t)dec_popc(v[p][(2 * q) / KA], xr[(2 * q) % KA]);
                        if (2 * q + 1 < KS * KA) d[p][q] |= (uint32_t)dec_popc(v[p][(2 * q + 1) / KA % KS], xr[(2 * q + 1) % KA]) << 16;
                    }
                for (int off = SEG >> 1; off > 0; off >>= 1) {
#pragma unroll
                    for (int p = 0; p < 2; ++p)
#pragma unroll
                        for (int q = 0; q < PAIRS; ++q) d[p][q] += __shfl_xor_sync(0xffffffffu, d[p][q], off);
                }
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int row = r + p * stride;
                    if (row < rows) {
                        float y = 0.0f;
#pragma unroll
                        for (int i = 0; i < KS; ++i) {
                            const float al = sWsA[row * KS + i];
#pragma unroll
                            for (int j = 0; j < KA; ++j) {
                                const int q = i * KA + j, n = (int)((d[p][q >> 1] >> (16 * (q & 1))) & 0xffffu);
                                y += al * beta[j] * (float)(H - 2 * n);
                            }
                        }
                        dec_max(mv, mi, y + sBs[row], r0 + row);
                    }
                }
            }
            dec_warp_max(mv, mi);
            if (lane == 0) { sMaxV[warp] = mv; sMaxI[warp] = mi; }
            __syncthreads();
            if (warp == 0) {
                mv = lane < DEC_WARPS ? sMaxV[lane] : -INFINITY;
                mi = lane < DEC_WARPS ? sMaxI[lane] : 0x7fffffff;
                dec_warp_max(mv, mi);
                if (lane < DEC_COPIES) {
                    unsigned long long* out = reinterpret_cast<unsigned long long*>(a.best + ((size_t)(t & 1) * DEC_COPIES + lane) * gridDim.x + blockIdx.x);
                    dec_store(out, __float_as_uint(mv), (uint32_t)(t + 1));
                    dec_store(out + 1, (uint32_t)mi, (uint32_t)(t + 1));
                }
            }
        }

        // ---- 4. W_h h_hat of the own units for the next token (beside the flight of the maxima) ----
        for (int ul = warp; ul < units; ul += DEC_WARPS) {
            const float y = dec_unit(sWh + (size_t)ul * R * CHH, sHA + ul * R, k_w, sH, sHb, KA, CHH, H);
            if (lane < 4) sPre[4 * ul + lane] = y;
        }

        // ---- 5. the next token ----
        if (t >= 0) {
            float mv = -INFINITY;
            int mi = 0x7fffffff;
            for (int q = tid; q < (int)gridDim.x; q += DEC_THREADS) {
                const ulonglong2* in = a.best_polled + ((size_t)(t & 1) * DEC_COPIES + my_copy) * gridDim.x + q;
                ulonglong2 v = make_ulonglong2(0, 0);
                bool there = false;                 // (each half is validated by its own tag)
                for (unsigned spins = 0; !there && spins < DEC_POLL_LIMIT; ++spins) {
                    v = dec_load2(in);
                    there = (uint32_t)(v.x >> 32) == (uint32_t)(t + 1) && (uint32_t)(v.y >> 32) == (uint32_t)(t + 1);
                }
                gave_up |= !there;
                dec_max(mv, mi, __uint_as_float((uint32_t)v.x), (int)(uint32_t)v.y);
            }
            dec_warp_max(mv, mi);
            __syncthreads();                        // (the first use of the slots has been read)
            if (lane == 0) { sMaxV[warp] = mv; sMaxI[warp] = mi; }
            if (__syncthreads_or(gave_up)) { gave_up = 1; break; }
            mv = sMaxV[lane & (DEC_WARPS - 1)]; mi = sMaxI[lane & (DEC_WARPS - 1)];
            dec_warp_max(mv, mi);
            token = mi;
            if (blockIdx.x == 0 && tid == 0) a.tokens[t + 1] = mi;
        }
    }
    if (gave_up) {
        if (tid == 0) atomicExch(a.status, 1u);
        return;
    }
    for (int q = tid; q < units; q += DEC_THREADS) { a.h[u0 + q] = sHn[q]; a.c[u0 + q] = sC[q]; }
}

struct DecodePlan { int grid, upc, rpc, resident; size_t smem; };

// Split of the units and the vocabulary over one CTA per SM; false when the fixed part does not fit a CTA's shared memory.
bool decode_plan(const DecodeSequence& d, DecodePlan* out)
{
    if (d.H > DEC_THREADS * DEC_EPT) return false;          // one byte of every plane per thread
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
    DecodePlan p;
    p.grid = sms < DECODE_MAX_CTAS ? sms : DECODE_MAX_CTAS;
    p.upc = (d.H + p.grid - 1) / p.grid;
    p.rpc = (d.vocab + p.grid - 1) / p.grid;
    const size_t CHI = words_per_row(d.I) / 4, CHH = words_per_row(d.H) / 4, R = 4 * (size_t)d.k_w;
    const size_t fixed = (p.upc * R + AMQ_MAX_K) * (CHI + CHH) * 16 + (size_t)p.rpc * (d.k_s + 1) * 4 + p.upc * (2 * R + 10) * 4 +
                         8 * 4 + DEC_WARPS * 8 + 16 + sizeof(QuantScratch<AMQ_MAX_K, DEC_WARPS>);
    const size_t limit = 200 * 1024, row = d.k_s * CHH * 16;
    if (fixed > limit) return false;
    const size_t fit = (limit - fixed) / row;
    p.resident = fit < (size_t)p.rpc ? (int)fit : p.rpc;
    p.smem = fixed + p.resident * row;
    *out = p;
    return true;
}

template <int KS, int KA>
amq_status decode_launch(const DecodeArgs& a, const DecodePlan& p, cudaStream_t st)
{
    auto kernel = decode_persistent_kernel<KS, KA>;
    AMQ_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem));
    DecodeArgs args = a;
    void* params[] = {&args};
    AMQ_CUDA_TRY(cudaLaunchCooperativeKernel((void*)kernel, dim3((unsigned)p.grid), dim3(DEC_THREADS), params, p.smem, st));
    __atomic_fetch_add(&g_kernel_launches, 1ull, __ATOMIC_RELAXED);
    return AMQ_OK;
}

template <int KS>
amq_status decode_launch_ka(const DecodeArgs& a, int k_a, const DecodePlan& p, cudaStream_t st)
{
    switch (k_a) {
        case 1: return decode_launch<KS, 1>(a, p, st);
        case 2: return decode_launch<KS, 2>(a, p, st);
        case 3: return decode_launch<KS, 3>(a, p, st);
        case 4: return decode_launch<KS, 4>(a, p, st);
    }
    return AMQ_ERR_UNSUPPORTED;
}

}  // namespace

bool decode_persistent_supported(const DecodeSequence& d)
{
    DecodePlan p;
    return decode_plan(d, &p);
}

amq_status launch_decode_persistent(const DecodeSequence& d, cudaStream_t st)
{
    DecodePlan p;
    if (!decode_plan(d, &p)) return AMQ_ERR_UNSUPPORTED;
    uint32_t* status = nullptr;
    const amq_status s = tc_status_word(&status);
    if (s != AMQ_OK) return s;
    DecodeArgs a{};
    a.We = reinterpret_cast<const uint4*>(d.We); a.We_alpha = d.We_alpha; a.vocab = d.vocab; a.I = d.I; a.k_e = d.k_e;
    a.Wi = reinterpret_cast<const uint4*>(d.Wi); a.Wi_alpha = d.Wi_alpha;
    a.Wh = reinterpret_cast<const uint4*>(d.Wh); a.Wh_alpha = d.Wh_alpha;
    a.bias = d.bias; a.H = d.H; a.k_w = d.k_w;
    a.Ws = reinterpret_cast<const uint4*>(d.Ws); a.Ws_alpha = d.Ws_alpha; a.bias_s = d.bias_s;
    a.T = d.T; a.steps = d.steps; a.tokens = d.tokens; a.h = d.h; a.c = d.c;
    a.hx = d.exchange; a.hx_stride = persistent_exchange_stride(d.H);
    a.best = reinterpret_cast<ulonglong2*>(d.exchange + 2 * DEC_COPIES * a.hx_stride);
    a.hx_polled = a.hx + (d.late == 1 ? DEC_COPIES * a.hx_stride : 0);
    a.best_polled = a.best + (d.late == 2 ? DEC_COPIES * p.grid : 0);
    a.status = status;
    a.CHI = words_per_row(d.I) / 4; a.CHH = words_per_row(d.H) / 4;
    a.upc = p.upc; a.rpc = p.rpc; a.resident = p.resident;
    // no word of an earlier call may carry a tag of this one
    AMQ_CUDA_TRY(cudaMemsetAsync(d.exchange, 0, decode_exchange_bytes(d.H), st));
    switch (d.k_s) {
        case 1: return decode_launch_ka<1>(a, d.k_a, p, st);
        case 2: return decode_launch_ka<2>(a, d.k_a, p, st);
        case 3: return decode_launch_ka<3>(a, d.k_a, p, st);
        case 4: return decode_launch_ka<4>(a, d.k_a, p, st);
    }
    return AMQ_ERR_UNSUPPORTED;
}

}  // namespace amq
