// Pieces shared by the two kernels that run a batch of sequences in one cooperative launch (amq_rnn_batched.cu, amq_rnn_resident.cu):
// the counters the CTAs of a block of vectors wait on, and the on-line quantization of one vector by a team of warps.
#pragma once

#include "amq_common.cuh"
#include "amq_quantize_device.cuh"

namespace amq {

constexpr unsigned SEQ_POLL_LIMIT = 1u << 21;   // looks at a counter before giving up (a second or so)

// One thread, after a CTA barrier: the release covers what the whole CTA has written before the barrier.
__device__ __forceinline__ void seq_publish(uint32_t* counter)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(counter) : "memory");
}

// What a counter reads once `ctas` CTAs have published `timesteps` times since it was cleared, modulo 2^32: with 148 CTAs a counter wraps
// after 29 million timesteps (and the product leaves the range of int after half of that).
__device__ __forceinline__ uint32_t seq_target(int timesteps, int ctas) { return (uint32_t)timesteps * (uint32_t)ctas; }

// A counter is never more than a timestep's CTAs away from what is waited for, so the sign of the difference tells across a wrap.
__device__ __forceinline__ bool seq_wait(const uint32_t* counter, uint32_t target)
{
    for (unsigned i = 0; i < SEQ_POLL_LIMIT; ++i) {
        uint32_t v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
        if ((int32_t)(v - target) >= 0) return true;
    }
    return false;
}

// The vectors z = [x ; h] of a timestep and where their planes go.
struct SeqVectors {
    int n, wpr, H, xn, T;       // xn: elements that come from x (0: z = h)
    uint32_t* zcodes; float* zbeta;
    size_t row_bytes, half_bytes;       // distance of two plane-rows, of two 16-byte pieces of one
};

// *p where `there`, else 0: a predicated load, so that several of them are in flight (as branches they are taken one after the other: GRU 2048,
// 256 sequences, 2/3 bits, 35 steps streamed 1249 us against 1242).
__device__ __forceinline__ float seq_load_if(const float* p, bool there)
{
    float v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@p ld.global.cg.f32 %0, [%1];\n\t}"
                 : "=f"(v) : "l"(p), "r"((int)there) : "memory");
    return v;
}

// Where h is in memory as it is.
struct SeqNoWords {
    static constexpr void* words = nullptr;
    template <int EPT> __device__ __forceinline__ bool gather(const SeqVectors&, int, int, float (&)[EPT]) const { return true; }
};

// Quantize one vector with a team of warps, thread g of the team owning the elements EPT g .. EPT g + EPT - 1.  Elements of h come from `h`,
// or from `words` (whose gather may fail: false) where there are some.  PREDICATED: elements that are no whole 16-byte pieces by predicated
// loads, otherwise by branches, which threads past the end do not enter (the resident form without words: GRU 128/128, 3530 sequences, 2/2 bits,
// 8 steps 189 us against 193, LSTM 159/259, 1644 sequences 186 against 190, one step of GRU 64/479, two sequences 14.6 against 14.8).
template <int KA, int EPT, int NW, bool PREDICATED = true, typename Words = SeqNoWords>
__device__ __forceinline__ bool seq_quantize(const SeqVectors& a, const float* x, const float* h, int vector,
                                             QuantScratch<KA, NW>& sc, const QuantTeam& team, int& parity, const Words& words = Words{})
{
    const int n = a.n, g = team.warp * 32 + ((int)threadIdx.x & 31), t0 = g * EPT;
    float w[EPT];
    uint32_t valid = 0;
    const float* xr = x + (size_t)vector * a.xn;
    const float* hr = h + (size_t)vector * a.H - a.xn;
    const int end = words.words ? a.xn : n;         // elements read as they are
#pragma unroll
    for (int q = 0; q < EPT / 4; ++q) {
        const int t = t0 + 4 * q;
        const float* p = (t < a.xn ? xr : hr) + t;
        const bool one_piece = t + 3 < end && (t + 3 < a.xn || t >= a.xn) && (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
        if (one_piece) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(p));        // (h: written by other SMs)
            w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
            valid |= 0xFu << (4 * q);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float* from = (t + e < a.xn ? xr : hr) + t + e;
                if (PREDICATED) w[4 * q + e] = seq_load_if(from, t + e < end);
                else w[4 * q + e] = t + e < end ? __ldcg(from) : 0.0f;
                valid |= (t + e < n ? 1u : 0u) << (4 * q + e);
            }
        }
    }
    const bool ok = words.words ? words.gather(a, vector, t0, w) : true;
    float beta[KA];
    uint32_t bits[KA];
    quantize_group<KA, EPT, NW>(w, valid, n, quant_padding_consecutive(n, EPT), a.T, beta, bits, sc, nullptr, &parity, team);
    if (t0 < a.wpr * 32) {
        uint8_t* dst = reinterpret_cast<uint8_t*>(a.zcodes) + (size_t)vector * KA * a.row_bytes + (size_t)(t0 >> 7) * a.half_bytes + ((t0 >> 3) & 15);
#pragma unroll
        for (int i = 0; i < KA; ++i)
            if (EPT == 8) dst[i * a.row_bytes] = (uint8_t)bits[i];
            else *reinterpret_cast<uint16_t*>(dst + i * a.row_bytes) = (uint16_t)bits[i];
    }
    if (g < KA) {
        float b = beta[0];
#pragma unroll
        for (int i = 1; i < KA; ++i) b = (g == i) ? beta[i] : b;
        a.zbeta[(size_t)vector * KA + g] = b;
    }
    return ok;
}

__device__ __forceinline__ float seq_logistic(float v) { return 1.0f / (1.0f + __expf(-v)); }

}  // namespace amq
