// Device-side body of the alternating multi-bit quantizer (Algorithm 2), shared by the row quantizer kernel and by the
// recurrent kernels, which quantize [x ; h] in place.
//
// A "group" of threads owns one vector; every thread holds EPT of its elements in registers (which ones is
// the caller's choice).  Algorithm 1 is evaluated in its data-parallel form (the remark on operating on all
// entries at once, Sec. 3): every element descends the tree over the 2^k - 1 midpoints of the ascending level
// table with k comparisons.  The table is antisymmetric, so a decision is the sign of w minus the midpoint of |w|'s side; decisions are
// gathered as words of bits, and a plane is a logic function of those words (the decision itself when the levels ascend by
// code).  Bulk quantization of 32768 x 1024 at 3 bits: 104 us with a leaf index and a table look-up per element and plane, 78 us
// this way (2.0 TB/s of input and planes; bound by issue slots: the reductions, then the decisions).
//
// Instruction economy of the inner loops (they decide the throughput of bulk quantization): inputs are
// canonicalised (-0.0 -> +0.0), after which "r >= 0" is exactly "sign bit clear" for every residue the
// greedy step can produce, so a sign plane is gathered with one funnel shift per element, a residue is
// updated as r - copysign(alpha, r) with one logic operation and one add, and +-w for the refit sums is one
// logic operation; the refit sums of a cycle are accumulated in the same pass that assigns the codes.
// A warp of its own (bulk quantization) is bound by the integer pipe, 64 lanes a clock, and by issue slots, while the fp32 pipe has 128
// lanes and two-wide instructions: there one logic operation makes s = +-1 of a sign bit, a residue is r - a s, |r| is s r and
// the refit sums add s w, multiply-adds (the products are exact: rounded as the plain sums, which are taken in the same order: the same
// bits as a team's way of writing it), two elements wide where they are no sums, and a word of
// sign bits is the exact sum of s 2^j over sixteen elements.  32768 x 1024 at 3 bits 78 -> 66 us, at 2 bits 58 -> 42.  A team's
// quantizer is a chain of dependent operations, which the multiply-adds make longer: LSTM sequence 1024, one sequence, 154 -> 159 us,
// decoding 674 -> 730; there it stays as it was.
// Elements past the end of the vector are zeros that take part in every loop unmasked: their bits are
// cleared at the end, they add nothing to B^T w, the Gram matrix is counted on masked words, and their known
// contribution to the greedy |r| sums (all of them follow the trajectory of a zero element) is subtracted.
// Threads that hold no element of the vector at all leave their |r| sums out instead, so that what is
// subtracted stays a few elements' worth whatever the size of the group (the subtraction of a large known
// sum from a rounded one would cost accuracy on short vectors).
//
// Arithmetic: sums over the vector are fp32 (per thread, then a fixed butterfly over the warp, then the
// per-warp partials in a fixed tree, so results are reproducible run to run); the Gram matrix B^T B is exact
// integer arithmetic; the k x k solve is fp64 for k >= 3 (k = 3: through the exact integer adjugate) and error-compensated fp32 for k = 2 (the products
// n c_i and g c_j are split exactly with fused multiply-adds, so cancellation costs nothing); levels,
// midpoints and comparisons are fp32.
//
// When the group is a whole CTA, a reduction costs ONE barrier: lane 0 of every warp leaves the warp's
// partial sums in shared memory, and after the barrier every thread adds up all partials itself and
// repeats the per-vector scalar work (solve, sorted level table) redundantly.  In the recurrent kernels the
// quantizer sits on the latency path of each timestep, and a second barrier plus a round trip through
// shared memory for "one warp computes, all read" costs more than the repeated arithmetic.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "amq_pairs.cuh"

namespace amq {

constexpr int QUANT_MAX_WARPS = 16;

// Whether a group sorts its levels through shared memory and descends the table element by element: teams at four bits, where the
// instructions of the in-register sort and of the leaf functions are on the critical path of one vector (LSTM sequence 1024, one
// sequence, 35 steps, 4 bits: 302 us with them, 271 us with the table; at 3 bits 204 against 211 us).  A warp of its own
// (NW = 1) has other rows' warps to hide them behind, and no scratch.
constexpr bool quant_level_table(int K, int NW) { return K == 4 && NW > 1; }

// Shared-memory scratch of one group of NW warps (NW = 1: a single warp, which needs none).
template <int K, int NW>
struct __align__(16) QuantScratch {
    static constexpr int V = 1 + K + K * (K - 1) / 2;
    static constexpr int SLOTS = NW > 1 ? ((NW + 3) / 4) * 4 : 4;
    float red[2][V][SLOTS];             // [reduction parity][value][warp]: per-warp partial sums
    static constexpr bool TABLE = quant_level_table(K, NW);
    float level[TABLE ? NW : 1][TABLE ? 1 << K : 1];        // per-warp scratch of the level sort
    int code[TABLE ? NW : 1][TABLE ? 1 << K : 1];
};

// The threads of a group of several warps: the whole CTA, or some consecutive warps of it with a hardware barrier of their own.
struct QuantTeam {
    int warp, bar, threads;         // this warp's number in the team, barrier, threads of the team
    __device__ __forceinline__ static QuantTeam cta() { return QuantTeam{(int)(threadIdx.x >> 5), 0, (int)blockDim.x}; }
    __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, %1;" :: "r"(bar), "r"(threads) : "memory"); }
    __device__ __forceinline__ int sync_or(int flag) const
    {
        int out;
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.or.pred q, %2, %3, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                     : "=r"(out) : "r"(flag), "r"(bar), "r"(threads) : "memory");
        return out;
    }
};

// To be called once by every thread of a team before its first quantize_group (no barrier needed
// afterwards): partial-sum slots of warps that do not exist are read as zeros by every reduction.
template <int K, int NW>
__device__ __forceinline__ void quant_scratch_init(QuantScratch<K, NW>& sc, const QuantTeam& team = QuantTeam::cta())
{
    constexpr int V = QuantScratch<K, NW>::V, SLOTS = QuantScratch<K, NW>::SLOTS;
    const int warps = team.threads >> 5;
    float* flat = &sc.red[0][0][0];
    for (int idx = team.warp * 32 + (threadIdx.x & 31); idx < 2 * V * SLOTS; idx += team.threads)
        if ((idx % SLOTS) >= warps) flat[idx] = 0.0f;
}

// Sums over the warp of VF floats, every lane gets all of them.  Four values at a time are reduced and scattered over the lanes at
// once (2 + 1 + 3 shuffles instead of 20) and gathered again; the additions pair the same lanes in the same order as a butterfly
// over distances 16, 8, 4, 2, 1 on each value, so the result is that butterfly's bit for bit.
template <int VF>
__device__ __forceinline__ void warp_sums(float (&f)[VF], int lane, bool gather)
{
    constexpr unsigned ALL = 0xffffffffu;
#pragma unroll
    for (int i = 0; i + 2 < VF; i += 4) {           // three or four values (a missing one rides along as a copy)
        const float v0 = f[i], v1 = f[i + 1], v2 = f[i + 2], v3 = i + 3 < VF ? f[i + 3 < VF ? i + 3 : 0] : 0.0f;
        const bool up16 = (lane & 16) != 0, up8 = (lane & 8) != 0;
        float a = up16 ? v2 : v0, b = up16 ? v3 : v1;               // kept by this half
        a += __shfl_xor_sync(ALL, up16 ? v0 : v2, 16);
        b += __shfl_xor_sync(ALL, up16 ? v1 : v3, 16);
        float c = up8 ? b : a;
        c += __shfl_xor_sync(ALL, up8 ? a : b, 8);
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) c += __shfl_xor_sync(ALL, c, off);
        if (gather) {
            f[i] = __shfl_sync(ALL, c, 0); f[i + 1] = __shfl_sync(ALL, c, 8); f[i + 2] = __shfl_sync(ALL, c, 16);
            if (i + 3 < VF) f[i + 3 < VF ? i + 3 : 0] = __shfl_sync(ALL, c, 24);
        } else {
            f[i] = c;                               // value i + lane / 8
        }
    }
    constexpr int REST = VF % 4 == 3 ? 0 : VF % 4;
#pragma unroll
    for (int i = VF - REST; i < VF; ++i) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) f[i] += __shfl_xor_sync(ALL, f[i], off);
    }
}

// Totals over the group of VF floats and VI ints (ints are carried exactly); every thread of the group holds
// them afterwards.  NW > 1: the group is a team and the call contains exactly one barrier of it; when `flag`
// is given, that barrier also ORs *flag over the team (every thread gets the result).
template <int VF, int VI, int K, int NW>
__device__ __forceinline__ void group_totals(float (&f)[VF], int (&iv)[VI > 0 ? VI : 1], QuantScratch<K, NW>& sc,
                                             int parity, int* flag, const QuantTeam& team)
{
    const int lane = threadIdx.x & 31;
    warp_sums<VF>(f, lane, NW == 1);
#pragma unroll
    for (int i = 0; i < VI; ++i) iv[i] = __reduce_add_sync(0xffffffffu, iv[i]);
    if (NW == 1) return;
    constexpr int SLOTS = QuantScratch<K, NW>::SLOTS;
    const int warp = team.warp;
    constexpr int FULL = VF % 4 == 3 ? VF : VF / 4 * 4;             // values that were reduced in fours
    if ((lane & 7) == 0) {
#pragma unroll
        for (int i = 0; i < FULL; i += 4)
            if (i + 3 < VF || lane < 24) sc.red[parity][i + (lane >> 3)][warp] = f[i];
    }
    if (lane == 0) {
#pragma unroll
        for (int i = FULL; i < VF; ++i) sc.red[parity][i][warp] = f[i];
#pragma unroll
        for (int i = 0; i < VI; ++i) sc.red[parity][VF + i][warp] = __int_as_float(iv[i]);
    }
    if (flag) *flag = team.sync_or(*flag);
    else team.sync();
    if constexpr (SLOTS == 4) {
        // Up to four warps: every thread reads the four partials of a value with one load and adds them in the order of the butterfly
        // below (a step of 576 units at 3 bits: 4.8 us, 5.4 us with the butterfly, whose shuffles are one after the other).
#pragma unroll
        for (int i = 0; i < VF; ++i) {
            const float4 r = *reinterpret_cast<const float4*>(sc.red[parity][i]);
            f[i] = (r.x + r.y) + (r.z + r.w);
        }
#pragma unroll
        for (int i = 0; i < VI; ++i) {
            const int4 r = *reinterpret_cast<const int4*>(sc.red[parity][VF + i]);
            iv[i] = (r.x + r.y) + (r.z + r.w);
        }
        return;
    }
    // Every warp adds up the partials of all warps: eight lanes per value, each with the partial of one warp or of two neighbours
    // (teams of up to sixteen warps), a butterfly over distances 1, 2, 4, and one shuffle per value to hand the total to all lanes.
    // (Every thread reading every partial itself took 14 to 28 128-bit loads per reduction, most of its 1300 to 2000 clocks.)
    static_assert(SLOTS <= 16, "two partials per lane");
    const bool two = team.threads > 256;
    auto partial = [&](int value) {
        const float* r = sc.red[parity][value];
        return two ? *reinterpret_cast<const float2*>(r + 2 * (lane & 7)) : make_float2((lane & 7) < SLOTS ? r[lane & 7] : 0.0f, 0.0f);
    };
#pragma unroll
    for (int i = 0; i < VF; i += 4) {
        const int v = i + (lane >> 3) < VF ? i + (lane >> 3) : VF - 1;
        const float2 q = partial(v);
        float c = two ? q.x + q.y : q.x;
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k < VF) f[i + k < VF ? i + k : 0] = __shfl_sync(0xffffffffu, c, 8 * k);
    }
#pragma unroll
    for (int i = 0; i < VI; i += 4) {
        const int v = i + (lane >> 3) < VI ? i + (lane >> 3) : VI - 1;
        const float2 q = partial(VF + v);
        int c = __float_as_int(q.x) + (two ? __float_as_int(q.y) : 0);
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k < VI) iv[i + k < VI ? i + k : 0] = __shfl_sync(0xffffffffu, c, 8 * k);
    }
}

// Least-squares solve of Eq. 5, G a = c with G = B^T B (G_ii = n, integer off-diagonals in gram[], row
// major upper triangle).  Leaves `a` untouched and returns false when a pivot of Gaussian elimination with
// partial pivoting falls below 1e-9 * n (reading for a singular system: skip the refit).  k = 2 and k = 3 solve
// through the exact integer adjugate (same rule, evaluated on exact quantities); k = 4 eliminates in fp64.
template <int K>
__device__ __forceinline__ bool solve_refit(const float (&c)[K], const int (&gram)[K > 1 ? K * (K - 1) / 2 : 1], int n,
                                            float (&a)[K])
{
    if (K == 1) {
        if (n <= 0) return false;
        a[0] = c[0] / (float)n;
        return true;
    }
    if (K == 2) {
        // pivots of the elimination are n and (n^2 - g^2) / n: the second is below 1e-9 n only when the
        // integer n^2 - g^2 is zero (n <= 8192), i.e. b_1 = +-b_2.  Cramer's rule on the exact integers; each
        // numerator n c_i - g c_j is formed without cancellation error: t = fl(g c_j), e = g c_j - t exactly
        // (fused multiply-add), fl(n c_i - t) rounds once relative to the RESULT, then e is taken off.
        const int g = gram[0];
        const int det = n * n - g * g;                       // |.| <= 2^26: exact in int
        if (det == 0) return false;
        const float fn = (float)n, fg = (float)g;            // exact (<= 8192)
        const float rdet = __fdividef(1.0f, (float)det);     // |det| <= 2^26: in range of the fast reciprocal
        const float t0 = fg * c[1], e0 = fmaf(fg, c[1], -t0);
        const float t1 = fg * c[0], e1 = fmaf(fg, c[0], -t1);
        a[0] = (fmaf(fn, c[0], -t0) - e0) * rdet;
        a[1] = (fmaf(fn, c[1], -t1) - e1) * rdet;
        return true;
    }
    if (K == 3) {
        // Adjugate of the Gram matrix: its entries and the determinant are integers below 2^53, exact in fp64, so the only
        // roundings are those of the three-term sums and of the division, and the dependent chain is a third of the
        // elimination's (the solve is per-vector scalar work that every warp repeats; on the batched cells' on-line
        // quantizer it was a visible part of a timestep).  The singularity rule is the elimination's, evaluated on the same
        // exact quantities: its second pivot is max(|n^2 - g01^2|, |n g12 - g01 g02|) / n and its third
        // |det| / (n x second pivot), whichever row the pivoting takes.
        const double n_ = (double)n, g01 = (double)gram[0], g02 = (double)gram[1], g12 = (double)gram[2];
        const double A00 = n_ * n_ - g12 * g12, A01 = g02 * g12 - g01 * n_, A02 = g01 * g12 - g02 * n_;
        const double A11 = n_ * n_ - g02 * g02, A12 = g01 * g02 - g12 * n_, A22 = n_ * n_ - g01 * g01;
        const double det = n_ * A00 + g01 * A01 + g02 * A02;
        const double tiny = 1e-9 * n_;
        const double pivot2n = fmax(fabs(A22), fabs(A12));          // n x the second pivot
        if (!(pivot2n >= tiny * n_) || !(fabs(det) >= tiny * pivot2n)) return false;
        // reciprocal of the determinant (an integer below 2^40 in magnitude): the fp32 one, refined by two Newton steps r (2 - d r) in
        // fp64, a fifth of the latency of the fp64 division (the solve is on the critical path of every vector)
        double rd = (double)__fdividef(1.0f, (float)det);
        rd = fma(rd, fma(-det, rd, 1.0), rd);
        rd = fma(rd, fma(-det, rd, 1.0), rd);
        const double c0 = (double)c[0], c1 = (double)c[1], c2 = (double)c[2];
        a[0] = (float)((A00 * c0 + A01 * c1 + A02 * c2) * rd);
        a[1] = (float)((A01 * c0 + A11 * c1 + A12 * c2) * rd);
        a[2] = (float)((A02 * c0 + A12 * c1 + A22 * c2) * rd);
        return true;
    }
    double G[K][K + 1];
    {
        int q = 0;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            G[i][i] = (double)n;
            G[i][K] = (double)c[i];
#pragma unroll
            for (int j = i + 1; j < K; ++j) { G[i][j] = (double)gram[q]; G[j][i] = (double)gram[q]; ++q; }
        }
    }
    const double tiny = 1e-9 * (double)n;
    double rp[K];
#pragma unroll
    for (int col = 0; col < K; ++col) {
        // bring the largest |entry| of the column to the pivot row by conditional swaps (static indices
        // only, so G stays in registers); the first maximum wins, as in a plain search
#pragma unroll
        for (int row = col + 1; row < K; ++row) {
            if (fabs(G[row][col]) > fabs(G[col][col])) {
#pragma unroll
                for (int j = 0; j <= K; ++j) { double t = G[col][j]; G[col][j] = G[row][j]; G[row][j] = t; }
            }
        }
        const double p = G[col][col];
        if (!(fabs(p) >= tiny) || p == 0.0) return false;
        rp[col] = 1.0 / p;
#pragma unroll
        for (int row = col + 1; row < K; ++row) {
            const double fct = G[row][col] * rp[col];
#pragma unroll
            for (int j = col; j <= K; ++j) G[row][j] -= fct * G[col][j];
        }
    }
    double sol[K];
#pragma unroll
    for (int i = K - 1; i >= 0; --i) {
        double s = G[i][K];
#pragma unroll
        for (int j = i + 1; j < K; ++j) s -= G[i][j] * sol[j];
        sol[i] = s * rp[i];
    }
#pragma unroll
    for (int i = 0; i < K; ++i) a[i] = (float)sol[i];
    return true;
}

// Levels that already ascend by code index (K >= 3): the usual case, a_1 > a_2 + a_3 (+ ..) > .. > 0, in which code bit i of an element
// is the i-th decision of the tree itself and no level has to be ranked.  v and -v are levels together and round alike, so the
// table is antisymmetric about its middle: the upper half decides, and the midpoints come out as the general table's, bit for bit.
// Fills the upper midpoints thr[2^(K-1) - 1 ..] and returns whether the levels do ascend.
template <int K>
__device__ __forceinline__ bool ascending_levels(const float (&alpha)[K], float (&thr)[(1 << K) - 1])
{
    constexpr int M = 1 << K;
    float v[M / 2];
#pragma unroll
    for (int c = 0; c < M / 2; ++c) {
        float s = alpha[0];
#pragma unroll
        for (int i = 1; i < K; ++i) s += ((c >> (K - 1 - i)) & 1) ? alpha[i] : -alpha[i];
        v[c] = s;
    }
    bool up = v[0] >= 0.0f;
    thr[M / 2 - 1] = 0.0f;
#pragma unroll
    for (int c = 0; c + 1 < M / 2; ++c) {
        up = up && v[c] <= v[c + 1];
        thr[M / 2 + c] = (v[c] + v[c + 1]) * 0.5f;
    }
    return up;
}

// The same for any coefficients, K >= 3: of every pair of levels v, -v the one in the upper half of the table (at v = 0 the one of the
// larger code index), sorted by (value, code index); its codes and the upper midpoints.
template <int K>
__device__ __forceinline__ void upper_levels(const float (&alpha)[K], float (&thr)[(1 << K) - 1], uint32_t (&code)[1 << (K - 1)])
{
    constexpr int M = 1 << K, M2 = M / 2;
    float v[M2];
#pragma unroll
    for (int c = 0; c < M2; ++c) {
        float s = alpha[0];
#pragma unroll
        for (int i = 1; i < K; ++i) s += ((c >> (K - 1 - i)) & 1) ? alpha[i] : -alpha[i];
        const bool flip = s < 0.0f;                 // (code M2 + c is the larger index of its pair)
        v[c] = flip ? -s : s;
        code[c] = flip ? (uint32_t)(M2 - 1 - c) : (uint32_t)(M2 + c);
    }
    auto order = [&](int i, int j) {                // compare and exchange
        const bool swap = v[i] > v[j] || (v[i] == v[j] && code[i] > code[j]);
        const float a = v[i], b = v[j];
        const uint32_t ca = code[i], cb = code[j];
        v[i] = swap ? b : a; v[j] = swap ? a : b;
        code[i] = swap ? cb : ca; code[j] = swap ? ca : cb;
    };
    // odd-even merge sort of four, or of twice four
#pragma unroll
    for (int h = 0; h < M2; h += 4) { order(h, h + 1); order(h + 2, h + 3); order(h, h + 2); order(h + 1, h + 3); order(h + 1, h + 2); }
    if constexpr (K == 4) {
        order(0, M2 - 4); order(1, M2 - 3); order(2, M2 - 2); order(3, M2 - 1);
        order(2, M2 - 4); order(3, M2 - 3);
        order(1, 2); order(3, M2 - 4); order(M2 - 3, M2 - 2);
    }
    thr[M2 - 1] = 0.0f;
#pragma unroll
    for (int c = 0; c + 1 < M2; ++c) thr[M2 + c] = (v[c] + v[c + 1]) * 0.5f;
}

// Algorithm 1 for one element, K >= 3, over an antisymmetric table: decision i compares w with the midpoint of the half, quarter, .. it
// is in (">=" goes up); d[i] = w minus that midpoint, whose sign bit is the inverted decision, collected in below[i] (i >= 1; decision 0
// is the sign of w).  The midpoints of the lower half are the negatives of the upper ones.
template <int K, int EPT>
__device__ __forceinline__ void tree_decisions(float w, const float (&thr)[(1 << K) - 1], uint32_t (&below)[K], uint32_t* d = nullptr)
{
    constexpr int M = 1 << K, M2 = M / 2;
    constexpr uint32_t SIGN = 0x80000000u;
    const uint32_t wb = __float_as_uint(w), sw = wb & SIGN;
    const uint32_t d1 = __float_as_uint(w - __uint_as_float(__float_as_uint(thr[M2 - 1 + M2 / 2]) | sw));
    const bool out1 = (int)(wb ^ d1) >= 0;          // the decision agrees with the sign: outer part of the half
    const float t2 = out1 ? thr[M2 - 1 + M2 / 2 + M2 / 4] : thr[M2 - 1 + M2 / 4];
    const uint32_t d2 = __float_as_uint(w - __uint_as_float(__float_as_uint(t2) | sw));
    below[1] = __funnelshift_l(d1, below[1], 1);
    below[2] = __funnelshift_l(d2, below[2], 1);
    if (d) { d[1] = d1; d[2] = d2; }
    if constexpr (K == 4) {
        const bool out2 = (int)(wb ^ d2) >= 0;
        const float hi = out2 ? thr[M - 2] : thr[M - 4], lo = out2 ? thr[M2 + 2] : thr[M2];
        const uint32_t d3 = __float_as_uint(w - __uint_as_float(__float_as_uint(out1 ? hi : lo) | sw));
        below[K - 1] = __funnelshift_l(d3, below[K - 1], 1);
        if (d) d[K - 1] = d3;
    }
}

// The sorted level table, K = 4, lane c < 2^K ranking its own level among all: the 2^K - 1 midpoints and, per plane, the signs along the
// table (bit p of plane[i]: sign, 1 = +1, of plane i at sorted level p).  One full warp, with scratch of its own.
template <int K>
__device__ __forceinline__ void level_table(const float (&alpha)[K], int lane, float (&thr)[(1 << K) - 1],
                                            uint32_t (&plane)[K], float* sc_level, int* sc_code)
{
    constexpr int M = 1 << K;
    __syncwarp();
    if (lane < M) {
        float mine = 0.0f;
#pragma unroll
        for (int i = 0; i < K; ++i) mine += ((lane >> (K - 1 - i)) & 1) ? alpha[i] : -alpha[i];
        int rank = 0;
#pragma unroll
        for (int c = 0; c < M; ++c) {
            float v = 0.0f;
#pragma unroll
            for (int i = 0; i < K; ++i) v += ((c >> (K - 1 - i)) & 1) ? alpha[i] : -alpha[i];
            rank += (v < mine || (v == mine && c < lane)) ? 1 : 0;
        }
        sc_level[rank] = mine;
        sc_code[rank] = lane;
    }
    __syncwarp();
#pragma unroll
    for (int p = 0; p < M - 1; ++p) thr[p] = (sc_level[p] + sc_level[p + 1]) * 0.5f;
    // lane p holds the code at sorted position p, one ballot per plane
    const int code = lane < M ? sc_code[lane] : 0;
#pragma unroll
    for (int i = 0; i < K; ++i) plane[i] = __ballot_sync(0xffffffffu, ((code >> (K - 1 - i)) & 1) != 0);
}

// Algorithm 1 for one element: index of the leaf (sorted level) the descent over the midpoints reaches.
// The midpoints are non-decreasing; ">=" goes to the upper half.
template <int K>
__device__ __forceinline__ int bst_leaf(float x, const float (&thr)[(1 << K) - 1])
{
    const bool c1 = x >= thr[7];
    const bool c2 = x >= (c1 ? thr[11] : thr[3]);
    const float hi3 = c2 ? thr[13] : thr[9], lo3 = c2 ? thr[5] : thr[1];
    const bool c3 = x >= (c1 ? hi3 : lo3);
    const float q3 = c3 ? thr[14] : thr[12], q2 = c3 ? thr[10] : thr[8];
    const float q1 = c3 ? thr[6] : thr[4], q0 = c3 ? thr[2] : thr[0];
    const float hi4 = c2 ? q3 : q2, lo4 = c2 ? q1 : q0;
    const bool c4 = x >= (c1 ? hi4 : lo4);
    return (c1 ? 8 : 0) + (c2 ? 4 : 0) + (c3 ? 2 : 0) + (c4 ? 1 : 0);
}

// +1.0 or -1.0 with the sign of x
__device__ __forceinline__ float unit_sign(float x) { return __uint_as_float((__float_as_uint(x) & 0x80000000u) | 0x3f800000u); }

// Signs s = +-1 of a thread's elements gathered as a word (bit j: s_j = +1).  Up to sixteen terms s_j 2^j plus 2^16 - 1 are twice that
// word, exactly; halved and added to 2^23 it stands in the low bits of the sum.
template <int EPT>
struct SignWord {
    static constexpr int PER = EPT < 16 ? EPT : 16, PARTS = (EPT + 15) / 16;
    float acc[PARTS];
    __device__ __forceinline__ SignWord()
    {
#pragma unroll
        for (int i = 0; i < PARTS; ++i) acc[i] = (float)((1 << PER) - 1);
    }
    __device__ __forceinline__ void add(int j, float s) { acc[j / 16] = fmaf(s, (float)(1 << (j % 16)), acc[j / 16]); }
    __device__ __forceinline__ uint32_t word() const
    {
        const uint32_t lo = __float_as_uint(fmaf(acc[0], 0.5f, 8388608.0f));
        if (PARTS == 1) return lo & ((1u << PER) - 1u);
        return __byte_perm(lo, __float_as_uint(fmaf(acc[PARTS - 1], 0.5f, 8388608.0f)), 0x5410);
    }
};

// Codes of a thread's elements for levels that ascend by code index, three bits: plane i is decision i of the tree, the sign of w less the
// midpoint it compares with (the midpoints of the lower half are the negatives of the upper ones, `thr`).  SUMS: also csum[i] = sum of
// b_i w, for which an element's own midpoints are chosen; without them every decision of a level is gathered as a word of bits and the
// words are chosen from, which takes fewer instructions.
template <int EPT, bool SUMS>
__device__ __forceinline__ void ascending_pass(const float (&w)[EPT], const f32x2 (&w2)[EPT / 2], const float (&thr)[7],
                                               uint32_t positive, float abs_w, uint32_t valid, uint32_t (&bits)[3], float (&csum)[3])
{
    constexpr int K = 3, M2 = 4;
    const float t1 = thr[M2 - 1 + M2 / 2], t2o = thr[M2 - 1 + M2 / 2 + M2 / 4], t2i = thr[M2 - 1 + M2 / 4];
    bits[0] = positive & valid;
    csum[0] = abs_w;
    if constexpr (SUMS) {
        float sum[K];
        SignWord<EPT> plane[K];
#pragma unroll
        for (int i = 1; i < K; ++i) sum[i] = 0.0f;
#pragma unroll
        for (int p = EPT / 2 - 1; p >= 0; --p) {
            const f32x2 sw = pack2(unit_sign(w[2 * p]), unit_sign(w[2 * p + 1]));
            const f32x2 d1 = fma2(sw, pack2(-t1, -t1), w2[p]);
            float ea, eb, da, db;
            unpack2(mul2(sw, d1), ea, eb);          // sign clear: the decision agrees with the sign of w, outer part of the half
            unpack2(d1, da, db);
            const bool oa = (int)__float_as_uint(ea) >= 0, ob = (int)__float_as_uint(eb) >= 0;
            {
                const float sa = unit_sign(da), sb = unit_sign(db);
                sum[1] = fmaf(sb, w[2 * p + 1], sum[1]);
                sum[1] = fmaf(sa, w[2 * p], sum[1]);
                plane[1].add(2 * p, sa);
                plane[1].add(2 * p + 1, sb);
            }
            const f32x2 d2 = fma2(sw, pack2(oa ? -t2o : -t2i, ob ? -t2o : -t2i), w2[p]);
            unpack2(d2, da, db);
            {
                const float sa = unit_sign(da), sb = unit_sign(db);
                sum[2] = fmaf(sb, w[2 * p + 1], sum[2]);
                sum[2] = fmaf(sa, w[2 * p], sum[2]);
                plane[2].add(2 * p, sa);
                plane[2].add(2 * p + 1, sb);
            }
        }
#pragma unroll
        for (int i = 1; i < K; ++i) {
            csum[i] = sum[i];
            bits[i] = plane[i].word() & valid;
        }
    } else {
        constexpr int WORDS = M2 - 1;               // midpoints of the upper half
        uint32_t below[WORDS];
#pragma unroll
        for (int c = 0; c < WORDS; ++c) below[c] = 0u;
#pragma unroll
        for (int p = EPT / 2 - 1; p >= 0; --p) {
            const f32x2 sw = pack2(unit_sign(w[2 * p]), unit_sign(w[2 * p + 1]));
#pragma unroll
            for (int c = 0; c < WORDS; ++c) {
                float da, db;
                unpack2(fma2(sw, pack2(-thr[M2 + c], -thr[M2 + c]), w2[p]), da, db);
                below[c] = __funnelshift_l(__float_as_uint(db), below[c], 1);
                below[c] = __funnelshift_l(__float_as_uint(da), below[c], 1);
            }
        }
        // decision i agrees with the sign of w: the outer part
        const uint32_t b1 = below[M2 / 2 - 1], o1 = positive ^ b1;
        const uint32_t b2 = (o1 & below[M2 / 2 + M2 / 4 - 1]) | (~o1 & below[M2 / 4 - 1]);
        bits[1] = ~b1 & valid;
        bits[2] = ~b2 & valid;
#pragma unroll
        for (int i = 1; i < K; ++i) csum[i] = 0.0f;
    }
}

// Elements past the end of the vector inside the threads that do hold some of it, for the two ownership patterns in
// use: thread g owns the EPT consecutive elements from g * EPT; lane l of a warp owns the elements j * 32 + l.
__host__ __device__ inline int quant_padding_consecutive(int n, int ept) { return (n + ept - 1) / ept * ept - n; }
__host__ __device__ inline int quant_padding_strided32(int n, int ept) { return (n >= 32 ? 32 : n) * ept - n; }

// The sorted table of two bits in closed form.  The tree's two decisions are the sign of w and w against the midpoint of its half; which
// plane is which decision, and its sign, follow from the coefficients.
struct TwoLevels {
    float mid;                      // >= 0
    bool first, sa, sb;
    __device__ __forceinline__ TwoLevels(float a0, float a1)
    {
        const float A = fabsf(a0), B = fabsf(a1), d = A - B;
        mid = 0.5f * ((A + B) + fabsf(d));
        sa = a0 < 0.0f; sb = a1 < 0.0f;
        first = d > 0.0f || (d == 0.0f && !sa);
        if ((A + B) == fabsf(d)) { if (first) sb = false; else sa = false; }
    }
    // c1, c2: words of the two decisions; abs_w, s1: their sums with w
    __device__ __forceinline__ void planes(uint32_t c1, uint32_t c2, uint32_t valid, float abs_w, float s1, uint32_t (&bits)[2], float (&csum)[2]) const
    {
        bits[0] = ((first ? c1 : c2) ^ (sa ? 0xffffffffu : 0u)) & valid;
        bits[1] = ((first ? c2 : c1) ^ (sb ? 0xffffffffu : 0u)) & valid;
        const float sum0 = first ? abs_w : s1, sum1 = first ? s1 : abs_w;
        csum[0] = sa ? -sum0 : sum0;
        csum[1] = sb ? -sum1 : sum1;
    }
};

// The table of three bits.  With the coefficients' magnitudes A >= B >= C the levels of its upper half are, in order, |A - B - C|, A - B + C,
// A + B - C and A + B + C: the planes of A, B and C are the tree's three decisions, but for the elements at the innermost level on either
// side, all of whose signs are the opposite ones where A < B + C.  So any order of the coefficients costs the four values (no codes
// travel with them) and a permutation of the finished words.  (On z = [x ; h] the levels seldom ascend by code: with the codes sorted along
// and the planes evaluated leaf by leaf a cycle's codes took a team of eight warps 1000 to 1130 clocks, where ascending levels take 300 to 470.)
// Levels that tie go by the order of their codes, and rounded sums of coefficients that differ by less than the rounding may tie or even come in
// another order than the exact ones.  `regular`: the smallest magnitude, the differences of any two and the innermost level are all above
// 2^-20 of the sum S, so that no two levels, each two sums within 2^-24 S of the exact ones, change places or meet.  Anything else,
// infinities and NaN among it, is sorted: the same codes as without ThreeLevels, always.  (Told from the magnitudes and not from the sorted
// levels, whose chain is the longer one.  35 steps of LSTM 1024, one sequence, 3/3 bits: 206 us without the question, 209.5 with it, 211.3
// from the sorted levels, 232 with every table sorted; 64 sequences 374, 378, 377, 396; the sorting as a call of its own, behind the pass,
// or sharing its loop over the elements: no faster there and slower in amq_quantize.)
struct ThreeLevels {
    float inner, mid, outer;        // midpoints of the upper half
    int rank[3];                    // 0: the largest magnitude; among equals the smaller index first
    bool neg[3], flip, regular;
    __device__ __forceinline__ ThreeLevels(const float (&a)[3])
    {
        const float m0 = fabsf(a[0]), m1 = fabsf(a[1]), m2 = fabsf(a[2]);
        rank[0] = (m1 > m0) + (m2 > m0); rank[1] = (m0 >= m1) + (m2 > m1); rank[2] = (m0 >= m2) + (m1 >= m2);
#pragma unroll
        for (int i = 0; i < 3; ++i) neg[i] = a[i] < 0.0f;
        // (each value rounded as the sum in the order of the planes)
        const float less = a[0] - a[1], more = a[0] + a[1];
        const float v0 = fabsf(less - a[2]), v1 = fabsf(less + a[2]), v2 = fabsf(more - a[2]), v3 = fabsf(more + a[2]);
        const float l1 = fminf(v0, v1), h1 = fmaxf(v0, v1), l2 = fminf(v2, v3), h2 = fmaxf(v2, v3);
        const float x = fmaxf(l1, l2), y = fminf(h1, h2), q0 = fminf(l1, l2), q1 = fminf(x, y), q2 = fmaxf(x, y), q3 = fmaxf(h1, h2);
        inner = (q0 + q1) * 0.5f; mid = (q1 + q2) * 0.5f; outer = (q2 + q3) * 0.5f;
        flip = ((rank[0] == 0 ? m0 : -m0) + (rank[1] == 0 ? m1 : -m1)) + (rank[2] == 0 ? m2 : -m2) < 0.0f;
        const float least = fminf(fminf(m0, fabsf(m0 - m1)), fminf(m1, fabsf(m1 - m2)));
        regular = fminf(fminf(least, q0), fminf(m2, fabsf(m0 - m2))) > ((m0 + m1) + m2) * 0x1p-20f;     // (false where the sum is infinite or NaN)
    }
    // Codes of a thread's elements; `sums`: also csum[i] = sum of b_i w.
    template <int EPT>
    __device__ __forceinline__ void pass(const float (&w)[EPT], uint32_t positive, float abs_w, uint32_t valid, bool sums,
                                         uint32_t (&bits)[3], float (&csum)[3]) const
    {
        constexpr uint32_t SIGN = 0x80000000u;
        uint32_t below1 = 0u, below2 = 0u;
        float s1 = 0.0f, s2 = 0.0f;
#pragma unroll
        for (int j = EPT - 1; j >= 0; --j) {
            const uint32_t wb = __float_as_uint(w[j]), sw = wb & SIGN;
            const uint32_t d1 = __float_as_uint(w[j] - __uint_as_float(__float_as_uint(mid) | sw));
            const float t2 = (int)(wb ^ d1) >= 0 ? outer : inner;           // the decision agrees with the sign: outer half
            const uint32_t d2 = __float_as_uint(w[j] - __uint_as_float(__float_as_uint(t2) | sw));
            below1 = __funnelshift_l(d1, below1, 1);
            below2 = __funnelshift_l(d2, below2, 1);
            if (sums) {
                s1 += __uint_as_float(wb ^ (d1 & SIGN));
                s2 += __uint_as_float(wb ^ (d2 & SIGN));
            }
        }
        uint32_t plane[3] = {positive, ~below1, ~below2};
        float sum[3] = {abs_w, s1, s2};
        if (flip) {
            const uint32_t leaf = (positive ^ plane[1]) & (positive ^ plane[2]);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                plane[i] ^= leaf;
                if (sums) {                         // (element by element, in the order of the other sums)
                    sum[i] = 0.0f;
#pragma unroll
                    for (int j = EPT - 1; j >= 0; --j) sum[i] += __uint_as_float(__float_as_uint(w[j]) ^ (~(plane[i] << (31 - j)) & SIGN));
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const uint32_t b = rank[i] == 0 ? plane[0] : rank[i] == 1 ? plane[1] : plane[2];
            const float c = rank[i] == 0 ? sum[0] : rank[i] == 1 ? sum[1] : sum[2];
            bits[i] = (neg[i] ? ~b : b) & valid;
            csum[i] = neg[i] ? -c : c;
        }
    }
};

// Codes of K >= 3 bits, levels in any order.  The table is still antisymmetric (v and -v are levels together, of complementary codes, and
// ties are ordered alike), so the tree's decisions are the same comparisons with the sorted upper half; a plane is a function of the
// leaf, evaluated on whole words of decision bits.  `sums`: also csum[i] = sum of b_i w.
template <int K, int EPT>
__device__ __forceinline__ void sorted_pass(const float (&w)[EPT], const float (&alpha)[K], uint32_t positive, uint32_t valid, bool sums,
                                            float (&thr)[(1 << K) - 1], uint32_t (&bits)[K], float (&csum)[K])
{
    constexpr uint32_t SIGN = 0x80000000u;
    constexpr int M2 = 1 << (K - 1);
    uint32_t code[M2];
    upper_levels<K>(alpha, thr, code);
    uint32_t below[K];
#pragma unroll
    for (int i = 0; i < K; ++i) below[i] = 0u;
#pragma unroll
    for (int j = EPT - 1; j >= 0; --j) tree_decisions<K, EPT>(w[j], thr, below);
    // minterms of the leaf within the half: bit i of the leaf = decision i agrees with the sign of w
    uint32_t leaf[M2];
    {
        const uint32_t u1 = positive ^ below[1], u2 = positive ^ below[2];          // (below: decision bits inverted)
        const uint32_t q3 = u1 & u2, q2 = u1 & ~u2, q1 = ~u1 & u2, q0 = ~(u1 | u2);
        if constexpr (K == 3) {
            leaf[0] = q0; leaf[1] = q1; leaf[2] = q2; leaf[3] = q3;
        } else {
            const uint32_t u3 = positive ^ below[K - 1];
            leaf[0] = q0 & ~u3; leaf[1] = q0 & u3; leaf[2] = q1 & ~u3; leaf[3] = q1 & u3;
            leaf[M2 - 4] = q2 & ~u3; leaf[M2 - 3] = q2 & u3; leaf[M2 - 2] = q3 & ~u3; leaf[M2 - 1] = q3 & u3;
        }
    }
#pragma unroll
    for (int i = 0; i < K; ++i) {
        uint32_t f = 0u;
#pragma unroll
        for (int q = 0; q < M2; ++q) f |= leaf[q] & (0u - ((code[q] >> (K - 1 - i)) & 1u));
        const uint32_t pb = ~(positive ^ f);        // the lower half has the complementary codes
        bits[i] = pb & valid;
        if (sums) {
            float cs = 0.0f;
#pragma unroll
            for (int j = EPT - 1; j >= 0; --j) cs += __uint_as_float(__float_as_uint(w[j]) ^ (~(pb << (31 - j)) & SIGN));
            csum[i] = cs;
        }
    }
}

// Three bits, coefficients in any order: the same codes and sums as sorted_pass gives, by way of ThreeLevels where that is sure.
template <int EPT>
__device__ __forceinline__ void three_bit_codes(const float (&w)[EPT], const float (&alpha)[3], uint32_t positive, float abs_w, uint32_t valid,
                                                bool sums, float (&thr)[7], uint32_t (&bits)[3], float (&csum)[3])
{
    const ThreeLevels t(alpha);
    if (t.regular) t.template pass<EPT>(w, positive, abs_w, valid, sums, bits, csum);
    else sorted_pass<3, EPT>(w, alpha, positive, valid, sums, thr, bits, csum);
}

// quantize_group of a warp of its own: the same steps with two-wide multiply-adds (see above).
template <int K, int EPT>
__device__ __forceinline__ void quantize_warp(const float (&w_in)[EPT], uint32_t valid, int n, int pad_elems, int T, float (&alpha)[K],
                                              uint32_t (&bits)[K], QuantScratch<K, 1>& sc)
{
    constexpr int NG = K * (K - 1) / 2;
    static_assert(EPT % 2 == 0 && EPT <= 32, "");
    const QuantTeam none_team{0, 0, 32};
    const int nvalid = __popc(valid);
    const float inv_n = 1.0f / (float)n;
    const float padding = (float)pad_elems;
    const bool holds_some = valid != 0;
    float w[EPT];
    f32x2 w2[EPT / 2];
#pragma unroll
    for (int p = 0; p < EPT / 2; ++p) {
        w2[p] = add2(pack2(w_in[2 * p], w_in[2 * p + 1]), 0ull);  // -0.0 -> +0.0
        unpack2(w2[p], w[2 * p], w[2 * p + 1]);
    }

    float last_abs = 0.0f, csum[K], abs_w = 0.0f;
    uint32_t positive = 0;
    float rho = 0.0f;
    {
        f32x2 r2[EPT / 2];
#pragma unroll
        for (int p = 0; p < EPT / 2; ++p) r2[p] = w2[p];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            float part = 0.0f;
            if (i == 0) {                                         // (|w| is an operand modifier, the word a funnel shift per element)
                uint32_t neg = 0;
#pragma unroll
                for (int j = EPT - 1; j >= 0; --j) {
                    part += fabsf(w[j]);
                    neg = __funnelshift_l(__float_as_uint(w[j]), neg, 1);
                }
                positive = ~neg;
                bits[0] = positive & valid;
                csum[0] = abs_w = part;
            } else {
                float cs = 0.0f;
                SignWord<EPT> plane;
#pragma unroll
                for (int p = EPT / 2 - 1; p >= 0; --p) {
                    float ra, rb;
                    unpack2(r2[p], ra, rb);
                    const float sa = unit_sign(ra), sb = unit_sign(rb);
                    part += fabsf(rb); part += fabsf(ra);
                    cs = fmaf(sb, w[2 * p + 1], cs);              // b_i w
                    cs = fmaf(sa, w[2 * p], cs);
                    plane.add(2 * p, sa);
                    plane.add(2 * p + 1, sb);
                }
                bits[i] = plane.word() & valid;
                csum[i] = cs;
            }
            part = holds_some ? part : 0.0f;
            if (i == K - 1 && T > 0) { last_abs = part; alpha[i] = 0.0f; break; }
            float tot[1] = {part};
            int none[1] = {0};
            group_totals<1, 0, K, 1>(tot, none, sc, 0, nullptr, none_team);
            const float a = (tot[0] - padding * fabsf(rho)) * inv_n;
            alpha[i] = a;
            const uint32_t ab = __float_as_uint(a);               // a >= 0, but for a rounding of a vanishing one
            rho -= __uint_as_float(ab | (__float_as_uint(rho) & 0x80000000u));
            if (i == K - 1) break;                                // (T = 0: no residue is needed any more)
            const uint32_t sign = ~ab & 0x80000000u;              // (a team takes a negative coefficient off every residue as it is)
            const f32x2 minus = pack2(-a, -a);
#pragma unroll
            for (int p = 0; p < EPT / 2; ++p) {                   // r - a sign(r)
                float ra, rb;
                unpack2(r2[p], ra, rb);
                r2[p] = fma2(pack2(__uint_as_float((__float_as_uint(ra) & sign) | 0x3f800000u), __uint_as_float((__float_as_uint(rb) & sign) | 0x3f800000u)),
                             minus, r2[p]);
            }
        }
    }

    for (int it = 0; it < T; ++it) {
        float fsum[1 + K];
        int gram[NG > 0 ? NG : 1];
        fsum[0] = last_abs;
#pragma unroll
        for (int i = 0; i < K; ++i) fsum[1 + i] = csum[i];
        {
            int q = 0;
#pragma unroll
            for (int i = 0; i < K; ++i)
#pragma unroll
                for (int j = i + 1; j < K; ++j)
                    gram[q++] = nvalid - 2 * __popc((bits[i] ^ bits[j]) & valid);
            if (NG == 0) gram[0] = 0;
        }
        group_totals<1 + K, NG, K, 1>(fsum, gram, sc, 0, nullptr, none_team);
        if (it == 0) alpha[K - 1] = (fsum[0] - padding * fabsf(rho)) * inv_n;
        {
            float c[K];
#pragma unroll
            for (int i = 0; i < K; ++i) c[i] = fsum[1 + i];
            solve_refit<K>(c, gram, n, alpha);
        }
        last_abs = 0.0f;
        const bool more = it + 1 < T;
        if constexpr (K == 1) {
            bits[0] = (alpha[0] < 0.0f ? ~positive : positive) & valid;
            csum[0] = alpha[0] < 0.0f ? -abs_w : abs_w;
        } else if constexpr (K == 2) {
            const TwoLevels t(alpha[0], alpha[1]);
            const f32x2 minus = pack2(-t.mid, -t.mid);
            uint32_t below = 0;
            float s1 = 0.0f;
            if (more) {
                SignWord<EPT> plane;
#pragma unroll
                for (int p = EPT / 2 - 1; p >= 0; --p) {
                    float da, db;
                    unpack2(fma2(pack2(unit_sign(w[2 * p]), unit_sign(w[2 * p + 1])), minus, w2[p]), da, db);
                    const float sa = unit_sign(da), sb = unit_sign(db);
                    s1 = fmaf(sb, w[2 * p + 1], s1);
                    s1 = fmaf(sa, w[2 * p], s1);
                    plane.add(2 * p, sa);
                    plane.add(2 * p + 1, sb);
                }
                below = ~plane.word();
            } else {
#pragma unroll
                for (int p = EPT / 2 - 1; p >= 0; --p) {
                    float da, db;
                    unpack2(fma2(pack2(unit_sign(w[2 * p]), unit_sign(w[2 * p + 1])), minus, w2[p]), da, db);
                    below = __funnelshift_l(__float_as_uint(db), below, 1);
                    below = __funnelshift_l(__float_as_uint(da), below, 1);
                }
            }
            t.planes(positive, ~below, valid, abs_w, s1, bits, csum);
        } else {
            float thr[(1 << K) - 1];
            if (ascending_levels<K>(alpha, thr)) {
                if (more) ascending_pass<EPT, true>(w, w2, thr, positive, abs_w, valid, bits, csum);
                else ascending_pass<EPT, false>(w, w2, thr, positive, abs_w, valid, bits, csum);
            } else {
                three_bit_codes<EPT>(w, alpha, positive, abs_w, valid, more, thr, bits, csum);
            }
        }
    }
}

// Quantize the vector held in w[] (positions past the end of the vector must hold 0 and have their bit
// clear in `valid`; `pad_elems` = how many such positions lie in threads whose `valid` is not zero).  NW = 1: the group is the calling warp; NW > 1: the group is the whole CTA of up to NW
// warps (quant_scratch_init must have run).  On return alpha[i] are the coefficients and bit j of bits[i] is
// the sign (1 = +1) of element j of this thread in plane i.
//
// The greedy step needs k dependent reductions (each coefficient is the mean |residue| left by the
// previous one, Eq. 3-4); the sign plane of the last greedy bit does not depend on its own coefficient,
// so that last reduction travels together with the sums of the first refit (Eq. 5): k + T - 1 group
// reductions in all for T >= 1, with the values Algorithm 2 prescribes; each is one CTA barrier when the
// group is the CTA.  `flag` (CTA groups only, may be NULL): ORed over the CTA by the first of those barriers,
// so a caller can fold a "some thread gave up waiting for its input" vote into it; `parity` (CTA groups
// only): which half of the double-buffered partial-sum scratch the first reduction uses, updated on return,
// so that consecutive calls keep alternating.
template <int K, int EPT, int NW>
__device__ __forceinline__ void quantize_group(const float (&w_in)[EPT], uint32_t valid, int n, int pad_elems, int T,
                                               float (&alpha)[K], uint32_t (&bits)[K], QuantScratch<K, NW>& sc,
                                               int* flag = nullptr, int* parity_io = nullptr,
                                               const QuantTeam& team = QuantTeam::cta())
{
    // (at four bits the warp's form gained 3 % on 32768 x 1024 and lost 7 % on 1704 x 896, where a row's chain of operations is what counts)
    if constexpr (NW == 1 && K <= 3) {
        quantize_warp<K, EPT>(w_in, valid, n, pad_elems, T, alpha, bits, sc);
        return;
    }
    constexpr int M = 1 << K;
    constexpr int NG = K * (K - 1) / 2;
    constexpr uint32_t SIGN = 0x80000000u;
    const int nvalid = __popc(valid);
    const float inv_n = 1.0f / (float)n;
    const float padding = (float)pad_elems;                      // zero elements past the end that are summed along
    const bool holds_some = valid != 0;
    int parity = parity_io ? *parity_io : 0;

    float w[EPT];
#pragma unroll
    for (int j = 0; j < EPT; ++j) w[j] = w_in[j] + 0.0f;          // -0.0 -> +0.0: from here on "x >= 0" is "sign bit clear"

    // ---- greedy initialisation, Eq. 3-4 (and, for T > 0, B^T w of the first refit in the same pass) ----
    float last_abs = 0.0f, csum[K], abs_w = 0.0f;                 // abs_w: this thread's sum |w|
    uint32_t positive = 0;                                        // bit j: w[j] >= 0
    float rho = 0.0f;                                             // residue of a zero element (the padding)
    {
        float r[EPT];
#pragma unroll
        for (int j = 0; j < EPT; ++j) r[j] = w[j];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            float part = 0.0f, cs = 0.0f;
            uint32_t neg = 0;
#pragma unroll
            for (int j = EPT - 1; j >= 0; --j) {
                const uint32_t rb = __float_as_uint(r[j]);
                part += fabsf(r[j]);
                neg = __funnelshift_l(rb, neg, 1);                // sign bit of r[j] enters at bit 0
                if (i > 0) cs += __uint_as_float(__float_as_uint(w[j]) ^ (rb & SIGN));     // b_i * w (i = 0: |w|)
            }
            bits[i] = ~neg & valid;
            if (i == 0) positive = ~neg;
            csum[i] = i > 0 ? cs : part;
            if (i == 0) abs_w = part;
            part = holds_some ? part : 0.0f;
            if (i == K - 1 && T > 0) { last_abs = part; alpha[i] = 0.0f; break; }
            float tot[1] = {part};
            int none[1] = {0};
            group_totals<1, 0, K, NW>(tot, none, sc, parity, flag, team);
            flag = nullptr;
            parity ^= 1;
            const float a = (tot[0] - padding * fabsf(rho)) * inv_n;
            alpha[i] = a;
            const uint32_t ab = __float_as_uint(a);               // a >= 0
            rho -= __uint_as_float(ab | (__float_as_uint(rho) & SIGN));
#pragma unroll
            for (int j = 0; j < EPT; ++j)
                r[j] -= __uint_as_float(ab | (__float_as_uint(r[j]) & SIGN));      // r - copysign(a, r)
        }
    }

    // ---- T alternating cycles ----
    for (int it = 0; it < T; ++it) {
        // least-squares refit, Eq. 5: G = B^T B (exact integers), c = B^T w (summed while the codes were assigned)
        float fsum[1 + K];
        int gram[NG > 0 ? NG : 1];
        fsum[0] = last_abs;
#pragma unroll
        for (int i = 0; i < K; ++i) fsum[1 + i] = csum[i];
        {
            int q = 0;
#pragma unroll
            for (int i = 0; i < K; ++i)
#pragma unroll
                for (int j = i + 1; j < K; ++j)
                    gram[q++] = nvalid - 2 * __popc((bits[i] ^ bits[j]) & valid);
            if (NG == 0) gram[0] = 0;
        }
        group_totals<1 + K, NG, K, NW>(fsum, gram, sc, parity, flag, team);
        flag = nullptr;
        parity ^= 1;
        float thr[M - 1];
        {
            if (it == 0) alpha[K - 1] = (fsum[0] - padding * fabsf(rho)) * inv_n;   // the last greedy coefficient
            float c[K];
#pragma unroll
            for (int i = 0; i < K; ++i) c[i] = fsum[1 + i];
            solve_refit<K>(c, gram, n, alpha);
        }
        last_abs = 0.0f;
        const bool more = it + 1 < T;

        if constexpr (K == 1) {
            // levels -a, a: the sign plane, or its opposite for a < 0
            bits[0] = (alpha[0] < 0.0f ? ~positive : positive) & valid;
            csum[0] = alpha[0] < 0.0f ? -abs_w : abs_w;
            continue;
        }
        if constexpr (K == 2) {
            const TwoLevels t(alpha[0], alpha[K - 1]);
            const uint32_t mid = __float_as_uint(t.mid);
            uint32_t below = 0;
            float s1 = 0.0f;
#pragma unroll
            for (int j = EPT - 1; j >= 0; --j) {
                const uint32_t wb = __float_as_uint(w[j]);
                const uint32_t db = __float_as_uint(w[j] - __uint_as_float(mid | (wb & SIGN)));
                below = __funnelshift_l(db, below, 1);
                if (more) s1 += __uint_as_float(wb ^ (db & SIGN));
            }
            t.planes(positive, ~below, valid, abs_w, s1, bits, csum);
            continue;
        }
        if constexpr (QuantScratch<K, NW>::TABLE) {
            uint32_t plane[K], pos_bits[K];
            level_table<K>(alpha, threadIdx.x & 31, thr, plane, sc.level[team.warp], sc.code[team.warp]);
#pragma unroll
            for (int i = 0; i < K; ++i) { pos_bits[i] = 0u; csum[i] = 0.0f; }
#pragma unroll
            for (int j = EPT - 1; j >= 0; --j) {
                const int sh = 31 - bst_leaf<K>(w[j], thr);
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    const uint32_t y = plane[i] << sh;             // sign of plane i at this leaf, in the top bit
                    pos_bits[i] = __funnelshift_l(y, pos_bits[i], 1);
                    if (more) csum[i] += __uint_as_float(__float_as_uint(w[j]) ^ (~y & SIGN));
                }
            }
#pragma unroll
            for (int i = 0; i < K; ++i) bits[i] = pos_bits[i] & valid;
            continue;
        }
        if constexpr (K == 3 && EPT < 32) {
            three_bit_codes<EPT>(w, alpha, positive, abs_w, valid, more, thr, bits, csum);
        } else if constexpr (K >= 3) {
            // A warp's rows of four bits, and bulk rows of more than 1024 at three bits, 32 elements a thread: they nearly always ascend, and a
            // thread's registers count (8192 x 3000 at 3 bits 72 us this way, 82 to 84 with ThreeLevels for all or for the other rows).
            if (ascending_levels<K>(alpha, thr)) {
                uint32_t below[K];
                float sum[K];
#pragma unroll
                for (int i = 0; i < K; ++i) { below[i] = 0u; sum[i] = 0.0f; }
#pragma unroll
                for (int j = EPT - 1; j >= 0; --j) {
                    uint32_t d[K];
                    tree_decisions<K, EPT>(w[j], thr, below, d);
                    if (more) {
#pragma unroll
                        for (int i = 1; i < K; ++i) sum[i] += __uint_as_float(__float_as_uint(w[j]) ^ (d[i] & SIGN));
                    }
                }
                bits[0] = positive & valid;
                csum[0] = abs_w;
#pragma unroll
                for (int i = 1; i < K; ++i) { bits[i] = ~below[i] & valid; csum[i] = sum[i]; }
            } else {
                sorted_pass<K, EPT>(w, alpha, positive, valid, more, thr, bits, csum);
            }
        }
    }
    if (parity_io) *parity_io = parity;
}

// Pack the sign bits of a group into words: word (j * G/32 + warp-in-group) of plane i is the ballot
// over the warp of bit j.  `out` points at the k planes of the vector (global or shared memory).
template <int K, int EPT>
__device__ __forceinline__ void pack_group(const uint32_t (&bits)[K], int lane, int warp_in_group,
                                           int warps_per_group, int wpr, uint32_t* out)
{
#pragma unroll
    for (int i = 0; i < K; ++i) {
        uint32_t mine = 0;
#pragma unroll
        for (int j = 0; j < EPT; ++j) {
            const uint32_t word = __ballot_sync(0xffffffffu, (bits[i] >> j) & 1u);
            if (lane == j) mine = word;
        }
        if (lane < EPT) {
            const int q = lane * warps_per_group + warp_in_group;
            if (q < wpr) out[i * wpr + q] = mine;
        }
    }
}

}  // namespace amq
