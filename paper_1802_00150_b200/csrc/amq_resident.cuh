// Tensor-core product with a RESIDENT activation operand: the pieces shared by the batched product (amq_bgemm_resident.cu) and
// the batched sequence kernel (amq_rnn_batched.cu).
//
// A CTA owns a block of TB activation vectors.  Their k_a planes are expanded ONCE, over the whole length of the vectors, into
// E2M1 nibbles in shared memory (N rows of n / 2 bytes, row (g, j, e) = plane j of vector 8 g + e; positions past the end of a
// vector hold zero nibbles, which add nothing to a dot product), and stay there while packed weight rows stream past: expander warps turn 512 bit positions of
// 128 plane-rows per pipeline step into tensor memory, one warp issues the MMAs (kind::mxf4, unit block scales, M = 128), and
// epilogue warps fold finished accumulators.  Against expanding both operands stage by stage this takes the activation
// operand's shared-memory stores (40-60 % of a stage's, repeated for every weight tile) out of the main loop.
//
// The k_w planes of a tile of 128 weight rows are k_w accumulators one after the other in a ring, not neighbouring lanes of one
// accumulator: a lane of tensor memory IS a weight row, so an epilogue thread adds up the planes of its row in registers
// and lanes store consecutive rows.  (The former layout, k_w plane-rows side by side, needed a pass through shared memory per
// tile that took longer than the tile's MMAs.)
//
// Nibbles.  Output word s of a packed word keeps its bits s, s + 4, .., s + 28, as the sign of 1.0 on both operands (bit 1 = -1: a dot
// product of +-1 vectors does not see the common sign).  A shift and one logic operation per word.  (Weight nibbles that keep the bits
// in place, {0, 2} by block scales, save the shifts but make the accumulator the dot product less a constant of the operand row: the
// epilogue, which is the busiest role, had to add it back, and the expansion of the activations to count it.)
//
// Along K the vector is cut into slots of 256 positions (128 bytes of every expanded row, 128-byte swizzle: eight rows per 1024
// bytes).  For the GRU, whose candidate keeps the columns [0, I) and [I, n) apart, the slot that holds column I exists twice,
// once with only the x columns and once with only the h columns, so any I works and the x part is slots [0, nx), the h part
// [nx, NS); a full product runs over all of them.
//
// Pace, measured in isolation (one CTA per SM): 240 clocks per slot at N <= 96, 265 at N = 128 (256 is the tensor pipe's own
// time), bound by the issue and synchronisation of the steps below N = 96 (an MMA takes 46 clocks however small N is).
//
// Code size matters as much as anything above: with the operand's expansion inlined into every role and its loops unrolled the kernels
// were 95 and 210 KB of instructions, and every role waited for instruction fetches (some ten clocks per instruction).  Bodies that
// run once per pass appear once and are not unrolled.
#pragma once

#include "amq_common.cuh"
#include "amq_tcgen05.cuh"

namespace amq {

// Roles of a CTA: groups of four expander warps (which take the pipeline steps in turn), epilogue warps (lane quarter = warp mod 4,
// SPLIT warps per quarter, groups of eight vectors in turn), one warp that issues the MMAs, others.  The epilogue warp
// that polls for its group is on another scheduler than the issuing warp.
template <int GROUPS_, int EPI_WARPS_, int OUT_WARPS_>
struct ResRoles {
    static constexpr int GROUPS = GROUPS_, EXP_WARPS = 4 * GROUPS_, EPI_WARPS = EPI_WARPS_, SPLIT = EPI_WARPS_ / 4,
                         MMA_WARP = EXP_WARPS + EPI_WARPS, POLL_WARP = EXP_WARPS + 1, OUT_WARPS = OUT_WARPS_, THREADS = 32 * (MMA_WARP + 1 + OUT_WARPS_);
};
constexpr int RES_STAGE_COLS = 64;                  // tensor-memory columns of a stage: two slots of the weight operand
constexpr int RES_MAX_STAGES = 4;
constexpr int RES_MAX_RING = 2;                     // accumulator buffers
constexpr int RES_TMEM_COLS = 512;
constexpr int RES_ROW_BYTES = 256 * 4;              // coefficient of an operand row
constexpr int RES_ALPHA_BYTES = 2 * AMQ_MAX_K * 128 * 4;         // weight coefficients of a tile, double-buffered
constexpr int RES_SMEM_LIMIT = 225 * 1024;

enum ResCell { RES_PLAIN = 0, RES_LSTM = 1, RES_GRU = 2 };

struct ResProblem {
    const uint32_t* W; const float* Walpha; int k_w, wpr;
    int vec32;          // every plane-row is whole 32-byte pieces (256-bit loads)
    int cell;           // ResCell
    int units;          // rows of a plain product (a tile is 128 of them), hidden units of a cell (a tile is 32: lane quarter = gate)
    int n, I;           // vector length; first column of the h part (GRU)
    int NS, nx, xw;     // slots; slots of the x part (0: no split); whole x slots before the doubled one
    int TB, N, ring;    // activation vectors per CTA, operand rows (TB * k_a rounded up to 16), accumulator buffers
    int stages;         // weight-operand stages in tensor memory
    int batch;
};

__device__ __forceinline__ int res_slot_word(const ResProblem& p, int s) { return 8 * (s < p.nx ? s : p.xw + s - p.nx); }

// weight row of lane r of tile `tile`; -1: none.  The lane quarters of a GRU's tile are r, z and the candidate's x and h parts.
template <int CELL>
__device__ __forceinline__ int res_row(const ResProblem& p, int tile, int r)
{
    if (CELL == RES_PLAIN) { const int u = tile * 128 + r; return u < p.units ? u : -1; }
    const int u = tile * 32 + (r & 31), q = r >> 5;
    return u < p.units ? ((p.cell == RES_GRU && q == 3) ? 2 : q) * p.units + u : -1;
}

// Synchronisation block in shared memory.
struct ResSync {
    uint64_t full[RES_MAX_STAGES], empty[RES_MAX_STAGES];           // stage filled / read by the MMAs
    uint64_t tfull[RES_MAX_RING], tempty[RES_MAX_RING];     // accumulator complete / read out
    uint64_t yfull, yempty;                                 // results of a tile staged / stored (plain product)
    uint32_t tmem_slot;
    int failed;                                             // a bounded wait ran out
};

template <typename R>
__device__ __forceinline__ void res_sync_init(ResSync& sy)
{
#pragma unroll 1
    for (int g = 0; g < RES_MAX_STAGES; ++g) { mbar_init(smem_u32(&sy.full[g]), 4); mbar_init(smem_u32(&sy.empty[g]), 1); }
#pragma unroll 1
    for (int q = 0; q < RES_MAX_RING; ++q) { mbar_init(smem_u32(&sy.tfull[q]), 1); mbar_init(smem_u32(&sy.tempty[q]), R::EPI_WARPS); }
    mbar_init(smem_u32(&sy.yfull), R::EPI_WARPS); mbar_init(smem_u32(&sy.yempty), R::OUT_WARPS);
    sy.failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// barrier of `threads` threads; true when `bad` is true in any of them
__device__ __forceinline__ bool res_bar(int id, int threads, bool bad)
{
    uint32_t out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.or.pred q, %2, %3, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(out) : "r"((uint32_t)bad), "r"(id), "r"(threads) : "memory");
    return out != 0;
}
template <typename R> __device__ __forceinline__ bool res_epi_bar(bool bad) { return res_bar(1, 32 * R::EPI_WARPS, bad); }

// Wait of a whole group of warps on one mbarrier: one warp polls, the others wait at a hardware barrier.  (With every warp polling,
// the polls alone took half of the SM's issue slots and the synchronisation of a slot, without any work in it, 370 clocks.)
__device__ __forceinline__ bool res_group_wait(ResSync& sy, uint32_t bar, uint32_t parity, bool polls, int id, int threads)
{
    bool ok = true;
    if (polls) {
        ok = mbar_wait(bar, parity);
        if (!ok) *(volatile int*)&sy.failed = 1;
    }
    return !res_bar(id, threads, !ok);
}

// ---- activation operand ---------------------------------------------------------------------------------------------------

// bits n .. 31 (all of them for n <= 0, none for n >= 32)
__device__ __forceinline__ uint32_t upper_bits(int n) { return n >= 32 ? 0u : 0xffffffffu << (n < 0 ? 0 : n); }

// 256 bit positions of one packed row -> the 128 nibble bytes of operand row `row` in one slot.  `lo`, `hi`: valid element range; whole
// slots inside it need no masks.
__device__ __forceinline__ void res_expand_row(uint32_t slot_addr, int row, const uint32_t (&w)[8], int first, int lo, int hi)
{
    const uint32_t base = slot_addr + (uint32_t)row * 128u;
    if (lo <= first && first + 256 <= hi) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                uint32_t y[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) y[q] = ((w[4 * h + q] << (3 - s)) & 0x88888888u) | 0x22222222u;
                st_shared_v4(base + (uint32_t)(((4 * h + s) ^ (row & 7)) << 4), y[0], y[1], y[2], y[3]);
            }
        return;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t vm[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = first + 32 * (4 * h + q);
            // bits of the word inside [lo, hi): everything from lo - e up, less everything from hi - e up
            vm[q] = upper_bits(lo - e) & ~upper_bits(hi - e);
        }
#pragma unroll 1
        for (int s = 0; s < 4; ++s) {
            uint32_t y[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                y[q] = (((w[4 * h + q] << (3 - s)) & 0x88888888u) | 0x22222222u) & (((vm[q] >> s) & 0x11111111u) * 15u);       // nibble i: bit 4 i + s
            st_shared_v4(base + (uint32_t)(((4 * h + s) ^ (row & 7)) << 4), y[0], y[1], y[2], y[3]);
        }
    }
}

// operand row -> (vector of the block, plane): rows of a group of eight vectors are plane-major
template <int KA> __device__ __forceinline__ int res_row_vector(int row) { return row / (8 * KA) * 8 + (row & 7); }
template <int KA> __device__ __forceinline__ int res_row_plane(int row) { return row / 8 % KA; }

// Expand the planes of vectors b0 .. b0 + TB - 1 (all threads of the CTA; rows past the batch are zero nibbles).  The caller makes the
// stores visible to the MMAs: every thread executes the proxy fence at the end, then a CTA barrier.  `row_step`, `piece_step`: distance, in
// 16-byte pieces, of two plane-rows and of two pieces of one.  AHEAD (row, slot) pairs at a time:
// their loads overlap.
template <int KA, int AHEAD>
__device__ __forceinline__ void res_expand_activations(const ResProblem& p, const uint32_t* xcodes, size_t row_step, size_t piece_step, int b0, uint32_t sB)
{
    const int N = p.N;
    int row = (int)threadIdx.x % N, slot = (int)threadIdx.x / N;
    const int drow = (int)blockDim.x % N, dslot = (int)blockDim.x / N;
#pragma unroll 1
    while (slot < p.NS) {
        uint32_t w[AHEAD][8];
        int rows[AHEAD], slots[AHEAD];
        bool live[AHEAD];
#pragma unroll
        for (int a = 0; a < AHEAD; ++a) {
            const int b = b0 + res_row_vector<KA>(row), j = res_row_plane<KA>(row), w0 = res_slot_word(p, slot < p.NS ? slot : 0);
            rows[a] = row; slots[a] = slot;
            live[a] = slot < p.NS && row < p.TB * KA && b < p.batch;
#pragma unroll
            for (int q = 0; q < 8; ++q) w[a][q] = 0;
            if (live[a]) {
                const uint4* src = reinterpret_cast<const uint4*>(xcodes) + ((size_t)b * KA + j) * row_step + (size_t)(w0 >> 2) * piece_step;
                const uint4 v0 = __ldcg(src);               // (other SMs wrote the planes: not through the read-only path)
                w[a][0] = v0.x; w[a][1] = v0.y; w[a][2] = v0.z; w[a][3] = v0.w;
                if (w0 + 4 < p.wpr) { const uint4 v1 = __ldcg(src + piece_step); w[a][4] = v1.x; w[a][5] = v1.y; w[a][6] = v1.z; w[a][7] = v1.w; }
            }
            row += drow; slot += dslot;
            if (row >= N) { row -= N; ++slot; }
        }
#pragma unroll
        for (int a = 0; a < AHEAD; ++a) {
            if (slots[a] >= p.NS) break;
            const bool in_x = slots[a] < p.nx;
            const int lo = (p.nx > 0 && !in_x) ? p.I : 0, hi = !live[a] ? 0 : (in_x ? p.I : p.n);
            res_expand_row(sB + (uint32_t)(slots[a] * N * 128), rows[a], w[a], res_slot_word(p, slots[a]) * 32, live[a] ? lo : 0, hi);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---- weight operand -------------------------------------------------------------------------------------------------------

// The steps of a tile (two consecutive slots of one plane each) as a table in shared memory, two words per step: word offset in
// the row's planes, bit 29: no such slot, bit 30: the slot has only 16 bytes of the row, bit 31: it belongs to the h part of a split.
constexpr int RES_TABLE = AMQ_MAX_K * 34;           // AMQ_MAX_N / 256 + 1 slots, in pairs
constexpr uint32_t RES_STEP_NONE = 1u << 29, RES_STEP_HALF = 1u << 30, RES_STEP_H = 1u << 31;

// (Not through the read-only path: with an overlapped launch the kernel before may still be writing the weights when this one starts.)
__device__ __forceinline__ uint4 res_load(const uint4* p)
{
    uint4 v;
    asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// One group's share of the CTA's steps: the steps of all tiles in order are dealt to the groups in turn.  Thread = plane-row.  The
// packed words of a step are fetched one of the group's steps ahead.  (Every instruction counts here: the expander warps
// issue about one in ten clocks beside the other roles, and a group has three steps' time, some 1500 clocks, per step.)
template <typename R, int CELL>
struct ResFeeder {
    const uint32_t* row;            // plane 0 of this thread's row in the cursor's tile (a lane without a weight row takes the last one:
                                    // its accumulators are read by nobody)
    int i, n;                       // the cursor's step in its tile, steps of a tile
    int it, nitems;                 // tile counter of the CTA
    int tile0, tile_step;
    uint4 v[2][2];                  // the next step's packed words, and its table entries
    uint2 e;
    bool live;                      // there is a next step

    __device__ __forceinline__ void tile(const ResProblem& p, int r)
    {
        const int wr = res_row<CELL>(p, tile0 + it * tile_step, r);
        row = p.W + (size_t)(wr < 0 ? p.units - 1 : wr) * (p.k_w * p.wpr);
    }
    // position on the first own step of a pass over `tiles` tiles first, first + step, ..; `skip` steps of other groups come first
    __device__ __forceinline__ void start(const ResProblem& p, const uint32_t* table, int first, int step, int tiles, int r, int skip)
    {
        it = 0; nitems = tiles; tile0 = first; tile_step = step;
        n = p.k_w * ((p.NS + 1) >> 1); i = skip;
        if (nitems > 0) tile(p, r);
        next_tile(p, r);
        fetch(p, table, r);
    }
    __device__ __forceinline__ void next_tile(const ResProblem& p, int r)
    {
#pragma unroll 1
        while (i >= n && it < nitems) {
            i -= n;
            if (++it < nitems) tile(p, r);
        }
    }
    // whether this lane's row is zero in the slot of table entry `entry` (a GRU's candidate rows)
    __device__ __forceinline__ static bool zero_row(const ResProblem& p, uint32_t entry, int r)
    {
        return CELL != RES_PLAIN && p.cell == RES_GRU && (r >> 5) == ((entry & RES_STEP_H) ? 2 : 3);
    }
    // packed words of the cursor's step, and on to the group's next step
    __device__ __forceinline__ void fetch(const ResProblem& p, const uint32_t* table, int r)
    {
        live = it < nitems;
        if (!live) return;
        e = *reinterpret_cast<const uint2*>(table + 2 * i);
        const uint4* src0 = reinterpret_cast<const uint4*>(row + (e.x & (RES_STEP_NONE - 1)));
        const uint4* src1 = reinterpret_cast<const uint4*>(row + (e.y & (RES_STEP_NONE - 1)));
        if (p.vec32) {
            asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(v[0][0].x), "=r"(v[0][0].y), "=r"(v[0][0].z), "=r"(v[0][0].w),
                           "=r"(v[0][1].x), "=r"(v[0][1].y), "=r"(v[0][1].z), "=r"(v[0][1].w) : "l"(src0));
            asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(v[1][0].x), "=r"(v[1][0].y), "=r"(v[1][0].z), "=r"(v[1][0].w),
                           "=r"(v[1][1].x), "=r"(v[1][1].y), "=r"(v[1][1].z), "=r"(v[1][1].w) : "l"(src1));
        } else {        // (a missing half keeps whatever was there: it meets zeros of the activation operand)
            v[0][0] = res_load(src0);
            if (!(e.x & RES_STEP_HALF)) v[0][1] = res_load(src0 + 1);
            v[1][0] = res_load(src1);
            if (!(e.y & RES_STEP_HALF)) v[1][1] = res_load(src1 + 1);
        }
        i += R::GROUPS;
        if (i >= n) next_tile(p, r);
    }
};

// fill the table (all threads; a CTA barrier follows)
__device__ __forceinline__ void res_fill_table(const ResProblem& p, uint32_t* table)
{
    const int per_plane = (p.NS + 1) & ~1;
#pragma unroll 1
    for (int q = threadIdx.x; q < p.k_w * per_plane; q += blockDim.x) {
        const int plane = q / per_plane, s = q - plane * per_plane, w0 = res_slot_word(p, s);
        table[q] = s >= p.NS ? RES_STEP_NONE | RES_STEP_HALF          // (offset 0: loads what is there, used by nobody)
            : (uint32_t)(plane * p.wpr + w0) | (w0 + 8 > p.wpr ? RES_STEP_HALF : 0u) | (p.nx > 0 && s >= p.nx ? RES_STEP_H : 0u);
    }
}

// 256 bit positions of this lane's row -> 32 tensor-memory columns (the same order inside a slot as the activation rows)
__device__ __forceinline__ void res_store_slot(uint32_t taddr, const uint4& a, const uint4& b, bool zero)
{
    const uint32_t one = zero ? 0u : 0x22222222u, keep = zero ? 0u : 0xffffffffu;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t w[4] = {h ? b.x : a.x, h ? b.y : a.y, h ? b.z : a.z, h ? b.w : a.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] &= keep;                   // (all ones where no row can be zero: nothing is executed)
        uint32_t y[16];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int t = 0; t < 4; ++t) y[4 * t + q] = ((w[q] << (3 - t)) & 0x88888888u) | one;
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
            :: "r"(taddr + 16 * h), "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]),
               "r"(y[8]), "r"(y[9]), "r"(y[10]), "r"(y[11]), "r"(y[12]), "r"(y[13]), "r"(y[14]), "r"(y[15]) : "memory");
    }
}

struct ResFeedState { int stage; uint32_t parity; };       // the group's next stage and the parity of its "empty" barrier: start {group, 1}

// The expander warps' part of one pass (f has been started).  False when a wait ran out.
template <typename R, int CELL>
__device__ __forceinline__ bool res_feed(const ResProblem& p, ResSync& sy, const uint32_t* table, ResFeeder<R, CELL>& f, uint32_t tmem, ResFeedState& st)
{
    const int r = (int)threadIdx.x & 127;
    const uint32_t taddr = tmem + ((uint32_t)(r & 96) << 16) + (uint32_t)(p.ring * p.N + 16);
#pragma unroll 1
    while (f.live) {
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&sy.empty[st.stage]), st.parity))) { *(volatile int*)&sy.failed = 1; return false; }
        const uint32_t t = taddr + (uint32_t)(st.stage * RES_STAGE_COLS);
        res_store_slot(t, f.v[0][0], f.v[0][1], f.zero_row(p, f.e.x, r));
        if (!(f.e.y & RES_STEP_NONE)) res_store_slot(t + 32, f.v[1][0], f.v[1][1], f.zero_row(p, f.e.y, r));
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&sy.full[st.stage])) : "memory");
        f.fetch(p, table, r);                       // (into the registers just expanded)
        st.stage += R::GROUPS;
        if (st.stage >= p.stages) { st.stage -= p.stages; st.parity ^= 1u; }
    }
    return true;
}

// ---- MMA issue ------------------------------------------------------------------------------------------------------------

struct ResIssueState { int stage; uint32_t full_parity; int ring; uint32_t ring_parity; };      // start: {0, 0, 0, 1}

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}

// The issuing warp's part of one pass over `nitems` tiles (whole warp, one elected lane issues).
__device__ __forceinline__ bool res_issue(const ResProblem& p, ResSync& sy, int nitems, uint32_t tmem, uint32_t sB, ResIssueState& st)
{
    const bool issues = elect_one();
    const uint32_t idesc = (1u << 7) | (1u << 10) | ((uint32_t)(p.N >> 3) << 17) | (1u << 23) | (8u << 24);     // E2M1, E8M0, M 128
    const uint64_t desc = smem_desc(sB);
    const uint32_t lo = (uint32_t)desc, hi = (uint32_t)(desc >> 32), slot_units = (uint32_t)(p.N * 8);      // N * 128 bytes / 16
    const uint32_t sf = tmem + (uint32_t)(p.ring * p.N), a0 = sf + 16;
    const uint32_t full0 = smem_u32(&sy.full[0]), empty0 = smem_u32(&sy.empty[0]);
    // The next step's barrier is looked at between the two halves of a step, while the MMAs of the first half are in the queue: with the
    // look after the last MMA the tensor pipe ran dry for 250-400 clocks between steps.
    bool ready = false;
#pragma unroll 1
    for (int it = 0; it < nitems; ++it) {
#pragma unroll 1
        for (int plane = 0; plane < p.k_w; ++plane) {
            if (!mbar_wait(smem_u32(&sy.tempty[st.ring]), st.ring_parity)) { *(volatile int*)&sy.failed = 1; return false; }
            const uint32_t acc = tmem + (uint32_t)(st.ring * p.N);
            uint32_t b = lo;
#pragma unroll 1
            for (int s = 0; s < p.NS; s += 2) {
                if (!ready && !mbar_wait(full0 + 8 * st.stage, st.full_parity)) { *(volatile int*)&sy.failed = 1; return false; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a = a0 + (uint32_t)(st.stage * RES_STAGE_COLS), empty = empty0 + 8 * st.stage;
                if (issues) mma_mxf4_stage_ta(acc, a, b, hi, idesc, s != 0 ? 1u : 0u, sf);
                if (++st.stage == p.stages) { st.stage = 0; st.full_parity ^= 1u; }
                ready = mbar_test(full0 + 8 * st.stage, st.full_parity);
                if (issues) {
                    if (s + 1 < p.NS) mma_mxf4_stage_ta(acc, a + 32, b + slot_units, hi, idesc, 1u, sf);
                    mma_commit(empty);
                }
                b += 2 * slot_units;
            }
            if (issues) mma_commit(smem_u32(&sy.tfull[st.ring]));
            __syncwarp();
            if (++st.ring == p.ring) { st.ring = 0; st.ring_parity ^= 1u; }
        }
    }
    return true;
}

// ---- accumulators ---------------------------------------------------------------------------------------------------------
//
// An epilogue warp reads its 32 rows in the m16n8 layout: a thread then holds, of every group of eight vectors, the two vectors
// 2 (lane mod 4) + {0, 1} for the four rows lane / 4 + 8 i.  A pair of vectors shares every instruction, and the coefficients of its
// vectors stay in registers for a whole pass.

struct ResDrainState { int ring; uint32_t parity; };        // start: {0, 0}

// Activation coefficients of this thread's vectors.
template <typename R, int KA, int NG>
__device__ __forceinline__ void res_load_beta(const ResProblem& p, const float* sBeta, int sub, f32x2 (&beta)[NG][KA])
{
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int j = 0; j < KA; ++j) {
            const int c = (R::SPLIT * g + sub) * 8 * KA + 8 * j + 2 * ((int)threadIdx.x & 3);
            beta[g][j] = c < p.N ? *reinterpret_cast<const f32x2*>(sBeta + c) : 0ull;
        }
}

// One tile: the k_w accumulators of this warp's 32 rows, y[g][i] = sum over planes of alpha * sum_j beta_j D_j for row lane / 4 + 8 i
// and the two vectors, D_j = the accumulators (exact integers).  `sAlpha`: coefficients [plane][128] of the tile.
template <typename R, int KA, int NG>
__device__ __forceinline__ bool res_drain_tile(const ResProblem& p, ResSync& sy, const float* sAlpha, int quarter, int sub, uint32_t tmem,
                                               const f32x2 (&beta)[NG][KA], ResDrainState& st, f32x2 (&y)[NG][4])
{
    const int lane = (int)threadIdx.x & 31;
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int i = 0; i < 4; ++i) y[g][i] = 0ull;
#pragma unroll 1
    for (int plane = 0; plane < p.k_w; ++plane) {
        f32x2 al[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float v = sAlpha[plane * 128 + quarter * 32 + (lane >> 2) + 8 * i];
            al[i] = pack2(v, v);
        }
        if (!res_group_wait(sy, smem_u32(&sy.tfull[st.ring]), st.parity, threadIdx.x >> 5 == R::POLL_WARP, 1, 32 * R::EPI_WARPS)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(st.ring * p.N);
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const int gg = R::SPLIT * g + sub;
            if (gg * 8 >= p.TB) break;
            f32x2 v[4][KA];
            tmem_ld_pairs<KA>(acc + (uint32_t)(gg * 8 * KA), v);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                f32x2 s = mul2(beta[g][0], v[i][0]);
#pragma unroll
                for (int j = 1; j < KA; ++j) s = fma2(beta[g][j], v[i][j], s);
                y[g][i] = fma2(al[i], s, y[g][i]);
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&sy.tempty[st.ring])) : "memory");
        if (++st.ring == p.ring) { st.ring = 0; st.parity ^= 1u; }
    }
    return true;
}

// ---- host -----------------------------------------------------------------------------------------------------------------

inline int res_sm_count()
{
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0) return v;
    return 1;
}

// shared memory: operand, coefficients, synchronisation block, and what the caller adds behind them
inline size_t res_smem_bytes(const ResProblem& p)
{
    return (size_t)p.NS * p.N * 128 + RES_ROW_BYTES + RES_ALPHA_BYTES + RES_TABLE * 4 + sizeof(ResSync);
}

// block of TB vectors: operand rows and accumulator buffers; false when they fit neither tensor nor shared memory
template <typename R>
inline bool res_set_block(ResProblem& p, int TB, int k_a, size_t more_smem = 0)
{
    p.TB = TB;
    p.N = (TB * k_a + 15) / 16 * 16;
    if (p.N > 256 || p.NS > 33) return false;
    // two accumulator buffers where that leaves a stage per group
    p.ring = (RES_TMEM_COLS - 16 - 2 * p.N) / RES_STAGE_COLS >= R::GROUPS ? 2 : 1;
    const int stages = (RES_TMEM_COLS - 16 - p.ring * p.N) / RES_STAGE_COLS;
    p.stages = stages < RES_MAX_STAGES ? stages : RES_MAX_STAGES;
    return res_smem_bytes(p) + more_smem <= (size_t)RES_SMEM_LIMIT;
}

// estimated clocks per slot of 128 plane-rows (measured: 240 up to N = 96, 265 at N = 128, then the tensor pipe's own pace); with
// one accumulator buffer the MMAs of the next plane wait while the epilogue reads the last one out
inline double res_slot_clocks(const ResProblem& p)
{
    const double t = 2.0 * p.N + 10.0 > 240.0 ? 2.0 * p.N + 10.0 : 240.0;
    return p.ring > 1 ? t : t + 600.0 / p.NS;
}

}  // namespace amq
