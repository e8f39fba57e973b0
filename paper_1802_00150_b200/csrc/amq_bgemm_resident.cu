// Batched binary product (Sec. 4, Fig. 3 right; y = sum_i sum_j alpha_i beta_j D_ij + bias) with a resident activation operand
// (amq_resident.cuh).  One CTA per SM; the work is the list of (block of vectors, tile of 128 weight rows) pairs, dealt out in
// equal contiguous shares, so that a CTA expands the activation operand once or twice and streams weight tiles past it.
//
// What bounds it: per tile of 128 rows (32768 x 1024, 512 vectors, 3/2 bits: some 5500 clocks, 3080 of them the tensor pipe's) the chain
// commit - poll - barrier - read - release of every accumulator, and the issue slots that the roles share with the warp that issues the
// MMAs.  That product took 59.8 us with a constant of every operand row added back in the epilogue (twice the instructions, and its
// loads kept the load/store unit busy) and the polling warp on the issuing warp's scheduler; 52.5 us now (behind a flush of L2 65.6 and 59.4).  Outputs leave through shared
// memory as 16-byte pieces.
#include "amq_resident.cuh"

namespace amq {

namespace {

struct ResGemmParams {
    ResProblem p;
    const uint32_t* xcodes; const float* xbeta; const float* bias;
    float* y; int ldy;
    int mtiles, blocks;         // tiles of 128 rows, blocks of TB vectors
    int b_bytes;                // expanded activation operand
    int early_weights;          // the kernel before does not write the weights: they may be fetched before it is through
    uint32_t* status;           // set when a bounded wait ran out
};

// Row stride of the results staged for the stores: 8 mod 32 words for two vectors (conflict-free in the m16n8 layout), 16-byte rows.
constexpr int Y_LD = 132;
// groups of eight vectors per epilogue thread: TB <= 64, or 32 (registers)
__host__ __device__ constexpr int res_ng(int k_a) { return k_a <= 2 ? 2 : 1; }

using R = ResRoles<3, 16, 3>;

// VEC: every row of the result starts on 16 bytes.  (Two kernels, not two paths in one: the registers and instructions of all the roles of a
// kernel of 1024 threads count for each role.  Without VEC a thread stores its four rows one by one; contiguous 128-byte stores, or
// 16-byte pieces shifted against the rows, were slower at most sizes: up to 35 % for rows of 2000 and more.)
template <int KA, bool VEC>
__global__ void __launch_bounds__(R::THREADS, 1)
bgemm_resident_kernel(const __grid_constant__ ResGemmParams a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const ResProblem& p = a.p;
    constexpr int NG = res_ng(KA);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float* sBeta = reinterpret_cast<float*>(smem_raw + a.b_bytes);                  // [256] per operand row
    float* sAlpha = sBeta + 256;                                                    // [2][4][128]
    uint32_t* table = reinterpret_cast<uint32_t*>(sAlpha + 2 * AMQ_MAX_K * 128);
    float* sY = reinterpret_cast<float*>(table + RES_TABLE);                        // [TB][Y_LD] results of a tile
    ResSync& sy = *reinterpret_cast<ResSync*>(sY + p.TB * Y_LD);
    const uint32_t sB = smem_u32(smem_raw);

    // this CTA's share of the (block, tile) list; a pass is the part of it that lies in one block of vectors
    const long long total = (long long)a.blocks * a.mtiles;
    long long w = total * blockIdx.x / gridDim.x;
    const long long w_end = total * (blockIdx.x + 1) / gridDim.x;
    auto pass_tiles = [&](long long at) {
        const int tile0 = (int)(at % a.mtiles);
        return (int)(w_end - at < a.mtiles - tile0 ? w_end - at : a.mtiles - tile0);
    };

    if (tid == 0) res_sync_init<R>(sy);
    res_fill_table(p, table);
    if (warp == R::MMA_WARP) {
        if (!a.early_weights) grid_dependency_wait();       // (a foreign kernel in front may still want tensor memory)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&sy.tmem_slot)), "r"((uint32_t)RES_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xffffffffu, sy.tmem_slot, 0);
    if (warp < 4) write_unit_scales(tmem, p.ring * p.N, warp);
    __syncthreads();

    // expand the activations of block bb; all threads, ends with a CTA barrier
    auto load_block = [&](int bb) {
        const int b0 = bb * p.TB;
        for (int q = tid; q < p.N; q += R::THREADS) {
            const int b = b0 + res_row_vector<KA>(q), j = res_row_plane<KA>(q);
            sBeta[q] = q < p.TB * KA && b < p.batch ? __ldcg(a.xbeta + (size_t)b * KA + j) : 0.0f;
        }
        res_expand_activations<KA, 1>(p, a.xcodes, (size_t)(p.wpr >> 2), 1, b0, sB);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    // Every role runs its own loop over the passes (the registers of one role are then not held through another's code); a pass
    // ends with a barrier, after which every MMA that read the operand has completed (the epilogue has waited for all
    // accumulators), so the operand may be overwritten.
    bool ok = true;
    if (warp < R::EXP_WARPS) {
        const int r = (warp & 3) * 32 + lane, steps_per_tile = p.k_w * ((p.NS + 1) >> 1);
        int first_step = 0;                         // pipeline steps so far, mod the number of groups
        ResFeedState fs{warp >> 2, 1u};
        ResFeeder<R, RES_PLAIN> feed;
        auto start = [&](long long at) {
            feed.start(p, table, (int)(at % a.mtiles), 1, pass_tiles(at), r, ((warp >> 2) - first_step + R::GROUPS) % R::GROUPS);
        };
        if (!a.early_weights) grid_dependency_wait();
        if (w < w_end) start(w);                    // (no kernel of a chain writes the weights)
        grid_dependency_wait();                     // the planes and coefficients may come from the preceding kernel
        while (w < w_end) {
            load_block((int)(w / a.mtiles));
            ok = res_feed(p, sy, table, feed, tmem, fs);
            const int tiles = pass_tiles(w);
            w += tiles;
            first_step = (int)((first_step + (long long)tiles * steps_per_tile) % R::GROUPS);
            if (w < w_end) start(w);
            if (__syncthreads_or(!ok)) { ok = false; break; }
        }
    } else if (warp == R::MMA_WARP) {
        ResIssueState issue{0, 0, 0, 1};
        grid_dependency_wait();
        while (w < w_end) {
            load_block((int)(w / a.mtiles));
            const int tiles = pass_tiles(w);
            ok = res_issue(p, sy, tiles, tmem, sB, issue);
            w += tiles;
            if (__syncthreads_or(!ok)) { ok = false; break; }
        }
    } else if (warp < R::MMA_WARP) {
        const int te = tid - 32 * R::EXP_WARPS, quarter = warp & 3, sub = (warp - R::EXP_WARPS) >> 2, rl = quarter * 32 + (lane >> 2);
        ResDrainState drain{0, 0};
        uint32_t y_parity = 1;
        // coefficients of a tile's rows: thread te takes one of the 128 k_w, a tile ahead
        auto alpha_of = [&](int tile) {
            const int row = tile * 128 + (te & 127), plane = te >> 7;
            return plane < p.k_w && row < p.units ? __ldcg(p.Walpha + (size_t)row * p.k_w + plane) : 0.0f;
        };
        grid_dependency_wait();
        while (w < w_end) {
            const int bb = (int)(w / a.mtiles), tile0 = (int)(w % a.mtiles), tiles = pass_tiles(w);
            float next_alpha = alpha_of(tile0);
            load_block(bb);
            f32x2 beta[NG][KA];
            res_load_beta<R, KA, NG>(p, sBeta, sub, beta);
            for (int t = 0; t < tiles; ++t) {
                float* sa = sAlpha + (t & 1) * AMQ_MAX_K * 128;
                sa[te] = next_alpha;
                if (res_epi_bar<R>(!ok)) { ok = false; break; }        // (also: everybody is past the tile before last, whose buffer this is)
                if (t + 1 < tiles) next_alpha = alpha_of(tile0 + t + 1);
                f32x2 y[NG][4];
                ok = res_drain_tile<R, KA, NG>(p, sy, sa, quarter, sub, tmem, beta, drain, y);
                // Results leave through shared memory and three warps of their own: in this layout a store from the registers is four
                // 32-byte pieces, and stores from the epilogue warps held them up for longer than a tile's MMAs take.
                if (ok && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&sy.yempty), y_parity))) { *(volatile int*)&sy.failed = 1; ok = false; }
                y_parity ^= 1u;
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    const int e = (R::SPLIT * g + sub) * 8 + 2 * (lane & 3);
                    if (e >= p.TB) break;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float y0, y1;
                        unpack2(y[g][i], y0, y1);
                        sY[e * Y_LD + rl + 8 * i] = y0;
                        sY[(e + 1) * Y_LD + rl + 8 * i] = y1;
                    }
                }
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&sy.yfull)) : "memory");
            }
            w += tiles;
            if (__syncthreads_or(!ok)) { ok = false; break; }
        }
    } else {
        uint32_t y_parity = 0;
        while (w < w_end) {
            const int bb = (int)(w / a.mtiles), tile0 = (int)(w % a.mtiles), b0 = bb * p.TB, tiles = pass_tiles(w);
            grid_dependency_wait();
            load_block(bb);
            const int last = p.batch - b0 < p.TB ? p.batch - b0 : p.TB;
            for (int t = 0; t < tiles && ok; ++t) {
                const int row = (tile0 + t) * 128 + 4 * lane;
                float4 bias = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (a.bias) {
                    if (row < p.units) bias.x = __ldcg(a.bias + row);
                    if (row + 1 < p.units) bias.y = __ldcg(a.bias + row + 1);
                    if (row + 2 < p.units) bias.z = __ldcg(a.bias + row + 2);
                    if (row + 3 < p.units) bias.w = __ldcg(a.bias + row + 3);
                }
                ok = __all_sync(0xffffffffu, mbar_wait_relaxed(smem_u32(&sy.yfull), y_parity, &sy.failed));
                y_parity ^= 1u;
                if (!ok) { *(volatile int*)&sy.failed = 1; break; }
                const bool vec = VEC && row + 3 < p.units;
#pragma unroll 4
                for (int e = warp - R::MMA_WARP - 1; e < last; e += R::OUT_WARPS) {
                    float4 v = *reinterpret_cast<const float4*>(sY + e * Y_LD + 4 * lane);
                    v.x += bias.x; v.y += bias.y; v.z += bias.z; v.w += bias.w;
                    float* out = a.y + (size_t)(b0 + e) * a.ldy + row;
                    if (vec) {
                        *reinterpret_cast<float4*>(out) = v;
                    } else {
                        if (row < p.units) out[0] = v.x;
                        if (row + 1 < p.units) out[1] = v.y;
                        if (row + 2 < p.units) out[2] = v.z;
                        if (row + 3 < p.units) out[3] = v.w;
                    }
                }
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&sy.yempty)) : "memory");
            }
            w += tiles;
            if (__syncthreads_or(!ok)) { ok = false; break; }
        }
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

struct ResGemmPlan { ResGemmParams a; int grid; size_t smem; bool vec_out; };

bool plan(const GemmArgs& g, int sms, ResGemmPlan* out)
{
    if (g.epilogue != EPI_Y) return false;
    ResGemmParams a{};
    ResProblem& p = a.p;
    p.W = g.Wcodes; p.Walpha = g.Walpha; p.k_w = g.k_w; p.wpr = words_per_row(g.n);
    p.vec32 = p.wpr % 8 == 0 && (reinterpret_cast<uintptr_t>(g.Wcodes) & 31) == 0;
    p.cell = RES_PLAIN; p.units = g.m;
    p.n = g.n; p.NS = (g.n + 255) / 256; p.batch = g.batch;
    a.mtiles = (g.m + 127) / 128;
    // block of vectors: the size with the least estimated time (shares of tiles x steps, plus the expansion of the operand,
    // which a share pays at least once); sizes whose operand does not fit shared memory are out (n > 28000 or so: none fits)
    double best = 0.0;
    for (int TB = 8; TB <= 8 * res_ng(g.k_a) * R::SPLIT; TB += 8) {
        ResProblem q = p;
        if (!res_set_block<R>(q, TB, g.k_a, (size_t)TB * Y_LD * 4)) break;
        const long long blocks = (g.batch + TB - 1) / TB, per_cta = (blocks * a.mtiles + sms - 1) / sms;
        const double expand = (double)q.N * q.NS * 128 / 80.0 + 1500.0;
        const double t = (double)per_cta * q.k_w * q.NS * res_slot_clocks(q) + expand * (1.0 + (double)per_cta / a.mtiles);
        if (best == 0.0 || t < best) { best = t; a.p = q; a.blocks = (int)blocks; }
        if (TB >= g.batch) break;
    }
    if (best == 0.0) return false;
    a.b_bytes = a.p.NS * a.p.N * 128;
    a.xcodes = g.xcodes; a.xbeta = g.xbeta; a.bias = g.bias; a.y = g.y; a.ldy = g.ldy;
    const long long total = (long long)a.blocks * a.mtiles;
    out->grid = (int)(total < sms ? total : sms);
    out->smem = res_smem_bytes(a.p) + (size_t)a.p.TB * Y_LD * 4;
    a.early_weights = !g.from_entry;
    out->vec_out = (reinterpret_cast<uintptr_t>(g.y) & 15) == 0 && g.ldy % 4 == 0;
    out->a = a;
    return true;
}

template <int KA>
amq_status launch(const ResGemmPlan& pl, bool overlap, cudaStream_t st)
{
    auto kernel = pl.vec_out ? bgemm_resident_kernel<KA, true> : bgemm_resident_kernel<KA, false>;
    AMQ_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem));
    AMQ_CUDA_TRY(launch_kernel(kernel, dim3((unsigned)pl.grid), dim3(R::THREADS), pl.smem, st, overlap, pl.a));
    AMQ_LAUNCH_CHECK();
    return AMQ_OK;
}

}  // namespace

double gemm_resident_clocks(const GemmArgs& g, int sms)
{
    // from 16 vectors on always; for 2..15 vectors when the weight matrix is large enough that the CUDA-core kernel's tile loop
    // costs more than this kernel's set-up
    if (sms < 1) sms = res_sm_count();
    ResGemmPlan pl;
    const bool big = (long long)g.m * g.k_w * words_per_row(g.n) >= (1ll << 17);
    if (!(g.batch >= 16 || (g.batch >= 2 && big)) || !plan(g, sms, &pl)) return 0.0;
    const ResProblem& p = pl.a.p;
    const double tiles = (double)(((long long)pl.a.blocks * pl.a.mtiles + sms - 1) / sms), passes = 1.0 + (tiles - 1.0) / pl.a.mtiles;
    return passes * (15600.0 + 7.4 * p.N * p.NS) + 23.8 * p.k_w * p.NS +
           tiles * (p.k_w * (1.11 * p.NS * res_slot_clocks(p) + 0.3 * p.N + 607.0) + 31.0 * p.TB);
}

amq_status launch_binary_gemm_resident(const GemmArgs& g, cudaStream_t st)
{
    ResGemmPlan pl;
    if (!plan(g, res_sm_count(), &pl)) return AMQ_ERR_UNSUPPORTED;
    amq_status s = tc_status_word(&pl.a.status);
    if (s != AMQ_OK) return s;
    switch (g.k_a) {
        case 1: return launch<1>(pl, g.overlap_with_previous || g.from_entry, st);
        case 2: return launch<2>(pl, g.overlap_with_previous || g.from_entry, st);
        case 3: return launch<3>(pl, g.overlap_with_previous || g.from_entry, st);
        case 4: return launch<4>(pl, g.overlap_with_previous || g.from_entry, st);
    }
    return AMQ_ERR_UNSUPPORTED;
}

}  // namespace amq
