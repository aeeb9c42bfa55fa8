// Projection GEMM for prompt passes (Algorithm 1's LLM(prompt)): hundreds to thousands of rows at once, so the product is
// bound by the tensor cores, not by reading the weights:  out[row][n] = sum_k W[n][k] * (a_hi[row][k] + a_lo[row][k]).
//
// A CTA owns an output tile of 256 features x T rows and walks the whole contraction dimension; T is the pass's rows cut into
// equal tiles of at most 256.  Per 64-wide k-block it brings two 128-feature weight blocks (the storage the decode projections
// stream, see ClPlan: the 256 features are neighbours in storage order, one linear copy per segment they belong to) and the T
// rows' hi and lo activation tiles (TMA boxes of 64 rows) into shared memory - 96 KB for sixteen 128 x 256 x 16 MMAs at T = 256 -
// and accumulates W0 x hi, W0 x lo into one 256-column accumulator in tensor memory and W1 x hi, W1 x lo into a second one:
// every activation byte is used against 256 features, every weight byte against T rows.  The first weight blocks are requested
// while the kernel before is still running.  Tiles that share a weight pair run on neighbouring CTAs at the same time, so a
// weight block crosses HBM once per prompt pass and is served from L2 otherwise.  A projection with fewer tiles than would keep
// every SM busy is also cut along K into `ksplit` equal parts (the same cut for every tile): part s leaves its sums in
// partial-sum slab s and the consumers add the slabs in order, as they add the decode projections' parts.  A projection whose
// tiles fill some rounds of CTAs and a fraction of one more has the tiles of that last round alone cut, so that the round takes
// a fraction of a tile's time on all SMs instead of a whole tile's time on some.
//
// Measured per launch (tiles of 256 rows and up to three parts before): 7B down, 250 rows 87 -> 43 us; 1.1B, 333 rows: QKV 27 ->
// 17, O 27 -> 16, gate-up 48 -> 33, down 52 -> 28; 7B at 1536 rows 199 + 91 + 346 + 185 us, 1.50 PFLOP/s over the layer.
#include "internal.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <vector>

typedef __nv_bfloat16 bf16;

namespace {

using namespace tc;

constexpr int PF_TILE_TOK = 256;
// Epilogue warps.  A finishing epilogue (below) is an exponential and a division per value and stands between two tiles' products, whose accumulators
// take all of tensor memory: sixteen warps, four per scheduler, hide each other's latencies.  us per prompt with eight and with sixteen: 1.1B 300
// tokens 2189 -> 2142, 512 3001 -> 2928, 1500 6493 -> 6256; 7B (8 layers) 1536 tokens 8140 -> 7950, 2000 10900 -> 10450; 1024 wide 600 tokens 1721 -> 1663.  Where sums are
// only stored, sixteen win nothing at 256 rows and lose 1 to 2 % at 100 (more threads to start, the same stores).
__host__ __device__ constexpr int pf_epi_warps(bool gu) { return gu ? 16 : 8; }
__host__ __device__ constexpr int pf_threads(bool gu) { return 64 + 32 * pf_epi_warps(gu); }          // warp 0: producer, warp 1: MMA issuer + tensor-memory owner, the others: epilogue
constexpr int PF_BLOCK = 16384;          // one 128 x 64 bf16 weight tile
constexpr int PF_BOX = 8192;             // 64 rows x 64 bf16 of the activations
constexpr int PF_SMEM = 224 * 1024;
constexpr int PF_MAX_STAGES = 4;
constexpr int PF_ERR_TIMEOUT = 205;

// a k-block of a tile: W0, W1, the rows' hi boxes, their lo boxes
__host__ __device__ constexpr int pf_stage_bytes(int boxes) { return 2 * PF_BLOCK + 2 * boxes * PF_BOX; }

struct PfArgs {
    float* out; int ld;
    int rows;
    int k_blocks, n_ft, n_tt, ksplit;
    int tile_rows, boxes, stages;
    int tail_from, tail_split;         // output tiles from tail_from on are cut into tail_split parts instead of ksplit
    size_t seg_stride;                 // elements between the partial-sum slabs of two K parts
    ClPlan plan;
    bf16 *act_hi, *act_lo;             // gate-up: the activations of tiles in one part, [row][F] as two terms
    int* err;
};

constexpr int PF_GROUPS = PF_BLOCK * 2 / 1024;           // groups of 8 features per output tile
constexpr int PF_TILE_FT = 8 * PF_GROUPS;

// rows of a tile when the pass is cut into n_tt: a multiple of 16 (the products' N)
int pf_tile_rows(int rows, int n_tt) { return ((rows + n_tt - 1) / n_tt + 15) / 16 * 16; }

// work item -> (output tile, K part, parts of that tile); K part fastest
__device__ __forceinline__ void pf_item(const PfArgs& g, int item, int& ot, int& ks, int& parts) {
    const int uniform = g.tail_from * g.ksplit;
    if (item < uniform) { ot = item / g.ksplit; ks = item - ot * g.ksplit; parts = g.ksplit; }
    else { const int j = item - uniform; ot = g.tail_from + j / g.tail_split; ks = j % g.tail_split; parts = g.tail_split; }
}

// GU: the gate-up projection.  A tile in one part is finished here: eight lanes hold gate features, the next eight their up features, so
// that a lane pair turns two rows' sums into one activation each.  That writes half of the sums' bytes, and nobody reads the sums again.
template <bool GU>
__global__ void __launch_bounds__(pf_threads(GU), 1)
gemm_pf_kernel(const unsigned char* __restrict__ w, const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
               const __grid_constant__ PfArgs g) {
    extern __shared__ __align__(1024) unsigned char pf_smem_raw[];
    __shared__ uint64_t bar_full[PF_MAX_STAGES], bar_empty[PF_MAX_STAGES], bar_acc_full, bar_acc_empty;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ const unsigned char* piece_src[PF_GROUPS];             // the tile's groups as runs inside one segment
    __shared__ int piece_step[PF_GROUPS], piece_at[PF_GROUPS], piece_bytes[PF_GROUPS];

    pdl_trigger();
    unsigned char* smem = pf_smem_raw + ((1024u - (smem_u32(pf_smem_raw) & 1023u)) & 1023u);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_tiles = g.tail_from * g.ksplit + (g.n_ft * g.n_tt - g.tail_from) * g.tail_split;     // work items

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < PF_MAX_STAGES; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
        mbar_init(&bar_acc_full, 1); mbar_init(&bar_acc_empty, pf_epi_warps(GU));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *((volatile uint32_t*)&tmem_slot);
    volatile int* abortp = &abort_flag;

    const int stage_size = pf_stage_bytes(g.boxes);

    if (warp == 0) {
        if (elect_one()) {
            const uint64_t pol_w = policy_evict_last(), pol_a = policy_evict_last();    // both are re-read by other CTAs: keep them in L2
            int stage = 0, issued = 0, ahead = 0;          // ahead: steps of the first item whose weights are already on their way
            uint32_t phase = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
                int ot, ks, parts;
                pf_item(g, tile, ot, ks, parts);
                const int ft = ot / g.n_tt, tt = ot - ft * g.n_tt;
                const int row0 = tt * g.tile_rows;
                const int g_begin = ft * PF_GROUPS, g_end = min(g_begin + PF_GROUPS, cl_groups(g.plan));
                int pieces = 0;
                for (int grp = g_begin; grp < g_end; ++pieces) {
                    const ClRun r = cl_run(g.plan, grp, 0);
                    const int n = min(r.run, g_end - grp);
                    piece_src[pieces] = w + r.at;
                    piece_step[pieces] = r.step * 1024;
                    piece_at[pieces] = (grp - g_begin) * 1024;
                    piece_bytes[pieces] = n * 1024;
                    grp += n;
                }
                const uint32_t stage_bytes = (uint32_t)((g_end - g_begin) * 1024 + 2 * g.boxes * PF_BOX);
                const int kb_begin = ks * g.k_blocks / parts, kb_end = (ks + 1) * g.k_blocks / parts;
                auto weights = [&](int kb, int s) {
                    unsigned char* st = smem + (size_t)s * stage_size;
                    mbar_expect_tx(&bar_full[s], stage_bytes);
                    for (int i = 0; i < pieces; ++i)
                        bulk_load(st + piece_at[i], piece_src[i] + (size_t)kb * piece_step[i], (uint32_t)piece_bytes[i], &bar_full[s], pol_w);
                };
                if (issued == 0) {
                    for (; ahead < min(g.stages, kb_end - kb_begin); ++ahead) weights(kb_begin + ahead, ahead);
                    pdl_wait();                            // the activations come from the kernel before
                }
                for (int kb = kb_begin; kb < kb_end; ++kb) {
                    if (issued >= ahead) {
                        ok = mbar_wait(&bar_empty[stage], phase ^ 1u, abortp);
                        if (!ok) break;
                        weights(kb, stage);
                    }
                    unsigned char* act = smem + (size_t)stage * stage_size + 2 * PF_BLOCK;
                    for (int i = 0; i < g.boxes; ++i) {
                        tma_load_2d(act + i * PF_BOX, &map_hi, kb * 64, row0 + 64 * i, &bar_full[stage], pol_a);
                        tma_load_2d(act + (g.boxes + i) * PF_BOX, &map_lo, kb * 64, row0 + 64 * i, &bar_full[stage], pol_a);
                    }
                    ++issued;
                    if (++stage == g.stages) { stage = 0; phase ^= 1u; }
                }
            }
            if (!ok) {
                // gave up: let every copy already issued land before the CTA may exit
                for (int i = max(0, issued - g.stages); i < issued; ++i)
                    for (unsigned spin = 0; spin < WAIT_LIMIT && !mbar_try_wait(&bar_full[i % g.stages], (uint32_t)((i / g.stages) & 1)); ++spin) {}
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            // fp32 accumulate, bf16 x bf16, both operands K-major, M = 128 (weight features), N = the tile's rows
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.tile_rows >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
            int stage = 0;
            uint32_t phase = 0;
            int done_tiles = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++done_tiles) {
                ok = mbar_wait(&bar_acc_empty, (uint32_t)((done_tiles & 1) ^ 1), abortp);      // the epilogue has read the previous tile
                if (!ok) break;
                tc_fence_after();
                int ot, ks, parts;
                pf_item(g, tile, ot, ks, parts);
                const int kb_begin = ks * g.k_blocks / parts, kb_end = (ks + 1) * g.k_blocks / parts;
                for (int kb = kb_begin; kb < kb_end; ++kb) {
                    ok = mbar_wait(&bar_full[stage], phase, abortp);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sb = smem_u32(smem + (size_t)stage * stage_size);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint64_t dw = make_smem_desc(sb + j * PF_BLOCK);
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            const uint64_t da = make_smem_desc(sb + 2 * PF_BLOCK + half * g.boxes * PF_BOX);       // the boxes lie one after the other
#pragma unroll
                            for (int k16 = 0; k16 < 4; ++k16) {
                                const uint64_t adv = (uint64_t)(k16 * 2);
                                tc_mma_bf16(tmem_base + (uint32_t)(j * 256), dw + adv, da + adv, idesc, ((kb - kb_begin) | half | k16) ? 1u : 0u);
                            }
                        }
                    }
                    tc_commit(&bar_empty[stage]);
                    if (++stage == g.stages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                tc_commit(&bar_acc_full);
            }
        }
    } else {
        // an accumulator's 16 rows at a time are one warp's of each lane quarter, in turn
        const int quad = warp & 3, acc = ((warp - 2) >> 2) & 1, first = (warp - 2) >> 3 << 4, step = 2 * pf_epi_warps(GU);
        int done_tiles = 0;
        bool ok = true;
        pdl_wait();                                        // the sums of the projection before have been read
        for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++done_tiles) {
            int ot, ks, parts;
            pf_item(g, tile, ot, ks, parts);
            const int ft = ot / g.n_tt, tt = ot - ft * g.n_tt;
            ok = mbar_wait(&bar_acc_full, (uint32_t)(done_tiles & 1), abortp);
            if (!ok) break;
            tc_fence_after();
            const int row0 = tt * g.tile_rows;
            const int n_pos = cl_groups(g.plan) * 8, pos = (2 * ft + acc) * 128 + quad * 32 + lane;
            const uint32_t col = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * 256);
            const int n_rows = (2 * ft + acc) * 128 < n_pos ? min(g.tile_rows, g.rows - row0) : 0;
            if (GU && parts == 1) {
                const int side = (lane >> 3) & 1, f = (pos >> 4) * 8 + (pos & 7);               // 0: this lane holds gate sums, 1: up sums
#pragma unroll 1
                for (int c0 = first; c0 < n_rows; c0 += step) {
                    float v[16];
                    tc_ld16(col + (uint32_t)c0, v);
                    const size_t at = (size_t)(row0 + c0) * g.plan.F + f;
#pragma unroll
                    for (int r = 0; r < 16; r += 2) {                                           // the gate lane takes row r, the up lane row r + 1
                        const float other = __shfl_xor_sync(0xffffffffu, side ? v[r] : v[r + 1], 8);
                        const float gte = side ? other : v[r], up = side ? v[r + 1] : other;
                        const float a = gte / (1.0f + expf(-gte)) * up;
                        if (f < g.plan.F && c0 + r + side < n_rows) {
                            const bf16 hi = __float2bfloat16_rn(a);
                            g.act_hi[at + (size_t)(r + side) * g.plan.F] = hi;
                            g.act_lo[at + (size_t)(r + side) * g.plan.F] = __float2bfloat16_rn(a - __bfloat162float(hi));
                        }
                    }
                }
            } else {
                const int n = pos < n_pos ? cl_feature(g.plan, pos) : g.plan.N;
#pragma unroll 1
                for (int c0 = first; c0 < n_rows; c0 += step) {
                    float v[16];
                    tc_ld16(col + (uint32_t)c0, v);
                    if (n < g.plan.N) {
                        float* out = g.out + (size_t)ks * g.seg_stride + (size_t)(row0 + c0) * g.ld + n;
#pragma unroll
                        for (int r = 0; r < 16; ++r)
                            if (c0 + r < n_rows) out[(size_t)r * g.ld] = v[r];
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_acc_empty);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) atomicExch(g.err, PF_ERR_TIMEOUT);
}

}  // namespace

// Cycles on the busiest CTA when the work items go to the CTAs round robin, and of the partial sums' way through memory.  The gate-up
// projection's are counted like the others', although it finishes the tiles that are left whole: a credit for that left tiles whole
// where they fill few SMs, and what sixteen warps per SM then do behind the last product costs more than the kernel it saves.  us per
// prompt with the credit and without: 7B (8 layers) 140 tokens 1585 and 1489, 1.1B 200 tokens 2000 and 1915, 512 wide (8 layers) 290
// tokens 568 and 503, 4096 wide with 14336 gate features (8 layers) 370 tokens 2790 and 2640 (runs differ by 4 %); equal within the runs' spread at 200 tokens of the
// tiny model and 300 of the last one; from 600 rows on the two cut alike nearly everywhere.
static long long pf_cost(int n_ft, int rows, int k_blocks, int num_sms, const PfSchedule& s) {
    const int T = pf_tile_rows(rows, s.n_tt), n_ot = n_ft * s.n_tt, boxes = (T + 63) / 64;
    // a k-block: 16 products of T / 2 cycles, or its bytes at about 48 a cycle and SM; an item: its epilogue and about a microsecond
    const int step = std::max(8 * T, pf_stage_bytes(boxes) / 48), item = 48 * T + 2000;
    const int uniform = s.tail_from * s.ksplit, tail = (n_ot - s.tail_from) * s.tail_split, grid = std::min(num_sms, uniform + tail);
    const long long a = (long long)((k_blocks + s.ksplit - 1) / s.ksplit) * step + item;
    const long long b = (long long)((k_blocks + s.tail_split - 1) / s.tail_split) * step + item;
    // CTA i gets every grid-th item from i on: the counts of both kinds change at two places only
    long long worst = 0;
    for (int i : {0, uniform % grid, (uniform + tail) % grid}) {
        const int nu = (uniform - i + grid - 1) / grid, n = (uniform + tail - i + grid - 1) / grid;
        worst = std::max(worst, nu * a + (n - nu) * b);
    }
    // a sum is written, read and added: 8 bytes at about 3000 a cycle for the device
    const long long sums = (long long)rows * PF_TILE_FT * ((long long)uniform + tail) / std::max(1, s.n_tt) * 8 / 3000;
    return worst + sums;
}

// The rows' tiles and the cut along K with the least cost: every tile in up to max_parts parts, or the tiles of the last, partly
// filled round alone in 2 to 4.
PfSchedule gemm_pf_schedule(int n_ft, int rows, int k_blocks, int num_sms, int max_parts) {
    PfSchedule best{1, n_ft, 1, 1};
    long long best_cost = -1;
    const int least = (rows + PF_TILE_TOK - 1) / PF_TILE_TOK;
    for (int n_tt = least; n_tt <= least + 1; ++n_tt) {
        const int n_ot = n_ft * n_tt, full = n_ot / num_sms;
        auto consider = [&](PfSchedule c) {
            const long long cost = pf_cost(n_ft, rows, k_blocks, num_sms, c);
            if (best_cost < 0 || cost < best_cost) { best = c; best_cost = cost; }
        };
        for (int s = 1; s <= std::min(max_parts, k_blocks); ++s) consider({s, n_ot, 1, n_tt});
        const int from = (full * num_sms / n_tt) * n_tt;                // whole feature pairs stay uncut
        if (from > 0 && from < n_ot)
            for (int s = 2; s <= std::min(std::min(max_parts, 4), k_blocks); ++s) consider({1, from, s, n_tt});
    }
    return best;
}

PfSchedule prompt_schedule(const anpd_model* m, const Workspace& ws, int kind, int rows) {
    return gemm_pf_schedule((m->plan[kind].m_tiles + 1) / 2, rows, m->cl[kind].kb, m->num_sms, std::min(PF_MAX_PARTS, 3 * ws.r_max / rows));
}

anpd_status gemm_pf_enqueue(const ClPlan& plan, const unsigned char* w, const CUtensorMap& map_hi, const CUtensorMap& map_lo, int rows,
                            float* out, int ld, size_t seg_stride, bf16* act_hi, bf16* act_lo, PfSchedule sched, int num_sms, int* err, cudaStream_t st, Profiler* prof) {
    static bool attr_set[64] = {false};
    if (first_call_on_device(attr_set)) {
        CUDA_TRY(cudaFuncSetAttribute(gemm_pf_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, PF_SMEM));
        CUDA_TRY(cudaFuncSetAttribute(gemm_pf_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, PF_SMEM));
    }
    PfArgs g;
    g.out = out; g.ld = ld; g.rows = rows;
    g.plan = plan; g.k_blocks = plan.kb;
    g.n_ft = (plan.n_units * plan.gpu + PF_GROUPS - 1) / PF_GROUPS;
    g.n_tt = sched.n_tt;
    g.tile_rows = pf_tile_rows(rows, g.n_tt);
    g.boxes = (g.tile_rows + 63) / 64;
    g.stages = std::min(PF_MAX_STAGES, (PF_SMEM - 1024) / pf_stage_bytes(g.boxes));
    const int smem = g.stages * pf_stage_bytes(g.boxes) + 1024;
    g.ksplit = sched.ksplit; g.tail_from = sched.tail_from; g.tail_split = sched.tail_split; g.seg_stride = seg_stride;
    g.act_hi = act_hi; g.act_lo = act_lo;
    g.err = err;
    const bool gu = act_hi && sched.ksplit == 1;            // (with every tile cut along K there is nothing to finish)
    const int grid = std::min(num_sms, sched.tail_from * sched.ksplit + (g.n_ft * g.n_tt - sched.tail_from) * sched.tail_split);
    LAUNCH(prof, st, KC_GEMM, 2.0 * (double)plan.N * (double)plan.K,
           (launch_k(gu ? gemm_pf_kernel<true> : gemm_pf_kernel<false>, grid, pf_threads(gu), (size_t)smem, st, w, map_hi, map_lo, g)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}
