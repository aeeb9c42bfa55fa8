// All layers of a single sequence's step (8 rows), and the vocabulary behind them, in one kernel that stays on the device: clusters of four
// CTAs, one CTA per SM, launched cooperatively.  Each cluster owns a range of every projection's features, its four CTAs a quarter of the
// contraction dimension each; they exchange partial sums over distributed shared memory, as in gemm_cl.cu, and what a phase leaves for the
// next (QKV, attention, O, gate-up, down) goes from cluster to cluster through global memory, which L2 holds.
//
// What bounds it: HBM for wide models (7B: 405 MB of weights per layer, 57 us at the 7.1 TB/s that 128 CTAs draw), for narrow ones the chain of
// five hand-overs per layer.  As a kernel per projection a hand-over took about 3 us: the last CTA's exit and the boundary behind it, tensor
// memory and barriers set up again, code from a cold instruction cache, a weight ring that starts empty or half an SM wide.  Here the ring runs
// through: the weight thread walks all layers' weights, and the cache's pages between them, and never waits for an activation.  us per step:
// 1.1B at 512 keys 729 -> 516, 1024 wide (16 layers) 380 -> 259, 7B (16 layers and the head) at 77 keys 1294 -> 1047 to 1080, at 1536 1382 -> 1200 to
// 1240, tiny (2 x 256) 48 -> 41.6.
//
// Hand-over.  The exchange buffers hold nothing but all-ones words until their values are written, and no value is one (a NaN that
// arithmetic or a rounding to bf16 leaves has its top bit clear): the words are their own flags.  A reader polls the very data it needs, with
// relaxed loads from L2, and no fence stands between a store and its use.  Measured with 16 KB per CTA, a round of store, poll and copy takes
// 1.2 us (1.5 to 2.0 beside a saturated weight stream); through flags with release and acquire it took 2.9, beside the stream 10.  After use
// the words are set back, by a warp that does nothing else and fences: there are two copies, by the layer's parity, and the copy of
// layer l - 1 is set back while layer l's gate-up runs.  Everybody has read all of it by then: this CTA's O results need its cluster's four
// quarters of the attention, these every cluster's QKV results, and no CTA pushes sums of QKV before it has read what l - 1 left.  And no
// sums of layer l's down projection leave this CTA before that is done (jan_done): every CTA's QKV of layer l + 1, the next to write there,
// needs them.  What the last layer leaves is set back at the start (its readers were those of the step before), ahead of this CTA's first sums of
// QKV, which every later result needs.  The workers meet that warp at the start and, without waiting for it, behind every O projection and at the
// vocabulary; they wait for jan_done between any two of these, so that no meeting begins before the one before is over.
// So are the others protected: a CTA's pushes of phase p + 2 into the region of the exchange that phase p used need results of
// phase p + 1 that need all results of phase p.  This needs every cluster to own features and every CTA k-blocks of every projection.
//
// Wide projections.  A cluster's features come in tiles of up to 128 and the weights tile by tile, each through all of K: a tile's sums are
// exchanged and finished (a quarter of its units by each CTA, the quarters taking turns) while the next one's weights still arrive, and only
// the last one's exchange stands behind the phase.  The activations of up to 24 k-blocks stay in their slots meanwhile; beyond
// that the tiles take turns every 24.  us per step against all tiles of a k-block together: 1.1B 627 -> 597, 1024 wide 291 -> 264,
// 7B (16 layers) at 77 keys 1147 -> 1138, 13B (8 layers) 947 -> 931.
//
// Narrow tiles.  A product reads 128 rows of weights from shared memory whatever they hold, beside the copies that fill the ring (350 cycles per
// 16 KB stage then, 160 alone).  Where a cluster has 64 or 32 features of the residual stream, the two or four k-blocks of a stage are rows of one
// product, its columns the activations of all of them, and the sums that count lie where a k-block's rows meet its columns: a half or a quarter
// of the products.  1.1B: O 2185 -> 1665 cycles, down 6344 -> 4856, 551 -> 539 us per step; 1024 wide 264 -> 262.
//
// The keys and values of the step itself reach the attention the same way; the pages are copied in before they can hold them (any time:
// they are as old as the step before), and the rows are put into the copy.
//
// Code.  A worker runs through some 60 KB of code per layer, so loops stay rolled unless they index registers (1.1B 520 -> 517 us per step);
// results' places worked out once and kept (3 KB of code more) or before the parts arrive lost 0.7 and 3 %.
//
// Values are those of gemm_cl.cu and attn_dec.cu: the same cut of K, the same order of parts, pages, warps and CTAs, and so equal bit for bit -
// but where products are packed (their k-blocks' sums meet at the end), beyond 4096 features (two tiles of the residual stream: a row's sum of
// squares comes in other groups),
// and for query heads of dimension 64 that share a kv head (a warp takes the products of one of them, not of two).
// Every wait is bounded and reports through the error flag; a handle that has failed once refuses all further results.  What can fail is to hear from
// another CTA: a wait for the cluster's sums that runs out raises abort_flag, a poll the handle's error too, and all others of either kind look at both.
// The CTA then goes through the rest of the step as ever, with whatever its buffers hold: ring, products and the setting back wait for nobody else,
// are in order whatever the values, and leave no copy or product under way behind them.  Only the exchange in the cluster stops, so that no
// barrier is counted on that has not come round.
#include "step_dev.cuh"

#include <algorithm>
#include <cstdlib>

namespace {

using namespace tc;

constexpr int SC_THREADS = 384;          // warp 0: weights and pages, 1: products, 2: exchange buffers, 3-10: workers, 11: L2 prefetch
constexpr int SC_WORKERS = 256;
constexpr int SC_STAGE = 16384;          // one slot of the ring: at most 16 groups of 8 features x 64 inputs, or part of a page
constexpr int SC_MAX_STAGES = 10;        // (what the shared memory holds beside the activations)
constexpr int SC_SMEM = 220 * 1024;      // of dynamic shared memory; the static arrays take 7 KB
constexpr int SC_AKB = 8, SC_ACT_SLOTS = 3;      // k-blocks of an activation slot, slots
constexpr int SC_ACT_SLOT = SC_AKB * ANPD_ROWS * 256;
constexpr int SC_CHUNK = SC_AKB * SC_ACT_SLOTS;  // k-blocks whose activations are there at once: tile by tile through all of them
constexpr int SC_MAX_TILES = 8;          // tiles of 128 features a projection may hold
constexpr unsigned SC_POLL_LIMIT = 1u << 21;
constexpr int SC_ERR_TIMEOUT = 209;

// Attention: a query head per item, 8 query vectors (with two heads of dimension 64 that share a kv head per item only half of the CTAs have
// one where there are 32: 1.1B at 512 keys 541 -> 525 us per step, at 3000 638 -> 575; 1536 wide 260 -> 250); the hi and lo terms of the queries, and of the weights, are the 16 rows of a tile.
template <int HD> struct ScCfg {
    static constexpr int NV = 8, WARPS = 8;                  // query vectors; warps, each with 16 keys of a page
    static constexpr int OP = HD + 4;                        // padded row
    static constexpr int QP = HD * 2 + 16;                   // bytes per staged query row
    static constexpr int V4 = HD / 4;
    static constexpr int KST = HD / 64;                      // ring stages of a page's K; as many of its V^T
    static constexpr int SLOTS = WARPS * NV * OP * 4;        // the warps' results and the queries lie where the activations go
    static_assert(SLOTS + 2 * NV * QP <= SC_ACT_SLOTS * SC_ACT_SLOT, "attention's buffers take the activations' place");
};

// kps: k-blocks of a stage; pack: how many of them one product takes side by side (see the kernel), 1 or kps
struct ScKind { int kb, gpu, n_units, seg, tiles, kps, pack, K, f_own_max, shift, red; };
// a projection as this cluster and CTA see it: tiles, k-blocks, where the weights start and the bytes from a k-block to the next
struct ScGeo { int T, nk, kb_lo, n_st, step; unsigned long long w_off; };
// a tile: its groups, the first one (of the cluster's), the units that each rank has finished before it, this CTA's units of it
struct ScTile { short groups, g0, before[CL_CTAS], own_n; int own_first; };

struct ScArgs {
    ScKind k[GK_COUNT];
    const unsigned char* w[GK_COUNT];    // the first layer's; the others follow `layer_step` bytes apart
    const float *attn_norm, *ffn_norm, *final_norm;
    size_t layer_step;
    unsigned* entered;                   // CTAs that have requested all weights before a projection, over all steps
    int L, ncl, stages, tmem_cols, red_bytes, ahead;
    // what the embedding left
    const unsigned char* img0;
    const float *x0, *ss0;
    // exchanged between CTAs: two copies, by the layer's parity, then what the last layer leaves
    unsigned char* xch;
    unsigned copy_bytes, fin_bytes, o_h2, o_ao, o_act, o_q, o_kv, o_ssa, o_ssb, o_fss;
    int d, Hq, Hkv, n_out;
    float inv_d, eps, q_scale;
    const int *row_pos, *row_slot, *row_seq, *row_ok, *hole_lo, *hole_hi;
    int tree;
    const float *rope_cos, *rope_sin;
    const int* page_table;
    int pages_per_seq, total_pages;
    bf16 *kpool, *vpool;
    int C, split, items;                 // attention: CTAs per item, items (query heads) that share a kv head, items
    float* out; float* amax_val; int* amax_idx;
    int* err;
};

__device__ __forceinline__ uint4 ld_relaxed4(const void* p) {
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_relaxed1(const void* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed1(void* p, uint32_t v) { asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ void st_relaxed2(void* p, uint2 v) { asm volatile("st.relaxed.gpu.global.v2.b32 [%0], {%1, %2};" ::"l"(p), "r"(v.x), "r"(v.y) : "memory"); }
constexpr uint32_t SC_EMPTY = 0xffffffffu;
__device__ __forceinline__ bool here(uint4 v) { return v.x != SC_EMPTY && v.y != SC_EMPTY && v.z != SC_EMPTY && v.w != SC_EMPTY; }
__device__ __forceinline__ void work_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void st_async2(uint32_t addr, uint32_t bar, float a, float b) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(a), "f"(b), "r"(bar) : "memory");
}
// four columns at `hi` and four at `lo` of this thread's tensor-memory lane, added
__device__ __forceinline__ void tc_ld4_sum(uint32_t hi, uint32_t lo, float* v) {
    uint32_t a[4], b[4];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%8];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4, %5, %6, %7}, [%9];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
        : "r"(hi), "r"(lo) : "memory");
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(a[i]) + __uint_as_float(b[i]);
}
// Bounded wait for something in this CTA, not begun where another one has run out.  (The flag is read ahead of the loop: 1.1B 515 -> 509 us per step.)
__device__ __forceinline__ bool sc_wait_at(uint32_t bar, uint32_t parity, volatile int* stuck_flag) {
    if (mbar_try_wait_at(bar, parity)) return true;
    if (*stuck_flag) return false;
#pragma unroll 1
    for (unsigned i = 0; i < WAIT_LIMIT; ++i)
        if (mbar_try_wait_at(bar, parity)) return true;
    *stuck_flag = 1;
    return false;
}
__device__ __forceinline__ bool sc_wait(uint64_t* bar, uint32_t parity, volatile int* stuck_flag) { return sc_wait_at(smem_u32(bar), parity, stuck_flag); }
// Bounded wait for what other CTAs of the cluster send: ends as soon as anybody in this CTA has given up, and soon after anybody at all has.
__device__ __forceinline__ void sc_wait_cluster(uint64_t* bar, uint32_t parity, volatile int* abort_flag, volatile int* err) {
#pragma unroll 1
    for (unsigned i = 0; i < WAIT_LIMIT; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (ok) return;
        if (*abort_flag || ((i & 255u) == 255u && *err)) break;
    }
    *abort_flag = 1;
}
__device__ __forceinline__ void fence_async_cta() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Units of tile t of a cluster's Uc.  Each rank finishes a quarter of every tile's units, the quarters taking turns.
__host__ __device__ inline int sc_tile_units(int Uc, int tiles, int t) { return Uc / tiles + (t < Uc % tiles ? 1 : 0); }

template <int HD>
__global__ void __launch_bounds__(SC_THREADS, 1) step_cl_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const __grid_constant__ ScArgs g) {
    typedef ScCfg<HD> Cfg;
    constexpr int NV = Cfg::NV, WARPS = Cfg::WARPS, OP = Cfg::OP, QP = Cfg::QP, V4 = Cfg::V4, KST = Cfg::KST;
    constexpr int KS = HD / 16, DT = HD / 8;
    constexpr int CC = CL_CTAS, rows = ANPD_ROWS;
    extern __shared__ __align__(1024) unsigned char sc_smem[];
    __shared__ uint64_t w_full[SC_MAX_STAGES], w_empty[SC_MAX_STAGES], a_full[SC_ACT_SLOTS], a_empty[SC_ACT_SLOTS];
    __shared__ uint64_t acc_full[SC_MAX_TILES], red_full[2][SC_MAX_TILES], att_full, jan_done;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_requested, s_phase, s_quit;         // copies of weights requested so far; all of them, or none will follow
    __shared__ int abort_flag, stuck_flag, s_issued;    // another CTA was not heard from; a wait inside this CTA ran out
    __shared__ float s_rstd[8], s_part[8][8];
    __shared__ int s_pos[8], s_slot[8], s_page[8], s_raw[8], s_idx[8][8];
    __shared__ ScGeo s_geo[GK_COUNT];
    __shared__ ScTile s_tile[GK_COUNT][SC_MAX_TILES];
    __shared__ int s_own[GK_COUNT];                     // units this CTA finishes
    __shared__ float2 rc[NV];                           // [CTA][VO] maximum and sum of the cluster's parts of this CTA's vectors
    __shared__ float sm_m[WARPS * NV], sm_l[WARPS * NV];
    __shared__ __align__(16) float recv[NV * HD];       // [CTA][VO][HD]

    unsigned char* ring = sc_smem + ((1024u - (smem_u32(sc_smem) & 1023u)) & 1023u);
    unsigned char* abuf = ring + (size_t)g.stages * SC_STAGE;
    unsigned char* redbuf = abuf + SC_ACT_SLOTS * SC_ACT_SLOT;
    float2* s_x = (float2*)(redbuf + g.red_bytes);      // this CTA's part of the residual stream, in pairs
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bid = (int)blockIdx.x, rank = bid % CC, cluster = bid / CC, ncta = g.ncl * CC;
    volatile int *abortp = &abort_flag, *stuckp = &stuck_flag;

    pdl_trigger();
    if (threadIdx.x < GK_COUNT) {                       // how this cluster and CTA cut each projection
        const ScKind& k = g.k[threadIdx.x];
        ScGeo e;
        const int ulo = cluster * k.n_units / g.ncl, uhi = (cluster + 1) * k.n_units / g.ncl, Uc = uhi - ulo, Gc = Uc * k.gpu;
        e.T = k.tiles;
        e.kb_lo = rank * k.kb / CC; e.nk = (rank + 1) * k.kb / CC - e.kb_lo;
        e.n_st = e.T == 1 ? (e.nk + k.kps - 1) / k.kps : e.nk * e.T;
        const int GS = k.seg == 1 ? k.n_units * k.gpu : Gc;               // groups of a k-block in its segment
        e.step = GS << 10;
        e.w_off = ((unsigned long long)ulo * k.gpu * (k.seg == 1 ? 1 : k.kb) + (unsigned long long)GS * e.kb_lo) * 1024;
        int before[CC] = {0, 0, 0, 0};
#pragma unroll 1
        for (int t = 0, u0 = 0; t < k.tiles; ++t) {
            ScTile& w = s_tile[threadIdx.x][t];
            const int un = sc_tile_units(Uc, k.tiles, t);
            w.groups = (short)(un * k.gpu); w.g0 = (short)(u0 * k.gpu);
            for (int r = 0; r < CC; ++r) {
                const int q = (r + t) & (CC - 1), lo = q * un / CC, n = (q + 1) * un / CC - lo;
                w.before[r] = (short)before[r];
                if (r == rank) { w.own_first = ulo + u0 + lo; w.own_n = (short)n; }
                before[r] += n;
            }
            u0 += un;
        }
        s_own[threadIdx.x] = before[rank];
        s_geo[threadIdx.x] = e;
    }
    if (threadIdx.x == 64) {
        abort_flag = 0; stuck_flag = 0; s_issued = 0; s_requested = 0; s_phase = 0; s_quit = 0;
#pragma unroll 1
        for (int s = 0; s < g.stages; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], WARPS); }
        for (int s = 0; s < SC_ACT_SLOTS; ++s) { mbar_init(&a_full[s], 8); mbar_init(&a_empty[s], 1); }
        for (int t = 0; t < SC_MAX_TILES; ++t) { mbar_init(&acc_full[t], 1); mbar_init(&red_full[0][t], 1); mbar_init(&red_full[1][t], 1); }
        mbar_init(&att_full, 1); mbar_init(&jan_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_cta();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"((uint32_t)g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cluster_arrive();                                   // waited for before the first push: every CTA's barriers are initialised then
    const uint32_t tmem_base = *((volatile uint32_t*)&tmem_slot);

    // attention: this CTA's item and its share of the pages (the row plan is older than the kernel before this one)
    const bool att = bid < g.items * g.C;
    const int arank = bid % g.C, hv = bid / g.C, kvh = hv / g.split;
    const int seq = g.row_seq[0], pos_lo = g.row_pos[0], pos_hi = (g.tree ? g.row_slot : g.row_pos)[rows - 1];
    const int n_pages = pos_hi / KV_PAGE + 1;
    const int my_pages = att && arank < n_pages ? (n_pages - arank + g.C - 1) / g.C : 0;
    const int pg_st = my_pages * 2 * KST;               // ring stages they take

    if (warp == 0) {
        // ---------------- weights and pages ----------------
        if (elect_one()) {
            const uint64_t pol_w = policy_evict_first(), pol_p = g.split > 1 ? policy_evict_last() : pol_w;       // pages are read again by the items that share the head
            const int* pages = g.page_table + (size_t)seq * g.pages_per_seq;
            // by address, with as few instructions per copy as it takes: 16 KB are due every 560 cycles, and faster behind a full ring
            const uint32_t full0 = smem_u32(&w_full[0]), empty_off = smem_u32(&w_empty[0]) - full0, full_end = full0 + 8u * (uint32_t)g.stages, ring0 = smem_u32(ring);
            uint32_t full = full0, dst = ring0, eph = 1;        // (a fresh barrier is through with the phase before its first)
            int turns = 0, requested = 0;
            bool ok = true;
            auto next = [&]() {
                full += 8u;
                dst += SC_STAGE;
                if (full == full_end) { full = full0; dst = ring0; eph ^= 1u; ++turns; }
            };
            auto weights = [&](int kd, const unsigned char* w) {
                const int nk = s_geo[kd].nk, T = s_geo[kd].T, step = s_geo[kd].step, kps = g.k[kd].kps;
                const unsigned char* src0 = w + s_geo[kd].w_off;
#pragma unroll 1
                for (int k0 = 0; k0 < nk && ok; k0 += SC_CHUNK, src0 += (size_t)SC_CHUNK * step) {
                    const int kn = min(SC_CHUNK, nk - k0);
#pragma unroll 1
                    for (int t = 0; t < T && ok; ++t) {
                        const unsigned char* src = src0 + ((int)s_tile[kd][t].g0 << 10);
                        const uint32_t kb_bytes = (uint32_t)s_tile[kd][t].groups << 10;
                        uint32_t bytes = (uint32_t)kps * kb_bytes;
                        const uint32_t src_step = kps > 1 ? bytes : (uint32_t)step;       // kps > 1 only where one tile holds all of the segment's groups
#pragma unroll 1
                        for (int k = kn; k > 0; k -= kps) {
                            if (k < kps) bytes = (uint32_t)k * kb_bytes;
                            if (!sc_wait_at(full + empty_off, eph, stuckp)) { ok = false; break; }
                            bulk_load_at(dst, src, bytes, full, pol_w);
                            mbar_arrive_at(full + empty_off, WARPS - 1);       // a page's stage is given back by its eight or four warps, a weight stage by one commit
                            src += src_step;
                            s_requested = ++requested;
                            next();
                        }
                    }
                }
            };
#pragma unroll 1
            for (int l = 0; l < g.L && ok; ++l) {
#pragma unroll 1
                for (int kd = 0; kd < 4 && ok; ++kd) {
                    weights(kd, g.w[kd] + (size_t)l * g.layer_step);
                    if (kd == GK_QKV) {
#pragma unroll 1
                        for (int i = 0, p = arank; i < my_pages && ok; ++i, p += g.C) {
                            const int row = (l * g.total_pages + pages[p]) * g.Hkv + kvh;
#pragma unroll 1
                            for (int s = 0; s < 2 * KST; ++s) {
                                if (!sc_wait_at(full + empty_off, eph, stuckp)) { ok = false; break; }
                                mbar_expect_tx_at(full, SC_STAGE);
                                if (s < KST) tma_load_2d_at(dst, &map_k, s * 64, row * KV_PAGE, full, pol_p);
                                else if (HD == 128) tma_load_2d_at(dst, &map_v, (s - KST) * 64, row * HD, full, pol_p);
                                else { tma_load_2d_at(dst, &map_v, 0, row * HD, full, pol_p); tma_load_2d_at(dst + HD * 128, &map_v, 64, row * HD, full, pol_p); }
                                if (HD == 128 && s >= KST) mbar_arrive_at(full + empty_off, WARPS / 2);       // half of the warps read it and give it back
                                s_requested = ++requested;
                                next();
                            }
                        }
                    }
                    atomicAdd(g.entered + 4 * l + kd + 1, 1u);
                    s_phase = 4 * l + kd + 1;
                }
            }
            if (ok) weights(GK_LM, g.w[GK_LM]);
            const int count = turns * g.stages + (int)((full - full0) >> 3);
            s_issued = count;
            s_quit = 1;
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- products ----------------
        if (elect_one()) {
            // fp32 accumulate, bf16 x bf16, both operands K-major, M = 128 features, N = 16 (hi terms, then lo terms)
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * rows) >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
            const uint64_t ring_d = make_smem_desc(smem_u32(ring)), act_d = make_smem_desc(smem_u32(abuf));
            const uint32_t stage_step = SC_STAGE >> 4, act_step = SC_ACT_SLOT >> 4, kb_step = (uint32_t)(rows * 256) >> 4;
            const uint32_t full0 = smem_u32(&w_full[0]), empty_off = smem_u32(&w_empty[0]) - full0, full_end = full0 + 8u * (uint32_t)g.stages;
            uint32_t full = full0, wph = 0;
            uint64_t w_d = ring_d;
            const uint32_t af0 = smem_u32(&a_full[0]), aempty_off = smem_u32(&a_empty[0]) - af0, af_end = af0 + 8u * SC_ACT_SLOTS;
            uint32_t afull = af0, aph = 0;
            uint64_t a_d = act_d;
            auto next_stage = [&]() {
                tc_commit_at(full + empty_off);
                w_d += stage_step;
                full += 8u;
                if (full == full_end) { full = full0; wph ^= 1u; w_d = ring_d; }
            };
            int kd = GK_QKV, l = 0;
#pragma unroll 1
            while (true) {
                const int nk = s_geo[kd].nk, T = s_geo[kd].T, kps = g.k[kd].kps, pack = g.k[kd].pack;
                uint32_t acc = 0;
#pragma unroll 1
                for (int k0 = 0; k0 < nk; k0 += SC_CHUNK) {
                    const int kn = min(SC_CHUNK, nk - k0);
                    uint32_t d_tmem = tmem_base;
#pragma unroll 1
                    for (int t = 0; t < T; ++t) {
                        const uint32_t kb_words = (uint32_t)s_tile[kd][t].groups << 6;
                        uint32_t af = afull, ap = aph, accumulate = acc;
                        uint64_t ad = a_d;
#pragma unroll 1
                        for (int ks = 0; ks < kn; ks += SC_AKB) {
                            if (t == 0) { sc_wait_at(af, ap, stuckp); tc_fence_after(); }
                            const int kend = min(SC_AKB, kn - ks);
                            uint64_t a = ad;
                            // a tile of fewer than 16 groups: the instruction reads whatever follows for the rows beyond, whose lanes nobody reads
#pragma unroll 1
                            for (int k = 0; k < kend; k += kps) {
                                sc_wait_at(full, wph, stuckp);
                                tc_fence_after();
                                const int n = min(kps, kend - k);
                                // packed: the stage's k-blocks are rows of one product, side by side, and its columns are the activations of all of
                                // them; of the sums, those count where a k-block's rows meet its own columns
                                tc_mma_k64(d_tmem, w_d, a, pack > 1 ? idesc + ((uint32_t)(n - 1) << 18) : idesc, accumulate);
                                accumulate = 1;
                                if (pack > 1) a += (uint32_t)n * kb_step;
                                else {
                                    a += kb_step;
                                    uint64_t w = w_d;
#pragma unroll 1
                                    for (int j = n; j > 1; --j) {
                                        w += kb_words;
                                        tc_mma_k64(d_tmem, w, a, idesc, 1u);
                                        a += kb_step;
                                    }
                                }
                                next_stage();
                            }
                            if (t == T - 1) tc_commit_at(af + aempty_off);
                            ad += act_step;
                            af += 8u;
                            if (af == af_end) { af = af0; ap ^= 1u; ad = act_d; }
                        }
                        if (k0 + kn == nk) tc_commit(&acc_full[t]);
                        d_tmem += (uint32_t)(2 * rows);
                        if (t == T - 1) { afull = af; aph = ap; a_d = ad; }
                    }
                    acc = 1;
                }
                if (kd == GK_LM) break;
                if (kd == GK_QKV) {                                     // the pages' stages are the workers'
                    int st = (int)((full - full0) >> 3) + pg_st;
                    wph ^= (uint32_t)(st / g.stages) & 1u;
                    st %= g.stages;
                    full = full0 + 8u * (uint32_t)st;
                    w_d = ring_d + stage_step * (uint32_t)st;
                }
                if (kd == GK_DOWN) { ++l; kd = l == g.L ? GK_LM : GK_QKV; } else ++kd;
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ---------------- exchange buffers: empty again once everybody has read them ----------------
        const unsigned slice = g.copy_bytes / (unsigned)ncta, fslice = g.fin_bytes / (unsigned)ncta;
#pragma unroll 1
        for (int l = 0; l <= g.L; ++l) {
            if (l) asm volatile("bar.sync 3, 288;" ::: "memory");      // this CTA is through the O projection of layer l (or has heard from every CTA's last layer)
            unsigned char* at = l ? g.xch + (size_t)((l - 1) & 1) * g.copy_bytes + (size_t)bid * slice : g.xch + 2 * (size_t)g.copy_bytes + (size_t)bid * fslice;
            const unsigned n = l ? slice : fslice;
#pragma unroll 1
            for (unsigned i = lane * 16u; i < n; i += 512u) *(uint4*)(at + i) = make_uint4(SC_EMPTY, SC_EMPTY, SC_EMPTY, SC_EMPTY);
            if (l == g.L) break;                                       // (the kernel's end makes these visible)
            __threadfence();
            __syncwarp();
            if (l == 0) {
                asm volatile("bar.sync 3, 288;" ::: "memory");         // the workers start
                asm volatile("bar.sync 3, 288;" ::: "memory");         // and are through the O projection
            }
            if (lane == 0) mbar_arrive(&jan_done);
        }
    } else if (warp == 11) {
        // ---------------- into L2 what the ring will ask for ----------------
        // While results go from phase to phase the ring is full and HBM would idle (7B: 10 us of a layer's 67); what is prefetched meanwhile comes in at
        // L2's rate behind the hand-over.  `ahead` copies at most beyond those requested, across projections - but into the one being requested only
        // once every CTA has requested all before it: CTAs are spread unevenly over the two dies (56 and 72 on one GPU, 60 and 68 on another), and those
        // of the emptier die would run ahead at the others' expense (7B at 1536 keys 1181 -> 1156 us).  us per step without prefetch and with: 1.1B at 512 keys
        // 590 -> 553, at 3000 683 -> 652, 7B (16 layers) at 77 keys 1142 -> 1075, from 1536 on the same within the runs' spread (1225, 1290).
        if (elect_one() && g.ahead > 0) {
            uint32_t all = ld_relaxed1(g.entered + 4 * g.L) + (uint32_t)ncta;       // the last phase's count is that of the step before
            int opened = 0;
            int idx = 0;                                // the walk's copy, of all weights
            auto prefetch = [](const void* src, uint32_t bytes) { asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory"); };
            auto turn = [&]() {                         // waits until copy idx is near enough; false: it has been requested
                if (idx < s_requested) return false;
#pragma unroll 1
                while (true) {
                    const int pr = s_requested, ph = s_phase;
                    if (idx < pr || s_quit) return false;
                    if (idx < pr + g.ahead) {
                        if (ph > opened && (int)(ld_relaxed1(g.entered + ph) - all) >= 0) opened = ph;
                        if (ph == opened) return true;
                    }
                    __nanosleep(40);
                }
            };
            int kd = GK_QKV, l = 0;
#pragma unroll 1
            while (!s_quit) {
                const int nk = s_geo[kd].nk, T = s_geo[kd].T, step = s_geo[kd].step, kps = g.k[kd].kps;
                const unsigned char* src0 = g.w[kd] + (kd == GK_LM ? 0 : (size_t)l * g.layer_step) + s_geo[kd].w_off;
#pragma unroll 1
                for (int k0 = 0; k0 < nk; k0 += SC_CHUNK, src0 += (size_t)SC_CHUNK * step) {
                    const int kn = min(SC_CHUNK, nk - k0);
#pragma unroll 1
                    for (int t = 0; t < T; ++t) {
                        const unsigned char* src = src0 + ((int)s_tile[kd][t].g0 << 10);
                        const uint32_t kb_bytes = (uint32_t)s_tile[kd][t].groups << 10, src_step = kps > 1 ? (uint32_t)kps * kb_bytes : (uint32_t)step;
#pragma unroll 1
                        for (int k = kn; k > 0; k -= kps, src += src_step, ++idx) {
                            if (turn()) prefetch(src, (uint32_t)min(k, kps) * kb_bytes);
                        }
                    }
                }
                if (kd == GK_QKV) idx += pg_st;         // the pages are left to the ring (prefetched too, 7B steps at 1536 keys took 1 % longer)
                if (kd == GK_LM) break;
                if (kd == GK_DOWN) { ++l; kd = l == g.L ? GK_LM : GK_QKV; } else ++kd;
            }
        }
        __syncwarp();
    } else {
        // ---------------- workers ----------------
        const int fw = warp - 3, ft = fw * 32 + lane, row = ft & 7;                  // worker warp and thread, its row
        const int quad = warp & 3;                                                   // a warp may only touch lanes 32 * (warp % 4) .. + 31
        const bool pushes = fw < 4;
        const int half = HD >> 1, upi = HD >> 4;
        const uint32_t red_addr = smem_u32(redbuf);
        const int VO = NV / g.C;                                                     // vectors a CTA finishes
        if (ft == 0) mbar_expect_tx(&att_full, (uint32_t)(g.C * VO * (HD * 4 + 8)));
        if (ft < 8) {
            const int slot = g.row_slot[ft];
            s_pos[ft] = g.row_pos[ft];
            s_raw[ft] = g.tree ? slot : g.row_pos[ft];
            s_slot[ft] = g.row_ok[ft] ? slot : -1;
            s_page[ft] = g.page_table[(size_t)g.row_seq[ft] * g.pages_per_seq + slot / KV_PAGE];
        }
        // A CTA's results in the order of its units over all tiles, 32 pairs each: item idx is thread idx % 256's.  The unit of an item
        // of tile t, and the features of the residual stream:
        auto unit_of = [&](int kd, int t, int idx) { return s_tile[kd][t].own_first + (idx >> 5) - s_tile[kd][t].before[rank]; };
        auto tile_of = [&](int kd, int idx) {
            int t = 0;
#pragma unroll 1
            while (t + 1 < s_geo[kd].T && (idx >> 5) >= s_tile[kd][t + 1].before[rank]) ++t;
            return t;
        };
        auto resid_feature = [&](int idx) { return unit_of(GK_O, tile_of(GK_O, idx), idx) * 8 + 2 * ((idx >> 3) & 3); };
        float2 cs0 = make_float2(0.f, 0.f), sn0 = cs0;         // the rotation of this thread's first item of QKV, the same in every layer
        if (ft < s_own[GK_QKV] * 32) {
            const int u = unit_of(GK_QKV, tile_of(GK_QKV, ft), ft);
            const size_t at = (size_t)g.row_pos[row] * half + (u % upi) * 8 + 2 * ((ft >> 3) & 3);
            cs0 = *(const float2*)(g.rope_cos + at);
            sn0 = *(const float2*)(g.rope_sin + at);
        }
        asm volatile("bar.sync 3, 288;" ::: "memory");       // (in the place of work_bar: the last layer's results are set back too)
        cluster_wait();
        pdl_wait();                                     // what the embedding left
#pragma unroll 1
        for (int idx = ft; idx < s_own[GK_O] * 32; idx += SC_WORKERS) s_x[idx] = *(const float2*)(g.x0 + (size_t)row * g.d + resid_feature(idx));

        int a_slot = 0, a_count = 0, p_st = 0;
        uint32_t a_ph = 1, p_par = 0, acc_par = 0, red_par = 0, att_par = 0;       // acc_par: a bit per tile; red_par: per region and tile
        const int st_rest = s_geo[GK_O].n_st + s_geo[GK_GU].n_st + s_geo[GK_DOWN].n_st + s_geo[GK_QKV].n_st;
        auto adv = [&](int n) {                          // stages consumed by others
            p_st += n;
            const int turns = p_st / g.stages;
            p_par ^= (uint32_t)turns & 1u;
            p_st -= turns * g.stages;
        };
        adv(s_geo[GK_QKV].n_st);
        auto gave_up = [&](unsigned i) {                // a poll that lasts: has anybody failed?
            if ((i & 255u) != 255u) return false;
            if (*abortp || *(volatile int*)g.err || i >= SC_POLL_LIMIT) { *abortp = 1; *(volatile int*)g.err = SC_ERR_TIMEOUT; return true; }
            return false;
        };

        // this CTA's k-blocks of an operand image, as the other CTAs write it, into the activation slots
        auto load_acts = [&](const unsigned char* img, int kd) {
            const int nk = s_geo[kd].nk, kb_lo = s_geo[kd].kb_lo, K = g.k[kd].K;
#pragma unroll 1
            for (int k0 = 0; k0 < nk; k0 += SC_AKB) {
                if (a_count >= SC_ACT_SLOTS) sc_wait(&a_empty[a_slot], a_ph, stuckp);
                const int chunks = min(SC_AKB, nk - k0) * 128;                       // of 16 bytes
                const unsigned char* src = img + (size_t)(kb_lo + k0) * (rows * 256) + ft * 16;
                unsigned char* dst = abuf + a_slot * SC_ACT_SLOT + ft * 16;
                uint4 v[4];
                uint32_t todo = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    v[j] = make_uint4(0u, 0u, 0u, 0u);
                    const int c = ft + j * SC_WORKERS;
                    // columns behind the last input meet zero weights: nobody writes them, they are zero here
                    if (c < chunks && (kb_lo + k0 + (c >> 7)) * 64 + (((c & 7) ^ ((c >> 3) & 7)) << 3) < K) todo |= 1u << j;
                }
#pragma unroll 1
                for (unsigned i = 0; todo; ++i) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) if (todo >> j & 1u) v[j] = ld_relaxed4(src + j * (SC_WORKERS * 16));
#pragma unroll
                    for (int j = 0; j < 4; ++j) if ((todo >> j & 1u) && here(v[j])) todo &= ~(1u << j);
                    if (gave_up(i)) break;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) if (ft + j * SC_WORKERS < chunks) *(uint4*)(dst + j * (SC_WORKERS * 16)) = v[j];
                fence_async_cta();
                __syncwarp();
                if (lane == 0) mbar_arrive(&a_full[a_slot]);
                ++a_count;
                if (++a_slot == SC_ACT_SLOTS) { a_slot = 0; a_ph ^= 1u; }
            }
        };

        auto attention = [&](int l, unsigned char* copy) {
            unsigned char* Qs = abuf + Cfg::SLOTS;
            float* sm_o = (float*)abuf;                                              // [warp][NV][OP]
            const int gid = lane >> 2, t = lane & 3;
            const unsigned char *qsrc = copy + g.o_q, *kvsrc = copy + g.o_kv;
            // the queries, and the step's own keys and values where this CTA has a page that holds them
            const int first_new = min(s_raw[0], s_raw[rows - 1]) / KV_PAGE;
            const bool own_new = my_pages > 0 && arank + (my_pages - 1) * g.C >= first_new;
            uint4 vnew;
            const int which = ft / HD, nr = (ft % HD) / (HD / 8), nc = (ft % HD) % (HD / 8);      // K or V, row, 16-byte chunk
            const bool has_q = ft < 2 * NV * (HD / 8), has_n = own_new && ft < 2 * HD;
            {
                const int qrow = ft / (HD / 8), c = ft % (HD / 8), vec = qrow & (NV - 1), term = qrow >= NV ? 1 : 0;
                const unsigned char* qp = qsrc + (((size_t)hv * 2 + term) * rows + vec) * (HD * 2) + c * 16;
                const unsigned char* np = kvsrc + (((size_t)kvh * 2 + which) * rows + nr) * (HD * 2) + nc * 16;
                uint4 vq = make_uint4(0u, 0u, 0u, 0u), vn = vq;
                bool tq = has_q, tn = has_n;
#pragma unroll 1
                for (unsigned i = 0; tq || tn; ++i) {
                    if (tq) vq = ld_relaxed4(qp);
                    if (tn) vn = ld_relaxed4(np);
                    if (tq && here(vq)) tq = false;
                    if (tn && here(vn)) tn = false;
                    if (gave_up(i)) break;
                }
                if (has_q) *(uint4*)(Qs + qrow * QP + c * 16) = vq;
            vnew = vn;
            }
            const int qpos = g.tree ? s_raw[gid] : pos_lo + gid, qhl = g.tree ? g.hole_lo[gid] : 0, qhh = g.tree ? g.hole_hi[gid] : 0;       // of this thread's row
            work_bar();
            // lane offsets of the ldmatrix addresses: matrix (lane / 8) of four
            const int mi = lane >> 3, lr = lane & 7;
            const uint32_t q_addr = smem_u32(Qs) + (uint32_t)((lr + 8 * (mi & 1)) * QP + (mi >> 1) * 16);
            const uint32_t kv_off = (uint32_t)((lr + 8 * (mi >> 1)) * 128), chunk0 = (uint32_t)(mi & 1);
            const uint32_t ring_addr = smem_u32(ring);
            const int key_page = fw * 16;

            float m_run = -CUDART_INF_F, l_run = 0.0f, o[DT][4];
#pragma unroll
            for (int d = 0; d < DT; ++d) { o[d][0] = 0.f; o[d][1] = 0.f; o[d][2] = 0.f; o[d][3] = 0.f; }
#pragma unroll 1
            for (int p = arank; p < n_pages; p += g.C) {
                const int st0 = p_st;                   // the page's stages, and their parities
                const uint32_t par0 = p_par;
                auto st = [&](int s) { return st0 + s >= g.stages ? st0 + s - g.stages : st0 + s; };
                auto par = [&](int s) { return st0 + s >= g.stages ? par0 ^ 1u : par0; };
                p_par = par(2 * KST);
                p_st = st(2 * KST);
#pragma unroll
                for (int s = 0; s < KST; ++s) sc_wait(&w_full[st(s)], par(s), stuckp);
                const int vs = HD == 128 ? KST + (key_page >> 6) : KST;
                if (p >= first_new) {                   // the cache's page is from before this step: the step's own rows go in here
#pragma unroll
                    for (int s = KST; s < 2 * KST; ++s) sc_wait(&w_full[st(s)], par(s), stuckp);
                    const int slot = s_slot[nr];
                    if (has_n && slot >= 0 && slot / KV_PAGE == p) {
                        const int at = slot % KV_PAGE, box = at >> 6;
                        if (which == 0) *(uint4*)(ring + st(KST == 2 && (nc >> 3) ? KST - 1 : 0) * SC_STAGE + at * 128 + (((nc & 7) ^ (at & 7)) << 4)) = vnew;
                        else {
                            unsigned char* vb = ring + st(KST == 2 && box ? 2 * KST - 1 : KST) * SC_STAGE + (KST == 2 ? 0 : box * (HD * 128)) + (at & 7) * 2;
                            const uint32_t e[4] = {vnew.x, vnew.y, vnew.z, vnew.w};
#pragma unroll
                            for (int i = 0; i < 8; ++i) *(unsigned short*)(vb + (nc * 8 + i) * 128 + ((((at & 63) >> 3) ^ i) << 4)) = (unsigned short)(e[i >> 1] >> (16 * (i & 1)));
                        }
                    }
                    fence_async_cta();                  // before a later copy into these stages
                    work_bar();
                }
                const int vst = st(vs);
                const uint32_t vpar = par(vs);
                if (p * KV_PAGE + key_page <= pos_hi) {
                    // two chains of products, added at the end: even and odd steps
                    float c[2][4], c2[2][4];
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int e = 0; e < 4; ++e) { c[j][e] = 0.f; c2[j][e] = 0.f; }
#pragma unroll
                    for (int k = 0; k < KS; ++k) {
                        uint32_t b[4], a[4];
                        const uint32_t kr = ring_addr + (uint32_t)st(k >> 2) * SC_STAGE + kv_off + (uint32_t)key_page * 128u;
                        ad_ldm4(kr + ((((uint32_t)((k & 3) * 2) + chunk0) ^ (uint32_t)lr) << 4), b);
                        ad_ldm4(q_addr + (uint32_t)(k * 32), a);
                        ad_mma(k & 1 ? c2[0] : c[0], a, b[0], b[1]);
                        ad_mma(k & 1 ? c2[1] : c[1], a, b[2], b[3]);
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int e = 0; e < 4; ++e) c[j][e] += c2[j][e];
                    __syncwarp();
                    if (lane == 0) {
#pragma unroll
                        for (int s = 0; s < KST; ++s) mbar_arrive(&w_empty[st(s)]);
                    }
                    float w[2][2], mx = -CUDART_INF_F;
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int key = p * KV_PAGE + key_page + 8 * j + 2 * t + e;
                            w[j][e] = (key <= qpos && !(key >= qhl && key < qhh)) ? c[j][e] + c[j][2 + e] : -CUDART_INF_F;
                            mx = fmaxf(mx, w[j][e]);
                        }
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                    const float m_new = fmaxf(m_run, mx);
                    const bool none = m_new == -CUDART_INF_F;
                    const float resc = none ? 1.0f : exp2f(m_run - m_new);
                    float wsum = 0.0f;
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int e = 0; e < 2; ++e) { w[j][e] = none ? 0.0f : exp2f(w[j][e] - m_new); wsum += w[j][e]; }
                    l_run = l_run * resc + wsum;                    // this lane's keys; the four lanes of a row are added at the end
                    m_run = m_new;
                    uint32_t ph[4];                                 // rows gid: hi terms, rows gid + 8: lo terms
#pragma unroll
                    for (int j = 0; j < 2; ++j) ph[2 * j] = ad_split(w[j][0], w[j][1], ph[2 * j + 1]);
                    if (__any_sync(0xffffffffu, resc != 1.0f)) {    // multiplying by 1 changes nothing
#pragma unroll
                        for (int d = 0; d < DT; ++d) { o[d][0] *= resc; o[d][1] *= resc; o[d][2] *= resc; o[d][3] *= resc; }
                    }
                    sc_wait(&w_full[vst], vpar, stuckp);
                    const uint32_t vr = ring_addr + (uint32_t)vst * SC_STAGE + kv_off + (HD == 128 ? 0u : (uint32_t)((key_page >> 6) * (HD * 128))) + ((((uint32_t)((key_page & 63) >> 3) + chunk0) ^ (uint32_t)lr) << 4);
#pragma unroll
                    for (int d = 0; d < DT / 2; ++d) {
                        uint32_t b[4];
                        ad_ldm4(vr + (uint32_t)(d * 16 * 128), b);
                        ad_mma(o[2 * d], ph, b[0], b[1]);
                        ad_mma(o[2 * d + 1], ph, b[2], b[3]);
                    }
                } else {
                    if (lane == 0) {
#pragma unroll
                        for (int s = 0; s < KST; ++s) mbar_arrive(&w_empty[st(s)]);
                    }
                    sc_wait(&w_full[vst], vpar, stuckp);
                }
                // only the stage that this warp has waited for: it counts towards the phase of this page, whatever lay there before
                __syncwarp();
                if (lane == 0) mbar_arrive(&w_empty[vst]);
            }
            // ---- the warps, in order ----
            l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
            l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
            if (t == 0) { sm_m[fw * NV + gid] = m_run; sm_l[fw * NV + gid] = l_run; }
            float* mine = sm_o + (size_t)fw * NV * OP;
#pragma unroll
            for (int d = 0; d < DT; ++d) *(float2*)(mine + gid * OP + 8 * d + 2 * t) = make_float2(o[d][0] + o[d][2], o[d][1] + o[d][3]);
            work_bar();
            // the result, as hi + lo terms in the O projection's operand image
            unsigned char* img = copy + g.o_ao;
            auto store = [&](int vec, int d4, float l_, float4 a) {
                const int k = hv * HD + 4 * d4;
                uint2 hi, lo;
                hi.x = ad_split(a.x / l_, a.y / l_, lo.x);
                hi.y = ad_split(a.z / l_, a.w / l_, lo.y);
                st_relaxed2(img + cl_img_offset(rows, vec, k), hi);
                st_relaxed2(img + cl_img_offset(rows, rows + vec, k), lo);
            };
#pragma unroll 1
            for (int idx = ft; idx < NV * V4; idx += SC_WORKERS) {
                const int vec = idx / V4, d4 = idx % V4;
                float mx = -CUDART_INF_F;
#pragma unroll
                for (int w = 0; w < WARPS; ++w) mx = fmaxf(mx, sm_m[w * NV + vec]);
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                float lsum = 0.0f;
#pragma unroll
                for (int w = 0; w < WARPS; ++w) {
                    const float m = sm_m[w * NV + vec], s = m == -CUDART_INF_F ? 0.0f : exp2f(m - mx);
                    const float4 x = *(const float4*)(sm_o + (size_t)(w * NV + vec) * OP + 4 * d4);
                    a.x = fmaf(x.x, s, a.x); a.y = fmaf(x.y, s, a.y); a.z = fmaf(x.z, s, a.z); a.w = fmaf(x.w, s, a.w);
                    lsum = fmaf(sm_l[w * NV + vec], s, lsum);
                }
                if (g.C == 1) { store(vec, d4, lsum, a); continue; }
                const int owner = vec / VO, at = arank * VO + vec % VO;
                const uint32_t cta = (uint32_t)(rank - arank + owner), bar = map_to_cta(smem_u32(&att_full), cta);
                st_async4(map_to_cta(smem_u32(recv + at * HD + 4 * d4), cta), bar, a.x, a.y, a.z, a.w);
                if (d4 == 0) st_async2(map_to_cta(smem_u32(&rc[at]), cta), bar, mx, lsum);
            }
            if (g.C > 1) {
                sc_wait_cluster(&att_full, att_par, abortp, g.err);
                att_par ^= 1u;
                if (ft == 0 && l + 1 < g.L && !*abortp) mbar_expect_tx(&att_full, (uint32_t)(g.C * VO * (HD * 4 + 8)));
#pragma unroll 1
                for (int idx = ft; idx < VO * V4; idx += SC_WORKERS) {
                    const int vo = idx / V4, d4 = idx % V4;
                    float m = -CUDART_INF_F, lsum = 0.0f;
                    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                    for (int k = 0; k < g.C; ++k)
                        ad_fold(m, lsum, a, rc[k * VO + vo].x, rc[k * VO + vo].y, *(const float4*)(recv + (k * VO + vo) * HD + 4 * d4));
                    store(arank * VO + vo, d4, lsum, a);
                }
            }
            work_bar();                                  // the activations go where the warps' results were
        };

        int kd = GK_QKV, l = 0;
#pragma unroll 1
        while (true) {
            unsigned char *copy = g.xch + (size_t)(l & 1) * g.copy_bytes, *prev = g.xch + (size_t)((l - 1) & 1) * g.copy_bytes, *fin = g.xch + 2 * (size_t)g.copy_bytes;
            if (kd == GK_O) {
                if (att) attention(l, copy);
                adv(st_rest);
            }
            const int T = s_geo[kd].T, shift = g.k[kd].shift, f_own_max = g.k[kd].f_own_max, pack = g.k[kd].pack;
            const bool resid = kd == GK_O || kd == GK_DOWN;
            const int region = resid ? 1 : 0;
            float2 gn = make_float2(0.f, 0.f);
            const float* gain = nullptr;
            if (resid) {
                gain = kd == GK_O ? (const float*)((const char*)g.ffn_norm + (size_t)l * g.layer_step) : l + 1 < g.L ? (const float*)((const char*)g.attn_norm + (size_t)(l + 1) * g.layer_step) : g.final_norm;
                if (ft < s_own[kd] * 32) gn = *(const float2*)(gain + resid_feature(ft));
            }
            if (ft < T && !*abortp) {                    // what the cluster will send here for each tile
                const int n = s_tile[kd][ft].own_n;
                mbar_expect_tx(&red_full[region][ft], (uint32_t)(n ? (n << shift) * CC * pack * 32 : CC * 16));
            }
            load_acts(kd == GK_QKV ? (l ? prev : g.img0) : kd == GK_LM ? fin : copy + (kd == GK_O ? g.o_ao : kd == GK_GU ? g.o_h2 : g.o_act), kd);
            // 1 / RMS of every row: a warp per row, 32 interleaved sums over the parts, then a tree over the lanes
            if (!resid) {
                float s = 0.0f;
                if (kd == GK_QKV && l == 0) s = lane == 0 ? g.ss0[fw] : 0.0f;
                else {
                    const unsigned char* src = (kd == GK_LM ? fin + g.o_fss : kd == GK_QKV ? prev + g.o_ssa : copy + g.o_ssb) + ((size_t)fw * ncta + lane) * 4;
                    uint32_t v[4];
                    uint32_t todo = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) if (lane + 32 * j < ncta) todo |= 1u << j;
                    const uint32_t mine = todo;
#pragma unroll 1
                    for (unsigned i = 0; todo; ++i) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) if (todo >> j & 1u) v[j] = ld_relaxed1(src + j * 128);
#pragma unroll
                        for (int j = 0; j < 4; ++j) if ((todo >> j & 1u) && v[j] != SC_EMPTY) todo &= ~(1u << j);
                        if (gave_up(i)) break;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) if (mine >> j & 1u) s += __uint_as_float(v[j]);
                }
#pragma unroll 1
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) s_rstd[fw] = rsqrtf(s * g.inv_d + g.eps);
            }
            if (!resid) work_bar();                      // the rows' 1 / RMS
            if (kd == GK_LM) asm volatile("bar.arrive 3, 288;" ::: "memory");        // (whose parts come from every CTA's last result)
            // the buffers of the layer before are empty again before anything that the next layer waits for leaves this CTA
            if (kd == GK_DOWN) sc_wait(&jan_done, (uint32_t)l & 1u, stuckp);
            const float* red = (const float*)(redbuf + g.k[kd].red);
            const int part_step = f_own_max * 8;
            auto sum = [&](int f) {                      // feature f of this CTA's share, this thread's row, parts in CTA order
                const float* s = red + f * 8 + row;
                return ((s[0] + s[part_step]) + s[2 * part_step]) + s[3 * part_step];
            };
            // Tile by tile: this CTA's sums go to whoever finishes the features, as soon as the products are through; then it finishes its own of
            // the tile before, whose parts have come in meanwhile.
            float ssq = 0.0f, best = -CUDART_INF_F;
            int bidx = 0x7fffffff;
            unsigned char* act = kd == GK_O ? copy + g.o_h2 : kd == GK_GU ? copy + g.o_act : l + 1 < g.L ? copy : fin;
            const float rs = resid ? 1.0f : s_rstd[row];
            auto finish = [&](int t) {
                const int lo = s_tile[kd][t].before[rank] * (kd == GK_LM ? 64 : 32), hi_ = lo + s_tile[kd][t].own_n * (kd == GK_LM ? 64 : 32);
                sc_wait_cluster(&red_full[region][t], (red_par >> (region * SC_MAX_TILES + t)) & 1u, abortp, g.err);
#pragma unroll 1
                for (int idx = lo + ((ft - lo) & (SC_WORKERS - 1)); idx < hi_; idx += SC_WORKERS) {
                    if (resid) {
                        const int f = 2 * (idx >> 3), n = unit_of(kd, t, idx) * 8 + (f & 7);
                        if (idx != ft) gn = *(const float2*)(gain + n);
                        float2 x = s_x[idx];
                        float2 v = make_float2(sum(f), sum(f + 1));
#pragma unroll 1
                        for (int q = 1; q < pack; ++q) { v.x += sum(f + q * CC * f_own_max); v.y += sum(f + 1 + q * CC * f_own_max); }
                        x.x += v.x; x.y += v.y;
                        s_x[idx] = x;
                        ssq += x.x * x.x + x.y * x.y;
                        uint32_t hi, lo2;
                        split2(x.x * gn.x, x.y * gn.y, hi, lo2);
                        st_relaxed1(act + cl_img_offset(rows, row, n), hi);
                        st_relaxed1(act + cl_img_offset(rows, rows + row, n), lo2);
                    } else if (kd == GK_GU) {
                        const int e = 2 * ((idx >> 3) & 3), f = (idx >> 5) * 16 + e, k = unit_of(kd, t, idx) * 8 + e;
                        float v[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float gte = sum(f + h) * rs, upv = sum(f + 8 + h) * rs;
                            v[h] = gte / (1.0f + expf(-gte)) * upv;
                        }
                        uint32_t hi, lo2;
                        split2(v[0], v[1], hi, lo2);
                        st_relaxed1(act + cl_img_offset(rows, row, k), hi);
                        st_relaxed1(act + cl_img_offset(rows, rows + row, k), lo2);
                    } else if (kd == GK_QKV) {
                        const int ul = idx >> 5, e = 2 * ((idx >> 3) & 3), u = unit_of(kd, t, idx), head = u / upi, i = (u - head * upi) * 8 + e;
                        float a[2], b[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) { a[h] = sum(ul * 16 + e + h) * rs; b[h] = sum(ul * 16 + 8 + e + h) * rs; }
                        if (head < g.Hq + g.Hkv) {
                            float2 cs = cs0, sn = sn0;
                            if (idx != ft) {
                                const size_t at = (size_t)s_pos[row] * half + i;
                                cs = *(const float2*)(g.rope_cos + at);
                                sn = *(const float2*)(g.rope_sin + at);
                            }
                            const float a0 = a[0] * cs.x - b[0] * sn.x, b0 = b[0] * cs.x + a[0] * sn.x;
                            const float a1 = a[1] * cs.y - b[1] * sn.y, b1 = b[1] * cs.y + a[1] * sn.y;
                            a[0] = a0; b[0] = b0; a[1] = a1; b[1] = b1;
                        }
                        if (head < g.Hq) {
                            // queries leave as two bf16 terms, already multiplied by log2(e) / sqrt(hd): [head][term][row][dim]
                            unsigned char* q = copy + g.o_q + ((size_t)(head * 2) * rows + row) * (HD * 2) + i * 2;
                            uint32_t hi, lo2;
                            split2(a[0] * g.q_scale, a[1] * g.q_scale, hi, lo2);
                            st_relaxed1(q, hi); st_relaxed1(q + rows * HD * 2, lo2);
                            split2(b[0] * g.q_scale, b[1] * g.q_scale, hi, lo2);
                            st_relaxed1(q + half * 2, hi); st_relaxed1(q + rows * HD * 2 + half * 2, lo2);
                        } else {
                            const bool is_k = head < g.Hq + g.Hkv;
                            const int kh = is_k ? head - g.Hq : head - g.Hq - g.Hkv, slot = s_slot[row];
                            const __nv_bfloat162 va = __floats2bfloat162_rn(a[0], a[1]), vb = __floats2bfloat162_rn(b[0], b[1]);
                            // for this step's attention [kv head][K, V][row][dim], and into the cache for later ones
                            unsigned char* n = copy + g.o_kv + ((size_t)(kh * 2 + (is_k ? 0 : 1)) * rows + row) * (HD * 2) + i * 2;
                            st_relaxed1(n, *(const uint32_t*)&va); st_relaxed1(n + half * 2, *(const uint32_t*)&vb);
                            if (slot >= 0) {
                                bf16* pg = (is_k ? g.kpool : g.vpool) + (((size_t)l * g.total_pages + s_page[row]) * g.Hkv + kh) * KV_PAGE * HD;
                                if (is_k) {                                   // K page: [position][dim]
                                    bf16* at = pg + (size_t)(slot % KV_PAGE) * HD + i;
                                    *(__nv_bfloat162*)at = va;
                                    *(__nv_bfloat162*)(at + half) = vb;
                                } else {                                      // V page, transposed: [dim][position]
                                    bf16* at = pg + (size_t)i * KV_PAGE + (slot % KV_PAGE);
                                    at[0] = va.x;
                                    at[KV_PAGE] = va.y;
                                    at[(size_t)half * KV_PAGE] = vb.x;
                                    at[(size_t)(half + 1) * KV_PAGE] = vb.y;
                                }
                            }
                        }
                    } else {                                                   // vocabulary: a unit is 64 items
                        const int f = idx >> 3, n = (s_tile[kd][t].own_first + (idx >> 6) - s_tile[kd][t].before[rank]) * 8 + (f & 7);
                        if (n >= g.n_out) continue;
                        const float v = sum(f) * rs;
                        if (g.out) g.out[(size_t)row * g.n_out + n] = v;
                        if (v > best) { best = v; bidx = n; }                   // ascending n: strict > keeps the lowest id
                    }
                }
            };
#pragma unroll 1
            for (int t = 0; t <= T; ++t) {
                if (t < T) {
                    // thread: a feature (tensor-memory lane) and four of the rows
                    // (packed: the lanes of the second k-block's rows hold the same features' sums over other k-blocks, in columns of their own)
                    const int lanes = (int)s_tile[kd][t].groups * 8, part = pack > 1 ? quad * 32 / lanes : 0;
                    const int un = s_tile[kd][t].groups >> (shift - 3), pos = quad * 32 + lane - part * lanes, u = pos >> shift;
                    const int b1 = un / 4, b2 = un / 2, b3 = 3 * un / 4, q = (u >= b1) + (u >= b2) + (u >= b3), owner = (q - t) & (CC - 1);
                    const int local = ((s_tile[kd][t].before[owner] + u - (q * un) / CC) << shift) + (pos & ((1 << shift) - 1));
                    const bool send = !*abortp;
                    sc_wait(&acc_full[t], (acc_par >> t) & 1u, stuckp);
                    tc_fence_after();
                    float v[4];
                    const uint32_t col = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)((t + part) * 2 * rows + (pushes ? 0 : 4));
                    tc_ld4_sum(col, col + 8u, v);
                    const uint32_t bar0 = smem_u32(&red_full[region][t]), to = red_addr + (uint32_t)(g.k[kd].red + ((part * CC + rank) * f_own_max + local) * 32 + (pushes ? 0 : 16));
                    if (pos < lanes && send) st_async4(map_to_cta(to, (uint32_t)owner), map_to_cta(bar0, (uint32_t)owner), v[0], v[1], v[2], v[3]);
                    // a CTA that finishes nothing of the tile hears from the others all the same: it is then behind them
                    if (ft < CC && send && (ft + 1) * un / CC == ft * un / CC) {
                        const uint32_t o = (uint32_t)((ft - t) & (CC - 1));
                        st_async4(map_to_cta(red_addr + (uint32_t)(g.k[kd].red + rank * 16), o), map_to_cta(bar0, o), 0.f, 0.f, 0.f, 0.f);
                    }
                    tc_fence_before();
                }
                if (t > 0) finish(t - 1);
            }
            acc_par ^= (1u << T) - 1u;
            red_par ^= ((1u << T) - 1u) << (region * SC_MAX_TILES);
            if (resid) {
                // the row's sum of squares over this CTA's features: one part
                ssq += __shfl_xor_sync(0xffffffffu, ssq, 8);
                ssq += __shfl_xor_sync(0xffffffffu, ssq, 16);
                if (lane < 8) s_part[fw][lane] = ssq;
                work_bar();
                if (ft < 8) {
                    float s = s_part[0][ft];
#pragma unroll
                    for (int w = 1; w < 8; ++w) s += s_part[w][ft];
                    unsigned char* ss = kd == GK_O ? copy + g.o_ssb : l + 1 < g.L ? copy + g.o_ssa : fin + g.o_fss;
                    st_relaxed1(ss + ((size_t)ft * ncta + bid) * 4, __float_as_uint(s));
                }
                if (kd == GK_O) asm volatile("bar.arrive 3, 288;" ::: "memory");
            } else if (kd == GK_LM) {
#pragma unroll 1
                for (int o = 8; o <= 16; o <<= 1) {
                    const float ov = __shfl_xor_sync(0xffffffffu, best, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
                    if (ov > best || (ov == best && oi < bidx)) { best = ov; bidx = oi; }
                }
                if (lane < 8) { s_part[fw][lane] = best; s_idx[fw][lane] = bidx; }
                work_bar();
                if (ft < 8) {
                    best = s_part[0][ft]; bidx = s_idx[0][ft];
                    for (int w = 1; w < 8; ++w)
                        if (s_part[w][ft] > best || (s_part[w][ft] == best && s_idx[w][ft] < bidx)) { best = s_part[w][ft]; bidx = s_idx[w][ft]; }
                    g.amax_val[(size_t)ft * ncta + bid] = best;
                    g.amax_idx[(size_t)ft * ncta + bid] = bidx;
                }
                break;
            }
            if (kd == GK_DOWN) { ++l; kd = l == g.L ? GK_LM : GK_QKV; } else ++kd;
        }
    }

    // Leaving: nothing is under way to a CTA that is through its last epilogue; the barrier only keeps a CTA whose wait ran out from leaving
    // under the others.
    if (warp < 3 || warp == 11) cluster_wait();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)g.tmem_cols) : "memory");
    }
    if (threadIdx.x == 0 && (abort_flag || stuck_flag)) {
        // gave up: let every copy already issued land before the CTA may exit
#pragma unroll 1
        for (int i = max(0, s_issued - g.stages); i < s_issued; ++i)
#pragma unroll 1
            for (unsigned spin = 0; spin < WAIT_LIMIT && !mbar_try_wait(&w_full[i % g.stages], (uint32_t)((i / g.stages) & 1)); ++spin) {}
        atomicExch(g.err, SC_ERR_TIMEOUT);
#pragma unroll 1
        for (int i = 0; i < 20; ++i) __nanosleep(20000);        // ... and what went to the cluster's other CTAs, for which nobody may be waiting, arrive
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
}

template <int HD>
anpd_status launch_step_cl(const anpd_kv* kv, const ScArgs& g, int smem, cudaStream_t st, Profiler* prof) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g.ncl * CL_CTAS); cfg.blockDim = dim3(SC_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[3];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL_CTAS; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;           // its CTAs wait for one another: all of them run, or none
    attr[1].val.cooperative = 1;
    attr[2].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[2].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (g_use_pdl && !t_no_pdl) ? 3 : 2;
    LAUNCH(prof, st, KC_GEMM, kv->m->streamed_bytes, (cudaLaunchKernelEx(&cfg, step_cl_kernel<HD>, kv->map_k, kv->map_v, g)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

// The kernel's function attributes on the current device, and whether the device holds all of its CTAs at once.  The limit of shared memory
// is the function's, for the handles of all models: the bound of every shape's need, so that no handle takes it from another.
template <int HD>
bool fits_step_cl(int ncl, int smem) {
    if (cudaFuncSetAttribute(step_cl_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, SC_SMEM) != cudaSuccess) { cudaGetLastError(); return false; }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ncl * CL_CTAS); cfg.blockDim = dim3(SC_THREADS); cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL_CTAS; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, step_cl_kernel<HD>, &cfg) != cudaSuccess) { cudaGetLastError(); return false; }
    return n >= ncl;
}

// Everything but the caller's pointers; the shared memory it takes.  False: the shape is not one for this kernel.
bool sc_args(const anpd_model* m, ScArgs* g, int* smem) {
    const anpd_model_config& c = m->cfg;
    *g = ScArgs{};
    g->ncl = m->cl[GK_QKV].ncl;
    const int ncta = g->ncl * CL_CTAS;
    int tiles_max = 1, red[2] = {0, 0};
#pragma unroll 1
    for (int k = 0; k < GK_COUNT; ++k) {
        const ClPlan& p = m->cl[k];
        ScKind& s = g->k[k];
        // every cluster has features to finish and every CTA k-blocks to multiply: nobody runs ahead of the exchange (see the kernel)
        if (p.n_units < g->ncl || p.kb < CL_CTAS) return false;
        const int groups = p.u_max * p.gpu, tiles = (groups + 15) / 16;
        if (tiles > SC_MAX_TILES) return false;
        s.kb = p.kb; s.gpu = p.gpu; s.n_units = p.n_units; s.seg = p.seg; s.tiles = tiles; s.K = p.K;
        s.kps = tiles == 1 && p.seg == p.ncl ? std::max(1, std::min(4, 16 / groups)) : 1;
        if (s.kps == 3) s.kps = 2;                       // a stage never straddles two activation slots
        if (tiles > 1 && p.n_units / g->ncl < tiles * CL_CTAS) return false;              // every CTA finishes units of every tile
        // the most units a CTA finishes, of the smaller and of the larger clusters
        int own_max = 0;
#pragma unroll 1
        for (int Uc = p.n_units / g->ncl; Uc <= p.u_max; ++Uc)
#pragma unroll 1
            for (int r = 0; r < CL_CTAS; ++r) {
                int own = 0;
#pragma unroll 1
                for (int t = 0; t < tiles; ++t) { const int un = sc_tile_units(Uc, tiles, t), q = (r + t) % CL_CTAS; own += (q + 1) * un / CL_CTAS - q * un / CL_CTAS; }
                own_max = std::max(own_max, own);
            }
        s.f_own_max = own_max * 8 * p.gpu;
        s.shift = p.gpu == 2 ? 4 : 3;
        // a stage's k-blocks fill whole warps' lanes, in every cluster alike, and every CTA has a full stage of them
        s.pack = (k == GK_O || k == GK_DOWN) && s.kps > 1 && p.n_units % g->ncl == 0 && groups % 4 == 0 && groups * s.kps <= 16 && p.kb >= CL_CTAS * s.kps ? s.kps : 1;
        s.red = k == GK_O || k == GK_DOWN ? 1 : 0;
        red[s.red] = std::max(red[s.red], CL_CTAS * s.pack * s.f_own_max * 32);
        tiles_max = std::max(tiles_max, tiles * s.pack);
    }
#pragma unroll 1
    for (int k = 0; k < GK_COUNT; ++k) g->k[k].red = g->k[k].red ? red[0] : 0;
    g->red_bytes = red[0] + red[1];
    g->tmem_cols = 32;
#pragma unroll 1
    while (g->tmem_cols < tiles_max * 2 * ANPD_ROWS) g->tmem_cols <<= 1;
    const int rest = SC_ACT_SLOTS * SC_ACT_SLOT + g->red_bytes + g->k[GK_O].f_own_max / 8 * 32 * (int)sizeof(float2) + 1024;
    g->stages = std::min(SC_MAX_STAGES, (SC_SMEM - rest) / SC_STAGE);
    if (g->stages < 5) return false;                     // a page and a stage of weights
    *smem = rest + g->stages * SC_STAGE;
    // How far the prefetch reaches, in copies: half a layer's, at most 24 (50 MB for all CTAs).  us per step with none, 16,
    // 24, 32 and 48: 1.1B (47 copies a layer and CTA) 592, 550, 553, 562, 662; 7B, 16 layers (203) 1136, 1055, 1043, 1034, 1035; 13B, 8 layers (368)
    // 903, 888, 870, 861, 865; 7B at 3000 keys 1287, -, 1290, 1320 (there the pages take what the prefetch takes).  A layer of less than 28 copies, three to four rings full, is better off without: 1280 wide (25) 227 -> 230, 1024 wide
    // (16) 263 -> 273, but 1536 wide (29) 262 -> 258.
    int copies = 0;
#pragma unroll 1
    for (int k = 0; k < GK_LM; ++k) {
        const int nk = (g->k[k].kb + CL_CTAS - 1) / CL_CTAS;
        copies += g->k[k].tiles == 1 ? (nk + g->k[k].kps - 1) / g->k[k].kps : nk * g->k[k].tiles;
    }
    g->ahead = copies < 28 ? 0 : std::min(24, copies / 2);
    g->L = c.n_layers; g->d = c.d_model; g->Hq = c.n_q_heads; g->Hkv = c.n_kv_heads; g->n_out = c.vocab;
    g->inv_d = 1.0f / (float)c.d_model; g->eps = c.rms_eps; g->q_scale = 1.4426950408889634f / sqrtf((float)c.head_dim);
    // the layers' tensors lie at one distance
    const LayerW& w = m->layers[0];
    g->w[GK_QKV] = w.wqkv; g->w[GK_O] = w.wo; g->w[GK_GU] = w.wgu; g->w[GK_DOWN] = w.wd; g->w[GK_LM] = m->lm_head;
    g->attn_norm = w.attn_norm; g->ffn_norm = w.ffn_norm; g->final_norm = m->final_norm;
    if (c.n_layers > 1) g->layer_step = (size_t)(m->layers[1].wqkv - w.wqkv);
#pragma unroll 1
    for (int l = 1; l < c.n_layers; ++l) {
        const LayerW& v = m->layers[l];
        const size_t at = (size_t)l * g->layer_step;
        if (v.wqkv != w.wqkv + at || v.wo != w.wo + at || v.wgu != w.wgu + at || v.wd != w.wd + at || (const char*)v.attn_norm != (const char*)w.attn_norm + at ||
            (const char*)v.ffn_norm != (const char*)w.ffn_norm + at) return false;
    }
    g->split = c.n_q_heads / c.n_kv_heads;
    g->items = c.n_q_heads;
    g->C = ad_cluster(m, g->items);
    if (g->items * g->C > ncta) return false;
    // exchange buffers
    auto up = [](size_t v, size_t to) { return (v + to - 1) / to * to; };
    const size_t ss = up((size_t)ncta * ANPD_ROWS * 4, 256), qrow = (size_t)2 * ANPD_ROWS * c.head_dim * 2;
    size_t at = cl_img_bytes(ANPD_ROWS, c.d_model);
    g->o_fss = (unsigned)at;
    g->fin_bytes = (unsigned)up(at + ss, (size_t)ncta * 16);
    auto put = [&](unsigned* o, size_t bytes) { *o = (unsigned)at; at += bytes; };
    put(&g->o_h2, cl_img_bytes(ANPD_ROWS, c.d_model)); put(&g->o_ao, cl_img_bytes(ANPD_ROWS, m->dq)); put(&g->o_act, cl_img_bytes(ANPD_ROWS, c.d_ffn));
    put(&g->o_q, c.n_q_heads * qrow); put(&g->o_kv, c.n_kv_heads * qrow); put(&g->o_ssa, ss); put(&g->o_ssb, ss);
    g->copy_bytes = (unsigned)up(at, (size_t)ncta * 16);
    return true;
}


}  // namespace

size_t step_cl_bytes(const anpd_model* m, int batch) {
    ScArgs g;
    int smem = 0;
    if (batch != 1 || !m->cl_all_fused || m->plain_gemm || !sc_args(m, &g, &smem)) return 0;
    // NV_COMPUTE_PROFILER_PERFWORKS_DIR: set for programs that run under Nsight Compute.  Its capture of one launch of this kernel (cooperative,
    // in clusters; 2025.2.1, driver 580.159) had not ended after ten minutes, where the same program alone takes seconds; the cause is not known.
    if (std::getenv("ANPD_STEP_CHAIN") || std::getenv("NV_COMPUTE_PROFILER_PERFWORKS_DIR")) return 0;
    const bool ok = m->cfg.head_dim == 128 ? fits_step_cl<128>(g.ncl, smem) : fits_step_cl<64>(g.ncl, smem);
    return ok ? 2 * (size_t)g.copy_bytes + g.fin_bytes + 4 * (4 * (size_t)g.L + 1) : 0;
}

anpd_status step_cl_enqueue(anpd_model* m, anpd_kv* kv, bool want_logits, bool tree) {
    Workspace& ws = kv->ws;
    ScArgs g;
    int smem = 0;
    if (!sc_args(m, &g, &smem)) return ANPD_ERR_STATE;
    g.img0 = ws.ci_h; g.x0 = ws.x; g.ss0 = ws.ss_cl_a;
    g.xch = ws.xch;
    g.entered = (unsigned*)(ws.xch + 2 * (size_t)g.copy_bytes + g.fin_bytes);
    g.row_pos = ws.row_pos; g.row_slot = ws.row_slot; g.row_seq = ws.row_seq; g.row_ok = ws.row_ok; g.hole_lo = ws.row_hole_lo; g.hole_hi = ws.row_hole_hi;
    g.tree = tree ? 1 : 0;
    g.rope_cos = kv->rope_cos; g.rope_sin = kv->rope_sin;
    g.page_table = kv->page_table; g.pages_per_seq = kv->pages_per_seq; g.total_pages = kv->total_pages;
    g.kpool = kv->kpool; g.vpool = kv->vpool;
    g.out = want_logits ? ws.logits : nullptr; g.amax_val = ws.amax_val_cl; g.amax_idx = ws.amax_idx_cl;
    g.err = ws.gemm_err;
    ws.amax_nblk = g.ncl * CL_CTAS;
    ws.amax_val_use = ws.amax_val_cl;
    ws.amax_idx_use = ws.amax_idx_cl;
    return m->cfg.head_dim == 128 ? launch_step_cl<128>(kv, g, smem, m->stream, &m->prof) : launch_step_cl<64>(kv, g, smem, m->stream, &m->prof);
}
