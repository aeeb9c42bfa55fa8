// Attention of a decode step, complete in one kernel: the 8 rows of a sequence's step against the paged cache, softmax, and the
// result as the O projection's operand image.
//
// What bounds it: the cache's pages from HBM at long contexts; at short ones a memory round trip, the merge and the launch.  A
// cluster of C CTAs takes one query head (or two that share a kv head) of one sequence: CTA v takes the pages p with p mod C == v.
// A producer thread brings pages in through a ring of TMA copies (those no kernel of this step writes before the dependency
// wait); eight warps compute, each on its 16 keys of every page.  Where more than two query heads share a kv head, several
// clusters read its pages (from L2 but for the first) and each computes a part of the heads.  One cluster of eight CTAs per kv head
// with four times the rows and twice the warps was slower, its chain of products per page being four times as long: 1.1B (8 query
// heads per kv head), per step, 827 -> 800 us at 512 keys, 891 -> 839 at 1400, 1024 -> 937 at 4000.  Head dimension 128 takes a
// cluster per query head whatever the group: 32 query heads, 8 layers and the head, 300 keys, against page partials on the tensor
// cores and a merging kernel: 16 / 8 / 4 kv heads 745 / 781 / 950 -> 698 / 684 / 683 us per step, at 4000 keys 850 / 871 / 997 ->
// 793 / 801 / 793.
//
// Order.  A warp takes its blocks in ascending order with a running maximum; the warps of a CTA are merged in warp order, the
// CTAs in rank order, each into the running result.  All of it depends on absolute key positions and on the handle (heads and
// sequences) only, and a masked key contributes an exact zero, so a row's result does not depend on the rows it shares the step
// with or on how far the cache reaches behind the row.
//
// mma.sync m16n8k16 (bf16, fp32 sums): with 8 or 16 query vectors the products are small beside the loads.  Queries and weights
// enter as two bf16 terms; with one query head the two terms of the 8 rows are the tile's 16 rows.  The scores are summed in two
// chains, which halves the wait for the products (7B at 1536 keys: 1104 -> 1089 us for 12 layers and the head).
#include "internal.h"
#include "step_dev.cuh"

#include <math_constants.h>

#include <algorithm>

typedef __nv_bfloat16 bf16;

// CTAs per item.
constexpr int AD_MAX_CLUSTER = 4;
int ad_cluster(const anpd_model* m, int heads) {
    const int resident = m->num_sms * 7 / 8;
    int cluster = AD_MAX_CLUSTER;
    while (cluster > 1 && heads * cluster > resident) cluster /= 2;
    return cluster;
}

namespace {

using namespace tc;

constexpr int AD_KEYS = 16;              // keys per block
constexpr int AD_MAX_CHUNKS = 6;
constexpr int AD_SMEM_PAIR = 111 * 1024; // two CTAs share an SM: another one of these, or one of the projection before or after
constexpr int AD_ERR_TIMEOUT = 208;

// HD: head dimension, G: query heads a CTA takes (1 or 2 of those that share a kv head)
template <int HD, int G> struct AdCfg {
    static constexpr bool STACK = G == 1;                    // hi and lo terms of the 8 vectors share a tile
    static constexpr int NV = STACK ? 8 : 16;                // query vectors of the CTA: one tile
    static constexpr int WARPS = 8;                          // compute warps, each with 16 keys of a page; one more loads
    static constexpr int COMPUTE = 32 * WARPS, THREADS = COMPUTE + 32;
    static constexpr int REGS = 112;
    static constexpr int OP = HD + 4;                        // padded row
    static constexpr int QP = HD * 2 + 16;                   // bytes per staged query row
    static constexpr int QROWS = STACK ? 16 : 32;
    static constexpr int V4 = HD / 4;
    static constexpr int CHUNK = KV_PAGE * HD * 2;           // one copy: the page's K or its V^T
    static constexpr int SLOTS = WARPS * NV * OP * 4;        // the warps' results
    static constexpr int REST = 1024 + NV * HD * 4 + 2 * WARPS * NV * 4 + 2 * NV * 4 + QROWS * QP;
    // Half an SM per CTA, in registers too, so that it starts beside a CTA of the projection before it and lets the next one start
    // beside it.  7B, step of a short context 2.80 -> 2.69 ms, at 4096 keys 3.25 -> 3.14.  The CTA has read its last page when the
    // warps' results are written: they take the ring's place.
    static constexpr int ROOM = AD_SMEM_PAIR - REST;
    static constexpr int CHUNKS = ROOM / CHUNK < AD_MAX_CHUNKS ? ROOM / CHUNK : AD_MAX_CHUNKS;
    static constexpr int RING = CHUNKS * CHUNK < SLOTS ? SLOTS : CHUNKS * CHUNK;
    static constexpr int SMEM = REST + RING;
};

struct AdArgs {
    const bf16 *q_hi, *q_lo;
    const int *page_table, *row_pos, *row_seq, *row_slot, *hole_lo, *hole_hi;      // row_slot and the holes: null outside two-candidate steps
    int pages_per_seq, Hkv, split, rows, layer_page0;      // split: CTA clusters that share a kv head, G of its query heads each
    unsigned char* img;
    int* err;
};

template <int N> __device__ __forceinline__ void ad_bar() { asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory"); }

template <int HD, int G>
__global__ void __launch_bounds__((AdCfg<HD, G>::THREADS)) __maxnreg__((AdCfg<HD, G>::REGS)) attn_dec_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const AdArgs g) {
    typedef AdCfg<HD, G> Cfg;
    constexpr bool STACK = Cfg::STACK;
    constexpr int NV = Cfg::NV, WARPS = Cfg::WARPS, COMPUTE = Cfg::COMPUTE, CHUNKS = Cfg::CHUNKS, OP = Cfg::OP, QP = Cfg::QP, V4 = Cfg::V4;
    constexpr int KS = HD / 16, DT = HD / 8, NR = STACK ? 1 : 2;      // NR: query vectors per thread
    constexpr int CHUNK = Cfg::CHUNK;
    extern __shared__ __align__(1024) unsigned char ad_smem[];
    __shared__ uint64_t full[AD_MAX_CHUNKS], empty[AD_MAX_CHUNKS];
    __shared__ int abort_flag, s_issued;
    unsigned char* ring = ad_smem + ((1024u - (smem_u32(ad_smem) & 1023u)) & 1023u);
    float* recv = (float*)(ring + Cfg::RING);               // [CTA][VO][HD], the cluster's parts of this CTA's vectors
    float* sm_m = recv + NV * HD;                       // [warp][NV]
    float* sm_l = sm_m + WARPS * NV;
    float* rc_m = sm_l + WARPS * NV;                        // [CTA][VO]
    float* rc_l = rc_m + NV;
    unsigned char* Qs = (unsigned char*)(rc_l + NV);
    float* sm_o = (float*)ring;                             // [warp][NV][OP]

    pdl_trigger();
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");          // waited for before the first remote store: every CTA runs then
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = blockIdx.x, C = gridDim.x, VO = NV / C, hv = blockIdx.y, kvh = hv / g.split, r0 = blockIdx.z * ANPD_ROWS;       // VO: vectors a CTA finishes
    // The row plan is older than the kernel before this one (the embedding kernel lets its successors start only after its own
    // dependency wait), so it may be read at once; so may pages below the first position this launch writes - the group's own
    // first, or the first of all rows where they are one sequence's (a prompt as short as a step of the batch).
    const int seq = g.row_seq[r0];
    const int first_new = g.row_pos[gridDim.z > 1 && g.row_seq[0] == g.row_seq[ANPD_ROWS] ? 0 : r0];
    const int pos_lo = g.row_pos[r0], pos_hi = (g.row_slot ? g.row_slot : g.row_pos)[r0 + ANPD_ROWS - 1];
    const int n_pages = pos_hi / KV_PAGE + 1;
    volatile int* abortp = &abort_flag;

    if (warp == WARPS) {
        if (elect_one()) {
            abort_flag = 0; s_issued = 0;
#pragma unroll
            for (int s = 0; s < AD_MAX_CHUNKS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], WARPS); }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncwarp();
    }
    __syncthreads();

    if (warp == WARPS) {
        // ---------------- pages ----------------
        if (elect_one()) {
            const uint64_t pol = g.split > 1 ? policy_evict_last() : policy_evict_first();       // read again by the clusters that share the head
            const int* pages = g.page_table + (size_t)seq * g.pages_per_seq;
            int stage = 0, count = 0;
            uint32_t phase = 1;
            bool waited = false, ok = true;
            for (int p = rank; p < n_pages && ok; p += C) {
                const int row = (g.layer_page0 + pages[p]) * g.Hkv + kvh;
                if (!waited && (p + 1) * KV_PAGE > first_new) { pdl_wait(); waited = true; }       // holds rows the kernel before writes
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    if (count >= CHUNKS && ok) ok = mbar_wait<1>(&empty[stage], phase, abortp);
                    if (!ok) break;
                    unsigned char* dst = ring + (size_t)stage * CHUNK;
                    mbar_expect_tx(&full[stage], CHUNK);
                    if (half == 0) {
#pragma unroll
                        for (int s = 0; s < HD / 64; ++s) tma_load_2d(dst + s * (KV_PAGE * 128), &map_k, s * 64, row * KV_PAGE, &full[stage], pol);
                    } else {
#pragma unroll
                        for (int s = 0; s < 2; ++s) tma_load_2d(dst + s * (HD * 128), &map_v, s * 64, row * HD, &full[stage], pol);
                    }
                    ++count;
                    if (++stage == CHUNKS) { stage = 0; phase ^= 1u; }
                }
            }
            s_issued = count;
        }
        __syncwarp();
    } else {
        const int gid = lane >> 2, t = lane & 3;
        pdl_wait();                                         // the queries come from the kernel before
        for (int idx = threadIdx.x; idx < Cfg::QROWS * (HD / 8); idx += COMPUTE) {
            const int row = idx / (HD / 8), c = idx % (HD / 8);
            const int vec = row & (NV - 1);
            const bf16* src = (row >= NV ? g.q_lo : g.q_hi) + ((size_t)(r0 + vec / G) * gridDim.y * G + hv * G + vec % G) * HD + c * 8;
            *(uint4*)(Qs + row * QP + c * 16) = *(const uint4*)src;
        }
        int qpos[NR], qhl[NR], qhh[NR];
#pragma unroll
        for (int h = 0; h < NR; ++h) {
            const int r = (gid + 8 * h) / G;
            qpos[h] = g.row_slot ? g.row_slot[r0 + r] : pos_lo + r;
            qhl[h] = g.row_slot ? g.hole_lo[r0 + r] : 0;
            qhh[h] = g.row_slot ? g.hole_hi[r0 + r] : 0;
        }
        ad_bar<COMPUTE>();
        // lane offsets of the ldmatrix addresses: matrix (lane / 8) of four
        const int mi = lane >> 3, lr = lane & 7;
        const uint32_t q_addr = smem_u32(Qs) + (uint32_t)((lr + 8 * (mi & 1)) * QP + (mi >> 1) * 16);
        const uint32_t kv_off = (uint32_t)((lr + 8 * (mi >> 1)) * 128), chunk0 = (uint32_t)(mi & 1);
        const uint32_t ring_addr = smem_u32(ring);

        float m_run[NR], l_run[NR], o[DT][4];
        // keys key_page .. + 15 of page p: its K chunk (given back after the last block's scores), its V chunk
        auto block = [&](int ck, int cv, uint32_t par_v, int key_page, int p) {
            // two chains of products, added at the end: even and odd steps, or hi and lo terms
            float c[2][4], c2[2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) { c[j][e] = 0.f; c2[j][e] = 0.f; }
            const uint32_t kr = ring_addr + (uint32_t)ck * (uint32_t)CHUNK + kv_off + (uint32_t)key_page * 128u;
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                uint32_t b[4], a[4];
                ad_ldm4(kr + (uint32_t)((k >> 2) * (KV_PAGE * 128)) + ((((uint32_t)((k & 3) * 2) + chunk0) ^ (uint32_t)lr) << 4), b);
                ad_ldm4(q_addr + (uint32_t)(k * 32), a);
                ad_mma(STACK && (k & 1) ? c2[0] : c[0], a, b[0], b[1]);
                ad_mma(STACK && (k & 1) ? c2[1] : c[1], a, b[2], b[3]);
                if (!STACK) {
                    ad_ldm4(q_addr + (uint32_t)(16 * QP + k * 32), a);
                    ad_mma(c2[0], a, b[0], b[1]);
                    ad_mma(c2[1], a, b[2], b[3]);
                }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) c[j][e] += c2[j][e];
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[ck]);         // the short ring waits for it
            uint32_t ph[4], pl[4];
            float resc[NR];
#pragma unroll
            for (int h = 0; h < NR; ++h) {
                float w[2][2], mx = -CUDART_INF_F;
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int key = p * KV_PAGE + key_page + 8 * j + 2 * t + e;
                        const float s = STACK ? c[j][e] + c[j][2 + e] : c[j][2 * h + e];
                        w[j][e] = (key <= qpos[h] && !(key >= qhl[h] && key < qhh[h])) ? s : -CUDART_INF_F;
                        mx = fmaxf(mx, w[j][e]);
                    }
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const float m_new = fmaxf(m_run[h], mx);
                const bool none = m_new == -CUDART_INF_F;
                resc[h] = none ? 1.0f : exp2f(m_run[h] - m_new);
                float sum = 0.0f;
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) { w[j][e] = none ? 0.0f : exp2f(w[j][e] - m_new); sum += w[j][e]; }
                l_run[h] = l_run[h] * resc[h] + sum;        // this lane's keys; the four lanes of a row are added at the end
                m_run[h] = m_new;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    uint32_t lo;
                    const uint32_t hi = ad_split(w[j][0], w[j][1], lo);
                    if (STACK) { ph[2 * j] = hi; ph[2 * j + 1] = lo; }       // rows gid: hi terms, rows gid + 8: lo terms
                    else { ph[2 * j + h] = hi; pl[2 * j + h] = lo; }
                }
            }
            const float ra = resc[0], rb = resc[NR - 1];
            if (__any_sync(0xffffffffu, ra != 1.0f || rb != 1.0f)) {        // multiplying by 1 changes nothing
#pragma unroll
                for (int d = 0; d < DT; ++d) { o[d][0] *= ra; o[d][1] *= ra; o[d][2] *= rb; o[d][3] *= rb; }
            }
            // rolled, this wait costs head dimension 128 registers it does not have at its cap (24 bytes spilled); 64 has them and loses 0.15 % of a
            // 1.1B step by the unrolled one's code (7B, 16 layers, 1536 keys: 1368 us per step with the spill, 1366 without, both +- 5)
            mbar_wait<HD == 128 ? 16 : 1>(&full[cv], par_v, abortp);
            const uint32_t vr = ring_addr + (uint32_t)cv * (uint32_t)CHUNK + kv_off + (uint32_t)((key_page >> 6) * (HD * 128)) + ((((uint32_t)((key_page & 63) >> 3) + chunk0) ^ (uint32_t)lr) << 4);
#pragma unroll
            for (int d = 0; d < DT / 2; ++d) {
                uint32_t b[4];
                ad_ldm4(vr + (uint32_t)(d * 16 * 128), b);
                ad_mma(o[2 * d], ph, b[0], b[1]);
                ad_mma(o[2 * d + 1], ph, b[2], b[3]);
                if (!STACK) { ad_mma(o[2 * d], pl, b[0], b[1]); ad_mma(o[2 * d + 1], pl, b[2], b[3]); }
            }
        };

        int stage = 0;
        uint32_t par = 0;
#pragma unroll
        for (int h = 0; h < NR; ++h) { m_run[h] = -CUDART_INF_F; l_run[h] = 0.0f; }
#pragma unroll
        for (int d = 0; d < DT; ++d) { o[d][0] = 0.f; o[d][1] = 0.f; o[d][2] = 0.f; o[d][3] = 0.f; }
        for (int p = rank; p < n_pages; p += C) {
            const int ck = stage;
            const uint32_t par_k = par;
            if (++stage == CHUNKS) { stage = 0; par ^= 1u; }
            const int cv = stage;
            const uint32_t par_v = par;
            if (++stage == CHUNKS) { stage = 0; par ^= 1u; }
            mbar_wait<1>(&full[ck], par_k, abortp);
            if (p * KV_PAGE + warp * AD_KEYS <= pos_hi) block(ck, cv, par_v, warp * AD_KEYS, p);
            else { if (lane == 0) mbar_arrive(&empty[ck]); mbar_wait<1>(&full[cv], par_v, abortp); }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[cv]);
        }
        ad_bar<COMPUTE>();                               // the slots' results go where the pages were
        // ---- the key slots, in slot order ----
#pragma unroll
        for (int h = 0; h < NR; ++h) {
            l_run[h] += __shfl_xor_sync(0xffffffffu, l_run[h], 1);
            l_run[h] += __shfl_xor_sync(0xffffffffu, l_run[h], 2);
            if (t == 0) { sm_m[warp * NV + gid + 8 * h] = m_run[h]; sm_l[warp * NV + gid + 8 * h] = l_run[h]; }
        }
        float* mine = sm_o + (size_t)warp * NV * OP;
#pragma unroll
        for (int d = 0; d < DT; ++d) {
            if (STACK) *(float2*)(mine + gid * OP + 8 * d + 2 * t) = make_float2(o[d][0] + o[d][2], o[d][1] + o[d][3]);
            else {
                *(float2*)(mine + gid * OP + 8 * d + 2 * t) = make_float2(o[d][0], o[d][1]);
                *(float2*)(mine + (gid + 8) * OP + 8 * d + 2 * t) = make_float2(o[d][2], o[d][3]);
            }
        }
        ad_bar<COMPUTE>();
        // the result, as hi + lo terms in the O projection's operand image
        auto store = [&](int vec, int d4, float l, float4 a) {
            const int row = r0 + vec / G, k = (hv * G + vec % G) * HD + 4 * d4;
            uint2 hi, lo;
            hi.x = ad_split(a.x / l, a.y / l, lo.x);
            hi.y = ad_split(a.z / l, a.w / l, lo.y);
            *(uint2*)(g.img + cl_img_offset(g.rows, row, k)) = hi;
            *(uint2*)(g.img + cl_img_offset(g.rows, g.rows + row, k)) = lo;
        };
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        for (int idx = threadIdx.x; idx < NV * V4; idx += COMPUTE) {
            const int vec = idx / V4, d4 = idx % V4;
            float mx = -CUDART_INF_F;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) mx = fmaxf(mx, sm_m[w * NV + vec]);
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            float l = 0.0f;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) {
                const float m = sm_m[w * NV + vec], s = m == -CUDART_INF_F ? 0.0f : exp2f(m - mx);
                const float4 x = *(const float4*)(sm_o + (size_t)(w * NV + vec) * OP + 4 * d4);
                a.x = fmaf(x.x, s, a.x); a.y = fmaf(x.y, s, a.y); a.z = fmaf(x.z, s, a.z); a.w = fmaf(x.w, s, a.w);
                l = fmaf(sm_l[w * NV + vec], s, l);
            }
            if (C == 1) { store(vec, d4, l, a); continue; }
            const int owner = vec / VO, at = rank * VO + vec % VO;
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(ad_map(recv + at * HD + 4 * d4, owner)), "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w) : "memory");
            if (d4 == 0) {
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(ad_map(rc_m + at, owner)), "f"(mx) : "memory");
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(ad_map(rc_l + at, owner)), "f"(l) : "memory");
            }
        }
        if (C > 1) {
            asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
            for (int idx = threadIdx.x; idx < VO * V4; idx += COMPUTE) {
                const int vo = idx / V4, d4 = idx % V4;
                float m = -CUDART_INF_F, l = 0.0f;
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                for (int k = 0; k < C; ++k)
                    ad_fold(m, l, a, rc_m[k * VO + vo], rc_l[k * VO + vo], *(const float4*)(recv + (k * VO + vo) * HD + 4 * d4));
                store(rank * VO + vo, d4, l, a);
            }
        }
    }
    // the loading warp takes part in the cluster barriers too
    if (warp == WARPS) {
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        if (C > 1) asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) {
        // gave up somewhere: let every copy already requested land before the CTA may exit
        for (int i = max(0, s_issued - CHUNKS); i < s_issued; ++i)
            for (unsigned spin = 0; spin < WAIT_LIMIT && !mbar_try_wait(&full[i % CHUNKS], (uint32_t)((i / CHUNKS) & 1)); ++spin) {}
        atomicExch(g.err, AD_ERR_TIMEOUT);
    }
}

// Clusters that share a kv head.
int ad_split(const anpd_model_config& c) {
    const int group = c.n_q_heads / c.n_kv_heads;
    return c.head_dim == 64 && group > 1 ? group / 2 : group;
}

template <int HD, int G>
anpd_status launch_attn_dec(anpd_model* m, anpd_kv* kv, AdArgs& a) {
    typedef AdCfg<HD, G> Cfg;
    static bool attr_set[64] = {false};
    if (first_call_on_device(attr_set)) CUDA_TRY(cudaFuncSetAttribute(attn_dec_kernel<HD, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM));
    // As many CTAs per head as find an SM each (about 7/8 of the SMs can hold clusters).  Two to an SM leave no room for the next
    // projection's CTAs, whose first weights then come late: one 13B sequence of 1000 tokens (8 layers and the head) 1098 us per
    // step with four CTAs per head, 1072 with two; at 4000 tokens 1255 and 1223; eight 1.1B sequences 1337 and 1230 (two, one); four
    // 7B sequences of 600 tokens (8 layers) 915 and 880, of 2000 tokens 1088 and 1040.  Never more than four: sixteen clusters of
    // eight crowd the O projection out (1.1B at 512 keys: 894, with four 800).
    const int cluster = ad_cluster(m, a.Hkv * a.split * kv->batch);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster, a.Hkv * a.split, kv->batch); cfg.blockDim = dim3(Cfg::THREADS); cfg.dynamicSmemBytes = Cfg::SMEM; cfg.stream = m->stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (g_use_pdl && !t_no_pdl) ? 2 : 1;
    LAUNCH(&m->prof, m->stream, KC_ATTN, 0, (cudaLaunchKernelEx(&cfg, attn_dec_kernel<HD, G>, kv->map_k, kv->map_v, (const AdArgs)a)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

}  // namespace

anpd_status attn_dec_enqueue(anpd_model* m, anpd_kv* kv, int layer, bool tree) {
    const anpd_model_config& c = m->cfg;
    Workspace& ws = kv->ws;
    AdArgs a;
    a.q_hi = ws.q_hi; a.q_lo = ws.q_lo;
    a.page_table = kv->page_table; a.row_pos = ws.row_pos; a.row_seq = ws.row_seq;
    a.row_slot = tree ? ws.row_slot : nullptr; a.hole_lo = tree ? ws.row_hole_lo : nullptr; a.hole_hi = tree ? ws.row_hole_hi : nullptr;
    a.pages_per_seq = kv->pages_per_seq; a.Hkv = c.n_kv_heads; a.rows = kv->batch * ANPD_ROWS;
    a.layer_page0 = layer * kv->total_pages;
    a.img = ws.ci_ao; a.err = ws.gemm_err;
    a.split = ad_split(c);
    switch (c.head_dim * 16 + c.n_q_heads / c.n_kv_heads) {
        case 64 * 16 + 1: return launch_attn_dec<64, 1>(m, kv, a);
        case 64 * 16 + 2: case 64 * 16 + 4: case 64 * 16 + 8: return launch_attn_dec<64, 2>(m, kv, a);
        case 128 * 16 + 1: case 128 * 16 + 2: case 128 * 16 + 4: case 128 * 16 + 8: return launch_attn_dec<128, 1>(m, kv, a);
    }
    return ANPD_ERR_ARG;
}
