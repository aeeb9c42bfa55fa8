// Projections of a decode step on sm_100a.  Four CTAs share a range of output features: they stream its weights once, each a
// quarter of the contraction dimension, so that a CTA reads a quarter of the activations only.
//
// One sequence (8 rows): the four are a cluster, add their partial sums over distributed shared memory and finish the projection
// themselves (rotary embedding and cache append, residual add, SwiGLU, vocabulary argmax): five kernels per layer with the
// attention, where partial sums through global memory and a kernel for every epilogue took ten.  RMSNorm is applied by the
// consumer: an O or down projection leaves x * gain as hi + lo terms and per-CTA sums of squares, the consumer's epilogue
// multiplies its results by the row's 1 / RMS.
// Several sequences (16 to 128 rows): partial sums per CTA in global memory, added by the consumers.  The exchange inside a
// cluster was built for these too and is slower there: 16 bytes per row and feature at about 14 bytes a cycle and SM take longer
// than the kernels they replace (13B width, eight sequences: 205 us per layer against 149).
//
// What bounds it: HBM, and beside it the hand-over between dependent kernels: about 1 us from a kernel's last store to the next
// one's first activation load, 0.5 us for that load, 1.5 us from the last product to the last store.  A layer of a step, attention
// included: 7B 405 MB of weights in 77 us at 77 keys (copy rate of the device: 62 us), 1.1B 88 MB in 31.5 us at 512 (13.5 us).
//
// Roles.  A weight thread keeps a ring of copies in flight; the first of them go out while the kernel before is still running (weights
// depend on nothing): all that the ring holds where CTAs share an SM, three where a step's CTA has one for itself (see CL_FIRST).
// An activation thread follows behind the dependency wait.  An MMA thread multiplies tiles of up to 128 features with the rows of
// the step (N operand: hi terms, then lo terms of the activations) into tensor memory.  Four warps read the accumulators and push each partial sum to the CTA that
// finishes its feature (st.async: data and arrival in one), eight add the parts in CTA order and apply the epilogue.
// The single threads must keep up with a 16 KB copy every 600 cycles: they are elected, not picked by lane number (see elect_one),
// walk their sequences with additions only (an integer division costs about a hundred cycles there) and keep only the low words
// of the operand descriptors.
//
// A row's result depends on its own inputs only: the cut of K, the order of the parts and every reduction tree depend on the
// matrix shape and the device.  Every wait is bounded and reports through the error flag.
#include "internal.h"
#include "step_dev.cuh"

#include <math_constants.h>

#include <algorithm>

typedef __nv_bfloat16 bf16;

namespace {

using namespace tc;

// warp 0: weights, warp 1: MMA issuer + tensor-memory owner, warp 2: activations, warps from 4 on: exchange and epilogue
__host__ __device__ constexpr int cl_threads(int R) { return R ? 384 : 256; }
constexpr int CL_MAX_STAGES = 16;
constexpr int CL_MAX_ACT = 8;
constexpr int CL_MAX_TILES = 8;          // tiles of 128 features a pass may hold
constexpr int CL_MAX_ROWS = 128;
constexpr int CL_STAGE_MAX = 16384;      // one copy: at most 16 groups of 8 features x 64 inputs
constexpr int CL_SMEM_PAIR = 112 * 1024; // two CTAs of this size share an SM
constexpr int CL_SMEM_MAX = 216 * 1024;
constexpr int CL_RING_BYTES = 8 * CL_STAGE_MAX;      // copies in flight per SM
// A CTA that has its SM for itself starts as the one before leaves, when the activations are about to be ready: its first ring, 128 KB
// requested at once, would stand in front of them (2.3 us at the device's rate).  So it requests a few stages, and the others once tensor
// memory is allocated, by when the activation thread is past its wait or about to be (a further wait for its first copy, of 500 to 6000
// cycles at most, changed nothing).  us per step against the whole ring at once: 7B (16 layers) at 77 keys 1311 -> 1295, at 1536 1389 ->
// 1374, 3072 wide (12 layers) 722 -> 712; 13B (8 layers) 987 -> 995.  Four stages give the same, two lost 5 us at 7B.
constexpr int CL_FIRST = 3;
constexpr int CL_ERR_TIMEOUT = 207;

struct ClArgs {
    const unsigned char* w;              // see ClPlan
    const unsigned char* act;            // operand image [k-block][2 * rows][64]
    int kb, gpu, n_units, ncl;
    int seg;                             // segments of the storage: ncl or 1
    int rows, passes, copies, two, kps, stages, stage_bytes, akb, act_slots, tmem_cols, acc_bufs, acc_cols;
    int f_own_max, first;                // first: stages requested before tensor memory is allocated
    // RMSNorm of the input
    const float* ss_in; int n_parts; float inv_d, eps;
    // rotary + append
    const int *row_pos, *row_slot, *row_seq, *row_ok;
    const float *rope_cos, *rope_sin; const int* page_table; int pages_per_seq, Hq, Hkv, hd; float q_scale;
    bf16 *q_hi, *q_lo, *kpool, *vpool;
    // residual
    float* x; const float* gain; float* ss_out; int d;
    unsigned char* act_out;              // operand image of the next projection (residual, SwiGLU)
    // vocabulary / plain output
    float* out; int n_out; float* amax_val; int* amax_idx;
    // partial sums of several sequences' rows: [CTA of the cluster][row][feature]
    float* part; size_t part_stride; int ld_part; ClPlan plan;
    int* err;
};

__device__ __forceinline__ void fin_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// R: 8 = a step of one sequence (8 rows, one pass, one chunk); 0 = rows, passes and chunks from the arguments.
// TMAX: most tiles of a sequence's step, 1 or CL_MAX_TILES: code is time here (see launch_step)
template <int EPI, int R, int TMAX>
__global__ void __launch_bounds__(cl_threads(R), 1) gemm_cl_kernel(const __grid_constant__ ClArgs g) {
    constexpr bool ONE = R && TMAX == 1;
    extern __shared__ __align__(1024) unsigned char cl_smem_raw[];
    __shared__ uint64_t w_full[CL_MAX_STAGES], w_empty[CL_MAX_STAGES], a_full[CL_MAX_ACT], a_empty[CL_MAX_ACT];
    __shared__ uint64_t acc_full[2], acc_empty[2], red_full;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag, s_issued[2];
    __shared__ float s_rstd[8], s_part[8][8];
    __shared__ int s_pos[8], s_slot[8], s_page[8], s_idx[8][8];

    const int rows = R ? R : g.rows, passes = R ? 1 : g.passes;
    unsigned char* ring = cl_smem_raw + ((1024u - (smem_u32(cl_smem_raw) & 1023u)) & 1023u);
    const int act_slot = g.akb * rows * 256;
    unsigned char* abuf = ring + (size_t)g.stages * g.stage_bytes;
    float* red = (float*)(abuf + (size_t)g.act_slots * act_slot);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int C = CL_CTAS;
    const int rank = (int)blockIdx.x % C, cluster = (int)blockIdx.x / C;            // a cluster is C consecutive CTAs
    const int ulo = (int)((unsigned)(cluster * g.n_units) / (unsigned)g.ncl), uhi = (int)((unsigned)((cluster + 1) * g.n_units) / (unsigned)g.ncl);     // at most 32 clusters, 2^21 units
    const int Uc = uhi - ulo, Gc = Uc * g.gpu;                                      // units and groups of the cluster
    const int GS = g.seg == 1 ? g.n_units * g.gpu : Gc;                             // groups of a k-block in its segment
    const int kb_lo = rank * g.kb / C, nk = (rank + 1) * g.kb / C - kb_lo;          // this CTA's k-blocks

    // Units [u0, u0 + up) of pass p (relative to the cluster), up * gpu groups in T copies per k-block: the first `rem` of them
    // have base + 1 groups, the others base.  One sequence: a copy is one tile of at most 16 groups.  Several: two tiles of half
    // the copy each where there are more than 16 groups (with twice the work behind a wait and a commit, the issuing thread keeps
    // up with the stream).
    auto pass_of = [&](int p, int& u0, int& up) {
        if (R) { u0 = 0; up = Uc; }
        else { u0 = p * Uc / passes; up = (p + 1) * Uc / passes - u0; }
    };

    auto copies_of = [&](int G) { return ONE ? min(1, G) : min(g.copies, G); };       // the same for every cluster and pass, though some have a unit less than others

    // ---- weight thread's walk over (pass, step, tile) ----
    const unsigned char* w_src = nullptr;
    int w_p = 0, w_k = 0, w_t = 0, w_T = 0, w_base = 0, w_rem = 0, w_G = 0;
    auto w_enter = [&]() {                              // start pass w_p, or a later one that has something to load
        for (; w_p < passes; ++w_p) {
            int u0, up;
            pass_of(w_p, u0, up);
            w_G = up * g.gpu;
            w_T = copies_of(w_G);
            if (w_T == 0 || nk == 0) continue;
            w_base = w_G / w_T; w_rem = w_G - w_base * w_T;
            w_k = 0; w_t = 0;
            w_src = g.w + ((size_t)ulo * g.gpu * (g.seg == 1 ? 1 : g.kb) + (size_t)GS * kb_lo + (size_t)u0 * g.gpu) * 1024;
            return;
        }
    };
    const uint64_t pol_w = policy_evict_first();
    auto w_issue = [&](int stage) {                     // load the current item into `stage` and move on
        const int n = min(g.kps, nk - w_k);
        const uint32_t bytes = (uint32_t)(n * (ONE ? Gc : w_base + (w_t < w_rem ? 1 : 0))) << 10;      // n > 1 only where one tile holds all of the segment's groups
        mbar_expect_tx(&w_full[stage], bytes);
        bulk_load(ring + stage * g.stage_bytes, w_src, bytes, &w_full[stage], pol_w);
        w_src += bytes;
        if (ONE || ++w_t == w_T) {
            w_t = 0;
            w_k += n;
            w_src += (size_t)(GS - (R ? Gc : w_G)) << 10;          // the k-block's other groups
            if (w_k >= nk) { ++w_p; if (!R) w_enter(); }
        }
    };
    int w_count = 0;

    constexpr int unit_shift = EPI == CL_QKV || EPI == CL_GU ? 4 : 3;               // features per unit: 8 * gpu
    const int o0 = rank * Uc / C, on = (rank + 1) * Uc / C - o0;                    // the cluster's units this CTA finishes (R = 8)

    if (warp == 0) {
        if (elect_one()) {
            if (!R) { abort_flag = 0; s_issued[0] = 0; s_issued[1] = 0; }
#pragma unroll 1
            for (int s = 0; s < g.stages; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], 1); }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            // the weights depend on nothing: the first of them are requested before anything else happens
            w_enter();
#pragma unroll 1
            for (; w_count < (R && !ONE ? g.first : g.stages) && w_p < passes; ++w_count) w_issue(w_count);
        }
        __syncwarp();
    } else if (R ? warp == 2 : threadIdx.x == 64) {
        if (!R || elect_one()) {
            if (R) { abort_flag = 0; s_issued[0] = 0; s_issued[1] = 0; }
#pragma unroll 1
            for (int s = 0; s < g.act_slots; ++s) { mbar_init(&a_full[s], 1); mbar_init(&a_empty[s], 1); }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        if (R) __syncwarp();
    } else if (threadIdx.x == 96) {
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 4); }
        mbar_init(&red_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (R) mbar_expect_tx(&red_full, (uint32_t)((on << unit_shift) * C * 32));       // what the cluster will send here
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    } else if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"((uint32_t)g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    // In a sequence's step the activation thread goes on at once, past the allocation of tensor memory (7B, 16 layers, 77 keys: 1329 ->
    // 1323 us; 1.1B's batches lost 4 %).
    if (!R) __syncthreads();
    else if (warp == 2) asm volatile("bar.arrive 2, %0;" ::"n"(cl_threads(R)) : "memory");
    else asm volatile("bar.sync 2, %0;" ::"n"(cl_threads(R)) : "memory");
    tc_fence_after();
    // Only now may the next kernel start beside this one: its tensor-memory allocation must not come before this CTA's.
    if (!R || warp != 2) pdl_trigger();
    if (R) cluster_arrive();                           // waited for before the first push: every CTA's barriers are initialised then
    const uint32_t tmem_base = *((volatile uint32_t*)&tmem_slot);
    volatile int* abortp = &abort_flag;

    if (warp == 0) {
        // ---------------- weights ----------------
        if (elect_one()) {
            if constexpr (R && !ONE) {                  // (one tile: the CTA is beside another, and the ring has gone out)
#pragma unroll 1
                for (; w_count < g.stages && w_p < passes; ++w_count) w_issue(w_count);
            }
            int stage = 0;
            uint32_t phase = 0;
#pragma unroll 1
            while (w_p < passes) {
                if (!mbar_wait<1>(&w_empty[stage], phase, abortp)) break;
                w_issue(stage);
                ++w_count;
                if (++stage == g.stages) { stage = 0; phase ^= 1u; }
            }
            s_issued[0] = w_count;
        }
        __syncwarp();
    } else if (warp == 2) {
        // ---------------- activations ----------------
        if (elect_one()) {
            const uint64_t pol_a = policy_evict_last();
            pdl_wait();
            int slot = 0, count = 0;
            uint32_t phase = 1;
            bool ok = true;
            for (int p = 0; p < passes && ok; ++p) {
                int u0, up;
                pass_of(p, u0, up);
                if (up == 0) continue;
#pragma unroll 1
                for (int k = 0; k < nk; k += g.akb) {
                    if (count >= g.act_slots) ok = mbar_wait<1>(&a_empty[slot], phase, abortp);
                    if (!ok) break;
                    const uint32_t bytes = (uint32_t)(min(g.akb, nk - k) * rows) * 256u;
                    mbar_expect_tx(&a_full[slot], bytes);
                    bulk_load(abuf + slot * act_slot, g.act + (size_t)(kb_lo + k) * rows * 256, bytes, &a_full[slot], pol_a);
                    ++count;
                    if (++slot == g.act_slots) { slot = 0; phase ^= 1u; }
                }
            }
            s_issued[1] = count;
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (elect_one()) {
            // fp32 accumulate, bf16 x bf16, both operands K-major, M = 128 features, N = 2 * rows (hi terms, then lo terms)
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * rows) >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
            const uint32_t ring_lo = smem_desc_lo(smem_u32(ring)), act_lo = smem_desc_lo(smem_u32(abuf));
            const uint32_t stage_step = (uint32_t)g.stage_bytes >> 4, act_step = (uint32_t)act_slot >> 4, kb_step = (uint32_t)(rows * 256) >> 4;
            const uint32_t full0 = smem_u32(&w_full[0]), empty_off = smem_u32(&w_empty[0]) - full0, full_end = full0 + 8u * (uint32_t)g.stages;
            uint32_t full = full0, wph = 0, w_lo = ring_lo;
            const uint32_t af0 = smem_u32(&a_full[0]), aempty_off = smem_u32(&a_empty[0]) - af0, af_end = af0 + 8u * (uint32_t)g.act_slots;
            const int akb = g.akb, kps = g.kps;
            int buf = 0;
            uint32_t afull = af0, aph = 0, eph = 1, a_lo = act_lo;
            // A wait that gave up has set the abort flag; the loops run on with whatever the buffers hold (every later wait is
            // short then), so that their trip counts depend on nothing the thread has to test.
            auto next_stage = [&]() {
                tc_commit_at(full + empty_off);
                w_lo += stage_step;
                full += 8u;
                if (full == full_end) { full = full0; wph ^= 1u; w_lo = ring_lo; }
            };
            for (int p = 0; p < passes; ++p) {
                int u0, up;
                pass_of(p, u0, up);
                const int G = up * g.gpu, T = copies_of(G), base = !R && T ? G / T : 0, rem = !R && T ? G - base * T : 0;
                if (p >= g.acc_bufs) mbar_wait<1>(&acc_empty[buf], eph, abortp);
                tc_fence_after();
                const uint32_t d0 = tmem_base + (uint32_t)(buf * g.acc_cols);
                uint32_t acc = 0;
                const int k_end = T > 0 ? nk : 0;
#pragma unroll 1
                for (int k0 = 0; k0 < k_end; k0 += akb) {
                    mbar_wait_at<1>(afull, aph, abortp);
                    const int kend = min(akb, nk - k0);
                    uint32_t a = a_lo;
                    // a tile of fewer than 16 groups: the instruction reads whatever follows for the rows beyond, whose lanes nobody reads
                    if (!R && g.two) {                                  // two tiles of one k-block per stage
#pragma unroll 1
                        for (int k = 0; k < kend; ++k) {
                            uint32_t d_tmem = d0;
#pragma unroll 1
                            for (int t = 0; t < T; ++t) {
                                const uint32_t first = (uint32_t)(base + (t < rem ? 2 : 1)) >> 1;       // groups of the copy's first tile
                                mbar_wait_at<1>(full, wph, abortp);
                                tc_fence_after();
                                tc_mma_k64(d_tmem, w_lo, a, idesc, acc);
                                tc_mma_k64(d_tmem + (uint32_t)(2 * rows), w_lo + (first << 6), a, idesc, acc);
                                next_stage();
                                d_tmem += (uint32_t)(4 * rows);
                            }
                            acc = 1;
                            a += kb_step;
                        }
                    } else if (!ONE && T > 1) {                         // one tile of one k-block per stage
#pragma unroll 1
                        for (int k = 0; k < kend; ++k) {
                            uint32_t d_tmem = d0;
#pragma unroll 1
                            for (int t = T; t > 0; --t) {
                                mbar_wait_at<1>(full, wph, abortp);
                                tc_fence_after();
                                tc_mma_k64(d_tmem, w_lo, a, idesc, acc);
                                next_stage();
                                d_tmem += (uint32_t)(2 * rows);
                            }
                            acc = 1;
                            a += kb_step;
                        }
                    } else {                                            // kps k-blocks of the only tile per stage
#pragma unroll 1
                        for (int k = 0; k < kend; k += kps) {
                            mbar_wait_at<1>(full, wph, abortp);
                            tc_fence_after();
                            tc_mma_k64(d0, w_lo, a, idesc, acc);
                            acc = 1;
                            a += kb_step;
                            uint32_t w = w_lo;
#pragma unroll 1
                            for (int j = min(kps, kend - k); j > 1; --j) {
                                w += (uint32_t)(G << 6);
                                tc_mma_k64(d0, w, a, idesc, 1u);
                                a += kb_step;
                            }
                            next_stage();
                        }
                    }
                    tc_commit_at(afull + aempty_off);
                    a_lo += act_step;
                    afull += 8u;
                    if (afull == af_end) { afull = af0; aph ^= 1u; a_lo = act_lo; }
                }
                tc_commit(&acc_full[buf]);
                if (++buf == g.acc_bufs) { buf = 0; eph ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp >= 4 && R) {
        // ---------------- exchange and epilogue, one sequence ----------------
        // warps 4-7 read the accumulators and push, warps 4-11 finish
        const int half = g.hd >> 1;
        const uint32_t red_addr = smem_u32(red), bar_addr = smem_u32(&red_full);
        const bool pushes = warp < 8;
        const int fw = warp - 4, ft = fw * 32 + lane, row = ft & 7;                  // finishing warp and thread, its row
        const int quad = warp & 3;                                                   // a warp may only touch lanes 32 * (warp % 4) .. + 31
        const int ufirst = ulo + o0, parts_out = (int)gridDim.x;

        // where this thread's feature of each tile goes: byte offset in the exchange buffer and the owner's rank
        uint32_t dst[TMAX + 1];
        const int tiles = copies_of(Gc);
        if (pushes) {
            const int base = tiles ? Gc / tiles : 0, rem = tiles ? Gc - base * tiles : 0;
            int t0 = 0;
#pragma unroll
            for (int t = 0; t < TMAX; ++t) {
                dst[t] = 0xffffffffu;
                if (t < tiles) {
                    const int gt = base + (t < rem ? 1 : 0);
                    if (quad * 32 + lane < gt * 8) {
                        const int f = t0 * 8 + quad * 32 + lane, u = f >> unit_shift, owner = ((u + 1) * C - 1) / Uc;
                        const int local = f - ((owner * Uc / C) << unit_shift);
                        dst[t] = ((uint32_t)owner << 24) | (uint32_t)((rank * g.f_own_max + local) * 32);
                    }
                    t0 += gt;
                }
            }
        }

        pdl_wait();
        // 1 / RMS of every row: a warp per row, 32 interleaved sums over the parts, then a tree over the lanes
        if (EPI != CL_RESID) {
            float s = 0.0f;
            for (int i = lane; i < g.n_parts; i += 32) s += g.ss_in[(size_t)fw * g.n_parts + i];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) s_rstd[fw] = g.n_parts ? rsqrtf(s * g.inv_d + g.eps) : 1.0f;
        }
        if (EPI == CL_QKV && ft < 8) {
            const int slot = g.row_slot[ft];
            s_pos[ft] = g.row_pos[ft];
            s_slot[ft] = g.row_ok[ft] ? slot : -1;
            s_page[ft] = g.page_table[g.row_seq[ft] * g.pages_per_seq + slot / KV_PAGE];
        }
        fin_bar();
        // what this thread's first item reads from global memory comes in under the weight stream
        float2 pf = make_float2(0.f, 0.f), pg = make_float2(0.f, 0.f);
        if (ft < on * 32) {
            if (EPI == CL_QKV) {
                const int u = ufirst + (ft >> 5), i = (u % (g.hd >> 4)) * 8 + 2 * ((ft >> 3) & 3);
                const size_t at = (size_t)s_pos[row] * half + i;
                pf = *(const float2*)(g.rope_cos + at);
                pg = *(const float2*)(g.rope_sin + at);
            }
            if (EPI == CL_RESID) {
                const int n = ufirst * 8 + 2 * (ft >> 3);
                pf = *(const float2*)(g.x + (size_t)row * g.d + n);
                pg = *(const float2*)(g.gain + n);
            }
        }
        if (EPI == CL_RESID || EPI == CL_GU) {          // the image's columns behind the last feature: one CTA, under the weight stream
            const int k_out = EPI == CL_RESID ? g.d : g.n_out >> 1;
            if ((k_out & 63) && blockIdx.x == 0 && ft < 128) cl_img_clear_tail(g.act_out, rows, ft >> 3, k_out, ft & 7);
        }
        cluster_wait();

        if (pushes) {
            mbar_wait<1>(&acc_full[0], 0, abortp);
            tc_fence_after();
            const uint32_t col0 = tmem_base + ((uint32_t)(quad * 32) << 16);
#pragma unroll
            for (int t = 0; t < TMAX; t += 2) {
                if (t >= tiles) break;
                // two tiles' columns in one load; the second repeats the first where there is none
                float v[2][8];
                const uint32_t ca = col0 + (uint32_t)(t * 16), cb = t + 1 < tiles ? ca + 16u : ca;
                if (ONE) tc_ld8_sum(ca, ca + 8u, v[0]);
                else tc_ld8_sum2(ca, ca + 8u, cb, cb + 8u, v[0], v[1]);
#pragma unroll
                for (int h = 0; h < (ONE ? 1 : 2); ++h) {
                    if (nk == 0)
#pragma unroll
                        for (int r = 0; r < 8; ++r) v[h][r] = 0.0f;
                    if (dst[t + h] != 0xffffffffu) {
                        const uint32_t owner = dst[t + h] >> 24, to = map_to_cta(red_addr + (dst[t + h] & 0xffffffu), owner), bar = map_to_cta(bar_addr, owner);
                        st_async4(to, bar, v[h][0], v[h][1], v[h][2], v[h][3]);
                        st_async4(to + 16u, bar, v[h][4], v[h][5], v[h][6], v[h][7]);
                    }
                }
            }
        }
        cluster_arrive();                               // nothing leaves for another CTA after the push
        mbar_wait_cluster(&red_full, 0, abortp);
        const int part_step = g.f_own_max * 8;
        auto sum = [&](int f) {                         // feature f of this CTA's share, this thread's row, parts in CTA order
            const float* s = red + f * 8 + row;
            return ((s[0] + s[part_step]) + s[2 * part_step]) + s[3 * part_step];
        };
        if (EPI == CL_RESID) {
            float ssq = 0.0f;
#pragma unroll 1
            for (int idx = ft; idx < on * 32; idx += 256) {
                const int f = 2 * (idx >> 3), n = ufirst * 8 + f;
                float2 x = pf, gn = pg;
                if (idx != ft) { x = *(const float2*)(g.x + (size_t)row * g.d + n); gn = *(const float2*)(g.gain + n); }
                x.x += sum(f); x.y += sum(f + 1);
                *(float2*)(g.x + (size_t)row * g.d + n) = x;
                ssq += x.x * x.x + x.y * x.y;
                uint32_t hi, lo;
                split2(x.x * gn.x, x.y * gn.y, hi, lo);
                *(uint32_t*)(g.act_out + cl_img_offset(rows, row, n)) = hi;
                *(uint32_t*)(g.act_out + cl_img_offset(rows, rows + row, n)) = lo;
            }
            // the row's sum of squares over this CTA's features: one part
            ssq += __shfl_xor_sync(0xffffffffu, ssq, 8);
            ssq += __shfl_xor_sync(0xffffffffu, ssq, 16);
            if (lane < 8) s_part[fw][lane] = ssq;
            fin_bar();
            if (ft < 8) {
                float s = s_part[0][ft];
#pragma unroll
                for (int w = 1; w < 8; ++w) s += s_part[w][ft];
                g.ss_out[(size_t)ft * parts_out + blockIdx.x] = s;
            }
        } else if (EPI == CL_GU) {
            const float rs = s_rstd[row];
#pragma unroll 1
            for (int idx = ft; idx < on * 32; idx += 256) {
                const int ul = idx >> 5, e = 2 * ((idx >> 3) & 3), f = ul * 16 + e, k = (ufirst + ul) * 8 + e;
                float v[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float gte = sum(f + h) * rs, upv = sum(f + 8 + h) * rs;
                    v[h] = gte / (1.0f + expf(-gte)) * upv;
                }
                uint32_t hi, lo;
                split2(v[0], v[1], hi, lo);
                *(uint32_t*)(g.act_out + cl_img_offset(rows, row, k)) = hi;
                *(uint32_t*)(g.act_out + cl_img_offset(rows, rows + row, k)) = lo;
            }
        } else if (EPI == CL_QKV) {
            const float rs = s_rstd[row];
            const int pos = s_pos[row], slot = s_slot[row], page = s_page[row], upi = g.hd >> 4;
#pragma unroll 1
            for (int idx = ft; idx < on * 32; idx += 256) {
                const int ul = idx >> 5, e = 2 * ((idx >> 3) & 3), u = ufirst + ul, head = u / upi, i = (u - head * upi) * 8 + e;
                float a[2], b[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) { a[h] = sum(ul * 16 + e + h) * rs; b[h] = sum(ul * 16 + 8 + e + h) * rs; }
                if (head < g.Hq + g.Hkv) {
                    float2 cs, sn;
                    if (idx == ft) { cs = pf; sn = pg; }
                    else { const size_t at = (size_t)pos * half + i; cs = *(const float2*)(g.rope_cos + at); sn = *(const float2*)(g.rope_sin + at); }
                    const float a0 = a[0] * cs.x - b[0] * sn.x, b0 = b[0] * cs.x + a[0] * sn.x;
                    const float a1 = a[1] * cs.y - b[1] * sn.y, b1 = b[1] * cs.y + a[1] * sn.y;
                    a[0] = a0; b[0] = b0; a[1] = a1; b[1] = b1;
                }
                if (head < g.Hq) {
                    // queries leave as two bf16 terms, already multiplied by log2(e) / sqrt(hd)
                    const size_t o = (size_t)row * g.Hq * g.hd + (size_t)head * g.hd + i;
                    uint32_t hi, lo;
                    split2(a[0] * g.q_scale, a[1] * g.q_scale, hi, lo);
                    *(uint32_t*)(g.q_hi + o) = hi; *(uint32_t*)(g.q_lo + o) = lo;
                    split2(b[0] * g.q_scale, b[1] * g.q_scale, hi, lo);
                    *(uint32_t*)(g.q_hi + o + half) = hi; *(uint32_t*)(g.q_lo + o + half) = lo;
                } else if (slot >= 0) {
                    const bool is_k = head < g.Hq + g.Hkv;
                    const int kvh = is_k ? head - g.Hq : head - g.Hq - g.Hkv;
                    bf16* pg_ = (is_k ? g.kpool : g.vpool) + ((size_t)page * g.Hkv + kvh) * KV_PAGE * g.hd;
                    if (is_k) {                                   // K page: [position][dim]
                        bf16* at = pg_ + (size_t)(slot % KV_PAGE) * g.hd + i;
                        *(__nv_bfloat162*)at = __floats2bfloat162_rn(a[0], a[1]);
                        *(__nv_bfloat162*)(at + half) = __floats2bfloat162_rn(b[0], b[1]);
                    } else {                                      // V page, transposed: [dim][position]
                        bf16* at = pg_ + (size_t)i * KV_PAGE + (slot % KV_PAGE);
                        at[0] = __float2bfloat16_rn(a[0]);
                        at[KV_PAGE] = __float2bfloat16_rn(a[1]);
                        at[(size_t)half * KV_PAGE] = __float2bfloat16_rn(b[0]);
                        at[(size_t)(half + 1) * KV_PAGE] = __float2bfloat16_rn(b[1]);
                    }
                }
            }
        } else {                                                       // vocabulary or plain output
            const float rs = s_rstd[row];
            float best = -CUDART_INF_F;
            int bidx = 0x7fffffff;
#pragma unroll 1
            for (int idx = ft; idx < on * 64; idx += 256) {
                const int f = idx >> 3, n = ufirst * 8 + f;
                if (n >= g.n_out) continue;
                const float v = sum(f) * rs;
                if (g.out) g.out[(size_t)row * g.n_out + n] = v;
                if (v > best) { best = v; bidx = n; }                   // ascending n: strict > keeps the lowest id
            }
            if (EPI == CL_LM) {
                for (int o = 8; o <= 16; o <<= 1) {
                    const float ov = __shfl_xor_sync(0xffffffffu, best, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
                    if (ov > best || (ov == best && oi < bidx)) { best = ov; bidx = oi; }
                }
                if (lane < 8) { s_part[fw][lane] = best; s_idx[fw][lane] = bidx; }
                fin_bar();
                if (ft < 8) {
                    best = s_part[0][ft]; bidx = s_idx[0][ft];
                    for (int w = 1; w < 8; ++w)
                        if (s_part[w][ft] > best || (s_part[w][ft] == best && s_idx[w][ft] < bidx)) { best = s_part[w][ft]; bidx = s_idx[w][ft]; }
                    g.amax_val[(size_t)ft * parts_out + blockIdx.x] = best;
                    g.amax_idx[(size_t)ft * parts_out + blockIdx.x] = bidx;
                }
            }
        }
    } else if (warp >= 4) {
        // ---------------- several sequences: this CTA's partial sums to global memory ----------------
        const int quad = warp & 3;
        pdl_wait();                                     // the kernel before may still read the buffer
        int buf = 0;
        uint32_t bph = 0;
        for (int p = 0; p < passes; ++p) {
            int u0, up;
            pass_of(p, u0, up);
            const int G = up * g.gpu, T = copies_of(G), base = T ? G / T : 0, rem = T ? G - base * T : 0, per = g.two ? 2 : 1;
            mbar_wait<1>(&acc_full[buf], bph, abortp);
            tc_fence_after();
            int t0 = (ulo + u0) * g.gpu;                // the tile's first group
            for (int t = 0; t < T * per; ++t) {
                const int gs = base + (t / per < rem ? 1 : 0), gt = per == 1 ? gs : (t & 1) ? gs >> 1 : (gs + 1) >> 1;
                const int pos = t0 * 8 + quad * 32 + lane;
                if (quad * 32 < gt * 8) {               // the whole warp agrees
                    const int n = quad * 32 + lane < gt * 8 ? cl_feature(g.plan, pos) : g.n_out;
                    float* dst = g.part + (size_t)rank * g.part_stride + n;
                    const uint32_t col = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * g.acc_cols + t * 2 * rows);
                    for (int r0 = 0; r0 < rows; r0 += 8) {
                        float v[8];
                        tc_ld8_sum(col + (uint32_t)r0, col + (uint32_t)(rows + r0), v);
                        if (n < g.n_out)
#pragma unroll
                            for (int r = 0; r < 8; ++r) dst[(size_t)(r0 + r) * g.ld_part] = nk == 0 ? 0.0f : v[r];
                    }
                }
                t0 += gt;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
            if (++buf == g.acc_bufs) { buf = 0; bph ^= 1u; }
        }
    }

    // Leaving: another CTA's pushes into this one have all arrived when the epilogue is through; the second cluster barrier only
    // keeps a CTA whose wait ran out from leaving under the others.
    if (R && warp < 4) { cluster_wait(); cluster_arrive(); }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)g.tmem_cols) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) {
        // gave up: let every copy already issued land before the CTA may exit
        for (int i = max(0, s_issued[0] - g.stages); i < s_issued[0]; ++i)
            for (unsigned spin = 0; spin < WAIT_LIMIT && !mbar_try_wait(&w_full[i % g.stages], (uint32_t)((i / g.stages) & 1)); ++spin) {}
        for (int i = max(0, s_issued[1] - g.act_slots); i < s_issued[1]; ++i)
            for (unsigned spin = 0; spin < WAIT_LIMIT && !mbar_try_wait(&a_full[i % g.act_slots], (uint32_t)((i / g.act_slots) & 1)); ++spin) {}
        atomicExch(g.err, CL_ERR_TIMEOUT);
    }
    if (R) {
        __syncwarp();
        cluster_wait();
    }
}

// Rows [row_off, row_off + rows) of a row-major [rows][K] source into the storage of the plan's matrix: a block takes a row at a
// time (its place is found once), a thread eight inputs at a time; eight threads write the row's 128 bytes of a k-block.
// WIDE: eight bf16 inputs in one load.  The source is the caller's and may start at any element (a tensor inside a larger buffer),
// so that takes a source on a 16-byte boundary (its rows are multiples of 16 bytes).
template <typename T, bool WIDE>
__global__ void __launch_bounds__(256) cl_retile_kernel(const T* __restrict__ src, int rows, int row_off, const ClPlan p, unsigned char* __restrict__ dst) {
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        const int pos = cl_position(p, row_off + r);
        const ClRun run = cl_run(p, pos >> 3, 0);
        const size_t step = (size_t)run.step * 1024;                                   // one k-block of the segment
        unsigned char* out = dst + run.at + (size_t)(pos & 7) * 128;
        for (int k8 = threadIdx.x; k8 < p.K / 8; k8 += blockDim.x) {
            const T* in = src + (size_t)r * p.K + 8 * k8;
            bf16 v[8];
            if (WIDE) *(uint4*)v = *(const uint4*)in;
            else {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = (bf16)in[e];
            }
            *(uint4*)(out + (size_t)(k8 >> 3) * step + (size_t)(((k8 & 7) ^ (pos & 7)) << 4)) = *(const uint4*)v;
        }
    }
}

// fp32 rows -> operand image (test hook)
__global__ void cl_image_kernel(const float* __restrict__ a, int rows, int K, unsigned char* __restrict__ img) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows * K; i += gridDim.x * blockDim.x) {
        const int r = i / K, k = i % K;
        const float v = a[i];
        const bf16 h = __float2bfloat16_rn(v);
        *(bf16*)(img + cl_img_offset(rows, r, k)) = h;
        *(bf16*)(img + cl_img_offset(rows, rows + r, k)) = __float2bfloat16_rn(v - __bfloat162float(h));
    }
}

template <int EPI, int R, int TMAX = CL_MAX_TILES>
anpd_status launch_cl(const ClArgs& g, int smem, cudaStream_t st, Profiler* prof, double bytes) {
    static bool attr_set[64] = {false};
    if (first_call_on_device(attr_set)) {
        CUDA_TRY(cudaFuncSetAttribute(gemm_cl_kernel<EPI, R, TMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, CL_SMEM_MAX));
        CUDA_TRY(cudaFuncSetAttribute(gemm_cl_kernel<EPI, R, TMAX>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g.ncl * CL_CTAS); cfg.blockDim = dim3(cl_threads(R)); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (R) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = CL_CTAS; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (g_use_pdl && !t_no_pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    LAUNCH(prof, st, KC_GEMM, bytes, (cudaLaunchKernelEx(&cfg, gemm_cl_kernel<EPI, R, TMAX>, g)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

// The instance of a sequence's step: what a kernel does not need is not in it.  Its code comes from a cold instruction cache, layer after
// layer; with one instance for any tile count and unrolled waits and loops (43 to 54 KB of code, now 25 to 46) us per step were: 1.1B at 512
// keys 776, now 744, tiny 55, now 48, 1024 wide (16 layers) 428, now 379, 7B (16 layers, 77 keys) 1317, now 1301.
template <int EPI>
anpd_status launch_step(const ClArgs& g, int smem, cudaStream_t st, Profiler* prof, double bytes) {
    return g.copies == 1 ? launch_cl<EPI, 8, 1>(g, smem, st, prof, bytes) : launch_cl<EPI, 8>(g, smem, st, prof, bytes);
}

}  // namespace

// Clusters that can be resident together, at most 32: the decoder family's dimensions are multiples of 32 units, so 32 clusters
// get equal shares, where the 33 a B200's 148 SMs hold would leave some with a unit more than the rest.
int cl_clusters() {
    if (cudaFuncSetAttribute(gemm_cl_kernel<CL_RAW, 8, CL_MAX_TILES>, cudaFuncAttributeMaxDynamicSharedMemorySize, CL_SMEM_MAX) != cudaSuccess) { cudaGetLastError(); return 0; }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(32 * CL_CTAS); cfg.blockDim = dim3(cl_threads(8)); cfg.dynamicSmemBytes = CL_SMEM_MAX;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL_CTAS; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_cl_kernel<CL_RAW, 8, CL_MAX_TILES>, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    return std::min(n, 32);
}

void cl_make_plan(ClPlan* p, int kind, int N, int K, int hd, int F, int ncl) {
    p->kind = kind; p->N = N; p->K = K; p->hd = hd; p->F = F;
    p->gpu = (kind == CL_QKV || kind == CL_GU) ? 2 : 1;
    p->n_units = (N + 8 * p->gpu - 1) / (8 * p->gpu);
    p->kb = (K + 63) / 64;
    p->ncl = ncl;
    p->u_max = (p->n_units + ncl - 1) / ncl;
    // One segment where the contraction is long and a cluster's tiles are (nearly) full: CTAs side by side read one window, and a
    // kernel that cuts the matrix its own way finds few seams (a stream-K cut over 148 CTAs, 13B width, 128 rows: gate-up 67.9 -> 63.7 us).
    // Per step of 7B, 8 layers: one sequence 733 -> 727 us, two 792 -> 774.  Short contractions and smaller tiles lost 1 to 2 % by it
    // (2560 wide 619 -> 630 us, 1.1B 793 -> 801): the weight thread then has more and smaller pieces to request.
    const int groups = p->n_units / ncl * p->gpu, tiles = (p->u_max * p->gpu + 15) / 16;
    p->seg = p->kb >= 64 && groups >= 13 * tiles ? 1 : ncl;
}

size_t cl_storage_bytes(const ClPlan& p) { return (size_t)p.n_units * p.gpu * p.kb * 1024; }

bool cl_fused(const ClPlan& p) { return p.u_max * p.gpu <= 16 * CL_MAX_TILES; }

int cl_parts(const ClPlan& p) { return p.ncl * CL_CTAS; }

anpd_status cl_retile_enqueue(const ClPlan& p, const void* src, bool src_is_f32, int rows, int row_off, unsigned char* dst, cudaStream_t st) {
    const int blocks = std::min(rows, 148 * 16);
    if (src_is_f32) cl_retile_kernel<float, false><<<blocks, 256, 0, st>>>((const float*)src, rows, row_off, p, dst);
    else if ((uintptr_t)src % 16 == 0) cl_retile_kernel<bf16, true><<<blocks, 256, 0, st>>>((const bf16*)src, rows, row_off, p, dst);
    else cl_retile_kernel<bf16, false><<<blocks, 256, 0, st>>>((const bf16*)src, rows, row_off, p, dst);
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

anpd_status cl_image_enqueue(const float* a_dev, int rows, int K, unsigned char* img, cudaStream_t st) {
    cl_image_kernel<<<64, 256, 0, st>>>(a_dev, rows, K, img);
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

// Passes over the activations: as few as tensor memory allows (2 * rows columns per tile; two to sixteen tiles).
static int cl_passes(const ClPlan& p, int rows) {
    const int tiles = 512 / (2 * rows);
    int passes = 1;
    while ((((p.u_max + passes - 1) / passes) * p.gpu + 31) / 32 * 2 > tiles) ++passes;
    return passes;
}

// the part of the arguments that both forms share, and the shared memory they leave for the ring
static anpd_status cl_args(ClArgs* g, const ClPlan& p, const unsigned char* w, const unsigned char* act, int rows, int passes, int red_bytes, int* smem) {
    *g = ClArgs{};
    g->w = w; g->act = act;
    g->kb = p.kb; g->gpu = p.gpu; g->n_units = p.n_units; g->ncl = p.ncl;
    g->rows = rows; g->passes = passes; g->n_out = p.N;
    const bool one = red_bytes > 0;                     // a single sequence
    const int up_max = (p.u_max + passes - 1) / passes, groups = up_max * p.gpu;
    const int tiles = one || groups <= 16 ? (groups + 15) / 16 : (groups + 31) / 32 * 2;
    // a cluster with few features: several k-blocks of its one tile make one copy
    const int nk = (p.kb + CL_CTAS - 1) / CL_CTAS;      // k-blocks of a CTA, at most
    g->seg = p.seg;
    g->kps = (passes == 1 && tiles == 1 && p.seg == p.ncl) ? std::max(1, std::min(std::min(4, 16 / groups), 64 / rows)) : 1;
    if (g->kps == 3) g->kps = 2;                        // a step never straddles two activation slots
    // A wait, a commit and the turn to the next activation slot cost the issuing thread as much as three to eight products.  So a CTA
    // of a sequence's step whose k-blocks fit one activation slot takes them in one, and one whose weights all fit the ring beside
    // another CTA has four k-blocks behind each wait.  1.1B (8 k-blocks: QKV, O, gate-up; ring: QKV, O): 807 -> 791 us per step at 512
    // keys, 941 -> 922 at 4000; the slot alone 800, the ring alone 799.
    const bool one_slot = one && nk > 4 && nk <= 8;
    const bool in_ring = one_slot && p.seg == p.ncl && tiles == 1 && 8 * groups * 1024 + 8 * rows * 256 + red_bytes + 1024 <= CL_SMEM_PAIR;
    if (in_ring) g->kps = 4;
    g->two = tiles > 1 && !one;
    g->copies = g->two ? tiles / 2 : tiles;
    g->stage_bytes = tiles == 1 ? groups * g->kps * 1024 : (groups + g->copies - 1) / g->copies * 1024;
    g->acc_cols = tiles * 2 * rows;
    g->acc_bufs = (passes > 1 && 2 * g->acc_cols <= 512) ? 2 : 1;
    g->tmem_cols = 32;
    while (g->tmem_cols < g->acc_bufs * g->acc_cols) g->tmem_cols <<= 1;
    // activation slots of 8 KB (one sequence) to 32 KB, a whole number of steps each
    int rest = 0;
    auto act_ring = [&](int akb, int slots) { g->akb = akb; g->act_slots = slots; rest = slots * akb * rows * 256 + red_bytes + 1024; };
    const int akb = std::max(g->kps, std::min(4, 128 / rows));
    if (one_slot) act_ring(8, 1);
    else act_ring(akb, std::max(2, std::min(CL_MAX_ACT, (one ? 24 : 96) * 1024 / (akb * rows * 256))));
    // Two CTAs of one sequence's projections share an SM where five copies in flight fit beside the rest: the next kernel's first
    // ring is then requested long before its turn.  With fewer in flight the stream itself is slower than that gain (7B, QKV
    // alone: 4 in flight 20.6 us, 8 and no second CTA 18.7), so such a projection takes the SM for itself.
    const bool pair = in_ring || (one && rest + 5 * g->stage_bytes <= CL_SMEM_PAIR);
    // with the SM to itself: half as many turns to the next slot (7B at 77 keys, 12 layers and the head: 1048.5 -> 1046.8)
    if (one && !pair && akb == 4) act_ring(8, one_slot ? 1 : 3);
    // beside another CTA: the same 24 KB as two slots of six k-blocks instead of three of four (1.1B, down projection, 22 k-blocks: 785 ->
    // 778 us per step); a step of kps k-blocks must not straddle two slots
    if (pair && nk > 8 && akb == 4 && g->kps <= 2) act_ring(6, 2);
    const int room = (pair ? CL_SMEM_PAIR : CL_SMEM_MAX) - rest;
    g->stages = std::min(CL_MAX_STAGES, std::min(room, CL_RING_BYTES) / g->stage_bytes);
    if (g->stages < 2) return ANPD_ERR_CAPACITY;
    g->first = one && !pair ? std::min(CL_FIRST, g->stages) : g->stages;
    // the M = 128 instruction reads 16 KB from the last tile of the last stage on, whatever the tile holds
    const int need = g->stages * g->stage_bytes + std::max(rest, CL_STAGE_MAX + 1024);
    // Two CTAs that share an SM take half of its shared memory each, whatever they need: with unequal halves the next kernel's
    // CTA finds the space its predecessor's predecessor left too small.
    *smem = pair ? std::max(need, CL_SMEM_PAIR) : need;
    return ANPD_OK;
}

anpd_status cl_enqueue(const ClPlan& p, const unsigned char* w, const unsigned char* act, const ClEpilogue& e, int* err, cudaStream_t st, Profiler* prof) {
    if (!cl_fused(p)) return ANPD_ERR_CAPACITY;
    ClArgs g;
    int smem = 0;
    const int f_own_max = (p.u_max + CL_CTAS - 1) / CL_CTAS * 8 * p.gpu;
    ANPD_TRY(cl_args(&g, p, w, act, ANPD_ROWS, 1, CL_CTAS * f_own_max * 32, &smem));
    g.f_own_max = f_own_max;
    g.ss_in = e.ss_in; g.n_parts = e.n_parts; g.inv_d = e.inv_d; g.eps = e.eps;
    g.row_pos = e.row_pos; g.row_slot = e.row_slot; g.row_seq = e.row_seq; g.row_ok = e.row_ok;
    g.rope_cos = e.rope_cos; g.rope_sin = e.rope_sin; g.page_table = e.page_table; g.pages_per_seq = e.pages_per_seq;
    g.Hq = e.Hq; g.Hkv = e.Hkv; g.hd = e.hd; g.q_scale = e.q_scale;
    g.q_hi = e.q_hi; g.q_lo = e.q_lo; g.kpool = e.kpool_l; g.vpool = e.vpool_l;
    g.x = e.x; g.gain = e.gain; g.ss_out = e.ss_out; g.d = e.d; g.act_out = e.act_out;
    g.out = e.out; g.amax_val = e.amax_val; g.amax_idx = e.amax_idx;
    g.err = err;
    const double bytes = 2.0 * (double)p.N * (double)p.K;
    switch (p.kind) {
        case CL_RAW: return launch_step<CL_RAW>(g, smem, st, prof, bytes);
        case CL_QKV: return launch_step<CL_QKV>(g, smem, st, prof, bytes);
        case CL_RESID: return launch_step<CL_RESID>(g, smem, st, prof, bytes);
        case CL_GU: return launch_step<CL_GU>(g, smem, st, prof, bytes);
        case CL_LM: return launch_step<CL_LM>(g, smem, st, prof, bytes);
    }
    return ANPD_ERR_ARG;
}

anpd_status cl_partial_enqueue(const ClPlan& p, const unsigned char* w, const unsigned char* act, int rows, float* part, size_t part_stride, int ld_part,
                               int* err, cudaStream_t st, Profiler* prof) {
    ClArgs g;
    int smem = 0;
    ANPD_TRY(cl_args(&g, p, w, act, rows, cl_passes(p, rows), 0, &smem));
    g.part = part; g.part_stride = part_stride; g.ld_part = ld_part; g.plan = p;
    g.err = err;
    return launch_cl<CL_RAW, 0>(g, smem, st, prof, 2.0 * (double)p.N * (double)p.K);
}
