// Verification forward of a LLaMA-style decoder over the rows of one step against the paged KV
// cache (paper Section 3.1, "Verification": one forward over the K+1 tokens), and the fused
// argmax / draft-compare / prefix-accept that ends the step (Algorithm 1's accept loop).
//
// Row-count invariance: every value a row produces depends on that row's inputs and absolute
// position only - never on how many rows share the launch, nor on which of them are real.  A
// greedy step (1 real row) and an ANPD step (K+1 real rows) therefore give bit-identical logits
// for the same position, which is what makes the two token streams identical.
#include "internal.h"

#include <math_constants.h>

typedef __nv_bfloat16 bf16;

namespace {

constexpr int ERR_TOKEN_RANGE = 101;
constexpr int ERR_KV_FULL = 102;
constexpr int ERR_CTX_FULL = 103;

__device__ __forceinline__ void split_bf16(float v, bf16& hi, bf16& lo) {
    hi = __float2bfloat16_rn(v);
    lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// ---------------------------------------------------------------------------------------------
// row plans
// ---------------------------------------------------------------------------------------------
// Rows of a sequence's step: row 0 the confirmed token at position P; rows 1..ka the first candidate at positions P+1..;
// with a second candidate (two-candidate mode) rows ka+1..ka+kb hold its tokens at positions P+1.. again, but their K/V go
// to the cache slots behind the first candidate's (slot = P + row), and they must not see the first candidate's slots.
__global__ void plan_decode_kernel(SeqState* seqs, int* row_tok, int* row_pos, int* row_seq, int* row_ok, int* row_slot,
                                   int* row_hole_lo, int* row_hole_hi, int vocab, int max_len, int two) {
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int b = i / ANPD_ROWS, r = i % ANPD_ROWS;
    SeqState& s = seqs[b];
    const int ka = s.draft_len, kb = two ? min(s.draft2_len, ANPD_K_MAX - ka) : 0;
    const bool real = r <= ka + kb;
    int tok = (r == 0) ? s.last_tok : (r <= ka ? s.draft[r - 1] : (real ? s.draft2[r - ka - 1] : 0));
    if (tok < 0 || tok >= vocab) { if (real) atomicExch(&s.error, ERR_TOKEN_RANGE); tok = 0; }
    const int slot = s.kv_len + r;
    const int pos = (r > ka && real) ? s.kv_len + (r - ka) : slot;
    if (slot >= max_len && real && s.active) atomicExch(&s.error, ERR_KV_FULL);
    row_tok[i] = tok;
    row_pos[i] = min(pos, max_len - 1);
    row_seq[i] = b;
    row_ok[i] = (slot < max_len) ? 1 : 0;
    row_slot[i] = min(slot, max_len - 1);
    row_hole_lo[i] = (r > ka && real) ? s.kv_len + 1 : 0;
    row_hole_hi[i] = (r > ka && real) ? s.kv_len + ka + 1 : 0;
}

// Rows of a prompt pass: n_seq sequences from `seq` on, `seg` rows each, positions from `start` on; prompts one behind the other.
__global__ void plan_prefill_kernel(const int* prompt, int seq, int start, int prompt_len, int rows, int n_seq, int seg,
                                    int* row_tok, int* row_pos, int* row_seq, int* row_ok, int* row_slot, int* row_hole_lo,
                                    int* row_hole_hi, int vocab, int max_len, SeqState* seqs) {
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows) return;
    const int s = min(i / seg, n_seq - 1), p = start + i - s * seg;
    int tok = (p < prompt_len) ? prompt[s * prompt_len + p] : 0;
    if (tok < 0 || tok >= vocab) { atomicExch(&seqs[seq + s].error, ERR_TOKEN_RANGE); tok = 0; }
    row_tok[i] = tok;
    row_pos[i] = min(p, max_len - 1);
    row_seq[i] = seq + s;
    row_ok[i] = (p < max_len && p < prompt_len) ? 1 : 0;
    row_slot[i] = min(p, max_len - 1);
    row_hole_lo[i] = 0;
    row_hole_hi[i] = 0;
}

// ---------------------------------------------------------------------------------------------
// embedding gather + first RMSNorm;  residual add + RMSNorm
// One 1024-thread block per row; every thread owns float4 chunks of the row and issues all of a
// chunk's loads (residual + every partial sum) before using any of them, so the kernel costs about
// one memory round trip.  The sum of squares is reduced in a fixed tree.
// ---------------------------------------------------------------------------------------------
constexpr int NORM_THREADS = 1024;
constexpr int NORM_THREADS_2 = 768;       // of a row of two chunks per thread
constexpr int NORM_MAX_CHUNKS = 4;        // float4 chunks per thread: rows up to 16384 wide

__device__ __forceinline__ float block_sum(float v, float* red /*[32]*/) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = (threadIdx.x & 31) < blockDim.x >> 5 ? red[threadIdx.x & 31] : 0.0f;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    __syncthreads();
    return t;
}

__device__ __forceinline__ void store_split4(const float4 v, bf16* hi_ptr, bf16* lo_ptr) {
    bf16 h[4], l[4];
    split_bf16(v.x, h[0], l[0]); split_bf16(v.y, h[1], l[1]); split_bf16(v.z, h[2], l[2]); split_bf16(v.w, h[3], l[3]);
    *(uint2*)hi_ptr = *(const uint2*)h;
    *(uint2*)lo_ptr = *(const uint2*)l;
}

__device__ __forceinline__ void add4(float4& a, const float4& p) { a.x += p.x; a.y += p.y; a.z += p.z; a.w += p.w; }

__global__ void __launch_bounds__(NORM_THREADS) embed_norm_kernel(const bf16* __restrict__ embed, const int* __restrict__ row_tok,
                                                                  const float* __restrict__ gain, float eps, int d,
                                                                  float* __restrict__ x, bf16* __restrict__ h_hi, bf16* __restrict__ h_lo,
                                                                  unsigned char* __restrict__ img) {
    // img: a decode step's operand image of gridDim.x rows instead of h_hi and h_lo.  The trigger comes after the wait here:
    // whatever starts behind this kernel may then read the row plan at once.
    pdl_wait();
    pdl_trigger();
    __shared__ float red[32];
    const int row = blockIdx.x, chunks = d >> 2;
    const bf16* e = embed + (size_t)row_tok[row] * d;
    float4 v[NORM_MAX_CHUNKS];
    float ss = 0.0f;
#pragma unroll
    for (int u = 0; u < NORM_MAX_CHUNKS; ++u) {
        const int c = threadIdx.x + u * NORM_THREADS;
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < chunks) {
            const uint2 raw = *(const uint2*)(e + 4 * c);
            const bf16* b = (const bf16*)&raw;
            v[u] = make_float4(__bfloat162float(b[0]), __bfloat162float(b[1]), __bfloat162float(b[2]), __bfloat162float(b[3]));
            *(float4*)(x + (size_t)row * d + 4 * c) = v[u];
            ss += v[u].x * v[u].x + v[u].y * v[u].y + v[u].z * v[u].z + v[u].w * v[u].w;
        }
    }
    cl_img_clear_row_tail(img, gridDim.x, row, d);
    const float rstd = rsqrtf(block_sum(ss, red) / (float)d + eps);
#pragma unroll
    for (int u = 0; u < NORM_MAX_CHUNKS; ++u) {
        const int c = threadIdx.x + u * NORM_THREADS;
        if (c < chunks) {
            const float4 g = *(const float4*)(gain + 4 * c);
            store_split4(make_float4(v[u].x * rstd * g.x, v[u].y * rstd * g.y, v[u].z * rstd * g.z, v[u].w * rstd * g.w),
                         img ? (bf16*)(img + cl_img_offset(gridDim.x, row, 4 * c)) : h_hi + (size_t)row * d + 4 * c,
                         img ? (bf16*)(img + cl_img_offset(gridDim.x, gridDim.x + row, 4 * c)) : h_lo + (size_t)row * d + 4 * c);
        }
    }
}

// Decode steps: x = E[tok]; the first projection's operand image receives x * gain as hi + lo terms, un-normalised (the consumer
// applies 1 / RMS); the row's sum of squares goes to ss[row] (one part).
__global__ void __launch_bounds__(NORM_THREADS) embed_cl_kernel(const bf16* __restrict__ embed, const int* __restrict__ row_tok,
                                                                const float* __restrict__ gain, int d, float* __restrict__ x,
                                                                unsigned char* __restrict__ img, int img_rows, float* __restrict__ ss) {
    // The trigger comes after the wait here: whatever starts behind this kernel may then read the row plan at once.
    pdl_wait();
    pdl_trigger();
    __shared__ float red[32];
    const int row = blockIdx.x, chunks = d >> 2;
    const bf16* e = embed + (size_t)row_tok[row] * d;
    float acc = 0.0f;
    for (int c = threadIdx.x; c < chunks; c += NORM_THREADS) {
        const uint2 raw = *(const uint2*)(e + 4 * c);
        const bf16* b = (const bf16*)&raw;
        const float4 g = *(const float4*)(gain + 4 * c);
        const float4 v = make_float4(__bfloat162float(b[0]), __bfloat162float(b[1]), __bfloat162float(b[2]), __bfloat162float(b[3]));
        *(float4*)(x + (size_t)row * d + 4 * c) = v;
        store_split4(make_float4(v.x * g.x, v.y * g.y, v.z * g.z, v.w * g.w), (bf16*)(img + cl_img_offset(img_rows, row, 4 * c)),
                     (bf16*)(img + cl_img_offset(img_rows, img_rows + row, 4 * c)));        // 4 elements never straddle a 16-byte chunk
        acc += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
    cl_img_clear_row_tail(img, img_rows, row, d);
    const float t = block_sum(acc, red);
    if (threadIdx.x == 0) ss[row] = t;
}

// Single-sequence steps (row-range projections): x = E[tok]; the first projection's operand image receives
// x * gain as hi + lo terms, un-normalised; the row's sum of squares goes to ss[0][row] (one partial).
__global__ void __launch_bounds__(NORM_THREADS) embed_img_kernel(const bf16* __restrict__ embed, const int* __restrict__ row_tok,
                                                                 const float* __restrict__ gain, int d, float* __restrict__ x,
                                                                 unsigned char* __restrict__ img, float* __restrict__ ss) {
    pdl_trigger();
    pdl_wait();
    __shared__ float red[32];
    const int row = blockIdx.x, chunks = d >> 2;
    const bf16* e = embed + (size_t)row_tok[row] * d;
    float acc = 0.0f;
    for (int c = threadIdx.x; c < chunks; c += NORM_THREADS) {
        const uint2 raw = *(const uint2*)(e + 4 * c);
        const bf16* b = (const bf16*)&raw;
        const float4 g = *(const float4*)(gain + 4 * c);
        const float v[4] = {__bfloat162float(b[0]), __bfloat162float(b[1]), __bfloat162float(b[2]), __bfloat162float(b[3])};
        const float gg[4] = {g.x, g.y, g.z, g.w};
        *(float4*)(x + (size_t)row * d + 4 * c) = make_float4(v[0], v[1], v[2], v[3]);
        bf16 hi[4], lo[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) { split_bf16(v[t] * gg[t], hi[t], lo[t]); acc += v[t] * v[t]; }
        *(uint2*)(img + act_img_offset(row, 4 * c)) = *(const uint2*)hi;               // 4 elements never straddle a 16-byte chunk
        *(uint2*)(img + act_img_offset(ANPD_ROWS + row, 4 * c)) = *(const uint2*)lo;
    }
    const float t = block_sum(acc, red);
    if (threadIdx.x == 0) ss[row] = t;
}

// x[row] += sum of the tile's partial sums (in segment order); then h = rmsnorm(x) * gain as hi + lo.  NCH chunks of four features per
// thread.  Rows run two and more to an SM, so that one row's sums travel while another's are reduced (1536 rows of 4096: 31 -> 19 us).
// A wider row takes as few threads as its chunks need: 1024 for 1280 chunks left most of them idle and the SM to one row (13B, ten
// layers, eight prompts of 512: 33.2 -> 32.2 ms).  Up to 1024 chunks a block of 1024 is the better one even where some idle (1.1B, 333 rows, 2275 against 2340 us).
// Above 6144 features two rows share an SM with four chunks per thread, which are as many round trips one after the other: where there
// are SMs enough for the rows, up to 1024 threads with two chunks are faster (8192 wide, two layers: steps of eight sequences 878 -> 850
// us, 7168 wide, two: 495 -> 488; prompts of 1500 tokens 7185 with four, 7255 with two).
struct NormShape { int chunks, threads, per_sm; };
inline NormShape norm_shape(int d, int rows, int num_sms) {
    if (d <= 4 * NORM_THREADS) return {1, NORM_THREADS, 2};
    const bool half = d <= 8 * NORM_THREADS_2, room = rows <= num_sms && d <= 8 * NORM_THREADS;
    const int n = half || room ? 2 : NORM_MAX_CHUNKS;
    return {n, (d / 4 + 32 * n - 1) / (32 * n) * 32, half ? 2 : 1};
}
template <int NCH, int MAX_THREADS, int PER_SM>
__global__ void __launch_bounds__(MAX_THREADS, PER_SM) resid_norm_kernel(float* __restrict__ x, const float* __restrict__ part,
                                                                  const int* __restrict__ seg_count, size_t split_stride, int ld_part,
                                                                  const float* __restrict__ gain, float eps, int d,
                                                                  bf16* __restrict__ h_hi, bf16* __restrict__ h_lo, int ns_min,
                                                                  unsigned char* __restrict__ img) {
    // img: a decode step's operand image of gridDim.x rows instead of h_hi and h_lo.
    // ns_min: partial sums every tile of this projection has; seg_count: null, or each tile's own count.
    pdl_trigger();
    constexpr int AT = PER_SM == 2 ? 4 : 8;
    __shared__ float red[32];
    const int row = blockIdx.x, chunks = d >> 2;
    float4 v[NCH], gn[NCH];
    // the norm's gain is a weight: nothing of this step writes it, so it is fetched before the dependency wait
#pragma unroll
    for (int u = 0; u < NCH; ++u) {
        const int c = threadIdx.x + u * blockDim.x;
        gn[u] = (c < chunks) ? *(const float4*)(gain + 4 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    pdl_wait();
    float ss = 0.0f;
#pragma unroll
    for (int u = 0; u < NCH; ++u) {
        const int c = threadIdx.x + u * blockDim.x;
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < chunks) {
            const float* pr = part + (size_t)row * ld_part + 4 * c;
            float4 acc = *(const float4*)(x + (size_t)row * d + 4 * c);
            const int ns = seg_count ? seg_count[(4 * c) >> 7] : ns_min;
            for (int s0 = 0; s0 < ns; s0 += AT) {
                float4 p[AT];
#pragma unroll
                for (int k = 0; k < AT; ++k)
                    p[k] = (s0 + k < ns) ? *(const float4*)(pr + (size_t)(s0 + k) * split_stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int k = 0; k < AT; ++k)
                    if (s0 + k < ns) add4(acc, p[k]);
            }
            v[u] = acc;
            *(float4*)(x + (size_t)row * d + 4 * c) = acc;
            ss += acc.x * acc.x + acc.y * acc.y + acc.z * acc.z + acc.w * acc.w;
        }
    }
    cl_img_clear_row_tail(img, gridDim.x, row, d);
    const float rstd = rsqrtf(block_sum(ss, red) / (float)d + eps);
#pragma unroll
    for (int u = 0; u < NCH; ++u) {
        const int c = threadIdx.x + u * blockDim.x;
        if (c < chunks) {
            const float4 g = gn[u];
            store_split4(make_float4(v[u].x * rstd * g.x, v[u].y * rstd * g.y, v[u].z * rstd * g.z, v[u].w * rstd * g.w),
                         img ? (bf16*)(img + cl_img_offset(gridDim.x, row, 4 * c)) : h_hi + (size_t)row * d + 4 * c,
                         img ? (bf16*)(img + cl_img_offset(gridDim.x, gridDim.x + row, 4 * c)) : h_lo + (size_t)row * d + 4 * c);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// QKV epilogue: reduce splits, rotary embedding, append K/V to the paged cache, keep q
// ---------------------------------------------------------------------------------------------
// Bound by latency (a decode step) or by the partial sums' way through L2 (a prompt pass): a thread owns four rotary pairs, requests
// the sums several at a time, and has fetched what does not depend on the kernel before - the row plan (older than that kernel, see
// embed_norm_kernel), cosines and sines - while it waits.
struct RopeSum { float4 a, b; };

template <int AT_ONCE>
__device__ __forceinline__ RopeSum rope_sum(const float* __restrict__ pr, int half, size_t split_stride, int ns) {
    RopeSum r;
    r.a = r.b = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < ns; s0 += AT_ONCE) {
        float4 pa[AT_ONCE], pb[AT_ONCE];
#pragma unroll
        for (int s = 0; s < AT_ONCE; ++s)
            if (s0 + s < ns) { pa[s] = *(const float4*)(pr + (s0 + s) * split_stride); pb[s] = *(const float4*)(pr + (s0 + s) * split_stride + half); }
#pragma unroll
        for (int s = 0; s < AT_ONCE; ++s)
            if (s0 + s < ns) { add4(r.a, pa[s]); add4(r.b, pb[s]); }
    }
    return r;
}

__device__ __forceinline__ void rope_rotate(RopeSum& v, float4 c, float4 s) {
    const float4 a = v.a, b = v.b;
    v.a = make_float4(a.x * c.x - b.x * s.x, a.y * c.y - b.y * s.y, a.z * c.z - b.z * s.z, a.w * c.w - b.w * s.w);
    v.b = make_float4(b.x * c.x + a.x * s.x, b.y * c.y + a.y * s.y, b.z * c.z + a.z * s.z, b.w * c.w + a.w * s.w);
}

// queries leave as two bf16 terms, already multiplied by log2(e) / sqrt(hd): the attention kernels take them as MMA operands and
// work with base-2 exponentials
__device__ __forceinline__ void rope_store_q(const RopeSum& v, float q_scale, bf16* hi, bf16* lo, int half) {
    store_split4(make_float4(v.a.x * q_scale, v.a.y * q_scale, v.a.z * q_scale, v.a.w * q_scale), hi, lo);
    store_split4(make_float4(v.b.x * q_scale, v.b.y * q_scale, v.b.z * q_scale, v.b.w * q_scale), hi + half, lo + half);
}

__device__ __forceinline__ uint2 pack_bf16x4(float4 v) {
    const __nv_bfloat162 x = __floats2bfloat162_rn(v.x, v.y), y = __floats2bfloat162_rn(v.z, v.w);
    uint2 r;
    r.x = *(const uint32_t*)&x; r.y = *(const uint32_t*)&y;
    return r;
}

// A step: a block takes the 8 rows of one sequence through the heads blockIdx.x, blockIdx.x + gridDim.x, ..., hd / 8 threads per
// row.  A V head goes through shared memory, so that eight lanes write the rows' eight positions of a dimension of the transposed
// page: single elements, a page row apart, were most of the kernel's time (7B, 16 sequences: 14.9 -> 8.5 us, 8: 9.0 -> 6.4).
// seg_count is fixed by the model here and read before the wait.
template <int HD>
__global__ void __launch_bounds__(HD) qkv_rope_append_kernel(const float* __restrict__ part, const int* __restrict__ seg_count, size_t split_stride, int ld_part,
                                       const int* __restrict__ row_pos, const int* __restrict__ row_slot, const int* __restrict__ row_seq,
                                       const int* __restrict__ row_ok, const float* __restrict__ rope_cos,
                                       const float* __restrict__ rope_sin, const int* __restrict__ page_table,
                                       int pages_per_seq, int Hq, int Hkv, float q_scale, bf16* __restrict__ q_hi,
                                       bf16* __restrict__ q_lo, bf16* __restrict__ kpool_l, bf16* __restrict__ vpool_l, int ns_min) {
    pdl_trigger();
    constexpr int half = HD / 2, TPR = HD / 8;
    __shared__ float tile[ANPD_ROWS][HD + 1];
    __shared__ int s_page[ANPD_ROWS], s_slot[ANPD_ROWS];
    const int r = threadIdx.x / TPR, i = threadIdx.x % TPR * 4, row = blockIdx.y * ANPD_ROWS + r;
    const size_t at = (size_t)row_pos[row] * half + i;
    const float4 c = *(const float4*)(rope_cos + at), sn = *(const float4*)(rope_sin + at);
    const int slot = row_slot[row];               // where the row lives in the cache (its position, except for a second candidate)
    const int page = page_table[row_seq[row] * pages_per_seq + slot / KV_PAGE], ok = row_ok[row];
    if (i == 0) { s_page[r] = ok ? page : -1; s_slot[r] = slot % KV_PAGE; }
    int ns = seg_count ? seg_count[(blockIdx.x * HD) >> 7] : ns_min;          // a head never straddles a 128-column tile
    pdl_wait();
    for (int head = blockIdx.x; head < Hq + 2 * Hkv; head += gridDim.x) {
        if (seg_count && head != (int)blockIdx.x) ns = seg_count[(head * HD) >> 7];
        RopeSum v = rope_sum<4>(part + (size_t)row * ld_part + (size_t)head * HD + i, half, split_stride, ns);
        if (head < Hq + Hkv) rope_rotate(v, c, sn);
        if (head < Hq) {
            const size_t o = (size_t)row * Hq * HD + head * HD + i;
            rope_store_q(v, q_scale, q_hi + o, q_lo + o, half);
        } else if (head < Hq + Hkv) {             // K page: [position][dim]
            if (!ok) continue;
            bf16* dst = kpool_l + (((size_t)page * Hkv + head - Hq) * KV_PAGE + slot % KV_PAGE) * HD + i;
            *(uint2*)dst = pack_bf16x4(v.a);
            *(uint2*)(dst + half) = pack_bf16x4(v.b);
        } else {                                  // V page is kept transposed: [dim][position]
            __syncthreads();
            tile[r][i] = v.a.x; tile[r][i + 1] = v.a.y; tile[r][i + 2] = v.a.z; tile[r][i + 3] = v.a.w;
            tile[r][i + half] = v.b.x; tile[r][i + half + 1] = v.b.y; tile[r][i + half + 2] = v.b.z; tile[r][i + half + 3] = v.b.w;
            __syncthreads();
            const int wr = threadIdx.x & (ANPD_ROWS - 1), pg = s_page[wr];
            if (pg < 0) continue;
            bf16* dst = vpool_l + ((size_t)pg * Hkv + head - Hq - Hkv) * KV_PAGE * HD + s_slot[wr];
#pragma unroll
            for (int dim = threadIdx.x / ANPD_ROWS; dim < HD; dim += HD / ANPD_ROWS) dst[(size_t)dim * KV_PAGE] = __float2bfloat16_rn(tile[wr][dim]);
        }
    }
}

// The same for a prompt pass (every `seg` rows are consecutive positions of one sequence, a multiple of 8, the first a multiple of the page):
// a block takes 32 rows of the heads blockIdx.x, blockIdx.x + gridDim.x, ... and keeps their cosines and sines; a V head goes
// through shared memory, so that the transposed page receives whole 16-byte runs of positions instead of single elements.  Per
// element the arithmetic is that of qkv_rope_append_kernel, in the same order.  7B: 80 rows 14 -> 6 us, 1536 rows 41 -> 36.
constexpr int ROPE_TILE_ROWS = 32;
constexpr int ROPE_BLOCKS = 12;                  // a step's blocks per SM
template <int HD>
__global__ void __launch_bounds__(256, 3) qkv_rope_append_tile_kernel(const float* __restrict__ part, const int* __restrict__ seg_count, size_t split_stride,
                                                                   int ld_part, int seg, const int* __restrict__ row_pos, const int* __restrict__ row_seq,
                                                                   const int* __restrict__ row_ok, const float* __restrict__ rope_cos,
                                                                   const float* __restrict__ rope_sin, const int* __restrict__ page_table,
                                                                   int pages_per_seq, int Hq, int Hkv, float q_scale, bf16* __restrict__ q_hi,
                                                                   bf16* __restrict__ q_lo, bf16* __restrict__ kpool_l, bf16* __restrict__ vpool_l, int ns_min) {
    pdl_trigger();
    __shared__ float tile[ROPE_TILE_ROWS][HD + 1];
    constexpr int half = HD / 2, TPR = HD / 8, PER = ROPE_TILE_ROWS * TPR / 256;
    const int tiles = (seg + ROPE_TILE_ROWS - 1) / ROPE_TILE_ROWS, tile0 = blockIdx.y % tiles * ROPE_TILE_ROWS;
    const int r0 = blockIdx.y / tiles * seg + tile0, i = threadIdx.x % TPR * 4;
    const int nr = min(ROPE_TILE_ROWS, seg - tile0);
    const int pos0 = row_pos[r0];                        // the tile's rows hold positions pos0, pos0 + 1, ... inside one page
    const int page = page_table[row_seq[r0] * pages_per_seq + pos0 / KV_PAGE];
    float4 c[PER], sn[PER];
    bool keep[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int r = u * (256 / TPR) + threadIdx.x / TPR;
        keep[u] = false;
        if (r < nr) {
            const size_t at = (size_t)row_pos[r0 + r] * half + i;
            c[u] = *(const float4*)(rope_cos + at); sn[u] = *(const float4*)(rope_sin + at);
            keep[u] = row_ok[r0 + r] != 0;
        }
    }
    pdl_wait();
    for (int head = blockIdx.x; head < Hq + 2 * Hkv; head += gridDim.x) {
        const bool is_q = head < Hq, is_k = !is_q && head < Hq + Hkv;
        bf16* pg = (is_k ? kpool_l : vpool_l) + ((size_t)page * Hkv + (is_q ? 0 : is_k ? head - Hq : head - Hq - Hkv)) * KV_PAGE * HD;
        const int count = seg_count ? seg_count[(head * HD) >> 7] : ns_min;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int r = u * (256 / TPR) + threadIdx.x / TPR;
            if (r >= nr) continue;
            RopeSum v = rope_sum<4>(part + (size_t)(r0 + r) * ld_part + (size_t)head * HD + i, half, split_stride, count);
            if (is_q || is_k) rope_rotate(v, c[u], sn[u]);
            if (is_q) {
                const size_t o = (size_t)(r0 + r) * Hq * HD + (size_t)head * HD + i;
                rope_store_q(v, q_scale, q_hi + o, q_lo + o, half);
            } else if (is_k) {                           // K page: [position][dim]
                if (!keep[u]) continue;
                bf16* dst = pg + (size_t)((pos0 + r) % KV_PAGE) * HD + i;
                *(uint2*)dst = pack_bf16x4(v.a);
                *(uint2*)(dst + half) = pack_bf16x4(v.b);
            } else {
                tile[r][i] = v.a.x; tile[r][i + 1] = v.a.y; tile[r][i + 2] = v.a.z; tile[r][i + 3] = v.a.w;
                tile[r][i + half] = v.b.x; tile[r][i + half + 1] = v.b.y; tile[r][i + half + 2] = v.b.z; tile[r][i + half + 3] = v.b.w;
            }
        }
        if (is_q || is_k) continue;
        __syncthreads();                                 // V page, transposed: [dim][position]; 8 positions = 16 bytes
        for (int idx = threadIdx.x; idx < (ROPE_TILE_ROWS / 8) * HD; idx += 256) {
            const int dim = idx % HD, r8 = (idx / HD) * 8;
            if (r8 >= nr) continue;
            bf16 v[8];
            bool all = true;
#pragma unroll
            for (int e = 0; e < 8; ++e) { v[e] = __float2bfloat16_rn(tile[r8 + e][dim]); all = all && row_ok[r0 + r8 + e] != 0; }
            bf16* dst = pg + (size_t)dim * KV_PAGE + (pos0 % KV_PAGE) + r8;
            if (all) *(uint4*)dst = *(const uint4*)v;
            else
                for (int e = 0; e < 8; ++e) if (row_ok[r0 + r8 + e]) dst[e] = v[e];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------
// attention: per (key page, kv head, group of 8 rows) partial softmax, then a combine in page order
//
// The partial kernel works on tensor cores (mma.sync m16n8k16, bf16 in, fp32 out).  A K page is
// [128 keys][hd] and a V page is stored transposed, [hd][128 keys], so both are the "column" operand
// of an MMA and each thread fetches 16 contiguous bytes per fragment.  A block first issues every
// 16-byte asynchronous copy of its K and V page into (row-padded, bank-conflict-free) shared memory,
// so one block keeps up to 64 KB in flight, then computes from shared memory.  The
// 8 rows x G query heads that share a kv head are the MMA's 16-row tiles.  q and the softmax weights
// enter as two bf16 terms each (hi + lo), so only the cache's own bf16 rounding is left.  A warp walks
// its 32-key blocks in position order with a running (max, sum, output); warps that split a page are
// merged in block order; pages are merged by the combine kernel in page order.  Every one of these
// orders is a function of absolute key positions only, and a masked key contributes an exact zero,
// so a row's result does not depend on which other rows share the launch.
//
// Fragment bookkeeping (g = lane / 4, t = lane % 4): a 16-byte load gives a thread 8 consecutive
// elements e0..e7 of the contraction dimension; (e0,e1),(e2,e3) feed one MMA and (e4,e5),(e6,e7) a
// second one, and the other operand is permuted the same way, which leaves the sum unchanged.  For
// QK^T the key a thread column maps to is chosen so that the score fragments are, as they stand,
// the P fragments the PV product needs: logical key 8j + 2t + e of a block is actual key 8t + 2j + e.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void mma_bf16_16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// (x, y) -> packed bf16 pair of the high parts; `lo` receives the packed pair of the remainders.
__device__ __forceinline__ uint32_t pack_split(float x, float y, uint32_t& lo) {
    const bf16 hx = __float2bfloat16_rn(x), hy = __float2bfloat16_rn(y);
    const bf16 lx = __float2bfloat16_rn(x - __bfloat162float(hx)), ly = __float2bfloat16_rn(y - __bfloat162float(hy));
    lo = (uint32_t)__bfloat16_as_ushort(lx) | ((uint32_t)__bfloat16_as_ushort(ly) << 16);
    return (uint32_t)__bfloat16_as_ushort(hx) | ((uint32_t)__bfloat16_as_ushort(hy) << 16);
}

constexpr int ATTN_THREADS = 128;
constexpr int KEY_BLOCK = 32;

template <int HD>
__global__ void __launch_bounds__(ATTN_THREADS) attn_partial_kernel(const bf16* __restrict__ q_hi, const bf16* __restrict__ q_lo,
                                                                    const bf16* __restrict__ kpool_l, const bf16* __restrict__ vtpool_l,
                                                                    const int* __restrict__ page_table, int pages_per_seq,
                                                                    const int* __restrict__ row_pos, const int* __restrict__ row_seq, int Hq,
                                                                    int Hkv, float* __restrict__ pm, float* __restrict__ pl,
                                                                    float* __restrict__ po, const int* __restrict__ row_slot,
                                                                    const int* __restrict__ row_hole_lo, const int* __restrict__ row_hole_hi) {
    pdl_trigger();
    pdl_wait();
    constexpr int SLABS = HD / 32;            // 32-wide slabs of the head dimension (two MMAs each)
    constexpr int DT = HD / 8;                // 8-wide tiles of the head dimension for P V
    constexpr int OP = HD + 4;                // padded row of the merge buffer
    constexpr int KPITCH = HD * 2 + 64;       // bytes per staged K row (64 bytes of padding: conflict-free 16-byte reads)
    constexpr int VPITCH = KV_PAGE * 2 + 64;  // bytes per staged V^T row
    extern __shared__ __align__(16) unsigned char attn_smem[];
    unsigned char* Ks = attn_smem;                                  // [KV_PAGE][KPITCH]
    unsigned char* Vs = attn_smem + KV_PAGE * KPITCH;               // [HD][VPITCH]
    float (*sm_o)[16][OP] = (float (*)[16][OP])Ks;                  // [4][16][OP], reuses the K staging area after the last MMA
    __shared__ float sm_m[4][16], sm_l[4][16], sm_w[4][16];

    const int G = Hq / Hkv;
    const int MT = (ANPD_ROWS * G + 15) / 16;             // 16-row tiles of query vectors: 1, 1, 2, 4 for G = 1, 2, 4, 8
    const int KG = 4 / MT;                                // warps that split the page's four key blocks
    const int c = blockIdx.x, kvh = blockIdx.y, r0 = blockIdx.z * ANPD_ROWS;
    // row_slot (two-candidate steps): a row sees the cache slots up to its own, except a hidden range; otherwise slot = position
    const int pos_lo = row_pos[r0], pos_hi = row_slot ? row_slot[r0 + ANPD_ROWS - 1] : row_pos[r0 + ANPD_ROWS - 1];
    if (c * KV_PAGE > pos_hi) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, t = lane & 3;
    const int mt = warp % MT, kg = warp / MT;
    const int page = page_table[row_seq[r0] * pages_per_seq + c];
    const bf16* Kg = kpool_l + ((size_t)page * Hkv + kvh) * KV_PAGE * HD;
    const bf16* Vg = vtpool_l + ((size_t)page * Hkv + kvh) * KV_PAGE * HD;

    // stage the part of the page that any row can see: whole 32-key blocks up to pos_hi
    {
        const int nblk = min(KV_PAGE / KEY_BLOCK, (pos_hi - c * KV_PAGE) / KEY_BLOCK + 1);
        constexpr int KCH = HD * 2 / 16;                  // 16-byte chunks per K row
        for (int i = threadIdx.x; i < nblk * KEY_BLOCK * KCH; i += ATTN_THREADS) {
            const int row = i / KCH, ch = i % KCH;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(Ks + row * KPITCH + ch * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(Kg + (size_t)row * HD + ch * 8) : "memory");
        }
        const int vch = nblk * (KEY_BLOCK * 2 / 16);      // chunks per V^T row that hold visible keys
        for (int i = threadIdx.x; i < HD * vch; i += ATTN_THREADS) {
            const int row = i / vch, ch = i % vch;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(Vs + row * VPITCH + ch * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(Vg + (size_t)row * KV_PAGE + ch * 8) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }

    // this thread's two query vectors (rows gid and gid + 8 of tile mt) and their positions
    int qpos[2], qhl[2] = {0, 0}, qhh[2] = {0, 0};
    uint32_t qh[SLABS][2][4], ql[SLABS][2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int qi = mt * 16 + gid + 8 * h;
        const bool valid = qi < ANPD_ROWS * G;
        const int r = valid ? qi / G : 0, hl = valid ? qi % G : 0;
        qpos[h] = valid ? (row_slot ? row_slot[r0 + r] : pos_lo + r) : -1;                // -1: padding row, sees no key
        if (valid && row_slot) { qhl[h] = row_hole_lo[r0 + r]; qhh[h] = row_hole_hi[r0 + r]; }
        const size_t qoff = (size_t)(r0 + r) * Hq * HD + (size_t)(kvh * G + hl) * HD + 8 * t;
#pragma unroll
        for (int s = 0; s < SLABS; ++s) {
            // 16 bytes = elements 8t..8t+7 of the slab: (e0,e1),(e2,e3) feed the slab's first MMA, (e4,e5),(e6,e7)
            // the second.  Register h holds row gid + 8h for logical k = 2t, 2t+1; register 2 + h for 2t+8, 2t+9.
            uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
            if (valid) { a = *(const uint4*)(q_hi + qoff + 32 * s); b = *(const uint4*)(q_lo + qoff + 32 * s); }
            qh[s][0][h] = a.x; qh[s][0][2 + h] = a.y; qh[s][1][h] = a.z; qh[s][1][2 + h] = a.w;
            ql[s][0][h] = b.x; ql[s][0][2 + h] = b.y; ql[s][1][h] = b.z; ql[s][1][2 + h] = b.w;
        }
    }

    float m_run[2] = {-CUDART_INF_F, -CUDART_INF_F}, l_run[2] = {0.f, 0.f};
    float o[DT][4];
#pragma unroll
    for (int d = 0; d < DT; ++d) { o[d][0] = 0.f; o[d][1] = 0.f; o[d][2] = 0.f; o[d][3] = 0.f; }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    for (int blk = kg; blk < KV_PAGE / KEY_BLOCK; blk += KG) {
        const int kb0 = c * KV_PAGE + blk * KEY_BLOCK;
        if (kb0 > pos_hi) break;
        // ---- scores of 16 query vectors x 32 keys ----
        float sc[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            sc[j][0] = 0.f; sc[j][1] = 0.f; sc[j][2] = 0.f; sc[j][3] = 0.f;
            const int key_local = blk * KEY_BLOCK + 8 * (gid >> 1) + 2 * j + (gid & 1);
            const unsigned char* kr = Ks + key_local * KPITCH + 16 * t;
#pragma unroll
            for (int s = 0; s < SLABS; ++s) {
                const uint4 kv = *(const uint4*)(kr + 64 * s);
                mma_bf16_16816(sc[j], qh[s][0], kv.x, kv.y);
                mma_bf16_16816(sc[j], ql[s][0], kv.x, kv.y);
                mma_bf16_16816(sc[j], qh[s][1], kv.z, kv.w);
                mma_bf16_16816(sc[j], ql[s][1], kv.z, kv.w);
            }
        }
        // ---- running softmax per row; sc[j][2h + e] belongs to row h, actual key kb0 + 8t + 2j + e ----
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float mx = -CUDART_INF_F;
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int key = kb0 + 8 * t + 2 * j + e;
                    const float v = (key <= qpos[h] && !(key >= qhl[h] && key < qhh[h])) ? sc[j][2 * h + e] : -CUDART_INF_F;
                    sc[j][2 * h + e] = v;
                    mx = fmaxf(mx, v);
                }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float m_new = fmaxf(m_run[h], mx);
            const bool none = (m_new == -CUDART_INF_F);
            const float resc = none ? 1.0f : exp2f(m_run[h] - m_new);
            float psum = 0.0f;
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float p = none ? 0.0f : exp2f(sc[j][2 * h + e] - m_new);
                    sc[j][2 * h + e] = p;
                    psum += p;
                }
            psum += __shfl_xor_sync(0xffffffffu, psum, 1);
            psum += __shfl_xor_sync(0xffffffffu, psum, 2);
            l_run[h] = l_run[h] * resc + psum;
            m_run[h] = m_new;
#pragma unroll
            for (int d = 0; d < DT; ++d) { o[d][2 * h] *= resc; o[d][2 * h + 1] *= resc; }
        }
        // ---- P fragments (hi + lo) for the two MMAs over this block's 32 keys ----
        uint32_t ph[2][4], plo[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            ph[u][0] = pack_split(sc[2 * u][0], sc[2 * u][1], plo[u][0]);            // row gid,     keys 8t + 4u + {0,1}
            ph[u][1] = pack_split(sc[2 * u][2], sc[2 * u][3], plo[u][1]);            // row gid + 8
            ph[u][2] = pack_split(sc[2 * u + 1][0], sc[2 * u + 1][1], plo[u][2]);    // row gid,     keys 8t + 4u + {2,3}
            ph[u][3] = pack_split(sc[2 * u + 1][2], sc[2 * u + 1][3], plo[u][3]);    // row gid + 8
        }
        // ---- O += P V : V^T rows are head dimensions, 16 bytes = keys 8t .. 8t+7 of the block ----
#pragma unroll
        for (int d = 0; d < DT; ++d) {
            const uint4 vv = *(const uint4*)(Vs + (8 * d + gid) * VPITCH + (blk * KEY_BLOCK + 8 * t) * 2);
            mma_bf16_16816(o[d], ph[0], vv.x, vv.y);
            mma_bf16_16816(o[d], plo[0], vv.x, vv.y);
            mma_bf16_16816(o[d], ph[1], vv.z, vv.w);
            mma_bf16_16816(o[d], plo[1], vv.z, vv.w);
        }
    }

    // ---- merge the warps that split this page (block order), write the page's partial ----
    __syncthreads();                                      // every warp is done reading the staged K rows
    if (t == 0) {
        sm_m[warp][gid] = m_run[0]; sm_m[warp][gid + 8] = m_run[1];
        sm_l[warp][gid] = l_run[0]; sm_l[warp][gid + 8] = l_run[1];
    }
#pragma unroll
    for (int d = 0; d < DT; ++d) {
        sm_o[warp][gid][8 * d + 2 * t] = o[d][0];
        sm_o[warp][gid][8 * d + 2 * t + 1] = o[d][1];
        sm_o[warp][gid + 8][8 * d + 2 * t] = o[d][2];
        sm_o[warp][gid + 8][8 * d + 2 * t + 1] = o[d][3];
    }
    __syncthreads();
    // weights of the merged warps, once per query vector
    if (threadIdx.x < MT * 16) {
        const int tile = threadIdx.x / 16, rowi = threadIdx.x % 16;
        float M = -CUDART_INF_F;
        for (int k = 0; k < KG; ++k) M = fmaxf(M, sm_m[k * MT + tile][rowi]);
        float L = 0.0f;
        for (int k = 0; k < KG; ++k) {
            const float mk = sm_m[k * MT + tile][rowi];
            const float w = (mk == -CUDART_INF_F) ? 0.0f : exp2f(mk - M);
            sm_w[k * MT + tile][rowi] = w;
            L = fmaf(sm_l[k * MT + tile][rowi], w, L);
        }
        const int qi = tile * 16 + rowi;
        if (qi < ANPD_ROWS * G) {
            const size_t out = ((size_t)(r0 + qi / G) * Hq + (kvh * G + qi % G)) * pages_per_seq + c;
            pm[out] = M;
            pl[out] = L;
        }
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < MT * 16 * (HD / 4); idx += ATTN_THREADS) {
        const int d4 = idx % (HD / 4), rowi = (idx / (HD / 4)) % 16, tile = idx / ((HD / 4) * 16);
        const int qi = tile * 16 + rowi;
        if (qi >= ANPD_ROWS * G) continue;
        float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = 0; k < KG; ++k) {
            const float w = sm_w[k * MT + tile][rowi];
            const float4 v = *(const float4*)&sm_o[k * MT + tile][rowi][4 * d4];
            O.x = fmaf(v.x, w, O.x); O.y = fmaf(v.y, w, O.y); O.z = fmaf(v.z, w, O.z); O.w = fmaf(v.w, w, O.w);
        }
        const size_t out = ((size_t)(r0 + qi / G) * Hq + (kvh * G + qi % G)) * pages_per_seq + c;
        *(float4*)(po + out * HD + 4 * d4) = O;
    }
}

// One block per (row, q head): fold the pages 0..pos/KV_PAGE, write the output as hi+lo.  The block is
// hd x 4 threads: thread (dim, k) adds the pages k, k+4, k+8, ... in ascending order, the four slices
// are then added in slice order - a fixed order for a given number of pages.  Page maxima and sums are
// fetched once by the first threads, so the kernel is about two memory round trips long.
constexpr int COMBINE_SLICES = 4;
constexpr int COMBINE_MAX_PAGES = 256;
__global__ void attn_combine_kernel(const float* __restrict__ pm, const float* __restrict__ pl, const float* __restrict__ po,
                                    const int* __restrict__ row_pos, int Hq, int hd, int pages_per_seq,
                                    bf16* __restrict__ ao_hi, bf16* __restrict__ ao_lo, unsigned char* __restrict__ img, int img_rows) {
    // row_pos: the rows' cache slots (= positions outside two-candidate steps)
    pdl_trigger();
    pdl_wait();
    __shared__ float s_w[COMBINE_MAX_PAGES];            // page maxima, then page weights
    __shared__ float s_l[COMBINE_MAX_PAGES];
    __shared__ float s_o[COMBINE_SLICES][128];
    __shared__ float s_L;
    const int row = blockIdx.x, head = blockIdx.y;
    const int dim = threadIdx.x % hd, slice = threadIdx.x / hd;
    const int nc = min(row_pos[row] / KV_PAGE + 1, COMBINE_MAX_PAGES);
    const size_t base = ((size_t)row * Hq + head) * pages_per_seq;
    for (int c = threadIdx.x; c < nc; c += blockDim.x) { s_w[c] = pm[base + c]; s_l[c] = pl[base + c]; }
    __syncthreads();
    float M = -CUDART_INF_F;
    for (int c = 0; c < nc; ++c) M = fmaxf(M, s_w[c]);
    __syncthreads();
    for (int c = threadIdx.x; c < nc; c += blockDim.x) s_w[c] = exp2f(s_w[c] - M);     // partial maxima are in the base-2 domain
    __syncthreads();
    if (threadIdx.x == 0) {
        float L = 0.0f;
        for (int c = 0; c < nc; ++c) L = fmaf(s_l[c], s_w[c], L);
        s_L = L;
    }
    float o = 0.0f;
    for (int c0 = slice; c0 < nc; c0 += 4 * COMBINE_SLICES) {
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + u * COMBINE_SLICES;
            v[u] = (c < nc) ? po[(base + c) * hd + dim] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + u * COMBINE_SLICES;
            if (c < nc) o = fmaf(v[u], s_w[c], o);
        }
    }
    s_o[slice][dim] = o;
    __syncthreads();
    if (slice == 0) {
        float t = s_o[0][dim];
        for (int k = 1; k < COMBINE_SLICES; ++k) t += s_o[k][dim];
        bf16 hi, lo;
        split_bf16(t / s_L, hi, lo);
        if (img_rows > 0) {                               // straight into the O projection's operand image
            *(bf16*)(img + cl_img_offset(img_rows, row, head * hd + dim)) = hi;
            *(bf16*)(img + cl_img_offset(img_rows, img_rows + row, head * hd + dim)) = lo;
        } else if (img) {                                 // the same for the row-range projections
            *(bf16*)(img + act_img_offset(row, head * hd + dim)) = hi;
            *(bf16*)(img + act_img_offset(ANPD_ROWS + row, head * hd + dim)) = lo;
        } else {
            const size_t out = (size_t)row * Hq * hd + head * hd + dim;
            ao_hi[out] = hi;
            ao_lo[out] = lo;
        }
    }
}

// The same for many rows (prefill passes), shaped for throughput: four warps per (row, q head), a lane owns hd/32
// consecutive dimensions and fetches them in one load per page.  Slices, page order within a slice, the order of the
// slices and the total weight are those of attn_combine_kernel, so the results are the same bits.
template <int VEC>
__global__ void __launch_bounds__(32 * COMBINE_SLICES) attn_combine_wide_kernel(const float* __restrict__ pm, const float* __restrict__ pl,
                                                                               const float* __restrict__ po, const int* __restrict__ row_pos,
                                                                               int Hq, int pages_per_seq, bf16* __restrict__ ao_hi,
                                                                               bf16* __restrict__ ao_lo, unsigned char* __restrict__ img, int img_rows) {
    pdl_trigger();
    pdl_wait();
    constexpr int hd = 32 * VEC;
    __shared__ float s_m[COMBINE_MAX_PAGES];
    __shared__ float s_l[COMBINE_MAX_PAGES];
    __shared__ float s_o[COMBINE_SLICES][hd];
    const int row = blockIdx.x, head = blockIdx.y;
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int nc = min(row_pos[row] / KV_PAGE + 1, COMBINE_MAX_PAGES);
    const size_t base = ((size_t)row * Hq + head) * pages_per_seq;
    for (int c = threadIdx.x; c < nc; c += blockDim.x) { s_m[c] = pm[base + c]; s_l[c] = pl[base + c]; }
    __syncthreads();
    float M = -CUDART_INF_F;
    for (int c = 0; c < nc; ++c) M = fmaxf(M, s_m[c]);
    float L = 0.0f;
    for (int c = 0; c < nc; ++c) L = fmaf(s_l[c], exp2f(s_m[c] - M), L);       // partial maxima are in the base-2 domain
    float o[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) o[e] = 0.0f;
    for (int c = slice; c < nc; c += COMBINE_SLICES) {
        const float w = exp2f(s_m[c] - M);
        const float* src = po + (base + c) * hd + lane * VEC;
        float v[VEC];
        if (VEC == 4) { const float4 t = *(const float4*)src; v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w; }
        else { const float2 t = *(const float2*)src; v[0] = t.x; v[1] = t.y; }
#pragma unroll
        for (int e = 0; e < VEC; ++e) o[e] = fmaf(v[e], w, o[e]);
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) s_o[slice][lane * VEC + e] = o[e];
    __syncthreads();
    if (slice == 0) {
        const size_t out = (size_t)row * Hq * hd + head * hd + lane * VEC;
        const int k = head * hd + lane * VEC;
        bf16* dst_hi = img_rows > 0 ? (bf16*)(img + cl_img_offset(img_rows, row, k)) : ao_hi + out;       // VEC elements never straddle a 16-byte chunk
        bf16* dst_lo = img_rows > 0 ? (bf16*)(img + cl_img_offset(img_rows, img_rows + row, k)) : ao_lo + out;
        bf16 h[VEC], l[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            float t = s_o[0][lane * VEC + e];
            for (int k = 1; k < COMBINE_SLICES; ++k) t += s_o[k][lane * VEC + e];
            split_bf16(t / L, h[e], l[e]);
        }
        if (VEC == 4) { *(uint2*)dst_hi = *(const uint2*)h; *(uint2*)dst_lo = *(const uint2*)l; }
        else { *(uint32_t*)dst_hi = *(const uint32_t*)h; *(uint32_t*)dst_lo = *(const uint32_t*)l; }
    }
}

// ---------------------------------------------------------------------------------------------
// SwiGLU epilogue of the gate/up projection
// ---------------------------------------------------------------------------------------------
// A thread owns CH chunks of four consecutive features (a block's width apart) and requests the sums every tile has (ns_min) several at
// a time; seg_count, null where all tiles have as many, tells of more.  Bound by those sums' way through L2; two chunks where the
// rows fill the device, one where parallelism is short.
template <int CH>
__global__ void __launch_bounds__(256, CH == 1 ? 4 : 5) swiglu_kernel(const float* __restrict__ part, const int* __restrict__ seg_count, size_t split_stride, int ld_part, int F, int from,
                                                     bf16* __restrict__ act_hi, bf16* __restrict__ act_lo, int ns_min, unsigned char* __restrict__ img) {
    // img: an operand image of gridDim.y rows instead of act_hi and act_lo; from: the projection has finished the features before it
    pdl_trigger();
    pdl_wait();
    const int row = blockIdx.y, j0 = from + 4 * (CH * blockIdx.x * blockDim.x + threadIdx.x);
    constexpr int AT = CH == 1 ? 4 : 1;
    const float* pr = part + (size_t)row * ld_part;
    if (blockIdx.x == 0) cl_img_clear_row_tail(img, gridDim.y, row, F);
    float4 g4[CH], u4[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) g4[c] = u4[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < ns_min; s0 += AT) {
        float4 pg[CH][AT], pu[CH][AT];
#pragma unroll
        for (int c = 0; c < CH; ++c)
#pragma unroll
            for (int s = 0; s < AT; ++s) {
                const int j = j0 + c * 4 * blockDim.x;
                if (s0 + s < ns_min && j < F) { pg[c][s] = *(const float4*)(pr + (s0 + s) * split_stride + j); pu[c][s] = *(const float4*)(pr + (s0 + s) * split_stride + F + j); }
            }
#pragma unroll
        for (int c = 0; c < CH; ++c)
#pragma unroll
            for (int s = 0; s < AT; ++s)
                if (s0 + s < ns_min && j0 + c * 4 * (int)blockDim.x < F) { add4(g4[c], pg[c][s]); add4(u4[c], pu[c][s]); }
    }
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        const int j = j0 + c * 4 * blockDim.x;
        if (j >= F) continue;
        if (seg_count)                                   // a 128-position storage tile holds 64 gate features and their up features
            for (int s = ns_min; s < seg_count[j >> 6]; ++s) { add4(g4[c], *(const float4*)(pr + s * split_stride + j)); add4(u4[c], *(const float4*)(pr + s * split_stride + F + j)); }
        const float gte[4] = {g4[c].x, g4[c].y, g4[c].z, g4[c].w}, up[4] = {u4[c].x, u4[c].y, u4[c].z, u4[c].w};
        bf16 hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) split_bf16(gte[e] / (1.0f + expf(-gte[e])) * up[e], hi[e], lo[e]);
        *(uint2*)(img ? (bf16*)(img + cl_img_offset(gridDim.y, row, j)) : act_hi + (size_t)row * F + j) = *(const uint2*)hi;
        *(uint2*)(img ? (bf16*)(img + cl_img_offset(gridDim.y, gridDim.y + row, j)) : act_lo + (size_t)row * F + j) = *(const uint2*)lo;
    }
}

// ---------------------------------------------------------------------------------------------
// LM-head epilogue: reduce splits, (optionally) keep logits, per-block argmax with ties to the lowest id
// ---------------------------------------------------------------------------------------------
constexpr int AMAX_COLS = 1024;
__global__ void __launch_bounds__(256) argmax_partial_kernel(const float* __restrict__ part, const int* __restrict__ seg_count, int n_parts, size_t split_stride,
                                                             int ld_part, int V, float* __restrict__ logits,
                                                             float* __restrict__ amax_val, int* __restrict__ amax_idx, int nblk) {
    pdl_trigger();
    pdl_wait();
    __shared__ float sv[8];
    __shared__ int si[8];
    const int row = blockIdx.y;
    const float* pr = part + (size_t)row * ld_part;
    float best = -CUDART_INF_F;
    int bidx = 0x7fffffff;
    const int v = blockIdx.x * AMAX_COLS + 4 * threadIdx.x;              // four consecutive features (the slabs' rows are padded)
    if (v < V) {
        float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const int ns = seg_count ? seg_count[v >> 7] : n_parts;
#pragma unroll 4
        for (int s = 0; s < ns; ++s) add4(z4, *(const float4*)(pr + s * split_stride + v));
        const float z[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (v + e >= V) break;
            if (logits) logits[(size_t)row * V + v + e] = z[e];
            if (z[e] > best) { best = z[e]; bidx = v + e; }     // ascending: strict > keeps the lowest id
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
        if (ov > best || (ov == best && oi < bidx)) { best = ov; bidx = oi; }
    }
    if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = best; si[threadIdx.x >> 5] = bidx; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w)
            if (sv[w] > best || (sv[w] == best && si[w] < bidx)) { best = sv[w]; bidx = si[w]; }
        amax_val[(size_t)row * nblk + blockIdx.x] = best;
        amax_idx[(size_t)row * nblk + blockIdx.x] = bidx;
    }
}

// Final argmax per row, draft compare, prefix accept, KV commit, token-buffer append.
__global__ void __launch_bounds__(256) accept_kernel(SeqState* seqs, const float* __restrict__ amax_val,
                                                     const int* __restrict__ amax_idx, int nblk, int mode,
                                                     const NgramDev* ctxs, int seq_arg, int last_row, int prompt_len, int two) {
    // a prompt pass: block b takes sequence seq_arg + b, whose last token's row is last_row + 8 b
    pdl_trigger();
    pdl_wait();
    __shared__ int pred[ANPD_ROWS];
    const int b = (mode == ACCEPT_PREFILL ? seq_arg : 0) + blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        const int row = (mode == ACCEPT_PREFILL) ? (last_row / ANPD_ROWS + blockIdx.x) * ANPD_ROWS + warp : b * ANPD_ROWS + warp;
        float best = -CUDART_INF_F;
        int bidx = 0x7fffffff;
        for (int i = lane; i < nblk; i += 32) {
            const float v = amax_val[(size_t)row * nblk + i];
            const int id = amax_idx[(size_t)row * nblk + i];
            if (v > best || (v == best && id < bidx)) { best = v; bidx = id; }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
            if (ov > best || (ov == best && oi < bidx)) { best = ov; bidx = oi; }
        }
        if (lane == 0) pred[warp] = bidx;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    SeqState& s = seqs[b];
    if (mode == ACCEPT_PREFILL) {
        const int nxt = pred[last_row % ANPD_ROWS];
        s.next_tok = nxt;
        s.kv_len = prompt_len;
        s.accepted_len = 0;
        if (ctxs) {
            const NgramDev& c = ctxs[b];
            const int T = c.state[0];
            if (T + 1 > c.max_ctx) { s.error = ERR_CTX_FULL; s.active = 0; return; }
            c.tokens[T] = nxt;
            c.state[0] = T + 1;
        }
        return;
    }
    int a = 0;
    const int ka = s.draft_len;
    while (a < ka && s.draft[a] == pred[a]) ++a;
    for (int r = 0; r < ANPD_ROWS; ++r) s.pred[r] = pred[r];
    // A second candidate (rows ka+1..ka+kb): its first token is judged by row 0's prediction, token j by the prediction of
    // its own row before (row ka+j).  It is kept when its accepted prefix is strictly longer; the first candidate wins ties.
    const int kb = two ? min(s.draft2_len, ANPD_K_MAX - ka) : 0;
    const int* chosen = s.draft;
    int nxt = pred[a];
    if (two) s.move_n = 0;
    if (kb > 0 && s.draft2[0] == pred[0]) {
        int ab = 1;
        while (ab < kb && s.draft2[ab] == pred[ka + ab]) ++ab;
        if (ab > a) {
            chosen = s.draft2;
            a = ab;
            nxt = pred[ka + ab];
            if (mode == ACCEPT_COMMIT && s.active) {           // its K/V rows sit behind the first candidate's: ask for the move
                s.move_from = s.kv_len + ka + 1;
                s.move_to = s.kv_len + 1;
                s.move_n = ab;
                s.alt_wins += 1;
            }
        }
    }
    s.accepted_len = a;
    s.next_tok = nxt;
    if (mode != ACCEPT_COMMIT || !s.active) return;
    s.kv_len += a + 1;
    s.steps += 1;
    s.drafted += ka + kb;
    s.accepted += a;
    s.hist[a] += 1;
    if (ctxs) {
        const NgramDev& c = ctxs[b];
        const int T = c.state[0];
        if (T + a + 1 > c.max_ctx) { s.error = ERR_CTX_FULL; s.active = 0; return; }
        for (int i = 0; i < a; ++i) c.tokens[T + i] = chosen[i];
        c.tokens[T + a] = nxt;
        c.state[0] = T + a + 1;
        if (T + a + 1 >= s.stop_at) s.active = 0;
    }
}

// Two-candidate steps: when the second candidate won, its accepted rows' K and V move from the slots behind the first
// candidate's to the positions they belong to (SeqState::move_*).  One thread per (layer, kv head, dim) walks the rows in
// ascending order, so overlapping ranges behave like memmove.  grid (layers * kv heads, batch), hd threads.
__global__ void kv_move_kernel(const SeqState* __restrict__ seqs, const int* __restrict__ page_table, int pages_per_seq, int Hkv, int hd,
                               size_t layer_elems, bf16* __restrict__ kpool, bf16* __restrict__ vpool) {
    pdl_trigger();
    pdl_wait();
    const SeqState& s = seqs[blockIdx.y];
    const int n = s.move_n;
    if (n <= 0) return;
    const int layer = blockIdx.x / Hkv, kvh = blockIdx.x % Hkv, i = threadIdx.x;
    for (int j = 0; j < n; ++j) {
        const int from = s.move_from + j, to = s.move_to + j;
        const size_t pf = ((size_t)page_table[blockIdx.y * pages_per_seq + from / KV_PAGE] * Hkv + kvh) * KV_PAGE * hd + layer * layer_elems;
        const size_t pt = ((size_t)page_table[blockIdx.y * pages_per_seq + to / KV_PAGE] * Hkv + kvh) * KV_PAGE * hd + layer * layer_elems;
        kpool[pt + (size_t)(to % KV_PAGE) * hd + i] = kpool[pf + (size_t)(from % KV_PAGE) * hd + i];
        vpool[pt + (size_t)i * KV_PAGE + (to % KV_PAGE)] = vpool[pf + (size_t)i * KV_PAGE + (from % KV_PAGE)];
    }
}

// ---------------------------------------------------------------------------------------------
// weight-streaming GEMM, plain version: one warp per output feature, 8 rows at a time
//   part[0][row][n] = sum_k W[n][k] * (a_hi[row][k] + a_lo[row][k])
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) gemm_rows8_kernel(const unsigned char* __restrict__ W, const bf16* __restrict__ a_hi,
                                                         const bf16* __restrict__ a_lo, int rows, const ClPlan plan,
                                                         float* __restrict__ part, int ld_part) {
    pdl_trigger();
    pdl_wait();
    const int n = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int N = plan.N, K = plan.K;
    if (n >= N) return;
    const int pos = cl_position(plan, n);
    for (int r0 = 0; r0 < rows; r0 += 8) {
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int k0 = lane * 8; k0 < K; k0 += 256) {
            const uint4 wv = *(const uint4*)(W + cl_weight_offset(plan, pos, k0));
            const bf16* w8 = (const bf16*)&wv;
            float wf[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) wf[e] = __bfloat162float(w8[e]);
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const uint4 hv = *(const uint4*)(a_hi + (size_t)(r0 + r) * K + k0);
                const uint4 lv = *(const uint4*)(a_lo + (size_t)(r0 + r) * K + k0);
                const bf16* h8 = (const bf16*)&hv;
                const bf16* l8 = (const bf16*)&lv;
                float a = acc[r];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    a = fmaf(wf[e], __bfloat162float(h8[e]), a);
                    a = fmaf(wf[e], __bfloat162float(l8[e]), a);
                }
                acc[r] = a;
            }
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            float a = acc[r];
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane == 0) part[(size_t)(r0 + r) * ld_part + n] = a;
        }
    }
}

// segment counts of a prompt-pass projection whose last tiles alone are cut along K
__global__ void fill_tail_segs_kernel(int* segs, int m_tiles, int first_cut, int parts) {
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m_tiles) segs[i] = i >= first_cut ? parts : 1;
}

// groups of 8 rows, `step` rows apart, from row `from` of the normalised activations on -> rows 0, 1, ... of a decode step's operand image
__global__ void rows_to_image_kernel(const bf16* __restrict__ h_hi, const bf16* __restrict__ h_lo, int from, int step, int d, unsigned char* __restrict__ img,
                                     int img_rows) {
    pdl_trigger();
    pdl_wait();
    const int r = blockIdx.x;
    const size_t src = (size_t)(from + r / ANPD_ROWS * step + r % ANPD_ROWS) * d;
    cl_img_clear_row_tail(img, img_rows, r, d);
    for (int i = threadIdx.x; i < d / 8; i += blockDim.x) {
        *(uint4*)(img + cl_img_offset(img_rows, r, 8 * i)) = ((const uint4*)(h_hi + src))[i];
        *(uint4*)(img + cl_img_offset(img_rows, img_rows + r, 8 * i)) = ((const uint4*)(h_lo + src))[i];
    }
}

// rows [from, from + 8) of the normalised activations -> rows [0, 8)
__global__ void move_rows_kernel(bf16* __restrict__ h_hi, bf16* __restrict__ h_lo, int from, int d) {
    pdl_trigger();
    pdl_wait();
    if (from == 0) return;
    const int r = blockIdx.x;
    for (int i = threadIdx.x; i < d / 8; i += blockDim.x) {
        ((uint4*)(h_hi + (size_t)r * d))[i] = ((const uint4*)(h_hi + (size_t)(from + r) * d))[i];
        ((uint4*)(h_lo + (size_t)r * d))[i] = ((const uint4*)(h_lo + (size_t)(from + r) * d))[i];
    }
}

// Whether the projections of a forward of `rows` rows run on the decode kernels (weights streamed once, several partial sums per
// output, operand images): decode steps, and prompt passes of up to CL_PROMPT_ROWS rows - as many as the tensor memory holds for
// it.  There the weights bound a pass and this kernel streams them better: 7B, pass of 77 tokens 8.7 -> 4.7 ms, of 128 5.5 ms,
// where 129 on the prompt GEMM take 5.9.
static bool cl_rows(const anpd_model* m, const anpd_kv* kv, int rows) {
    return !m->plain_gemm && (rows == kv->batch * ANPD_ROWS || rows <= CL_PROMPT_ROWS);
}

// One projection of a prompt pass, of a step of several sequences or, with the plain GEMM, of any forward.  Returns how many
// partial sums every output has and, where some 128-feature storage tiles have more, all tiles' counts.  finished: of a gate-up
// projection, the activations that it has written itself.
anpd_status gemm_enqueue(anpd_model* m, anpd_kv* kv, int kind, int layer, int rows, const int** seg_count_out, int* seg_min_out, int* finished = nullptr) {
    Workspace& ws = kv->ws;
    if (finished) *finished = 0;
    const ClPlan& plan = m->cl[kind];
    const unsigned char* W = kind == GK_LM ? m->lm_head : (kind == GK_QKV ? m->layers[layer].wqkv : kind == GK_O ? m->layers[layer].wo
                                                          : kind == GK_GU ? m->layers[layer].wgu : m->layers[layer].wd);
    const bf16 *a_hi = ws.h_hi, *a_lo = ws.h_lo;
    const CUtensorMap* maps = ws.map_h;
    if (kind == GK_O) { a_hi = ws.ao_hi; a_lo = ws.ao_lo; maps = ws.map_ao; }
    if (kind == GK_DOWN) { a_hi = ws.act_hi; a_lo = ws.act_lo; maps = ws.map_act; }
    if (m->plain_gemm) {
        *seg_count_out = nullptr;
        *seg_min_out = 1;
        return gemm_plain_enqueue(plan, W, a_hi, a_lo, rows, ws.part, ws.ld[kind], m->stream, &m->prof);
    }
    if (cl_rows(m, kv, rows)) {                        // a partial sum per CTA of a cluster
        const unsigned char* act = kind == GK_O ? ws.ci_ao : kind == GK_DOWN ? ws.ci_act : ws.ci_h;
        if (const GemmPlan* tc = tc_model_plan(m, kind, rows)) {
            *seg_count_out = tc->d_seg_count;
            *seg_min_out = tc->min_segs;
            return gemm_tc_model_enqueue(*tc, plan, W, act, rows, ws.part, (size_t)rows * ws.ld[kind], ws.ld[kind], ws.gemm_err, m->stream, &m->prof);
        }
        *seg_count_out = nullptr;
        *seg_min_out = CL_CTAS;
        // (no L2 prefetch for the projection after this one: two sequences, 13B, 8 layers 1103 -> 1066 us without, 7B 754 -> 746, larger batches equal)
        return cl_partial_enqueue(plan, W, act, rows, ws.part, (size_t)rows * ws.ld[kind], ws.ld[kind], ws.gemm_err, m->stream, &m->prof);
    }
    // a prompt pass: complete sums, or several per output
    const int m_tiles = m->plan[kind].m_tiles;
    if (ws.pf_rows != rows) {
        for (int k = 0; k < GK_LM; ++k)
            ws.pf_sched[k] = prompt_schedule(m, ws, k, rows);
        ws.pf_rows = rows;
    }
    const PfSchedule sched = ws.pf_sched[kind];
    if (sched.tail_split > 1) {                        // feature tiles from `first` on come in tail_split parts, the others in one
        const int first = 2 * (sched.tail_from / sched.n_tt), cfg = first * PF_MAX_PARTS + sched.tail_split;
        if (m->tail_cfg[kind] != cfg) {
            LAUNCH(&m->prof, m->stream, KC_OTHER, 0,
                   (launch_k(fill_tail_segs_kernel, (m_tiles + 127) / 128, 128, 0, m->stream, m->d_tail_segs[kind], m_tiles, first, sched.tail_split)));
            m->tail_cfg[kind] = cfg;
        }
        *seg_count_out = m->d_tail_segs[kind];
    } else {
        *seg_count_out = nullptr;
    }
    *seg_min_out = sched.ksplit;
    // a pair of storage tiles holds 128 gate features and their up features
    if (finished && sched.ksplit == 1) *finished = std::min(m->cfg.d_ffn, sched.tail_split > 1 ? 128 * (sched.tail_from / sched.n_tt) : m->cfg.d_ffn);
    return gemm_pf_enqueue(plan, W, maps[0], maps[1], rows, ws.part, ws.ld[kind], (size_t)rows * ws.ld[kind], finished ? ws.act_hi : nullptr, finished ? ws.act_lo : nullptr, sched, m->num_sms,
                           ws.gemm_err, m->stream, &m->prof);
}

template <int HD>
anpd_status attn_enqueue(anpd_model* m, anpd_kv* kv, int layer, int rows, int max_pos, unsigned char* img = nullptr, bool tree = false, int img_rows = 0, int n_seq = 1) {
    const anpd_model_config& c = m->cfg;
    Workspace& ws = kv->ws;
    const size_t layer_elems = (size_t)kv->total_pages * c.n_kv_heads * KV_PAGE * HD;
    const int chunks = max_pos / KV_PAGE + 1;
    const size_t smem = (size_t)KV_PAGE * (HD * 2 + 64) + (size_t)HD * (KV_PAGE * 2 + 64);
    static_assert(4 * 16 * (HD + 4) * sizeof(float) <= (size_t)KV_PAGE * (HD * 2 + 64), "merge buffer must fit in the K staging area");
    static bool attr_set[64] = {false};
    if (first_call_on_device(attr_set)) {
        CUDA_TRY(cudaFuncSetAttribute(attn_partial_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    }
    // a prompt pass: pages are folded in the kernel, nothing to merge (the older 16-row kernel knows one query head per kv head only)
    if (rows != kv->batch * ANPD_ROWS && kv->attn_pf) return attn_pf_enqueue(m, kv, layer, rows, img, n_seq);
    if (HD == 128 && kv->attn_tc && rows != kv->batch * ANPD_ROWS && c.n_q_heads == c.n_kv_heads) {
        ANPD_TRY(attn_prompt_enqueue(m, kv, layer, rows));
        if (img) LAUNCH(&m->prof, m->stream, KC_ATTN, 0, (launch_k(rows_to_image_kernel, rows, 256, 0, m->stream, ws.ao_hi, ws.ao_lo, 0, ANPD_ROWS, m->dq, img, rows)));
        return ANPD_OK;
    }
    if (HD == 128 && kv->attn_tc) {
        ANPD_TRY(attn_tc_enqueue(m, kv, layer, rows, max_pos, tree));
    } else {
        dim3 grid(chunks, c.n_kv_heads, rows / ANPD_ROWS);
        LAUNCH(&m->prof, m->stream, KC_ATTN, 0,
               (launch_k(attn_partial_kernel<HD>, grid, ATTN_THREADS, smem, m->stream, ws.q_hi, ws.q_lo, kv->kpool + layer * layer_elems,
                         kv->vpool + layer * layer_elems, kv->page_table, kv->pages_per_seq, ws.row_pos, ws.row_seq, c.n_q_heads,
                         c.n_kv_heads, ws.attn_m, ws.attn_l, ws.attn_o, tree ? ws.row_slot : (const int*)nullptr,
                         tree ? ws.row_hole_lo : (const int*)nullptr, tree ? ws.row_hole_hi : (const int*)nullptr)));
    }
    if (rows >= 64) LAUNCH(&m->prof, m->stream, KC_ATTN, 0,
           (launch_k(attn_combine_wide_kernel<HD / 32>, dim3(rows, c.n_q_heads), 32 * COMBINE_SLICES, 0, m->stream, ws.attn_m, ws.attn_l, ws.attn_o,
                     tree ? ws.row_slot : ws.row_pos, c.n_q_heads, kv->pages_per_seq, ws.ao_hi, ws.ao_lo, img, img_rows)));
    else LAUNCH(&m->prof, m->stream, KC_ATTN, 0,
           (launch_k(attn_combine_kernel, dim3(rows, c.n_q_heads), HD * COMBINE_SLICES, 0, m->stream, ws.attn_m, ws.attn_l, ws.attn_o, tree ? ws.row_slot : ws.row_pos, c.n_q_heads,
                                                                              HD, kv->pages_per_seq, ws.ao_hi, ws.ao_lo, img, img_rows)));
    return ANPD_OK;
}

}  // namespace

// Where the projections of several sequences' steps run as one stream-K sweep over all SMs and not on clusters.  The cluster form
// re-reads its activations once per pass and leaves four sums per value, which costs more the more rows there are; the sweep's
// sums are one more than a tile has CTAs, which a narrow or short matrix pays for.  us per step, cluster form and sweep: 13B (10
// layers) 16 sequences 2733 and 2409, 12 2345 and 2069, 8 1760 and 1749, 6 1606 and 1559; 7B (8 layers) 16 1460 and 1415, 12 1240 and
// 1168, 8 1000 and 998, 4 817 and 803, but 2 sequences 771 and 783; 1.1B, 8 sequences 1241 and 1341.
bool tc_model_fits(const GemmPlan& p, int rows) { return rows >= 32 && p.k_blocks >= 64 && p.max_segs <= 6; }
const GemmPlan* tc_model_plan(const anpd_model* m, int kind, int rows) { return tc_model_fits(m->plan[kind], rows) ? &m->plan[kind] : nullptr; }

anpd_status gemm_plain_enqueue(const ClPlan& p, const unsigned char* W, const bf16* a_hi, const bf16* a_lo, int rows, float* part, int ld_part,
                               cudaStream_t st, Profiler* prof) {
    LAUNCH(prof, st, KC_GEMM, 2.0 * (double)p.N * (double)p.K,
           (launch_k(gemm_rows8_kernel, (p.N + 7) / 8, 256, 0, st, W, a_hi, a_lo, rows, p, part, ld_part)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

anpd_status plan_decode_enqueue(anpd_model* m, anpd_kv* kv, bool two_candidates) {
    Workspace& ws = kv->ws;
    LAUNCH(&m->prof, m->stream, KC_OTHER, 0,
           (launch_k(plan_decode_kernel, kv->batch, ANPD_ROWS, 0, m->stream, kv->seq, ws.row_tok, ws.row_pos, ws.row_seq, ws.row_ok,
                                                                      ws.row_slot, ws.row_hole_lo, ws.row_hole_hi, m->cfg.vocab, kv->max_len,
                                                                      two_candidates ? 1 : 0)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

anpd_status plan_prefill_enqueue(anpd_model* m, anpd_kv* kv, int seq, int start, int prompt_len, int rows, int n_seq, int seg) {
    Workspace& ws = kv->ws;
    LAUNCH(&m->prof, m->stream, KC_OTHER, 0,
           (launch_k(plan_prefill_kernel, (rows + 127) / 128, 128, 0, m->stream, kv->d_prompt, seq, start, prompt_len, rows, n_seq, seg, ws.row_tok,
                                                                          ws.row_pos, ws.row_seq, ws.row_ok, ws.row_slot, ws.row_hole_lo,
                                                                          ws.row_hole_hi, m->cfg.vocab, kv->max_len, kv->seq)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

anpd_status accept_enqueue(anpd_model* m, anpd_kv* kv, int mode, const NgramDev* d_ctxs, int seq, int last_row, int prompt_len, bool two_candidates, int n_seq) {
    Workspace& ws = kv->ws;
    const int blocks = (mode == ACCEPT_PREFILL) ? n_seq : kv->batch;
    LAUNCH(&m->prof, m->stream, KC_OTHER, 0,
           (launch_k(accept_kernel, blocks, 256, 0, m->stream, kv->seq, ws.amax_val_use, ws.amax_idx_use,
                     ws.amax_nblk, mode, d_ctxs, seq, last_row, prompt_len, two_candidates ? 1 : 0)));
    if (two_candidates && mode == ACCEPT_COMMIT) {
        const anpd_model_config& c = m->cfg;
        LAUNCH(&m->prof, m->stream, KC_OTHER, 0,
               (launch_k(kv_move_kernel, dim3(c.n_layers * c.n_kv_heads, kv->batch), c.head_dim, 0, m->stream, (const SeqState*)kv->seq,
                         (const int*)kv->page_table, kv->pages_per_seq, c.n_kv_heads, c.head_dim,
                         (size_t)kv->total_pages * c.n_kv_heads * KV_PAGE * c.head_dim, kv->kpool, kv->vpool)));
    }
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

// The forward of a single-sequence step (8 rows) on the row-range projections: per layer QKV (+ rotary, append) ->
// attention -> page combine -> O (+ residual) -> gate/up (+ SwiGLU) -> down (+ residual); then the LM head (+ argmax).
static anpd_status forward_rr_enqueue(anpd_model* m, anpd_kv* kv, int max_pos, bool want_logits) {
    const anpd_model_config& c = m->cfg;
    Workspace& ws = kv->ws;
    cudaStream_t st = m->stream;
    Profiler* pf = &m->prof;
    const int d = c.d_model, hd = c.head_dim;
    const size_t layer_elems = (size_t)kv->total_pages * c.n_kv_heads * KV_PAGE * hd;
    LAUNCH(pf, st, KC_OTHER, 0, (launch_k(embed_img_kernel, ANPD_ROWS, NORM_THREADS, 0, st, m->embed, ws.row_tok, m->layers[0].attn_norm, d, ws.x,
                                          ws.img_h, ws.ss_a)));
    int parts_a = 1;                                   // partial sums of squares behind img_h: 1 after the embedding, then the down projection's CTAs
    for (int l = 0; l < c.n_layers; ++l) {
        const anpd_model::LayerRR& w = m->rr_layers[l];
        RREpiHost q;
        q.ss_in = ws.ss_a; q.n_parts_in = parts_a; q.inv_d_in = 1.0f / (float)d; q.eps = c.rms_eps;
        q.row_pos = ws.row_pos; q.row_seq = ws.row_seq; q.row_ok = ws.row_ok; q.rope_cos = kv->rope_cos; q.rope_sin = kv->rope_sin;
        q.page_table = kv->page_table; q.pages_per_seq = kv->pages_per_seq; q.Hq = c.n_q_heads; q.Hkv = c.n_kv_heads; q.hd = hd;
        q.q_scale = 1.4426950408889634f / sqrtf((float)hd);
        q.q_hi = ws.q_hi; q.q_lo = ws.q_lo; q.kpool_l = kv->kpool + l * layer_elems; q.vpool_l = kv->vpool + l * layer_elems;
        ANPD_TRY(rr_enqueue(RR_QKV, m->rr[GK_QKV], w.wqkv, ws.img_h, q, ws.gemm_err, st, pf));
        if (hd == 128) ANPD_TRY(attn_enqueue<128>(m, kv, l, ANPD_ROWS, max_pos, ws.img_ao));
        else ANPD_TRY(attn_enqueue<64>(m, kv, l, ANPD_ROWS, max_pos, ws.img_ao));
        RREpiHost o;
        o.x = ws.x; o.gain = m->layers[l].ffn_norm; o.ss_out = ws.ss_b; o.d = d; o.act_out = ws.img_h2;
        ANPD_TRY(rr_enqueue(RR_RESID, m->rr[GK_O], w.wo, ws.img_ao, o, ws.gemm_err, st, pf));
        RREpiHost gu;
        gu.ss_in = ws.ss_b; gu.n_parts_in = m->rr[GK_O].G; gu.inv_d_in = 1.0f / (float)d; gu.eps = c.rms_eps; gu.act_out = ws.img_act;
        ANPD_TRY(rr_enqueue(RR_GU, m->rr[GK_GU], w.wgu, ws.img_h2, gu, ws.gemm_err, st, pf));
        RREpiHost dn;
        dn.x = ws.x; dn.gain = (l + 1 < c.n_layers) ? m->layers[l + 1].attn_norm : m->final_norm; dn.ss_out = ws.ss_a; dn.d = d;
        dn.act_out = ws.img_h;
        ANPD_TRY(rr_enqueue(RR_RESID, m->rr[GK_DOWN], w.wd, ws.img_act, dn, ws.gemm_err, st, pf));
        parts_a = m->rr[GK_DOWN].G;
    }
    RREpiHost lm;
    lm.ss_in = ws.ss_a; lm.n_parts_in = parts_a; lm.inv_d_in = 1.0f / (float)d; lm.eps = c.rms_eps;
    lm.logits = want_logits ? ws.logits : nullptr; lm.amax_val = ws.amax_val_rr; lm.amax_idx = ws.amax_idx_rr; lm.V = c.vocab;
    ANPD_TRY(rr_enqueue(RR_LM, m->rr[GK_LM], m->rr_lm, ws.img_h, lm, ws.gemm_err, st, pf));
    ws.amax_nblk = m->rr[GK_LM].G;
    ws.amax_val_use = ws.amax_val_rr;
    ws.amax_idx_use = ws.amax_idx_rr;
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

// The vocabulary projection of the 8 rows whose operand image is ws.ci_h, and its argmax candidates.
static anpd_status lm_head_cl_enqueue(anpd_model* m, anpd_kv* kv, const float* ss, int n_parts, bool want_logits) {
    const anpd_model_config& c = m->cfg;
    Workspace& ws = kv->ws;
    ClEpilogue lm;
    lm.ss_in = ss; lm.n_parts = n_parts; lm.inv_d = 1.0f / (float)c.d_model; lm.eps = c.rms_eps;
    lm.out = want_logits ? ws.logits : nullptr; lm.amax_val = ws.amax_val_cl; lm.amax_idx = ws.amax_idx_cl;
    ANPD_TRY(cl_enqueue(m->cl[GK_LM], m->lm_head, ws.ci_h, lm, ws.gemm_err, m->stream, &m->prof));
    ws.amax_nblk = cl_parts(m->cl[GK_LM]);
    ws.amax_val_use = ws.amax_val_cl;
    ws.amax_idx_use = ws.amax_idx_cl;
    return ANPD_OK;
}

// The forward of a single sequence's step: per layer QKV (+ rotary, append), attention, O (+ residual), gate/up (+ SwiGLU), down
// (+ residual); then the LM head (+ argmax).  Every projection finishes its own results (gemm_cl.cu).
static anpd_status forward_cl_enqueue(anpd_model* m, anpd_kv* kv, int max_pos, bool want_logits, bool two_candidates) {
    const anpd_model_config& c = m->cfg;
    Workspace& ws = kv->ws;
    cudaStream_t st = m->stream;
    Profiler* pf = &m->prof;
    const int d = c.d_model, hd = c.head_dim, rows = ANPD_ROWS;
    const size_t layer_elems = (size_t)kv->total_pages * c.n_kv_heads * KV_PAGE * hd;
    LAUNCH(pf, st, KC_OTHER, 0, (launch_k(embed_cl_kernel, rows, NORM_THREADS, 0, st, m->embed, ws.row_tok, m->layers[0].attn_norm, d, ws.x,
                                          ws.ci_h, rows, ws.ss_cl_a)));
    if (ws.xch_bytes && !pf->on) return step_cl_enqueue(m, kv, want_logits, two_candidates);
    int parts_a = 1;                                   // sums of squares behind ci_h: one after the embedding, then the down projection's
    // No projection fetches the weights of the next one, or its own beyond its ring, into L2: the traffic stands in front of the activations and
    // of the other CTAs' last copies, and the code for it is as much as that of a product loop.  us per step with and without: 7B (16
    // layers) at 77 keys 1370 and 1348, 13B (8 layers) 1040 and 991, 1.1B at 512 keys 747 and 739, at 3000 838 and 834, 1.1B's
    // widths with 8192 gate features and 16 query heads of 128 (12 layers) 540 and 502; with 16 kv heads of 64 at 600 keys no more than the runs' own
    // spread (438 and 431 to 443).
    for (int l = 0; l < c.n_layers; ++l) {
        const LayerW& w = m->layers[l];
        ClEpilogue q;
        q.ss_in = ws.ss_cl_a; q.n_parts = parts_a; q.inv_d = 1.0f / (float)d; q.eps = c.rms_eps;
        q.row_pos = ws.row_pos; q.row_slot = ws.row_slot; q.row_seq = ws.row_seq; q.row_ok = ws.row_ok;
        q.rope_cos = kv->rope_cos; q.rope_sin = kv->rope_sin; q.page_table = kv->page_table; q.pages_per_seq = kv->pages_per_seq;
        q.Hq = c.n_q_heads; q.Hkv = c.n_kv_heads; q.hd = hd; q.q_scale = 1.4426950408889634f / sqrtf((float)hd);
        q.q_hi = ws.q_hi; q.q_lo = ws.q_lo; q.kpool_l = kv->kpool + l * layer_elems; q.vpool_l = kv->vpool + l * layer_elems;
        ANPD_TRY(cl_enqueue(m->cl[GK_QKV], w.wqkv, ws.ci_h, q, ws.gemm_err, st, pf));
        if (kv->attn_dec) ANPD_TRY(attn_dec_enqueue(m, kv, l, two_candidates));
        else if (hd == 128) ANPD_TRY(attn_enqueue<128>(m, kv, l, rows, max_pos, ws.ci_ao, two_candidates, rows));
        else ANPD_TRY(attn_enqueue<64>(m, kv, l, rows, max_pos, ws.ci_ao, two_candidates, rows));
        ClEpilogue o;
        o.x = ws.x; o.gain = w.ffn_norm; o.ss_out = ws.ss_cl_b; o.d = d; o.act_out = ws.ci_h2;
        ANPD_TRY(cl_enqueue(m->cl[GK_O], w.wo, ws.ci_ao, o, ws.gemm_err, st, pf));
        ClEpilogue gu;
        gu.ss_in = ws.ss_cl_b; gu.n_parts = cl_parts(m->cl[GK_O]); gu.inv_d = 1.0f / (float)d; gu.eps = c.rms_eps; gu.act_out = ws.ci_act;
        ANPD_TRY(cl_enqueue(m->cl[GK_GU], w.wgu, ws.ci_h2, gu, ws.gemm_err, st, pf));
        ClEpilogue dn;
        dn.x = ws.x; dn.gain = (l + 1 < c.n_layers) ? m->layers[l + 1].attn_norm : m->final_norm; dn.ss_out = ws.ss_cl_a; dn.d = d;
        dn.act_out = ws.ci_h;
        ANPD_TRY(cl_enqueue(m->cl[GK_DOWN], w.wd, ws.ci_act, dn, ws.gemm_err, st, pf));
        parts_a = cl_parts(m->cl[GK_DOWN]);
    }
    ANPD_TRY(lm_head_cl_enqueue(m, kv, ws.ss_cl_a, parts_a, want_logits));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

anpd_status forward_enqueue(anpd_model* m, anpd_kv* kv, int rows, int max_pos, bool head, bool want_logits, int head_row, bool two_candidates, int n_seq) {
    // the two fused variants know nothing of a second candidate's cache slots and mask
    if (m->rr_ready && kv->batch == 1 && rows == ANPD_ROWS && head && !m->plain_gemm && !two_candidates) return forward_rr_enqueue(m, kv, max_pos, want_logits);
    if (kv->step_ready && rows == kv->batch * ANPD_ROWS && head && !m->prof.on && !two_candidates) return step_kernel_enqueue(m, kv, max_pos, want_logits);
    const bool decode = rows == kv->batch * ANPD_ROWS && !m->plain_gemm;           // (or a prompt pass of as many rows)
    const NormShape norm = norm_shape(m->cfg.d_model, rows, m->num_sms);
    const auto resid_norm = norm.chunks == 1 ? resid_norm_kernel<1, NORM_THREADS, 2> : norm.chunks == NORM_MAX_CHUNKS ? resid_norm_kernel<NORM_MAX_CHUNKS, NORM_THREADS, 1>
                          : norm.per_sm == 2 ? resid_norm_kernel<2, NORM_THREADS_2, 2> : resid_norm_kernel<2, NORM_THREADS, 1>;
    const bool slab = cl_rows(m, kv, rows);
    if (decode && kv->batch == 1 && head && m->cl_all_fused) return forward_cl_enqueue(m, kv, max_pos, want_logits, two_candidates);
    const anpd_model_config& c = m->cfg;
    kv->ws.amax_nblk = kv->ws.amax_blocks;
    kv->ws.amax_val_use = kv->ws.amax_val;
    kv->ws.amax_idx_use = kv->ws.amax_idx;
    Workspace& ws = kv->ws;
    cudaStream_t st = m->stream;
    Profiler* pf = &m->prof;
    const int d = c.d_model, F = c.d_ffn, hd = c.head_dim, V = c.vocab;
    auto sstride = [&](int kind) { return (size_t)rows * ws.ld[kind]; };           // between the partial sums of an output (the K parts of a projection)
    const size_t layer_elems = (size_t)kv->total_pages * c.n_kv_heads * KV_PAGE * hd;
    const int* segs = nullptr;
    int seg_min = 1;                                   // partial sums every tile of the last projection has

    LAUNCH(pf, st, KC_OTHER, 0, (launch_k(embed_norm_kernel, rows, NORM_THREADS, 0, st, m->embed, ws.row_tok, m->layers[0].attn_norm, c.rms_eps, d,
                                                                      ws.x, ws.h_hi, ws.h_lo, slab ? ws.ci_h : nullptr)));
    for (int l = 0; l < c.n_layers; ++l) {
        const LayerW& w = m->layers[l];
        ANPD_TRY(gemm_enqueue(m, kv, GK_QKV, l, rows, &segs, &seg_min));
        if (rows != kv->batch * ANPD_ROWS) {            // a prompt pass
            // as many heads at once as keep every SM's 2048 threads busy, the others by the same blocks
            const int seg = rows / n_seq, tiles = n_seq * ((seg + ROPE_TILE_ROWS - 1) / ROPE_TILE_ROWS);
            const dim3 grid(std::min(c.n_q_heads + 2 * c.n_kv_heads, std::max(1, m->num_sms * 8 / tiles)), tiles);
            const float qs = 1.4426950408889634f / sqrtf((float)hd);
            if (hd == 128) LAUNCH(pf, st, KC_OTHER, 0,
                   (launch_k(qkv_rope_append_tile_kernel<128>, grid, 256, 0, st, ws.part, segs, sstride(GK_QKV), ws.ld[GK_QKV], seg, ws.row_pos, ws.row_seq, ws.row_ok,
                             kv->rope_cos, kv->rope_sin, kv->page_table, kv->pages_per_seq, c.n_q_heads, c.n_kv_heads, qs, ws.q_hi, ws.q_lo,
                             kv->kpool + l * layer_elems, kv->vpool + l * layer_elems, seg_min)));
            else LAUNCH(pf, st, KC_OTHER, 0,
                   (launch_k(qkv_rope_append_tile_kernel<64>, grid, 256, 0, st, ws.part, segs, sstride(GK_QKV), ws.ld[GK_QKV], seg, ws.row_pos, ws.row_seq, ws.row_ok,
                             kv->rope_cos, kv->rope_sin, kv->page_table, kv->pages_per_seq, c.n_q_heads, c.n_kv_heads, qs, ws.q_hi, ws.q_lo,
                             kv->kpool + l * layer_elems, kv->vpool + l * layer_elems, seg_min)));
        } else
        {
            const float qs = 1.4426950408889634f / sqrtf((float)hd);
            const dim3 grid(std::min(c.n_q_heads + 2 * c.n_kv_heads, std::max(1, m->num_sms * ROPE_BLOCKS / kv->batch)), kv->batch);
            LAUNCH(pf, st, KC_OTHER, 0,
                   (launch_k(hd == 128 ? qkv_rope_append_kernel<128> : qkv_rope_append_kernel<64>, grid, hd, 0, st, ws.part, segs, sstride(GK_QKV), ws.ld[GK_QKV],
                             ws.row_pos, ws.row_slot, ws.row_seq, ws.row_ok, kv->rope_cos, kv->rope_sin, kv->page_table, kv->pages_per_seq, c.n_q_heads,
                             c.n_kv_heads, qs, ws.q_hi, ws.q_lo, kv->kpool + l * layer_elems, kv->vpool + l * layer_elems, seg_min)));
        }
        unsigned char* ao_img = slab ? ws.ci_ao : nullptr;
        const int ao_rows = slab ? rows : 0;
        if (decode && kv->attn_dec) ANPD_TRY(attn_dec_enqueue(m, kv, l, two_candidates));
        else if (hd == 128) ANPD_TRY(attn_enqueue<128>(m, kv, l, rows, max_pos, ao_img, two_candidates, ao_rows, n_seq));
        else ANPD_TRY(attn_enqueue<64>(m, kv, l, rows, max_pos, ao_img, two_candidates, ao_rows, n_seq));
        ANPD_TRY(gemm_enqueue(m, kv, GK_O, l, rows, &segs, &seg_min));
        LAUNCH(pf, st, KC_OTHER, 0,
               (launch_k(resid_norm, rows, norm.threads, 0, st, ws.x, ws.part, segs, sstride(GK_O), ws.ld[GK_O], w.ffn_norm, c.rms_eps, d,
                                                       ws.h_hi, ws.h_lo, seg_min, slab ? ws.ci_h : nullptr)));
        int from = 0;
        ANPD_TRY(gemm_enqueue(m, kv, GK_GU, l, rows, &segs, &seg_min, &from));
        if (from < F) {
            const bool many = rows >= 256;
            LAUNCH(pf, st, KC_OTHER, 0,
                   (launch_k(many ? swiglu_kernel<2> : swiglu_kernel<1>, dim3(((F - from) / 4 + (many ? 511 : 255)) / (many ? 512 : 256), rows), 256, 0, st, ws.part, segs,
                             sstride(GK_GU), ws.ld[GK_GU], F, from, ws.act_hi, ws.act_lo, seg_min, slab ? ws.ci_act : nullptr)));
        }
        ANPD_TRY(gemm_enqueue(m, kv, GK_DOWN, l, rows, &segs, &seg_min));
        const float* next_gain = (l + 1 < c.n_layers) ? m->layers[l + 1].attn_norm : m->final_norm;
        LAUNCH(pf, st, KC_OTHER, 0,
               (launch_k(resid_norm, rows, norm.threads, 0, st, ws.x, ws.part, segs, sstride(GK_DOWN), ws.ld[GK_DOWN], next_gain, c.rms_eps, d,
                                                       ws.h_hi, ws.h_lo, seg_min, decode || (slab && l + 1 < c.n_layers) ? ws.ci_h : nullptr)));
    }
    if (!head) { CUDA_TRY(cudaGetLastError()); return ANPD_OK; }
    // A prompt pass needs the LM head for each sequence's last token only: the groups of 8 rows that hold them become the first rows of a decode
    // projection (the other rows of that launch, if any, are whatever the buffer holds; rows are independent).
    const int group = (head_row / ANPD_ROWS) * ANPD_ROWS;
    const bool prompt = rows != kv->batch * ANPD_ROWS;
    if (prompt && !m->plain_gemm) {
        const bool one = n_seq == 1 && cl_fused(m->cl[GK_LM]);
        const int img_rows = one ? ANPD_ROWS : kv->batch * ANPD_ROWS;
        LAUNCH(pf, st, KC_OTHER, 0,
               (launch_k(rows_to_image_kernel, n_seq * ANPD_ROWS, 256, 0, st, ws.h_hi, ws.h_lo, group, rows / n_seq, d, ws.ci_h, img_rows)));
        if (one) return lm_head_cl_enqueue(m, kv, nullptr, 0, want_logits);
    } else if (prompt) {
        LAUNCH(pf, st, KC_OTHER, 0, (launch_k(move_rows_kernel, ANPD_ROWS, 256, 0, st, ws.h_hi, ws.h_lo, group, d)));
    }
    rows = kv->batch * ANPD_ROWS;
    ANPD_TRY(gemm_enqueue(m, kv, GK_LM, 0, rows, &segs, &seg_min));
    LAUNCH(pf, st, KC_OTHER, 0,
           (launch_k(argmax_partial_kernel, dim3(ws.amax_blocks, rows), 256, 0, st, ws.part, segs, seg_min, sstride(GK_LM), ws.ld[GK_LM], V,
                                                                             want_logits ? ws.logits : nullptr, ws.amax_val,
                                                                             ws.amax_idx, ws.amax_blocks)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}
