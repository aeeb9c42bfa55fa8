// Multi-Level N-gram module on the GPU (paper Sections 3.1 and 3.2, Algorithm 2).
//
// Per level n two open-addressing hash tables live in device memory (small enough to stay in
// L2): the gram table holds, for every distinct n-gram of the committed tokens, its count and
// last position; the prefix table holds, for every distinct (n-1)-gram context, the successor
// Query would return, packed so that "better" is a plain 64-bit maximum.  Update is two
// order-independent passes (count, then best) built from atomics, so a parallel fold over the
// whole prompt (Initialize) and the fold of a step's few tokens give the state a sequential
// token-by-token Update would give.
//
// What bounds it: chains of dependent L2 accesses.  A fold's warp looks for its gram with one half and for the gram's context with
// the other, sixteen consecutive slots at a time, and requests a slot's whole key at once.  A query is one warp's work: every level
// probes with four or eight lanes, whose slots and successors come in one 16-byte load, and the longest level that knows the
// context answers - two accesses per drafted token and no barrier (a warp per level with block barriers before).  A call from the
// host is one kernel that takes the new tokens as an argument and leaves its results and a ticket in host memory, where the caller
// waits for the ticket: 51 calls (a prompt of 512 tokens, 25 drafts of 5, 24 updates) 1.55 -> 0.78 ms, with copies and a stream
// synchronisation per call before.
#include "internal.h"

#include <algorithm>
#include <atomic>
#include <cstring>
#include <map>
#include <new>
#include <vector>

namespace {

constexpr int NG_ERR_FULL = 1;      // probing ran through the whole table
constexpr int NG_ERR_MISSING = 2;   // a gram counted in pass 1 was not found in pass 2
constexpr unsigned FULL_MASK = 0xffffffffu;
constexpr int STEP_THREADS = 1024;
constexpr int NG_CALL_TOKENS = 32;  // tokens a call's kernel takes as its argument; a longer run goes through the bulk kernels
constexpr int NG_HOST_TICKET = 32;   // index in the host buffer, a cache line away from the results

constexpr int KEY_MAX = ANPD_N_MAX;

// Unrolled over the longest key, so that keys stay in registers: a query is one warp's chain of instructions, and the key's way through local
// memory was a fifth of it.  What a step with drafts takes beyond a greedy one, before and after (with one vote per query instead of two): tiny 7.4 -> 6.8 us,
// 1.1B, five drafts, 9.8 -> 7.2, two candidates 18.5 -> 16; 51 calls 790 -> 770 us.
__device__ __forceinline__ unsigned hash_tokens(const int* key, int len) {
    unsigned h = 0x811C9DC5u ^ (unsigned)len;
#pragma unroll
    for (int i = 0; i < KEY_MAX; ++i) {
        unsigned m = (h ^ (unsigned)key[i]) * 0x01000193u;
        m ^= m >> 15;
        h = i < len ? m : h;
    }
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return h;
}

static_assert(sizeof(GramSlot) == 16 && sizeof(PrefSlot) == 16, "both tables are probed with one stride");

// Whether the klen tokens from position ref - n (the slot's gram starts there) on are the key.
__device__ __forceinline__ bool key_equals(const int* tokens, int ref, int n, const int* key, int klen) {
    const int* sk = tokens + ref - n;
    int got[KEY_MAX];
#pragma unroll
    for (int i = 0; i < KEY_MAX; ++i) got[i] = i < klen ? sk[i] : 0;        // all requested before the first comparison
    bool same = true;
#pragma unroll
    for (int i = 0; i < KEY_MAX; ++i) same = same && (i >= klen || got[i] == key[i]);
    return same;
}

// Find or insert the n-gram that ends at position t (lanes 0-15, gram table) and its context, the first n - 1 of its tokens
// (lanes 16-31, prefix table), linear probing.  All 32 lanes call it; each half returns its slot, or -2 if the bounded probe ran out.
__device__ int fold_slots(const NgramDev& c, int t, int n) {
    const int lane = threadIdx.x & 31, half = lane >> 4, lig = lane & 15, mask = c.cap - 1, windows = c.cap >> 4;
    const int klen = n - half;
    int key[KEY_MAX];
#pragma unroll
    for (int i = 0; i < KEY_MAX; ++i) key[i] = i < n ? c.tokens[t - n + 1 + i] : 0;
    char* table = half ? (char*)c.pref[n] : (char*)c.gram[n];
    const int base = (int)(hash_tokens(key, klen) & (unsigned)mask);
    int result = -3, w = 0;
    for (int guard = 0; guard < windows * 17 && __any_sync(FULL_MASK, result == -3); ++guard) {
        const int slot = (base + w * 16 + lig) & mask;
        int* ref = (int*)(table + (size_t)slot * 16);
        const int r = *((volatile int*)ref);
        const bool match = r != 0 && key_equals(c.tokens, r, n, key, klen);
        const unsigned mm = (__ballot_sync(FULL_MASK, match) >> (16 * half)) & 0xffffu, em = (__ballot_sync(FULL_MASK, r == 0) >> (16 * half)) & 0xffffu;
        const int fm = mm ? __ffs(mm) - 1 : 16, fe = em ? __ffs(em) - 1 : 16;
        const bool take = result == -3 && fm >= fe && fe < 16;            // a hole before any match: claim it
        int won = 0;
        if (take && lig == fe) won = atomicCAS(ref, 0, t + 1) == 0 ? 1 : 0;
        won = __shfl_sync(FULL_MASK, won, fe & 15, 16);
        if (result == -3) {
            if (fm < fe) result = (base + w * 16 + fm) & mask;
            else if (fe == 16) { if (++w == windows) result = -2; }
            else if (won) result = (base + w * 16 + fe) & mask;           // otherwise another warp took the hole: look again
        }
    }
    return result == -3 ? -2 : result;
}

__device__ __forceinline__ unsigned long long pack_best(int policy, int count, int last, int succ) {
    const unsigned long long c = (policy == 0) ? (unsigned long long)count : 0ull;
    return (c << 44) | ((unsigned long long)last << 24) | (unsigned long long)(unsigned)succ;
}

struct FoldSlots { int gram, pref; };

__device__ __forceinline__ FoldSlots fold_find(const NgramDev& c, int t, int n) {
    const int s = fold_slots(c, t, n);
    return {__shfl_sync(FULL_MASK, s, 0), __shfl_sync(FULL_MASK, s, 16)};
}

// Pass 1 for the token at position t, level n: count the n-gram ending at t.
__device__ FoldSlots fold_count(const NgramDev& c, int t, int n) {
    if (t < n - 1) return {-1, -1};
    const FoldSlots s = fold_find(c, t, n);
    if ((threadIdx.x & 31) == 0) {
        if (s.gram < 0 || s.pref < 0) atomicExch(&c.state[2], NG_ERR_FULL);
        else { atomicAdd(&c.gram[n][s.gram].count, 1); atomicMax(&c.gram[n][s.gram].last, t); }
    }
    return s;
}

// Pass 2: with every count final, offer this n-gram's (count, last, successor) to its context.
__device__ void fold_best(const NgramDev& c, int t, int n, FoldSlots s) {
    if (t < n - 1 || s.gram < 0 || s.pref < 0) return;
    if ((threadIdx.x & 31) == 0) {
        const int cnt = *((volatile int*)&c.gram[n][s.gram].count), last = *((volatile int*)&c.gram[n][s.gram].last);
        atomicMax(&c.pref[n][s.pref].best, pack_best(c.policy, cnt, last, c.tokens[t]));
    }
}

template <int PASS>
__global__ void ngram_bulk_kernel(NgramDev c, int from, int to) {
    const int levels = c.n_max - c.n_min + 1;
    const int items = (to - from) * levels;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += warps) {
        const int t = from + it / levels, n = c.n_min + it % levels;
        if (PASS == 1) fold_count(c, t, n);
        else if (t >= n - 1) fold_best(c, t, n, fold_find(c, t, n));
    }
}

// A block folds the tokens [from, to) at all levels, both passes.
__device__ void block_fold(const NgramDev& c, int from, int to) {
    const int levels = c.n_max - c.n_min + 1, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, items = (to - from) * levels;
    FoldSlots first{-1, -1};
    for (int it = warp; it < items; it += nwarps) {
        const FoldSlots s = fold_count(c, from + it / levels, c.n_min + it % levels);
        if (it == warp) first = s;
    }
    __threadfence_block();
    __syncthreads();
    for (int it = warp; it < items; it += nwarps) {
        const int t = from + it / levels, n = c.n_min + it % levels;
        if (t >= n - 1) fold_best(c, t, n, it == warp ? first : fold_find(c, t, n));
    }
    __threadfence_block();
    __syncthreads();
}

// One back-off query by one warp on the last tokens of tail[0 .. avail): the levels' answers (-1: the level does not know its
// context), longest level first, are left in lanes 0, W, 2 W, ... (W lanes per level).
__device__ int query_levels(const NgramDev& c, const int* tail, int avail, int W) {
    const int lane = threadIdx.x & 31, group = lane / W, lig = lane % W, mask = c.cap - 1;
    const int n = c.n_max - group, klen = n - 1;
    const unsigned gmask = (1u << W) - 1u;
    bool pending = n >= c.n_min && avail >= klen;
    int key[KEY_MAX];
#pragma unroll
    for (int i = 0; i < KEY_MAX; ++i) key[i] = pending && i < klen ? tail[avail - klen + i] : 0;
    const int base = pending ? (int)(hash_tokens(key, klen) & (unsigned)mask) : 0;
    const PrefSlot* table = pending ? c.pref[n] : nullptr;
    int ans = -1;
    for (int w = 0; __any_sync(FULL_MASK, pending); ++w) {
        if (w * W >= c.cap) { if (pending && lig == 0) atomicExch(&c.state[2], NG_ERR_FULL); break; }
        int4 slot = make_int4(0, 0, 0, 0);
        if (pending) slot = __ldcg((const int4*)&table[(base + w * W + lig) & mask]);        // ref, pad, best
        const bool match = pending && slot.x != 0 && key_equals(c.tokens, slot.x, n, key, klen);
        // the first slot that holds the key or nothing decides
        const unsigned ends = (__ballot_sync(FULL_MASK, match || (pending && slot.x == 0)) >> (group * W)) & gmask;
        const int found = __shfl_sync(FULL_MASK, match ? slot.z & 0xFFFFFF : -1, ends ? __ffs(ends) - 1 : 0, W);       // the low word holds the successor
        if (pending && ends) { ans = found; pending = false; }
    }
    return lig == 0 ? ans : -1;
}

// Up to K chained queries by one warp from tail[0 .. avail) on, each answer appended to tail and to draft; `first` receives the
// levels' answers to the first one.  Returns the number of answers.
__device__ int draft_chain(const NgramDev& c, int* tail, int avail, int K, int* draft, int& first) {
    const int W = c.n_max - c.n_min + 1 <= 4 ? 8 : 4;
    int i = 0;
    for (; i < K; ++i) {
        const int ans = query_levels(c, tail, avail, W);
        if (i == 0) first = ans;
        const unsigned known = __ballot_sync(FULL_MASK, ans >= 0);
        if (!known) break;
        const int tok = __shfl_sync(FULL_MASK, ans, __ffs(known) - 1);     // longest level first
        if ((threadIdx.x & 31) == 0) { tail[avail] = tok; draft[i] = tok; }
        ++avail;
        __syncwarp();
    }
    return i;
}

// The last min(T, n_max - 1) tokens, by one warp.
__device__ __forceinline__ int load_tail(const NgramDev& c, int T, int* tail) {
    const int keep = min(T, c.n_max - 1), lane = threadIdx.x & 31;
    if (lane < keep) tail[lane] = c.tokens[T - keep + lane];
    __syncwarp();
    return keep;
}

// One block per sequence: fold the tokens committed since the last step, then draft K tokens (and a second candidate of up to K2).
__global__ void __launch_bounds__(STEP_THREADS) ngram_step_kernel(const NgramDev* ctxs, SeqState* seqs, int K, int K2) {
    pdl_trigger();
    pdl_wait();
    __shared__ NgramDev c;
    __shared__ int tail[ANPD_N_MAX - 1 + ANPD_K_MAX + 1];
    if (threadIdx.x < sizeof(NgramDev) / 4) ((int*)&c)[threadIdx.x] = ((const int*)(ctxs + blockIdx.x))[threadIdx.x];
    __syncthreads();
    SeqState& sq = seqs[blockIdx.x];
    const int T = c.state[0];
    block_fold(c, c.state[1], T);
    if (threadIdx.x >= 32) return;
    const int keep = load_tail(c, T, tail);
    const bool idle = T <= 0 || sq.active == 0;
    int first = -1, none = -1;
    const int drafted = idle ? 0 : draft_chain(c, tail, keep, K, sq.draft, first);
    // The second candidate: its first token is the answer of the longest level that disagrees with the first candidate's
    // first token; it then continues like the first one, by back-off queries on its own temporary context.
    int drafted2 = 0;
    if (K2 > 0 && drafted > 0) {
        const unsigned other = __ballot_sync(FULL_MASK, first >= 0 && first != tail[keep]);
        if (other) {
            const int alt = __shfl_sync(FULL_MASK, first, __ffs(other) - 1);
            __syncwarp();
            if (threadIdx.x == 0) { tail[keep] = alt; sq.draft2[0] = alt; }
            __syncwarp();
            drafted2 = 1 + draft_chain(c, tail, keep + 1, K2 - 1, sq.draft2 + 1, none);
        }
    }
    if (threadIdx.x == 0) {
        c.state[1] = T;
        sq.draft_len = drafted;
        sq.draft2_len = drafted2;
        sq.last_tok = (T > 0) ? c.tokens[T - 1] : 0;
    }
}

// A call from the host: append n_new tokens, fold up to the end from `from` on, draft K.  host: [0] error, [1] draft_len, [2 ..] draft,
// and the ticket once all of it is there.
struct NgramCall {
    int n0, n_new, from, K, ticket;
    int tok[NG_CALL_TOKENS];
};

__global__ void __launch_bounds__(STEP_THREADS) ngram_call_kernel(const __grid_constant__ NgramDev ctx, const __grid_constant__ NgramCall a, int* host) {
    __shared__ int tail[ANPD_N_MAX - 1 + ANPD_K_MAX + 1];
    __shared__ int draft[ANPD_K_MAX + 1];
    __shared__ NgramDev c;
    if (threadIdx.x < sizeof(NgramDev) / 4) ((int*)&c)[threadIdx.x] = ((const int*)&ctx)[threadIdx.x];
    if (threadIdx.x < a.n_new) ctx.tokens[a.n0 + threadIdx.x] = a.tok[threadIdx.x];
    const int T = a.n0 + a.n_new;
    if (threadIdx.x == 0) { ctx.state[0] = T; ctx.state[1] = T; }
    __threadfence_block();
    __syncthreads();
    block_fold(c, a.from, T);
    if (threadIdx.x >= 32) return;
    int first = -1, drafted = 0;
    if (a.K > 0) {
        const int keep = load_tail(c, T, tail);
        drafted = draft_chain(c, tail, keep, a.K, draft, first);
        if ((int)threadIdx.x < drafted) host[2 + threadIdx.x] = draft[threadIdx.x];
    }
    __threadfence_block();
    __syncwarp();
    if (threadIdx.x == 0) { host[0] = *((volatile int*)&c.state[2]); host[1] = drafted; }
    __threadfence_system();
    __syncwarp();
    if (threadIdx.x == 0) *((volatile int*)(host + NG_HOST_TICKET)) = a.ticket;
}

int next_pow2(int v) { int p = 64; while (p < v) p <<= 1; return p; }

}  // namespace

anpd_status ngram_enqueue_bulk(anpd_ngram* ctx, int from, int to, Profiler* prof, cudaStream_t on) {
    if (to <= from) return ANPD_OK;
    cudaStream_t st = on ? on : ctx->stream;
    const int levels = ctx->h.n_max - ctx->h.n_min + 1;
    const int items = (to - from) * levels;
    const int threads = 256, wpb = threads / 32;
    const int blocks = std::min((items + wpb - 1) / wpb, 148 * 8);
    LAUNCH(prof, st, KC_NGRAM, 0, (ngram_bulk_kernel<1><<<blocks, threads, 0, st>>>(ctx->h, from, to)));
    LAUNCH(prof, st, KC_NGRAM, 0, (ngram_bulk_kernel<2><<<blocks, threads, 0, st>>>(ctx->h, from, to)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

anpd_status ngram_enqueue_step(const NgramDev* d_ctxs, SeqState* d_seq, int batch, int K,
                               cudaStream_t st, Profiler* prof, int K2) {
    LAUNCH(prof, st, KC_NGRAM, 0, (launch_k(ngram_step_kernel, batch, STEP_THREADS, 0, st, d_ctxs, d_seq, K, K2)));
    CUDA_TRY(cudaGetLastError());
    return ANPD_OK;
}

anpd_status ngram_reset_enqueue(anpd_ngram* c) {
    CUDA_TRY(cudaMemsetAsync(c->slab, 0, c->slab_bytes, c->stream));
    c->n_tokens = 0;
    c->n_folded = 0;
    return ANPD_OK;
}

// ---------------------------------------------------------------------------------------------
// boundary
// ---------------------------------------------------------------------------------------------
extern "C" {

anpd_status anpd_ngram_create(const anpd_ngram_config* cfg, void* cuda_stream, anpd_ngram** out) {
    if (!cfg || !out) return ANPD_ERR_ARG;
    if (cfg->n_min < 2 || cfg->n_max < cfg->n_min || cfg->n_max > ANPD_N_MAX) return ANPD_ERR_RANGE;
    if (cfg->max_ctx < 1 || cfg->max_ctx > (1 << 20)) return ANPD_ERR_ARG;
    if (cfg->policy != 0 && cfg->policy != 1) return ANPD_ERR_ARG;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) { cudaGetLastError(); return ANPD_ERR_CUDA; }
    anpd_ngram* c = new (std::nothrow) anpd_ngram();
    if (!c) return ANPD_ERR_OOM;
    std::memset(&c->h, 0, sizeof(c->h));
    c->pinned = nullptr; c->ticket = 0; c->slab = nullptr; c->n_tokens = 0; c->n_folded = 0;
    c->stream = (cudaStream_t)cuda_stream;
    const int cap = next_pow2(2 * cfg->max_ctx);
    const int levels = cfg->n_max - cfg->n_min + 1;
    auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    const size_t tok_b = up(sizeof(int) * (size_t)cfg->max_ctx), st_b = 256;
    const size_t gram_b = up(sizeof(GramSlot) * (size_t)cap), pref_b = up(sizeof(PrefSlot) * (size_t)cap);
    c->slab_bytes = tok_b + st_b + levels * (gram_b + pref_b);
    if (cudaMalloc(&c->slab, c->slab_bytes) != cudaSuccess) { cudaGetLastError(); delete c; return ANPD_ERR_OOM; }
    if (cudaMallocHost((void**)&c->pinned, 256) != cudaSuccess) { cudaGetLastError(); cudaFree(c->slab); delete c; return ANPD_ERR_OOM; }
    char* p = (char*)c->slab;
    c->h.tokens = (int*)p; p += tok_b;
    c->h.state = (int*)p; p += st_b;
    for (int n = cfg->n_min; n <= cfg->n_max; ++n) {
        c->h.gram[n] = (GramSlot*)p; p += gram_b;
        c->h.pref[n] = (PrefSlot*)p; p += pref_b;
    }
    c->h.n_min = cfg->n_min; c->h.n_max = cfg->n_max; c->h.max_ctx = cfg->max_ctx;
    c->h.cap = cap; c->h.policy = cfg->policy;
    c->pinned[NG_HOST_TICKET] = 0;
    if (cudaMemsetAsync(c->slab, 0, c->slab_bytes, c->stream) != cudaSuccess ||
        cudaStreamSynchronize(c->stream) != cudaSuccess) {
        anpd_note_cuda_error(cudaGetLastError(), __FILE__, __LINE__);
        cudaFreeHost(c->pinned); cudaFree(c->slab); delete c;
        return ANPD_ERR_CUDA;
    }
    *out = c;
    return ANPD_OK;
}

anpd_status anpd_ngram_reset(anpd_ngram* c) {
    if (!c) return ANPD_ERR_ARG;
    ANPD_TRY(ngram_reset_enqueue(c));
    CUDA_TRY(cudaStreamSynchronize(c->stream));
    return ANPD_OK;
}

anpd_status anpd_ngram_destroy(anpd_ngram* c) {
    if (!c) return ANPD_ERR_ARG;
    cudaStreamSynchronize(c->stream);
    cudaFreeHost(c->pinned);
    cudaFree(c->slab);
    delete c;
    return ANPD_OK;
}

// Launches ngram_call_kernel and waits for its ticket.  The wait ends with the stream at the latest: a kernel that failed never
// writes the ticket, but the stream then reports why.
static anpd_status ngram_call(anpd_ngram* c, const int32_t* tokens, int n_new, int from, int K) {
    NgramCall a;
    a.n0 = c->n_tokens; a.n_new = n_new; a.from = from; a.K = K;
    a.ticket = ++c->ticket;
    for (int i = 0; i < NG_CALL_TOKENS; ++i) a.tok[i] = i < n_new ? tokens[i] : 0;
    const int levels = c->h.n_max - c->h.n_min + 1, items = (a.n0 + n_new - from) * levels;
    const int threads = std::min(STEP_THREADS, std::max(128, 32 * items));
    LAUNCH(nullptr, c->stream, KC_NGRAM, 0, (ngram_call_kernel<<<1, threads, 0, c->stream>>>(c->h, a, c->pinned)));
    CUDA_TRY(cudaGetLastError());
    volatile int* at = c->pinned + NG_HOST_TICKET;
    for (unsigned spin = 1; *at != a.ticket; ++spin) {
        if (spin % 2048 == 0) {
            const cudaError_t e = cudaStreamQuery(c->stream);
            if (e == cudaErrorNotReady) continue;
            CUDA_TRY(e);
            if (*at != a.ticket) return ANPD_ERR_CUDA;
        }
#if defined(__x86_64__)
        __builtin_ia32_pause();
#endif
    }
    std::atomic_thread_fence(std::memory_order_acquire);
    return ANPD_OK;
}

// Tokens that wait to be folded: a call's one block takes the few of a decoding loop's last step, the bulk kernels what a greedy loop
// leaves, the whole prompt and output (1500 tokens, 4 levels: an update 721 us in one block, 38 through the bulk kernels).
static anpd_status fold_backlog(anpd_ngram* c) {
    if (c->n_tokens - c->n_folded <= NG_CALL_TOKENS) return ANPD_OK;
    ANPD_TRY(ngram_enqueue_bulk(c, c->n_folded, c->n_tokens, nullptr));
    c->n_folded = c->n_tokens;
    return ANPD_OK;
}

anpd_status anpd_ngram_len(anpd_ngram* c, int* n_tokens) {
    if (!c || !n_tokens) return ANPD_ERR_ARG;
    *n_tokens = c->n_tokens;
    return ANPD_OK;
}

anpd_status anpd_ngram_update(anpd_ngram* c, const int32_t* new_tokens, int n_new) {
    if (!c || (n_new > 0 && !new_tokens) || n_new < 0) return ANPD_ERR_ARG;
    if (n_new == 0) return ANPD_OK;
    for (int i = 0; i < n_new; ++i)
        if (new_tokens[i] < 0 || new_tokens[i] >= (1 << 24)) return ANPD_ERR_RANGE;
    if (c->n_tokens + n_new > c->h.max_ctx) return ANPD_ERR_CAPACITY;
    ANPD_TRY(fold_backlog(c));
    const int from = c->n_tokens, to = from + n_new;
    // tokens a decoding loop committed in its last step are still waiting to be folded
    if (n_new <= NG_CALL_TOKENS) ANPD_TRY(ngram_call(c, new_tokens, n_new, c->n_folded, 0));
    else {
        CUDA_TRY(cudaMemcpyAsync(c->h.tokens + from, new_tokens, sizeof(int) * (size_t)n_new, cudaMemcpyHostToDevice, c->stream));
        ANPD_TRY(ngram_enqueue_bulk(c, c->n_folded, to, nullptr));
        c->n_tokens = to;
        const anpd_status rc = ngram_call(c, nullptr, 0, to, 0);
        c->n_tokens = from;
        ANPD_TRY(rc);
    }
    c->n_tokens = to;
    c->n_folded = to;
    return c->pinned[0] == 0 ? ANPD_OK : ANPD_ERR_CUDA;
}

anpd_status anpd_ngram_draft(anpd_ngram* c, int K, int32_t* draft, int* draft_len) {
    if (!c || !draft_len || (K > 0 && !draft)) return ANPD_ERR_ARG;
    if (K < 0 || K > ANPD_K_MAX) return ANPD_ERR_RANGE;
    if (c->n_tokens < 1) return ANPD_ERR_STATE;
    ANPD_TRY(fold_backlog(c));
    ANPD_TRY(ngram_call(c, nullptr, 0, c->n_folded, K));
    if (c->pinned[0] != 0) return ANPD_ERR_CUDA;
    c->n_folded = c->n_tokens;
    *draft_len = c->pinned[1];
    for (int i = 0; i < *draft_len; ++i) draft[i] = c->pinned[2 + i];
    return ANPD_OK;
}

static anpd_status dump_level(anpd_ngram* c, int n, std::vector<anpd_ngram_entry>& grams,
                              std::vector<anpd_ngram_entry>* bests) {
    if (n < c->h.n_min || n > c->h.n_max) return ANPD_ERR_RANGE;
    std::vector<int> tok((size_t)std::max(c->n_tokens, 1));
    std::vector<GramSlot> g((size_t)c->h.cap);
    std::vector<PrefSlot> p((size_t)c->h.cap);
    CUDA_TRY(cudaStreamSynchronize(c->stream));
    if (c->n_tokens > 0) CUDA_TRY(cudaMemcpy(tok.data(), c->h.tokens, sizeof(int) * (size_t)c->n_tokens, cudaMemcpyDeviceToHost));
    CUDA_TRY(cudaMemcpy(g.data(), c->h.gram[n], sizeof(GramSlot) * g.size(), cudaMemcpyDeviceToHost));
    CUDA_TRY(cudaMemcpy(p.data(), c->h.pref[n], sizeof(PrefSlot) * p.size(), cudaMemcpyDeviceToHost));
    auto less = [](const anpd_ngram_entry& a, const anpd_ngram_entry& b) {
        for (int i = 0; i < ANPD_N_MAX - 1; ++i) if (a.key[i] != b.key[i]) return a.key[i] < b.key[i];
        return a.succ < b.succ;
    };
    grams.clear();
    for (const GramSlot& s : g) {
        if (s.ref == 0) continue;
        anpd_ngram_entry e;
        const int t = s.ref - 1;
        for (int i = 0; i < ANPD_N_MAX - 1; ++i) e.key[i] = (i < n - 1) ? tok[t - n + 1 + i] : -1;
        e.succ = tok[t]; e.count = s.count; e.last_pos = s.last;
        grams.push_back(e);
    }
    std::sort(grams.begin(), grams.end(), less);
    if (bests) {
        bests->clear();
        for (const PrefSlot& s : p) {
            if (s.ref == 0) continue;
            anpd_ngram_entry e;
            const int t = s.ref - 1;
            for (int i = 0; i < ANPD_N_MAX - 1; ++i) e.key[i] = (i < n - 1) ? tok[t - n + 1 + i] : -1;
            e.succ = (int)(s.best & 0xFFFFFFull);
            e.last_pos = (int)((s.best >> 24) & 0xFFFFFull);
            e.count = 0;
            auto it = std::lower_bound(grams.begin(), grams.end(), e, less);
            if (it != grams.end() && !less(e, *it)) e.count = it->count;
            bests->push_back(e);
        }
        std::sort(bests->begin(), bests->end(), less);
    }
    return ANPD_OK;
}

anpd_status anpd_ngram_dump(anpd_ngram* c, int n, anpd_ngram_entry* out, int cap, int* n_entries) {
    if (!c || !n_entries) return ANPD_ERR_ARG;
    std::vector<anpd_ngram_entry> grams;
    ANPD_TRY(dump_level(c, n, grams, nullptr));
    if (out) {
        if ((int)grams.size() > cap) return ANPD_ERR_CAPACITY;
        std::copy(grams.begin(), grams.end(), out);
    }
    *n_entries = (int)grams.size();
    return ANPD_OK;
}

anpd_status anpd_ngram_dump_best(anpd_ngram* c, int n, anpd_ngram_entry* out, int cap, int* n_entries) {
    if (!c || !n_entries) return ANPD_ERR_ARG;
    std::vector<anpd_ngram_entry> grams, bests;
    ANPD_TRY(dump_level(c, n, grams, &bests));
    if (out) {
        if ((int)bests.size() > cap) return ANPD_ERR_CAPACITY;
        std::copy(bests.begin(), bests.end(), out);
    }
    *n_entries = (int)bests.size();
    return ANPD_OK;
}

}  // extern "C"
