// Decode step of SAS (Alg. 2): one new token per sequence, grouped-query
// attention with one block selection per query group (Sec. 5, inference
// implementation), over a paged KV cache holding one 64-token block per page.
//
//   dec_prep_kernel    appends k_new / v_new at position n-1, summarises the block
//                      that position closes (K~ = bf16(Wk mean K), App. B) and
//                      forms the group's gate query q~ = bf16(Wq_g [q_0; ...]).
//   dec_score_kernel   s_m = q~ . K~_m / sqrt(d_sel) for the C historical blocks
//                      (Alg. 2 step 1), CTAs of 256 blocks whose summary rows are
//                      staged in shared memory by bulk async copies.  Each CTA keeps
//                      the exact Top-K of its own blocks (ranks by counting, past
//                      kRankRows blocks a sort); the last CTA of a group selects the
//                      Top-K of those candidates (step 2) on the scores' order-
//                      preserving bit patterns, by counting ranks or, past kRankMax
//                      candidates, a radix select, ties to the lower block, and
//                      writes the kept list in ascending order.
//   dec_attn_tc_kernel split-KV attention over B_0 and the kept blocks (steps 3-4),
//                      d = 128: each CTA takes a few pages (K and V slices of 16 KB,
//                      TMA into a ring), two pages a step on the tensor cores.  A SAS
//                      list's CTAs form a cluster; every page pair leaves its own
//                      partial (max, sum, output) and the cluster merges them in list
//                      order, so that the result does not depend on how many CTAs a
//                      batch leaves for a list.  A dense list's CTA keeps an online
//                      softmax over its pages and the last CTA merges.
//   dec_attn_kernel    the same for d = 64 on the CUDA cores.
// The three kernels are chained with programmatic dependent launch: each one
// starts while its predecessor runs, does the work that needs none of the
// predecessor's results (barrier set-up, reading lengths and queries, the block
// summaries, the page of the current block) and then waits on the grid dependency.
// A decode step moves bytes, not flops, and is bound by latencies: at 8 sequences
// of 64K tokens (8 KV heads, K = 32) 36 us a step, against 12.6 us for its bytes.
#include <math_constants.h>

#include "internal.h"
#include "ptx.cuh"

namespace sas {
namespace {

constexpr int kBlk = 64;
constexpr int kStatusBadInput = 1;   // == SAS_ERR_INVALID_ARG
constexpr int kPrepThreads = 256;
constexpr int kScoreThreads = 256;
constexpr int kAttnThreads = 256;
constexpr int kStages = 3;
constexpr int kRankRows = 96;         // blocks of a score CTA ranked by counting; more are sorted (score kernel, us,
                                      // counting / sorting: 76 blocks 4.2 / 4.5, 129 6.4 / 5.5, 256 and 221 8.0 / 6.2)
constexpr int kRankMax = 256;         // candidates ranked by counting, one a thread; more take the radix select
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ bool bad_len(int n, const DecodeArgs& a) { return n < 1 || n > a.max_blocks * kBlk; }

// Programmatic dependent launch: wait until the preceding grid has completed
// and its writes are visible; allow the next grid to start launching.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Exclusive prefix sum over the 256 threads of a CTA (scan: 16 shared ints).
__device__ int block_excl_scan(int v, int* scan) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) scan[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < 8 ? scan[lane] : 0;
        const int own = w;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < 8) scan[8 + lane] = w - own;
    }
    __syncthreads();
    const int r = x - v + scan[8 + warp];
    __syncthreads();
    return r;
}

// One full block's summary (App. B): the mean of its 64 keys in fp32, projected
// by the KV head's Wk [d_sel][d] and rounded to bf16.  256 threads.
// red: 512 floats, kbar: 128 floats of shared memory.  Latency: a thread's key
// words and its warp's rows of Wk are all requested before the first is used
// (loaded one by one they made a step that closes a block wait 11 us on this).
template <int D>
__device__ void summarize_block_d(const bf16* Kt, const bf16* Wk, bf16* out, int d_sel, float* red, float* kbar) {
    constexpr int NW = D / 2;                    // bf16 pairs per key row
    constexpr int GROUPS = kPrepThreads / NW;    // 4 (d = 128) or 8 (d = 64) row groups
    constexpr int ROWS = kBlk / GROUPS;
    constexpr int OUTS = 128 / (kPrepThreads / 32);   // projection rows per warp, at most
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int wi = t % NW, rg = t / NW;
    const uint32_t* K32 = reinterpret_cast<const uint32_t*>(Kt);
    uint32_t kw[ROWS], ww[OUTS][NW / 32];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) kw[r] = __ldg(K32 + (rg * ROWS + r) * NW + wi);
#pragma unroll
    for (int k = 0; k < OUTS; ++k) {
        const int o = warp + k * (kPrepThreads / 32);
        const uint32_t* row = reinterpret_cast<const uint32_t*>(Wk + static_cast<size_t>(o) * D);
#pragma unroll
        for (int e = 0; e < NW / 32; ++e) ww[k][e] = o < d_sel ? __ldg(row + e * 32 + lane) : 0u;
    }
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        a0 += bf_lo(kw[r]);
        a1 += bf_hi(kw[r]);
    }
    red[rg * D + 2 * wi] = a0;
    red[rg * D + 2 * wi + 1] = a1;
    __syncthreads();
    if (t < D) {
        float s = 0.f;
        for (int g = 0; g < GROUPS; ++g) s += red[g * D + t];
        kbar[t] = s * (1.f / kBlk);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < OUTS; ++k) {
        const int o = warp + k * (kPrepThreads / 32);
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < NW / 32; ++e) {
            acc = fmaf(bf_lo(ww[k][e]), kbar[2 * (e * 32 + lane)], acc);
            acc = fmaf(bf_hi(ww[k][e]), kbar[2 * (e * 32 + lane) + 1], acc);
        }
        acc = warp_sum(acc);
        if (lane == 0 && o < d_sel) out[o] = __float2bfloat16_rn(acc);
    }
}
__device__ void summarize_block(const bf16* Kt, const bf16* Wk, bf16* out, int d, int d_sel, float* red,
                                float* kbar) {
    if (d == 128) summarize_block_d<128>(Kt, Wk, out, d_sel, red, kbar);
    else summarize_block_d<64>(Kt, Wk, out, d_sel, red, kbar);
}

// grid (B*Hkv, 1 + d_sel/8): y = 0 appends the token and updates the summary
// cache, y >= 1 computes 8 entries of the group's gate query (one per warp).
__global__ void __launch_bounds__(kPrepThreads) dec_prep_kernel(DecodeArgs a, int* status) {
    __shared__ float red[512];
    __shared__ __align__(16) float vec[1024];
    grid_dep_launch();   // the score kernel may start its set-up
    const int bh = blockIdx.x;
    const int b = bh / a.Hkv, g = bh - b * a.Hkv;
    const int n = __ldg(a.seq_lens + b);
    const int t = threadIdx.x;
    if (bad_len(n, a)) {
        if (t == 0 && blockIdx.y == 0) atomicExch(status, kStatusBadInput);
        return;
    }
    if (blockIdx.y == 0) {
        const int pos = n - 1, blk = pos / kBlk, slot = pos - blk * kBlk;
        const int32_t* row = a.block_table + static_cast<size_t>(b) * a.max_blocks;
        const int page = __ldg(row + blk);
        if (page < 0 || page >= a.num_pages) {
            if (t == 0) atomicExch(status, kStatusBadInput);
            return;
        }
        if (a.k_new != nullptr) {
            const int nu = a.d / 8;   // 16-byte units per row
            if (t < 2 * nu) {
                const bool isv = t >= nu;
                const int u = isv ? t - nu : t;
                const uint4* src =
                    reinterpret_cast<const uint4*>(static_cast<const bf16*>(isv ? a.v_new : a.k_new) +
                                                   static_cast<size_t>(bh) * a.d) + u;
                uint4* dst = reinterpret_cast<uint4*>(static_cast<bf16*>(isv ? a.V_cache : a.K_cache) +
                                                      ((static_cast<size_t>(page) * a.Hkv + g) * kBlk + slot) * a.d) + u;
                *dst = __ldg(src);
            }
        }
        if (!a.dense && slot == 0 && blk >= 1) {
            const int pp = __ldg(row + blk - 1);
            if (pp < 0 || pp >= a.num_pages) {
                if (t == 0) atomicExch(status, kStatusBadInput);
                return;
            }
            summarize_block(static_cast<const bf16*>(a.K_cache) + (static_cast<size_t>(pp) * a.Hkv + g) * kBlk * a.d,
                            static_cast<const bf16*>(a.Wk) + static_cast<size_t>(g) * a.d_sel * a.d,
                            static_cast<bf16*>(a.Ksum) + (static_cast<size_t>(bh) * a.max_blocks + blk - 1) * a.d_sel,
                            a.d, a.d_sel, red, vec);
        }
        return;
    }
    // gate query q~[o] = bf16(sum_e Wq_g[o][e] q_cat[e]), o = 8 (y-1) + warp.  The
    // warp's row of Wq_g (G*d <= 1024 bf16) is loaded in one go, 32 bytes a lane.
    const int GD = a.G * a.d;
    const int warp = t >> 5, lane = t & 31;
    const int o = (blockIdx.y - 1) * 8 + warp;
    const bool has_row = o < a.d_sel;
    const bf16* wrow = static_cast<const bf16*>(a.Wq) + (static_cast<size_t>(g) * a.d_sel + (has_row ? o : 0)) * GD;
    uint4 w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int e = (k * 32 + lane) * 8;
        w[k] = (has_row && e < GD) ? __ldg(reinterpret_cast<const uint4*>(wrow + e)) : make_uint4(0, 0, 0, 0);
    }
    const bf16* qg = static_cast<const bf16*>(a.q) + (static_cast<size_t>(b) * a.Hq + static_cast<size_t>(g) * a.G) * a.d;
    for (int e = t; e < GD; e += kPrepThreads) vec[e] = __bfloat162float(qg[e]);
    __syncthreads();
    if (!has_row) return;
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int e = (k * 32 + lane) * 8;
        if (e < GD) {
            const float4 x0 = *reinterpret_cast<const float4*>(vec + e);
            const float4 x1 = *reinterpret_cast<const float4*>(vec + e + 4);
            acc = fmaf(bf_lo(w[k].x), x0.x, acc);
            acc = fmaf(bf_hi(w[k].x), x0.y, acc);
            acc = fmaf(bf_lo(w[k].y), x0.z, acc);
            acc = fmaf(bf_hi(w[k].y), x0.w, acc);
            acc = fmaf(bf_lo(w[k].z), x1.x, acc);
            acc = fmaf(bf_hi(w[k].z), x1.y, acc);
            acc = fmaf(bf_lo(w[k].w), x1.z, acc);
            acc = fmaf(bf_hi(w[k].w), x1.w, acc);
        }
    }
    acc = warp_sum(acc);
    if (lane == 0) static_cast<bf16*>(a.qt)[static_cast<size_t>(bh) * a.d_sel + o] = __float2bfloat16_rn(acc);
}

// grid (max_blocks, B*Hkv): summary of full block m of every sequence (after a prefill).
__global__ void __launch_bounds__(kPrepThreads) dec_summarize_kernel(DecodeArgs a, int* status) {
    __shared__ float red[512];
    __shared__ float kbar[128];
    const int m = blockIdx.x, bh = blockIdx.y;
    const int b = bh / a.Hkv, g = bh - b * a.Hkv;
    const int n = __ldg(a.seq_lens + b);
    if (n < 0 || n > a.max_blocks * kBlk) {
        if (threadIdx.x == 0 && m == 0) atomicExch(status, kStatusBadInput);
        return;
    }
    if (m >= n / kBlk) return;
    const int page = __ldg(a.block_table + static_cast<size_t>(b) * a.max_blocks + m);
    if (page < 0 || page >= a.num_pages) {
        if (threadIdx.x == 0) atomicExch(status, kStatusBadInput);
        return;
    }
    summarize_block(static_cast<const bf16*>(a.K_cache) + (static_cast<size_t>(page) * a.Hkv + g) * kBlk * a.d,
                    static_cast<const bf16*>(a.Wk) + static_cast<size_t>(g) * a.d_sel * a.d,
                    static_cast<bf16*>(a.Ksum) + (static_cast<size_t>(bh) * a.max_blocks + m) * a.d_sel, a.d, a.d_sel,
                    red, kbar);
}

// ------------------------------------------------------------ scores + Top-K

struct ScoreSmem {
    size_t r0;   // staged summary rows; in the last CTA the candidates (keys, blocks)
    size_t qs, bars, misc, xchg, scan, hist, total;
};
__host__ __device__ inline ScoreSmem score_smem_layout(int nsplit, int topk, int d_sel) {
    ScoreSmem L;
    const size_t slab = static_cast<size_t>(8) * 32 * d_sel * 2;
    const size_t cand = (static_cast<size_t>(nsplit) * (topk > 0 ? topk : 1) + 4) * 8;
    L.r0 = ((slab > cand ? slab : cand) + 127) / 128 * 128;
    L.qs = L.r0;                  // d_sel bf16 (<= 256 bytes)
    L.bars = L.qs + 256;          // 8 mbarriers
    L.misc = L.bars + 64;         // flag, radix broadcast, per-warp counts (16 ints)
    L.xchg = L.misc + 64;         // 256 order keys
    L.scan = L.xchg + 256 * 4;    // 16 ints
    L.hist = L.scan + 128;        // 4096 ints of the radix select; kept for every size: two CTAs an
                                  // SM ran a step of 8 x 64K (36 us now) in 39.8 us, three (without them) in 44.3
    L.total = L.hist + 4096 * 4;
    return L;
}

// Order-preserving map of a finite float to uint32 (larger float, larger key);
// -0 is mapped like +0 so that equal scores stay ties.  Every finite float maps
// above 0, so 0 marks an empty candidate slot.
__device__ __forceinline__ uint32_t order_key(float f) {
    const uint32_t u = __float_as_uint(f == 0.f ? 0.f : f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Descending bitonic sort of 256 distinct 64-bit keys, one per thread of the
// CTA; returns the key that ends at position threadIdx.x.  Exchanges within a
// warp use shuffles, wider ones the 256-entry shared buffer xchg.
__device__ uint64_t bitonic256_desc(uint64_t c, uint64_t* xchg) {
    const int t = threadIdx.x;
#pragma unroll
    for (int k = 2; k <= 256; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            uint64_t o;
            if (j >= 32) {
                xchg[t] = c;
                __syncthreads();
                o = xchg[t ^ j];
                __syncthreads();
            } else {
                o = __shfl_xor_sync(0xffffffffu, c, j);
            }
            const bool keep_max = ((t & j) == 0) == ((t & k) == 0);
            c = keep_max ? (c > o ? c : o) : (c < o ? c : o);
        }
    }
    return c;
}

// How many of the M keys (16-byte aligned, the rest of the last four slots 0) rank
// ahead of key (>= 1) at position t: the larger ones, and the equal ones listed
// before it.  All lanes of a warp read the same four keys at a time; the
// position decides only for keys in the warp's own range, w0 .. w0 + 31.
__device__ __forceinline__ int rank_of(const uint32_t* keys, int M, uint32_t key, int t, int w0) {
    int r = 0;
    for (int j = 0; j < M; j += 4) {
        const uint4 k4 = *reinterpret_cast<const uint4*>(keys + j);
        // an equal key ranks ahead when listed before: compare with key - 1 there
        const bool own = j >= w0 && j < w0 + 32;
        const uint32_t all = key - (j < w0 ? 1u : 0u);
        r += k4.x > (own ? key - (j < t) : all);
        r += k4.y > (own ? key - (j + 1 < t) : all);
        r += k4.z > (own ? key - (j + 2 < t) : all);
        r += k4.w > (own ? key - (j + 3 < t) : all);
    }
    return r;
}

// Exact Top-K of at most kRankMax candidates in ascending block order by counting
// each one's rank (M^2 comparisons, about 1 us at 160 candidates, against 4 us of the
// radix select's three histogram passes; two candidates a thread lose: one sequence of
// 205325 tokens, 416 candidates: 28.2 us against 17.5 for the radix select); same
// arguments as select_candidates.
__device__ __forceinline__ void select_by_rank(const DecodeArgs& a, int bh, int M, const uint32_t* keys, const int32_t* idx,
                               int* scan) {
    const int K = a.topk, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int32_t* lst = a.list + static_cast<size_t>(bh) * 64;
    int32_t* so = a.sel_idx ? a.sel_idx + static_cast<size_t>(bh) * K : nullptr;
    const uint32_t k = t < M ? keys[t] : 0u;
    const bool take = k != 0 && rank_of(keys, M, k, t, t - lane) < K;
    const unsigned bal = __ballot_sync(0xffffffffu, take);
    if (lane == 0) scan[warp] = __popc(bal);
    __syncthreads();
    int total = 0;   // K, or fewer when a summary load gave up and left candidates empty
    for (int w = 0; w < kScoreThreads / 32; ++w) total += scan[w];
    if (take) {
        int pos = __popc(bal & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) pos += scan[w];
        const int m = idx[t];
        lst[pos] = m;
        if (so) so[pos] = m;
    }
    if (so)
        for (int e = total + t; e < K; e += kScoreThreads) so[e] = -1;
    if (t == 0) a.list_n[bh] = total;
}

// Exact Top-K of M candidates (keys[i], block idx[i]) listed in ascending block
// order, ties to the lower block: radix select of the K-th largest key tau in
// digits of 12, 10 and 10 bits, then every key > tau plus the first keys == tau,
// emitted in list order.  256 threads; K <= M.  Empty candidates (key 0) are never
// kept: with fewer than K others (a summary load that gave up) the list is shorter.
__device__ __forceinline__ void select_candidates(const DecodeArgs& a, int bh, int M, const uint32_t* keys, const int32_t* idx,
                                  int* hist, int* scan, int* bc) {
    const int K = a.topk;
    const int t = threadIdx.x, lane = t & 31;
    int32_t* lst = a.list + static_cast<size_t>(bh) * 64;
    int32_t* so = a.sel_idx ? a.sel_idx + static_cast<size_t>(bh) * K : nullptr;
    uint32_t prefix = 0, mask = 0;
    int r = K;
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
        const int width = pass == 0 ? 12 : 10;
        const int sh = pass == 0 ? 20 : (pass == 1 ? 10 : 0);
        const int nb = 1 << width;
        for (int i = t; i < nb; i += kScoreThreads) hist[i] = 0;
        __syncthreads();
        for (int base = 0; base < M; base += kScoreThreads) {
            const int i = base + t;
            bool in = false;
            int bin = 0;
            if (i < M) {
                const uint32_t k = keys[i];
                in = (k & mask) == prefix;
                bin = static_cast<int>((k >> sh) & static_cast<uint32_t>(nb - 1));
            }
            // lanes with the same bin add once (the first pass sees few distinct bins)
            const uint32_t peers = __match_any_sync(0xffffffffu, in ? bin : -1 - lane);
            if (in && lane == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
        }
        __syncthreads();
        const int per = nb / kScoreThreads;   // 16 or 4 bins per thread, highest digits first
        int s = 0;
        for (int j = 0; j < per; ++j) s += hist[nb - 1 - (t * per + j)];
        const int excl = block_excl_scan(s, scan);
        if (excl < r && excl + s >= r) {
            int cum = excl;
            for (int j = 0; j < per; ++j) {
                const int bin = nb - 1 - (t * per + j);
                const int c = hist[bin];
                if (cum + c >= r) {
                    bc[0] = bin;
                    bc[1] = r - cum;
                    break;
                }
                cum += c;
            }
        }
        __syncthreads();
        prefix |= static_cast<uint32_t>(bc[0]) << sh;
        mask |= static_cast<uint32_t>(nb - 1) << sh;
        r = bc[1];
    }
    const uint32_t tau = prefix;   // the K-th largest key; take the first r keys equal to it
    if (tau == 0) r = 0;
    // list-order emission: contiguous ranges of odd length per thread (conflict-free reads)
    const int per = ((M + kScoreThreads - 1) / kScoreThreads) | 1;
    const int lo = min(t * per, M), hi = min(lo + per, M);
    int eq = 0;
    for (int i = lo; i < hi; ++i) eq += keys[i] == tau;
    const int eq_base = block_excl_scan(eq, scan);
    int cnt = 0, er = eq_base;
    for (int i = lo; i < hi; ++i) {
        const uint32_t k = keys[i];
        if (k > tau) {
            ++cnt;
        } else if (k == tau) {
            if (er < r) ++cnt;
            ++er;
        }
    }
    int pos = block_excl_scan(cnt, scan);
    er = eq_base;
    for (int i = lo; i < hi; ++i) {
        const uint32_t k = keys[i];
        bool take = k > tau;
        if (k == tau) {
            take = er < r;
            ++er;
        }
        if (take) {
            lst[pos] = idx[i];
            if (so) so[pos] = idx[i];
            ++pos;
        }
    }
    if (t == kScoreThreads - 1) {   // the last range ends the list
        a.list_n[bh] = pos;
        if (so)
            for (int e = pos; e < K; ++e) so[e] = -1;
    }
}

// grid (nsplit_s, B*Hkv), launched as a programmatic dependent of the prep kernel.
template <int DSEL>
__global__ void __launch_bounds__(kScoreThreads) dec_score_kernel(DecodeArgs a, int* status, long long limit,
                                                                  float score_scale) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr int kRowBytes = DSEL * 2;
    constexpr int kSlab = 32 * kRowBytes;
    const ScoreSmem L = score_smem_layout(a.nsplit_s, a.topk, DSEL);
    uint8_t* stage = smem;
    uint4* qs = reinterpret_cast<uint4*>(smem + L.qs);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bars);
    int* misc = reinterpret_cast<int*>(smem + L.misc);
    uint32_t* xchg = reinterpret_cast<uint32_t*>(smem + L.xchg);
    const int bh = blockIdx.y;
    const int b = bh / a.Hkv;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        for (int w = 0; w < 8; ++w) mbar_init(&bars[w], 1);
        fence_barrier_init();
    }
    const int n = __ldg(a.seq_lens + b);
    const bool bad = bad_len(n, a);   // recorded by the prep kernel
    const int C = bad ? 0 : (n - 1) / kBlk;
    const int K = a.topk;
    const int Kc = K > 0 ? K : 1;
    const int m0 = blockIdx.x * kDecScoreChunk;
    const int rows_cta = max(0, min(kDecScoreChunk, C - m0));
    const bool scored = rows_cta > 0 && K > 0 && C > K;
    const int r0 = m0 + warp * 32;
    const int rows = scored ? max(0, min(32, C - r0)) : 0;
    // the summaries, but the one of a block this step closes (the prep kernel writes
    // it), are fetched while the prep kernel runs
    const bool closes = rows > 0 && (n - 1) % kBlk == 0 && r0 + rows == C;
    const bf16* ksrc = static_cast<const bf16*>(a.Ksum) + (static_cast<size_t>(bh) * a.max_blocks + r0) * DSEL;
    const int early = rows - (closes ? 1 : 0);
    __syncthreads();   // barriers initialised
    if (rows > 0 && lane == 0) {
        mbar_arrive_expect_tx(&bars[warp], static_cast<uint32_t>(rows) * kRowBytes);
        if (early > 0)
            bulk_load(stage + warp * kSlab, ksrc, static_cast<uint32_t>(early) * kRowBytes, &bars[warp]);
    }
    grid_dep_wait();     // q~ and the summary of a block closed by this step
    grid_dep_launch();   // the attention kernel may start its set-up
    if (bad) return;
    if (rows > early && lane == 0)
        bulk_load(stage + warp * kSlab + early * kRowBytes, ksrc + static_cast<size_t>(early) * DSEL, kRowBytes,
                  &bars[warp]);
    uint32_t key = 0;
    // this CTA's candidate slots: global, or (one CTA per group) its own shared
    // memory, the ranks' key buffer once they are counted
    const bool alone = a.nsplit_s == 1;
    const size_t cbase = (static_cast<size_t>(bh) * a.nsplit_s + blockIdx.x) * Kc;
    uint32_t* my_key = alone ? xchg : a.cand_key + cbase;
    int32_t* my_idx = alone ? reinterpret_cast<int32_t*>(xchg) + Kc : a.cand_idx + cbase;
    if (scored) {
        if (t < DSEL / 8) qs[t] = __ldg(reinterpret_cast<const uint4*>(a.qt) + static_cast<size_t>(bh) * (DSEL / 8) + t);
        __syncthreads();   // q~ in shared memory
        if (rows > 0) {
            const bool ok = mbar_wait_drain(&bars[warp], 0, limit, status);
            if (ok && lane < rows) {
                const uint4* krow = reinterpret_cast<const uint4*>(stage + warp * kSlab + lane * kRowBytes);
                constexpr int NCH = DSEL / 8;
                uint64_t acc = 0;
#pragma unroll
                for (int j = 0; j < NCH; ++j) {
                    const int c = (j + lane) & (NCH - 1);   // rotated: a quarter warp hits distinct banks
                    const uint4 kv = krow[c], qv = qs[c];
                    acc = fma_f32x2(f32x2(bf_lo(kv.x), bf_hi(kv.x)), f32x2(bf_lo(qv.x), bf_hi(qv.x)), acc);
                    acc = fma_f32x2(f32x2(bf_lo(kv.y), bf_hi(kv.y)), f32x2(bf_lo(qv.y), bf_hi(qv.y)), acc);
                    acc = fma_f32x2(f32x2(bf_lo(kv.z), bf_hi(kv.z)), f32x2(bf_lo(qv.z), bf_hi(qv.z)), acc);
                    acc = fma_f32x2(f32x2(bf_lo(kv.w), bf_hi(kv.w)), f32x2(bf_lo(qv.w), bf_hi(qv.w)), acc);
                }
                float s0, s1;
                f32x2_split(acc, s0, s1);
                key = order_key((s0 + s1) * score_scale);
            }
        }
        // local Top-K of this CTA's blocks: those with fewer than K ahead of them
        bool take = t < rows_cta && key != 0;
        if (rows_cta > K && rows_cta <= kRankRows) {
            xchg[t] = take ? key : 0u;
            __syncthreads();
            take = take && rank_of(xchg, (rows_cta + 3) & ~3, key, t, warp * 32) < K;
        } else if (rows_cta > K) {
            // sort the distinct keys (score key, then the lower block first) and keep
            // those at or above the K-th
            uint64_t* sx = reinterpret_cast<uint64_t*>(smem + L.hist);
            const uint64_t comp = (static_cast<uint64_t>(key) << 32) | (0xffffffffu - static_cast<uint32_t>(t));
            const uint64_t sorted = bitonic256_desc(comp, sx);
            __syncthreads();
            if (t == K - 1) sx[0] = sorted;
            __syncthreads();
            take = take && comp >= sx[0];
        }
        // compact the kept blocks in block order into this CTA's K candidate slots
        const unsigned bal = __ballot_sync(0xffffffffu, take);
        if (lane == 0) misc[8 + warp] = __popc(bal);
        __syncthreads();
        int off = 0, total = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const int c = misc[8 + w];
            off += w < warp ? c : 0;
            total += c;
        }
        if (take) {
            const int pos = off + __popc(bal & ((1u << lane) - 1u));
            my_key[pos] = key;
            my_idx[pos] = m0 + t;
        }
        for (int e = total + t; e < Kc; e += kScoreThreads) {
            my_key[e] = 0;
            my_idx[e] = -1;
        }
    } else if (K > 0 && C > K) {
        // no blocks in this CTA's range: empty candidate slots
        for (int e = t; e < Kc; e += kScoreThreads) {
            my_key[e] = 0;
            my_idx[e] = -1;
        }
    }
    if (alone) {
        __syncthreads();
    } else {
        // the last CTA of the group to finish selects
        __threadfence();
        __syncthreads();
        if (t == 0) {
            const int old = atomicAdd(a.cnt_sel + bh, 1);
            misc[0] = old == static_cast<int>(gridDim.x) - 1;
        }
        __syncthreads();
        if (!misc[0]) return;
        __threadfence();
        if (t == 0) a.cnt_sel[bh] = 0;   // zero again for the next launch
    }
    int32_t* lst = a.list + static_cast<size_t>(bh) * 64;
    int32_t* so = a.sel_idx ? a.sel_idx + static_cast<size_t>(bh) * K : nullptr;
    if (C <= K) {   // short history: every historical block is kept
        for (int e = t; e < K; e += kScoreThreads) {
            if (e < C) lst[e] = e;
            if (so) so[e] = e < C ? e : -1;
        }
        if (t == 0) a.list_n[bh] = C;
        return;
    }
    if (K == 0) {
        if (t == 0) a.list_n[bh] = 0;
        return;
    }
    const size_t gbase = static_cast<size_t>(bh) * a.nsplit_s * Kc;
    if (C <= kDecScoreChunk) {
        // one CTA held every block: its local Top-K is the group's, already in block
        // order (-1 past the blocks whose summaries arrived; K <= 64 < 256 threads)
        const int m = t < K ? (alone ? my_idx[t] : __ldcg(a.cand_idx + gbase + t)) : -1;
        if (t < K) {
            lst[t] = m;
            if (so) so[t] = m;
        }
        const int kept = __syncthreads_count(m >= 0);
        if (t == 0) a.list_n[bh] = kept;
        return;
    }
    const int M = ((C + kDecScoreChunk - 1) / kDecScoreChunk) * Kc;   // the splits that held blocks
    const int Mp = (M + 3) & ~3;
    uint32_t* ckeys = reinterpret_cast<uint32_t*>(stage);
    int32_t* cidx = reinterpret_cast<int32_t*>(stage) + Mp;
    for (int i = t; i < Mp; i += kScoreThreads) {
        ckeys[i] = i < M ? __ldcg(a.cand_key + gbase + i) : 0u;
        cidx[i] = i < M ? __ldcg(a.cand_idx + gbase + i) : -1;
    }
    if (M <= kRankMax) {
        __syncthreads();
        select_by_rank(a, bh, M, ckeys, cidx, reinterpret_cast<int*>(smem + L.scan));
        return;
    }
    select_candidates(a, bh, M, ckeys, cidx, reinterpret_cast<int*>(smem + L.hist),
                      reinterpret_cast<int*>(smem + L.scan), misc + 1);
}

// ---------------------------------------------------------------- attention

// Page of block blk of sequence b, whose own block is c.  -1, and nothing is read, for a
// block it does not have; -1 and the status word for a table entry outside the cache.
__device__ __forceinline__ int block_page(const DecodeArgs& a, int b, int blk, int c, int* status) {
    if (static_cast<unsigned>(blk) > static_cast<unsigned>(c)) return -1;
    const int page = __ldg(a.block_table + static_cast<size_t>(b) * a.max_blocks + blk);
    if (page >= 0 && page < a.num_pages) return page;
    atomicExch(status, kStatusBadInput);
    return -1;
}

// Shared-memory layout of the attention kernel for a ring of nst stages.
struct AttnLayout {
    size_t tile, q32, ps, red, alpha, lsum, bars, misc, ent, total;
};
__host__ __device__ inline AttnLayout attn_layout(int D, int G, int nst, int bpc) {
    AttnLayout L;
    L.tile = static_cast<size_t>(kBlk) * D * 2;     // one K or V page slice
    L.q32 = nst * 2 * L.tile;                        // fp32 queries [G][D]
    L.ps = L.q32 + static_cast<size_t>(G) * D * 4;   // probabilities [G][64]
    L.red = L.ps + static_cast<size_t>(G) * 64 * 4;  // [8 warps][8]
    L.alpha = L.red + 64 * 4;                        // [8], then merge max [8] and sum [8]
    L.lsum = L.alpha + 32 * 4;                       // [8 warps][8]
    L.bars = L.lsum + 64 * 4;                        // nst mbarriers
    L.misc = L.bars + 64;                            // flag
    L.ent = L.misc + 64;                             // entries: block, page (2 ints each)
    L.total = L.ent + static_cast<size_t>(bpc) * 8;
    return L;
}

// grid (nsplit_a, B*Hkv), a programmatic dependent of the score kernel (of the
// prep kernel in dense mode).  The group's list is the current block c first,
// then the kept blocks in ascending order (dense: blocks 0 .. c-1); this CTA
// takes entries [x*bpc, (x+1)*bpc).
template <int D, int G>
__global__ void __launch_bounds__(kAttnThreads) dec_attn_kernel(DecodeArgs a, int* status, long long limit,
                                                                float scale_log2) {
    constexpr int kNW = D / 2;                          // bf16 pairs per row
    constexpr int NQG = kAttnThreads / 64;              // head groups in the score step
    constexpr int HP = (G + NQG - 1) / NQG;             // heads per thread in the score step
    constexpr int NHG = kAttnThreads / kNW;             // head groups in the PV step
    constexpr int HPV = (G + NHG - 1) / NHG;            // heads per thread in the PV step
    constexpr int NCH = D / 8;                          // 16-byte chunks per row
    extern __shared__ __align__(128) uint8_t smem[];
    const int nst = a.nst;
    const AttnLayout Ly = attn_layout(D, G, nst, a.bpc);
    const int kTile = static_cast<int>(Ly.tile);
    float* q32 = reinterpret_cast<float*>(smem + Ly.q32);
    float* Ps = reinterpret_cast<float*>(smem + Ly.ps);
    float* red = reinterpret_cast<float*>(smem + Ly.red);
    float* alpha_s = reinterpret_cast<float*>(smem + Ly.alpha);
    float* lsum = reinterpret_cast<float*>(smem + Ly.lsum);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + Ly.bars);
    int* misc = reinterpret_cast<int*>(smem + Ly.misc);
    int* ent = reinterpret_cast<int*>(smem + Ly.ent);

    const int bh = blockIdx.y;
    const int b = bh / a.Hkv, g = bh - b * a.Hkv;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int n = __ldg(a.seq_lens + b);
    const bool bad = bad_len(n, a);   // recorded by the prep kernel
    const int c = bad ? 0 : (n - 1) / kBlk;
    const int j0 = blockIdx.x * a.bpc;
    const size_t head_off = static_cast<size_t>(g) * kBlk * D;   // this KV head's slice inside a page
    auto issue = [&](int jj) {
        const int s = jj % nst;
        const int page = ent[2 * jj + 1];
        uint8_t* dst = smem + s * 2 * kTile;
        if (page < 0) {
            mbar_arrive(&full[s]);
            return;
        }
        const size_t off = static_cast<size_t>(page) * a.Hkv * kBlk * D + head_off;
        mbar_arrive_expect_tx(&full[s], 2 * kTile);
        bulk_load(dst, static_cast<const bf16*>(a.K_cache) + off, kTile, &full[s]);
        bulk_load(dst + kTile, static_cast<const bf16*>(a.V_cache) + off, kTile, &full[s]);
    };

    // --- set-up that needs nothing from the preceding kernel
    if (t == 0) {
        for (int s = 0; s < nst; ++s) mbar_init(&full[s], 1);
        fence_barrier_init();
    }
    const bf16* qg = static_cast<const bf16*>(a.q) + (static_cast<size_t>(b) * a.Hq + static_cast<size_t>(g) * G) * D;
    for (int e = t; e < G * D; e += kAttnThreads) q32[e] = __bfloat162float(qg[e]);
    grid_dep_wait();   // the kept list
    if (bad) return;
    const int L = (a.dense ? c : __ldg(a.list_n + bh)) + 1;
    const int cnt = max(0, min(j0 + a.bpc, L) - j0);
    // (the current block, entry 0, is written by the preceding kernel, so every
    // page load waits for the grid dependency)
    const int first = 0;
    for (int jj = first + t; jj < cnt; jj += kAttnThreads) {
        const int j = j0 + jj;
        const int blk = j == 0 ? c : (a.dense ? j - 1 : __ldg(a.list + static_cast<size_t>(bh) * 64 + j - 1));
        ent[2 * jj] = blk;
        ent[2 * jj + 1] = block_page(a, b, blk, c, status);
    }
    __syncthreads();
    int issued = first;
    if (t == 0) {
        for (; issued < min(cnt, nst); ++issued) issue(issued);
    }

    const int k = t & 63, hh = t >> 6;           // score step: key k, heads hh*HP + u (keys of a head in warps 2hh, 2hh+1)
    const int wi = t % kNW, hg = t / kNW;        // PV step: column pair wi, heads hg*HPV + u
    float m_run[HP], l_part[HP];
#pragma unroll
    for (int u = 0; u < HP; ++u) {
        m_run[u] = -CUDART_INF_F;
        l_part[u] = 0.f;
    }
    uint64_t acc[HPV];
#pragma unroll
    for (int u = 0; u < HPV; ++u) acc[u] = 0;

    bool ok = true;
    int jj = 0;
    for (; jj < cnt; ++jj) {
        const int s = jj % nst;
        const bool got = mbar_wait_drain(&full[s], (jj / nst) & 1, limit, status);
        if (!__syncthreads_and(got)) {
            ok = false;
            break;
        }
        const int page = ent[2 * jj + 1];
        const int nvalid = page < 0 ? 0 : (ent[2 * jj] == c ? n - c * kBlk : kBlk);
        const uint8_t* Kt = smem + s * 2 * kTile;
        const uint8_t* Vt = Kt + kTile;

        // z = scale * q_h . k for this thread's key and heads (log2 units)
        float z[HP];
        {
            uint64_t az[HP];
#pragma unroll
            for (int u = 0; u < HP; ++u) az[u] = 0;
            const uint4* krow = reinterpret_cast<const uint4*>(Kt + k * D * 2);
#pragma unroll
            for (int jc = 0; jc < NCH; ++jc) {
                const int cc = (jc + k) & (NCH - 1);    // rotated chunk: no bank conflicts across keys
                const uint4 kv = krow[cc];
                const uint64_t k01 = f32x2(bf_lo(kv.x), bf_hi(kv.x));
                const uint64_t k23 = f32x2(bf_lo(kv.y), bf_hi(kv.y));
                const uint64_t k45 = f32x2(bf_lo(kv.z), bf_hi(kv.z));
                const uint64_t k67 = f32x2(bf_lo(kv.w), bf_hi(kv.w));
#pragma unroll
                for (int u = 0; u < HP; ++u) {
                    const int h = hh * HP + u;
                    if (h < G) {
                        const float4 qa = *reinterpret_cast<const float4*>(q32 + h * D + cc * 8);
                        const float4 qb = *reinterpret_cast<const float4*>(q32 + h * D + cc * 8 + 4);
                        az[u] = fma_f32x2(k01, f32x2(qa.x, qa.y), az[u]);
                        az[u] = fma_f32x2(k23, f32x2(qa.z, qa.w), az[u]);
                        az[u] = fma_f32x2(k45, f32x2(qb.x, qb.y), az[u]);
                        az[u] = fma_f32x2(k67, f32x2(qb.z, qb.w), az[u]);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < HP; ++u) {
                float z0, z1;
                f32x2_split(az[u], z0, z1);
                z[u] = k < nvalid ? (z0 + z1) * scale_log2 : -CUDART_INF_F;
            }
        }
#pragma unroll
        for (int u = 0; u < HP; ++u) {
            const float mx = warp_max(z[u]);
            if (lane == 0) red[warp * 8 + u] = mx;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < HP; ++u) {
            const int h = hh * HP + u;
            if (h < G) {
                const float mb = fmaxf(red[(2 * hh) * 8 + u], red[(2 * hh + 1) * 8 + u]);
                const float m_new = fmaxf(m_run[u], mb);
                const float alpha = m_run[u] == -CUDART_INF_F ? 0.f : fast_exp2(m_run[u] - m_new);
                const float p = z[u] == -CUDART_INF_F ? 0.f : fast_exp2(z[u] - m_new);
                l_part[u] = l_part[u] * alpha + p;
                m_run[u] = m_new;
                Ps[h * 64 + k] = p;
                if (k == 0) alpha_s[h] = alpha;
            }
        }
        __syncthreads();
        // O_h = alpha_h O_h + sum_k p_hk v_k for this thread's column pair
#pragma unroll
        for (int u = 0; u < HPV; ++u) {
            const int h = hg * HPV + u;
            if (h < G) {
                const float al = alpha_s[h];
                acc[u] = fma_f32x2(acc[u], f32x2(al, al), 0ull);
            }
        }
        const uint32_t* V32 = reinterpret_cast<const uint32_t*>(Vt);
#pragma unroll 4
        for (int kk = 0; kk < nvalid; ++kk) {
            const uint32_t w = V32[kk * kNW + wi];
            const uint64_t v2 = f32x2(bf_lo(w), bf_hi(w));
#pragma unroll
            for (int u = 0; u < HPV; ++u) {
                const int h = hg * HPV + u;
                if (h < G) {
                    const float p = Ps[h * 64 + kk];
                    acc[u] = fma_f32x2(f32x2(p, p), v2, acc[u]);
                }
            }
        }
        __syncthreads();   // the stage, Ps and red are free
        if (t == 0 && issued < cnt) {
            fence_proxy_async_smem();
            issue(issued);
            ++issued;
        }
    }
    if (!ok) {
        // let copies still in flight land before the CTA exits; report nothing
        if (t == 0)
            for (int q = jj; q < issued; ++q) mbar_wait_drain(&full[q % nst], (q / nst) & 1, limit, status);
#pragma unroll
        for (int u = 0; u < HP; ++u) {
            m_run[u] = -CUDART_INF_F;
            l_part[u] = 0.f;
        }
#pragma unroll
        for (int u = 0; u < HPV; ++u) acc[u] = 0;
    }

    // partial (max, sum, output) of this CTA per head
#pragma unroll
    for (int u = 0; u < HP; ++u) {
        const float ls = warp_sum(l_part[u]);
        if (lane == 0) lsum[warp * 8 + u] = ls;
    }
    __syncthreads();
    float* part = a.part + (static_cast<size_t>(bh) * a.nsplit_a + blockIdx.x) * G * (D + 2);
    if (k == 0) {
#pragma unroll
        for (int u = 0; u < HP; ++u) {
            const int h = hh * HP + u;
            if (h < G) {
                part[h * (D + 2)] = m_run[u];
                part[h * (D + 2) + 1] = lsum[(2 * hh) * 8 + u] + lsum[(2 * hh + 1) * 8 + u];
            }
        }
    }
#pragma unroll
    for (int u = 0; u < HPV; ++u) {
        const int h = hg * HPV + u;
        if (h < G) {
            float o0, o1;
            f32x2_split(acc[u], o0, o1);
            part[h * (D + 2) + 2 + 2 * wi] = o0;
            part[h * (D + 2) + 3 + 2 * wi] = o1;
        }
    }
    __threadfence();
    __syncthreads();
    if (t == 0) {
        const int old = atomicAdd(a.cnt_attn + bh, 1);
        misc[0] = old == static_cast<int>(gridDim.x) - 1;
    }
    __syncthreads();
    if (!misc[0]) return;
    __threadfence();
    if (t == 0) a.cnt_attn[bh] = 0;   // zero again for the next launch

    // Merge the partials of every head (only the splits the list reached).  The
    // (max, sum) pairs are staged in the free ring first, turned into weights
    // exp2(m_x - M) per head, then every thread sums its columns over the splits
    // with all loads independent.
    const int used = (L + a.bpc - 1) / a.bpc;
    const float* pg = a.part + static_cast<size_t>(bh) * a.nsplit_a * G * (D + 2);
    float* mw = reinterpret_cast<float*>(smem);    // [used][G][2]
    float* mM = alpha_s + 8;                       // [G] max
    float* mL = alpha_s + 16;                      // [G] sum
    for (int i = t; i < used * G; i += kAttnThreads) {
        const float* px = pg + static_cast<size_t>(i) * (D + 2);
        mw[2 * i] = __ldcg(px);
        mw[2 * i + 1] = __ldcg(px + 1);
    }
    __syncthreads();
    if (t < G) {
        float M = -CUDART_INF_F;
        for (int x = 0; x < used; ++x) M = fmaxf(M, mw[2 * (x * G + t)]);
        float ls = 0.f;
        for (int x = 0; x < used; ++x) {
            const float mx = mw[2 * (x * G + t)];
            const float w = mx == -CUDART_INF_F ? 0.f : fast_exp2(mx - M);
            ls = fmaf(w, mw[2 * (x * G + t) + 1], ls);
            mw[2 * (x * G + t)] = w;
        }
        mM[t] = M;
        mL[t] = ls;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < HPV; ++u) {
        const int h = hg * HPV + u;
        if (h >= G) continue;
        float o0 = 0.f, o1 = 0.f;
#pragma unroll 16
        for (int x = 0; x < used; ++x) {
            const float2 v = __ldcg(reinterpret_cast<const float2*>(pg + (static_cast<size_t>(x) * G + h) * (D + 2) + 2) + wi);
            const float w = mw[2 * (x * G + h)];
            o0 = fmaf(w, v.x, o0);
            o1 = fmaf(w, v.y, o1);
        }
        const float inv = 1.f / mL[h];
        const size_t orow = (static_cast<size_t>(b) * a.Hq + static_cast<size_t>(g) * G + h) * D;
        reinterpret_cast<uint32_t*>(static_cast<bf16*>(a.O) + orow)[wi] = pack_bf16x2(o0 * inv, o1 * inv);
        if (a.LSE != nullptr && wi == 0)
            a.LSE[static_cast<size_t>(b) * a.Hq + static_cast<size_t>(g) * G + h] = (mM[h] + log2f(mL[h])) / kLog2e;
    }
}

// -------------------------------------------------- attention on tensor cores (d = 128)
//
// A step takes two pages (128 keys) of the CTA's list:
//   S^T[128 keys][16] = Kpair[128 x 128] . Qpad[16 x 128]^T          tcgen05, M=128 N=16, K-major A and B
//   softmax over the 128 keys of every head (TMEM lane = key)
//   O^T[128 d][16]    = Vpair^T[128 d x 128 keys] . Ppad[16 x 128]^T  tcgen05, A MN-major (V as stored)
// Q and P are padded from G <= 8 heads to N = 16 rows of zeros.  K and V tiles
// sit in shared memory as [d half][128 keys][128 B] with the 128-byte swizzle,
// written by four 64 x 64 TMA boxes each (page 0 in rows 0-63, page 1 in
// rows 64-127); Q is [d half][16][128 B], P [key half][16][128 B], both
// swizzled by the threads that write them.  Every step's O^T is a fresh
// accumulator (thread t owns row d = t): a dense list's threads fold it into
// registers with the online-softmax rescale, a SAS list's store it as the pair's
// partial (2.2 KB a step at G = 4, merged from L2; the sums are stored while PV
// runs, the output behind the next loads).

constexpr int kTcThreads = 128;
constexpr int kTcTile = 2 * 128 * 128;          // bytes of one K (or V) tile of a step
constexpr int kTcStage = 2 * kTcTile;           // K and V
constexpr uint32_t kTcTmemCols = 64;            // S^T in columns 0-15, O^T in 32-47
constexpr int kMaxDecCluster = 16;              // needs the non-portable cluster size attribute
constexpr int kPairFloats = 136;                // partial of a page pair and head: max, -, -, -, sum of each warp, output

struct TcLayout {
    size_t q, p, red, alpha, lsum, bars, misc, ent, total;
};
__host__ __device__ inline TcLayout tc_layout(int nst, int bpc) {
    TcLayout L;
    L.q = static_cast<size_t>(nst) * kTcStage;   // 4096: [2][16][128 B]
    L.p = L.q + 4096;                            // 4096: [2][16][128 B]
    L.red = L.p + 4096;                          // [4 warps][16]
    L.alpha = L.red + 64 * 4;                    // [16] alpha, then merge max [16] and sum [16]
    L.lsum = L.alpha + 48 * 4;                   // [4 warps][16]
    L.bars = L.lsum + 64 * 4;                    // full[4], qk, pv
    L.misc = L.bars + 64;                        // flag, TMEM base
    L.ent = L.misc + 64;                         // entries: block, page
    L.total = L.ent + static_cast<size_t>(bpc) * 8 + 1024;   // + alignment slack
    return L;
}

// TMA loads of list entry e (a page of step e/2) into the step's stage: K and V,
// two 64 x 64 boxes each (the two halves of d); nothing for a missing page.
__device__ __forceinline__ void tc_load_page(uint8_t* smem, int nst, const int* ent, int e, const CUtensorMap* mapK,
                                             const CUtensorMap* mapV, uint64_t* full, int Hkv, int g) {
    const int page = ent[2 * e + 1];
    if (page < 0) return;
    const int s = (e >> 1) % nst, pg = e & 1;
    uint8_t* st = smem + static_cast<size_t>(s) * kTcStage;
    const int row = page * Hkv + g;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        tma_load_3d(st + h * 16384 + pg * 8192, mapK, &full[s], h * 64, 0, row);
        tma_load_3d(st + kTcTile + h * 16384 + pg * 8192, mapV, &full[s], h * 64, 0, row);
    }
}
__device__ __forceinline__ uint32_t tc_page_bytes(const int* ent, int e) {
    return ent[2 * e + 1] >= 0 ? 4u * 8192u : 0u;
}

// Three CTAs an SM at most (shared memory), so 168 registers a thread are there to take:
// without the second bound the compiler kept to 48, 56 and 64 (G = 1, 2, 4) and spilled
// (dense lists, 8 sequences of 64K tokens, G = 1, 2, 4: 1235, 640 and 349 us, with it
// 1194, 625 and 342; a SAS step of one sequence of 8K tokens 19.6 and 19.1).
template <int G, bool SAS>
__global__ void __launch_bounds__(kTcThreads, 3)
dec_attn_tc_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV, DecodeArgs a,
                   int* status, long long limit, float scale_log2) {
    constexpr int D = 128;
    constexpr uint32_t IDESC_S = idesc_bf16(128, 16, 0, 0);
    constexpr uint32_t IDESC_O = idesc_bf16(128, 16, 1, 0);
    extern __shared__ __align__(1024) uint8_t dsm[];
    // the swizzled tiles need 1024-byte alignment
    uint8_t* smem = dsm + ((1024u - (smem_u32(dsm) & 1023u)) & 1023u);
    const int nst = a.nst;
    const TcLayout Ly = tc_layout(nst, a.bpc);
    uint8_t* qs = smem + Ly.q;
    uint8_t* ps = smem + Ly.p;
    float* red = reinterpret_cast<float*>(smem + Ly.red);
    float* mM = reinterpret_cast<float*>(smem + Ly.alpha) + 16;
    float* mL = reinterpret_cast<float*>(smem + Ly.alpha) + 32;
    float* lsum = reinterpret_cast<float*>(smem + Ly.lsum);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + Ly.bars);
    uint64_t* qk_bar = full + 4;
    uint64_t* pv_bar = full + 5;
    int* misc = reinterpret_cast<int*>(smem + Ly.misc);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc + 4);
    int* ent = reinterpret_cast<int*>(smem + Ly.ent);

    const int bh = blockIdx.y;
    const int b = bh / a.Hkv, g = bh - b * a.Hkv;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int n = __ldg(a.seq_lens + b);
    const bool bad = bad_len(n, a);   // recorded by the prep kernel
    const int c = bad ? 0 : (n - 1) / kBlk;
#define SAS_TC_LOAD(e) tc_load_page(smem, nst, ent, (e), &mapK, &mapV, full, a.Hkv, g)

    // --- set-up that needs nothing from the preceding kernel
    if (t == 0) {
        for (int s = 0; s < nst; ++s) mbar_init(&full[s], 1);
        mbar_init(qk_bar, 1);
        mbar_init(pv_bar, 1);
        fence_barrier_init();
        tma_prefetch_desc(&mapK);
        tma_prefetch_desc(&mapV);
        // the current block (entry 0) was appended by the prep kernel, which the
        // score kernel waited for before letting this grid start, so its page can
        // load now (dense mode: the prep kernel precedes this one directly)
        if (SAS && !bad && blockIdx.x == 0) {
            int page = __ldg(a.block_table + static_cast<size_t>(b) * a.max_blocks + c);
            if (page < 0 || page >= a.num_pages) page = -1;   // recorded by the prep kernel
            ent[0] = c;
            ent[1] = page;
            mbar_expect_tx(&full[0], tc_page_bytes(ent, 0));
            SAS_TC_LOAD(0);
        }
    }
    if (warp == 0) {
        tmem_alloc(tmem_slot, kTcTmemCols);
        tmem_relinquish();
    }
    // Q rows (zero past G) and P (rows past G stay zero), 16-byte chunks swizzled
    const bf16* qg = static_cast<const bf16*>(a.q) + (static_cast<size_t>(b) * a.Hq + static_cast<size_t>(g) * G) * D;
    for (int i = t; i < 2 * 16 * 8; i += kTcThreads) {
        const int h = i >> 7, row = (i >> 3) & 15, ch = i & 7;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (row < G) v = __ldg(reinterpret_cast<const uint4*>(qg + row * D + h * 64 + ch * 8));
        *reinterpret_cast<uint4*>(qs + h * 2048 + row * 128 + ((ch ^ (row & 7)) << 4)) = v;
        *reinterpret_cast<uint4*>(ps + h * 2048 + row * 128 + (ch << 4)) = make_uint4(0, 0, 0, 0);
    }
    grid_dep_wait();   // the kept list
    const int L = bad ? 0 : (SAS ? __ldg(a.list_n + bh) : c) + 1;
    // a cluster shares its list's page pairs evenly (a short history has fewer than bpc / 2 a CTA)
    const int pairs = (L + 1) >> 1;
    const int per = SAS ? 2 * ((pairs + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x)) : a.bpc;
    const int j0 = blockIdx.x * per;
    const int cnt = bad ? 0 : max(0, min(j0 + per, L) - j0);
    const int first = SAS && blockIdx.x == 0 ? 1 : 0;   // entries set up before the wait
    for (int jj = first + t; jj < cnt; jj += kTcThreads) {
        const int j = j0 + jj;
        const int blk = j == 0 ? c : (SAS ? __ldg(a.list + static_cast<size_t>(bh) * 64 + j - 1) : j - 1);
        ent[2 * jj] = blk;
        ent[2 * jj + 1] = block_page(a, b, blk, c, status);
    }
    fence_proxy_async_smem();   // Q and P writes before the tensor cores read them
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int steps = (cnt + 1) >> 1;
    int issued = 0;   // steps whose loads are issued (thread 0)
    if (t == 0) {
        for (; issued < min(steps, nst); ++issued) {
            const int e0 = 2 * issued, e1 = e0 + 1;
            uint32_t bytes = 0;
            if (e0 >= first) bytes += tc_page_bytes(ent, e0);
            if (e1 < cnt) bytes += tc_page_bytes(ent, e1);
            mbar_arrive_expect_tx(&full[issued], bytes);
            if (e0 >= first) SAS_TC_LOAD(e0);
            if (e1 < cnt) SAS_TC_LOAD(e1);
        }
    }

    // dense: running maximum, sum and output of this CTA's pages; SAS: of one page pair,
    // stored before the next
    float m_run[G], l_part[G], o[G];
#pragma unroll
    for (int h = 0; h < G; ++h) {
        m_run[h] = -CUDART_INF_F;
        l_part[h] = 0.f;
        o[h] = 0.f;
    }
    float* pair_part = a.part + (static_cast<size_t>(bh) * a.nsplit_a * (a.bpc >> 1) + (j0 >> 1)) * G * kPairFloats;
    // the CTA's x-th pair: maximum and sum, while the second product runs, then the output
    auto store_sums = [&](int x) {
        // warp sums with warp_sum's pairs of lanes, the heads shared out on the way:
        // a lane ends with head (lane's top log2(G) bits)
        float v[G];
#pragma unroll
        for (int h = 0; h < G; ++h) v[h] = l_part[h];
        int o = 16;
#pragma unroll
        for (int half = G / 2; half > 0; half >>= 1, o >>= 1) {
            const bool upper = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < half; ++i) {
                const float send = upper ? v[i] : v[i + half];
                v[i] = (upper ? v[i + half] : v[i]) + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
#pragma unroll
        for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        float* px = pair_part + x * G * kPairFloats;
        if (lane % (32 / G) == 0) px[lane / (32 / G) * kPairFloats + 4 + warp] = v[0];
        if (t == 0) {
#pragma unroll
            for (int h = 0; h < G; ++h) px[h * kPairFloats] = m_run[h];
        }
    };
    auto store_output = [&](int x) {
#pragma unroll
        for (int h = 0; h < G; ++h) pair_part[(x * G + h) * kPairFloats + 8 + t] = o[h];
    };
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(warp * 32) << 16);
    bool ok = true;
    int j = 0;
    int pending = 0, pj = 0;   // 1: a QK commit outstanding, 2: a PV commit outstanding (of step pj)
    for (; j < steps; ++j) {
        const int s = j % nst;
        uint8_t* st = smem + static_cast<size_t>(s) * kTcStage;
        // Two CTA-wide barriers a step: everything else is ordered by the MMAs' commits.
        if (warp == 0) {
            // QK (whole warp; the elected lane issues).  Every thread has read the
            // previous S before the barrier ahead of the previous PV.
            ok = __all_sync(0xffffffffu, ok && mbar_wait_drain(&full[s], (j / nst) & 1, limit, status));
            tc_fence_after();
            if (ok && elect_one()) {
                const uint32_t kb = smem_u32(st), qb = smem_u32(qs);
#pragma unroll
                for (int k = 0; k < D / 16; ++k) {
                    const uint64_t da = smem_desc_sw128(kb + (k >> 2) * 16384 + (k & 3) * 32, 16, 1024);
                    const uint64_t db = smem_desc_sw128(qb + (k >> 2) * 2048 + (k & 3) * 32, 16, 1024);
                    umma_bf16(tmem, da, db, IDESC_S, k > 0);
                }
                umma_commit(qk_bar);
            }
            __syncwarp();
            if (ok) { pending = 1; pj = j; }
        }
        if (ok && !mbar_wait_drain(qk_bar, j & 1, limit, status)) ok = false;
        ok = __all_sync(0xffffffffu, ok);
        const int e0 = 2 * j, e1 = e0 + 1;
        const int nv0 = ent[2 * e0 + 1] < 0 ? 0 : (ent[2 * e0] == c ? n - c * kBlk : kBlk);
        const int nv1 = (e1 >= cnt || ent[2 * e1 + 1] < 0) ? 0 : (ent[2 * e1] == c ? n - c * kBlk : kBlk);
        tc_fence_after();
        const int key = t;                           // TMEM lane = key of the pair
        const bool valid = key < 64 ? key < nv0 : key - 64 < nv1;
        float z[G];
        if (ok) {
            uint32_t sr[16];
            tmem_ld16(lane_base, sr);
            tmem_wait_ld();
#pragma unroll
            for (int h = 0; h < G; ++h) {
                z[h] = valid ? __uint_as_float(sr[h]) * scale_log2 : -CUDART_INF_F;
                const float mx = warp_max(z[h]);
                if (lane == 0) red[warp * 16 + h] = mx;
            }
            // rows of a page past its valid keys (or of a missing page) get zero values,
            // so P = 0 there cannot meet a non-finite V
            if (nv0 < kBlk || nv1 < kBlk) {
                mbar_wait_drain(&full[s], (j / nst) & 1, limit, status);   // completed: QK has read the stage
                for (int i = t; i < 2 * 2 * 64 * 8; i += kTcThreads) {   // (page, half, row, chunk)
                    const int pg = i >> 10, h = (i >> 9) & 1, row = (i >> 3) & 63, ch = i & 7;
                    if (row >= (pg ? nv1 : nv0))
                        *reinterpret_cast<uint4*>(st + kTcTile + h * 16384 + pg * 8192 + row * 128 + (ch << 4)) =
                            make_uint4(0, 0, 0, 0);
                }
            }
        }
        if (!__syncthreads_and(ok)) {
            ok = false;
            break;
        }
        float alpha[G];
#pragma unroll
        for (int h = 0; h < G; ++h) {
            const float mb = fmaxf(fmaxf(red[h], red[16 + h]), fmaxf(red[32 + h], red[48 + h]));
            const float m_new = SAS ? mb : fmaxf(m_run[h], mb);
            alpha[h] = SAS || m_run[h] == -CUDART_INF_F ? 0.f : fast_exp2(m_run[h] - m_new);
            const float pr = z[h] == -CUDART_INF_F ? 0.f : fast_exp2(z[h] - m_new);
            l_part[h] = SAS ? pr : l_part[h] * alpha[h] + pr;
            m_run[h] = m_new;
            const int kh = key >> 6, ch = (key & 63) >> 3;
            *reinterpret_cast<bf16*>(ps + kh * 2048 + h * 128 + ((ch ^ (h & 7)) << 4) + ((key & 7) << 1)) =
                __float2bfloat16_rn(pr);
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        if (warp == 0) {
            tc_fence_after();
            if (elect_one()) {
                const uint32_t vb = smem_u32(st + kTcTile), pb = smem_u32(ps);
#pragma unroll
                for (int k = 0; k < 128 / 16; ++k) {
                    const uint64_t da = smem_desc_sw128(vb + k * 2048, 16384, 1024);
                    const uint64_t db = smem_desc_sw128(pb + (k >> 2) * 2048 + (k & 3) * 32, 16, 1024);
                    umma_bf16(tmem + 32, da, db, IDESC_O, k > 0);
                }
                umma_commit(pv_bar);
            }
            __syncwarp();
            pending = 2;
        }
        if (SAS) store_sums(j);
        if (!mbar_wait_drain(pv_bar, j & 1, limit, status)) ok = false;
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
            pending = 0;
            tc_fence_after();
            uint32_t orr[16];
            tmem_ld16(lane_base + 32, orr);
            tmem_wait_ld();
#pragma unroll
            for (int h = 0; h < G; ++h)
                o[h] = SAS ? __uint_as_float(orr[h]) : fmaf(o[h], alpha[h], __uint_as_float(orr[h]));
            tc_fence_before();
        }
        // (a warp that gave up here says so at the next step's barrier)
        // PV has read the stage: its next load can go out
        if (t == 0 && ok && issued < steps) {
            const int e0 = 2 * issued, e1 = e0 + 1;
            const int s2 = issued % nst;
            uint32_t bytes = tc_page_bytes(ent, e0);
            if (e1 < cnt) bytes += tc_page_bytes(ent, e1);
            mbar_arrive_expect_tx(&full[s2], bytes);
            SAS_TC_LOAD(e0);
            if (e1 < cnt) SAS_TC_LOAD(e1);
            ++issued;
        }
        if (SAS && ok) store_output(j);
    }
    if (!__syncthreads_and(ok)) {
        // let the tensor cores and the copies in flight finish before leaving
        if (t == 0) {
            if (pending == 1) mbar_wait_drain(qk_bar, pj & 1, limit, status);
            if (pending == 2) mbar_wait_drain(pv_bar, pj & 1, limit, status);
            for (int q = max(0, issued - nst); q < issued; ++q) mbar_wait_drain(&full[q % nst], (q / nst) & 1, limit, status);
        }
#pragma unroll
        for (int h = 0; h < G; ++h) {
            m_run[h] = -CUDART_INF_F;
            l_part[h] = 0.f;
            o[h] = 0.f;
        }
        if (SAS)
            for (int x = 0; x < steps; ++x) {
                store_sums(x);
                store_output(x);
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTcTmemCols);
    }

    if constexpr (SAS) {
        // the group's CTAs are one cluster: with every pair's partial stored, warp w of
        // CTA r merges heads r + S w, ... over the list's pairs in order (a lane takes
        // four of the output's columns).  Short rolled code: it runs once a CTA, so its
        // instructions come from L2 (unrolled over heads and pairs it took 2 to 7 us)
        cluster_sync();
        const int S = cluster_size();
        constexpr int kBatch = 17;   // pairs of 33 pages
        const float* base = a.part + static_cast<size_t>(bh) * a.nsplit_a * (a.bpc >> 1) * G * kPairFloats;
#pragma unroll 1
        for (int h = cluster_rank() + warp * S; h < G && !bad; h += (kTcThreads / 32) * S) {
            const float* ph = base + h * kPairFloats;
            // lane x: maximum and sum of pairs x and 32 + x (a list has at most 33)
            float w[2] = {-CUDART_INF_F, -CUDART_INF_F}, l[2] = {0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int x = 32 * i + lane;
                if (x < pairs) {
                    const float* px = ph + x * G * kPairFloats;
                    w[i] = __ldcg(px);
                    const float4 l4 = __ldcg(reinterpret_cast<const float4*>(px + 4));
                    l[i] = l4.x + l4.y + l4.z + l4.w;
                }
            }
            float M = 0.f, ls = 0.f;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
            for (int x0 = 0; x0 < pairs; x0 += kBatch) {
                float4 v[kBatch];
#pragma unroll
                for (int x = 0; x < kBatch; ++x)
                    v[x] = x0 + x < pairs ? __ldcg(reinterpret_cast<const float4*>(ph + (x0 + x) * G * kPairFloats + 8) + lane)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
                if (x0 == 0) {
                    M = warp_max(fmaxf(w[0], w[1]));
#pragma unroll
                    for (int i = 0; i < 2; ++i) w[i] = w[i] == -CUDART_INF_F ? 0.f : fast_exp2(w[i] - M);
                }
#pragma unroll
                for (int x = 0; x < kBatch; ++x) {
                    const int xx = x0 + x;
                    if (xx >= pairs) break;
                    const float wx = __shfl_sync(0xffffffffu, xx < 32 ? w[0] : w[1], xx & 31);
                    ls = fmaf(wx, __shfl_sync(0xffffffffu, xx < 32 ? l[0] : l[1], xx & 31), ls);
                    acc.x = fmaf(wx, v[x].x, acc.x);
                    acc.y = fmaf(wx, v[x].y, acc.y);
                    acc.z = fmaf(wx, v[x].z, acc.z);
                    acc.w = fmaf(wx, v[x].w, acc.w);
                }
            }
            const size_t at = static_cast<size_t>(b) * a.Hq + static_cast<size_t>(g) * G + h;
            reinterpret_cast<uint2*>(static_cast<bf16*>(a.O) + at * D)[lane] =
                make_uint2(pack_bf16x2(acc.x / ls, acc.y / ls), pack_bf16x2(acc.z / ls, acc.w / ls));
            if (a.LSE != nullptr && lane == 0) a.LSE[at] = (M + log2f(ls)) / kLog2e;
        }
        return;
    }
    // partial (max, sum, output) of this CTA per head
#pragma unroll
    for (int h = 0; h < G; ++h) {
        const float ls = warp_sum(l_part[h]);
        if (lane == 0) lsum[warp * 16 + h] = ls;
    }
    __syncthreads();
    float* part = a.part + (static_cast<size_t>(bh) * a.nsplit_a + blockIdx.x) * G * (D + 2);
#pragma unroll
    for (int h = 0; h < G; ++h) {
        if (t == 0) {
            part[h * (D + 2)] = m_run[h];
            part[h * (D + 2) + 1] = lsum[h] + lsum[16 + h] + lsum[32 + h] + lsum[48 + h];
        }
        part[h * (D + 2) + 2 + t] = o[h];
    }
    __threadfence();
    __syncthreads();
    if (t == 0) {
        const int old = atomicAdd(a.cnt_attn + bh, 1);
        misc[0] = old == static_cast<int>(gridDim.x) - 1;
    }
    __syncthreads();
    if (!misc[0]) return;
    __threadfence();
    if (t == 0) a.cnt_attn[bh] = 0;   // zero again for the next launch
    if (bad) return;

    // merge the partials of the splits the list reached
    const int used = (L + per - 1) / per;
    const float* pgp = a.part + static_cast<size_t>(bh) * a.nsplit_a * G * (D + 2);
    float* mw = reinterpret_cast<float*>(smem);    // [used][G][2], in the free stage
    for (int i = t; i < used * G; i += kTcThreads) {
        const float* px = pgp + static_cast<size_t>(i) * (D + 2);
        mw[2 * i] = __ldcg(px);
        mw[2 * i + 1] = __ldcg(px + 1);
    }
    __syncthreads();
    if (t < G) {
        float M = -CUDART_INF_F;
        for (int x = 0; x < used; ++x) M = fmaxf(M, mw[2 * (x * G + t)]);
        float ls = 0.f;
        for (int x = 0; x < used; ++x) {
            const float mx = mw[2 * (x * G + t)];
            const float w = mx == -CUDART_INF_F ? 0.f : fast_exp2(mx - M);
            ls = fmaf(w, mw[2 * (x * G + t) + 1], ls);
            mw[2 * (x * G + t)] = w;
        }
        mM[t] = M;
        mL[t] = ls;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < G; ++h) {
        float acc = 0.f;
#pragma unroll 8
        for (int x = 0; x < used; ++x)
            acc = fmaf(mw[2 * (x * G + h)], __ldcg(pgp + (static_cast<size_t>(x) * G + h) * (D + 2) + 2 + t), acc);
        const size_t orow = (static_cast<size_t>(b) * a.Hq + static_cast<size_t>(g) * G + h) * D;
        static_cast<bf16*>(a.O)[orow + t] = __float2bfloat16_rn(acc / mL[h]);
        if (a.LSE != nullptr && t == 0)
            a.LSE[static_cast<size_t>(b) * a.Hq + static_cast<size_t>(g) * G + h] = (mM[h] + log2f(mL[h])) / kLog2e;
    }
#undef SAS_TC_LOAD
}

// Launch with programmatic stream serialization: the kernel may start while
// the preceding kernel on the stream still runs (it waits with griddepcontrol).
// cluster > 1: the CTAs of a grid row form clusters of that many.
template <class... KArgs, class... Args>
cudaError_t launch_dependent(int cluster, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                             cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Raises the kernel's dynamic shared-memory limit to what these arguments need
// (called when a handle is created, so that a captured step sets nothing).
template <int D, int G>
cudaError_t prepare_attn_dg(const DecodeArgs& a) {
    const size_t smem = attn_layout(D, G, a.nst, a.bpc).total;
    return ensure_smem_attr(reinterpret_cast<const void*>(dec_attn_kernel<D, G>), smem);
}

template <int D, int G>
cudaError_t launch_attn_dg(const DecodeArgs& a, const KernelEnv& env) {
    const size_t smem = attn_layout(D, G, a.nst, a.bpc).total;
    cudaError_t e = prepare_attn_dg<D, G>(a);
    if (e != cudaSuccess) return e;
    dim3 grid(a.nsplit_a, a.B * a.Hkv);
    return launch_dependent(1, dec_attn_kernel<D, G>, grid, dim3(kAttnThreads), smem, env.stream, a, env.status,
                            env.limit, a.sm_scale * kLog2e);
}

template <int G, bool SAS>
cudaError_t prepare_attn_tc(const DecodeArgs& a) {
    const size_t smem = tc_layout(a.nst, a.bpc).total;
    return ensure_smem_attr(reinterpret_cast<const void*>(dec_attn_tc_kernel<G, SAS>), smem, false, true);
}

template <int G, bool SAS>
cudaError_t launch_attn_tc(const DecodeArgs& a, const KernelEnv& env) {
    cudaError_t e = prepare_attn_tc<G, SAS>(a);
    if (e != cudaSuccess) return e;
    CUtensorMap mk, mv;
    const uint64_t rows = static_cast<uint64_t>(a.num_pages) * a.Hkv;
    if (make_tmap_bf16_3d(&mk, a.K_cache, 128, kBlk, rows, 64, kBlk) != 0) return cudaErrorInvalidValue;
    if (make_tmap_bf16_3d(&mv, a.V_cache, 128, kBlk, rows, 64, kBlk) != 0) return cudaErrorInvalidValue;
    dim3 grid(a.nsplit_a, a.B * a.Hkv);
    return launch_dependent(SAS ? a.nsplit_a : 1, dec_attn_tc_kernel<G, SAS>, grid, dim3(kTcThreads),
                            tc_layout(a.nst, a.bpc).total, env.stream, mk, mv, a, env.status, env.limit,
                            a.sm_scale * kLog2e);
}

template <int D>
cudaError_t launch_attn_d(const DecodeArgs& a, const KernelEnv& env) {
    if constexpr (D == 128) {
        switch (a.G) {
            case 1: return a.dense ? launch_attn_tc<1, false>(a, env) : launch_attn_tc<1, true>(a, env);
            case 2: return a.dense ? launch_attn_tc<2, false>(a, env) : launch_attn_tc<2, true>(a, env);
            case 4: return a.dense ? launch_attn_tc<4, false>(a, env) : launch_attn_tc<4, true>(a, env);
            case 8: return a.dense ? launch_attn_tc<8, false>(a, env) : launch_attn_tc<8, true>(a, env);
        }
    } else {
        switch (a.G) {
            case 1: return launch_attn_dg<D, 1>(a, env);
            case 2: return launch_attn_dg<D, 2>(a, env);
            case 4: return launch_attn_dg<D, 4>(a, env);
            case 8: return launch_attn_dg<D, 8>(a, env);
        }
    }
    return cudaErrorInvalidValue;
}

template <int D>
cudaError_t prepare_attn_d(const DecodeArgs& a) {
    if constexpr (D == 128) {
        switch (a.G) {
            case 1: return a.dense ? prepare_attn_tc<1, false>(a) : prepare_attn_tc<1, true>(a);
            case 2: return a.dense ? prepare_attn_tc<2, false>(a) : prepare_attn_tc<2, true>(a);
            case 4: return a.dense ? prepare_attn_tc<4, false>(a) : prepare_attn_tc<4, true>(a);
            case 8: return a.dense ? prepare_attn_tc<8, false>(a) : prepare_attn_tc<8, true>(a);
        }
    } else {
        switch (a.G) {
            case 1: return prepare_attn_dg<D, 1>(a);
            case 2: return prepare_attn_dg<D, 2>(a);
            case 4: return prepare_attn_dg<D, 4>(a);
            case 8: return prepare_attn_dg<D, 8>(a);
        }
    }
    return cudaErrorInvalidValue;
}

template <int DSEL>
cudaError_t prepare_score_d(const DecodeArgs& a) {
    const size_t smem = score_smem_layout(a.nsplit_s, a.topk, DSEL).total;
    return ensure_smem_attr(reinterpret_cast<const void*>(dec_score_kernel<DSEL>), smem);
}

template <int DSEL>
cudaError_t launch_score_d(const DecodeArgs& a, const KernelEnv& env) {
    const size_t smem = score_smem_layout(a.nsplit_s, a.topk, DSEL).total;
    cudaError_t e = prepare_score_d<DSEL>(a);
    if (e != cudaSuccess) return e;
    dim3 grid(a.nsplit_s, a.B * a.Hkv);
    return launch_dependent(1, dec_score_kernel<DSEL>, grid, dim3(kScoreThreads), smem, env.stream, a, env.status,
                            env.limit, static_cast<float>(1.0 / sqrt(static_cast<double>(DSEL))));
}

}  // namespace

namespace {

// Clusters of S attention CTAs (a ring of nst stages, bpc pages each) that the device
// holds at once; 0 if it cannot say.
int attn_clusters_at_once(int S, int nst, int bpc, int G) {
    const void* f = G == 1   ? reinterpret_cast<const void*>(dec_attn_tc_kernel<1, true>)
                    : G == 2 ? reinterpret_cast<const void*>(dec_attn_tc_kernel<2, true>)
                    : G == 4 ? reinterpret_cast<const void*>(dec_attn_tc_kernel<4, true>)
                             : reinterpret_cast<const void*>(dec_attn_tc_kernel<8, true>);
    const size_t smem = tc_layout(nst, bpc).total;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {static_cast<unsigned>(S), 1, 1};
    cfg.gridDim = dim3(static_cast<unsigned>(S));
    cfg.blockDim = dim3(kTcThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (ensure_smem_attr(f, smem, false, true) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, f, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace

void decode_attn_split(int max_len, int d, bool dense, int groups, int G, int sms, int* nsplit, int* bpc, int* nst,
                       int* cluster) {
    int per;
    *cluster = 0;
    if (d == 128 && !dense) {
        // tensor-core kernel, a SAS list (at most 65 pages, taken by pairs): a cluster of
        // S <= 16 CTAs per group, as many as run at once.
        // Three CTAs of one 64 KB stage share an SM, but whole clusters have to find
        // room in a GPC, so the grid stays at 8/3 of the SMs (64 groups of 33 pages:
        // 28.8, 25.7, 23.6, 20.8 and 32.0 us with S = 3, 4, 5, 6 and 7; the device's own
        // count of clusters that fit stops earlier, 45.4 us a step for 39.8, now 36).  One
        // CTA per SM or fewer: up to three stages, so that a CTA's own loads overlap, and
        // there the device's count decides (8 groups of 49 pages: thirteen CTAs each did
        // not all find room and took 19.5 us, two waves).  (Before clusters: one page pair
        // per CTA and a merge by the last one to arrive; 64 groups took 2.4 waves and 36.5
        // us, now 19.0.  A partial per CTA, kept by online softmax and merged over
        // distributed shared memory, made the result depend on S: a step of 8 sequences
        // of 64K tokens 29.3 us against 29.7, 32 of 8K 73 against 77, 4 of 32K 32 against
        // 25, 1 of 8K 18.5 against 16.4.)
        const int fit = 8 * sms / (3 * (groups > 0 ? groups : 1));
        int S = fit < 1 ? 1 : (fit > kMaxDecCluster ? kMaxDecCluster : fit);
        const int pairs = (max_len + 1) / 2;
        for (;; --S) {
            const int steps = (pairs + S - 1) / S;
            S = (pairs + steps - 1) / steps;
            per = 2 * steps;
            const bool spread = static_cast<long long>(groups) * S <= sms;
            *nst = spread ? (steps < 3 ? steps : 3) : 1;
            if (S == 1 || !spread || attn_clusters_at_once(S, *nst, per, G) >= groups) break;
        }
        *cluster = 1;
    } else if (d == 128) {
        // dense lists: cut into at most 64 (128 past 2048 pages) pieces of whole
        // steps.  One stage, so that three CTAs share an SM and overlap one
        // another's loads (two stages and one CTA per SM measured slower).
        const int pieces = max_len <= 2048 ? 64 : 128;   // long lists: more CTAs pay for the larger merge
        per = max_len <= 96 ? 2 : 2 * ((max_len + 2 * pieces - 1) / (2 * pieces));
        *nst = 1;
    } else {
        // CUDA-core kernel: one page per CTA for a SAS list; long dense lists in
        // at most 64 pieces streamed through a 3-stage ring
        per = max_len <= 96 ? 1 : (max_len + 63) / 64;
        *nst = per < kStages ? per : kStages;
    }
    *bpc = per;
    *nsplit = (max_len + per - 1) / per;
}

size_t decode_part_floats(const DecodeArgs& a) {
    const size_t splits = static_cast<size_t>(a.nsplit_a) * a.G;
    return a.cluster ? splits * (a.bpc / 2) * kPairFloats : splits * (a.d + 2);
}

size_t decode_score_smem(int nsplit, int topk, int d_sel) { return score_smem_layout(nsplit, topk, d_sel).total; }

size_t decode_attn_smem(int d, int G, int nst, int bpc) {
    return d == 128 ? tc_layout(nst, bpc).total : attn_layout(d, G, nst, bpc).total;
}

cudaError_t decode_prepare(const DecodeArgs& a) {
    cudaError_t e = cudaSuccess;
    if (!a.dense) e = a.d_sel == 128 ? prepare_score_d<128>(a) : prepare_score_d<64>(a);
    if (e == cudaSuccess) e = a.d == 128 ? prepare_attn_d<128>(a) : prepare_attn_d<64>(a);
    return e;
}

cudaError_t launch_decode_prep(const DecodeArgs& a, const KernelEnv& env) {
    dim3 grid(a.B * a.Hkv, a.dense ? 1 : 1 + (a.d_sel + 7) / 8);
    dec_prep_kernel<<<grid, kPrepThreads, 0, env.stream>>>(a, env.status);
    return cudaGetLastError();
}

cudaError_t launch_decode_summarize(const DecodeArgs& a, const KernelEnv& env) {
    dim3 grid(a.max_blocks, a.B * a.Hkv);
    dec_summarize_kernel<<<grid, kPrepThreads, 0, env.stream>>>(a, env.status);
    return cudaGetLastError();
}

cudaError_t launch_decode_score(const DecodeArgs& a, const KernelEnv& env) {
    if (a.d_sel == 128) return launch_score_d<128>(a, env);
    if (a.d_sel == 64) return launch_score_d<64>(a, env);
    return cudaErrorInvalidValue;
}

cudaError_t launch_decode_attn(const DecodeArgs& a, const KernelEnv& env) {
    if (a.d == 128) return launch_attn_d<128>(a, env);
    if (a.d == 64) return launch_attn_d<64>(a, env);
    return cudaErrorInvalidValue;
}

}  // namespace sas
