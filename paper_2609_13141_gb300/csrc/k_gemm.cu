// Persistent warp-specialised bf16 GEMM on the 5th-generation tensor cores.
//
//   C = epi(A @ B^T + bias)        (fp32 accumulate, bf16 out)
//
// Used for the dense MLP sublayer (up-projection with an exact-GELU epilogue,
// then the down-projection).  Design:
//   * one CTA per SM, static round-robin over 128 x BN output tiles, grouped
//     along M so that concurrently running CTAs share operand tiles in L2;
//   * warp 0 streams 128x64 A and BNx64 B tiles with TMA (128-byte swizzle)
//     into a ring of shared-memory stages guarded by mbarriers;
//   * warp 1 (one lane) issues tcgen05.mma (M=128, N=BN, K=16) into one of
//     two TMEM accumulators and releases stages with tcgen05.commit;
//   * warps 2-5 drain the other accumulator (tcgen05.ld), apply bias/GELU in
//     fp32, write bf16 into a per-warp 128-byte-swizzled staging tile and send
//     each 32 x 64 block out with a TMA tensor store (per-thread row stores
//     scattered over 32 rows cost 6% of the GEMM), overlapping the next tile's
//     main loop.
// Problems whose tiles do not fill the chip take gemm_split_kernel: a cluster
// of CTAs splits one tile's K and adds the partial sums over distributed
// shared memory.  pick_shape() chooses between the two and their tile widths.
#include <mutex>

#include "internal.h"
#include "ptx.cuh"

namespace sas {
namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;
constexpr int kThreads = 192;

template <int BN>
struct GemmCfg {
    static constexpr int A_BYTES = kBM * kBK * 2;
    static constexpr int B_BYTES = BN * kBK * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = BN == 256 ? 4 : (BN == 128 ? 6 : 8);
    static constexpr int TMEM_COLS = 2 * BN;
    // per epilogue warp two 32-row x 64-column bf16 staging tiles (4 KB each)
    static constexpr int OFF_STAGING = STAGES * STAGE_BYTES;
    static constexpr int STAGING_BYTES = 4 * 2 * 4096;
    static constexpr int SMEM = OFF_STAGING + STAGING_BYTES + 1024;
    static constexpr uint32_t IDESC = idesc_bf16(kBM, BN, 0, 0);
};

// Split-K kernel: S CTAs of a cluster share one 128 x BN tile.
template <int BN>
struct SplitCfg {
    static constexpr int A_BYTES = kBM * kBK * 2;
    static constexpr int B_BYTES = BN * kBK * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = 4;                 // BN = 64: 96 KB, two CTAs per SM
    // after the main loop the ring holds the fp32 partial tile, rows padded so
    // that a warp's row-by-row writes spread over the banks
    static constexpr int PITCH = BN + 4;
    static_assert(kBM * PITCH * 4 <= STAGES * STAGE_BYTES, "partial tile");
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024;
    static constexpr uint32_t IDESC = idesc_bf16(kBM, BN, 0, 0);
};
constexpr int kMaxSplit = 8;                         // portable cluster size

struct GemmParams {
    bf16* C;
    const bf16* bias;
    int M, N, K;
    int gelu;
    int early_b;             // launched ahead of the kernel that writes A: B may be loaded before it ends
    int* status;
    long long limit;
};

// Programmatic dependent launch: lets the next kernel of the stream start its
// set-up / waits until the kernels this one depends on have completed.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr int kGroupM = 16;
// Every wait in this kernel sleeps while it waits (measured: 4.5% faster for the
// up-projection than polling, which takes issue slots from the epilogue warps).
constexpr uint32_t kSuspendNs = 1000;

__device__ __forceinline__ void tile_coords(int t, int m_tiles, int n_tiles, int& m, int& n) {
    const int group_span = kGroupM * n_tiles;
    const int g = t / group_span;
    const int first_m = g * kGroupM;
    const int gsize = min(m_tiles - first_m, kGroupM);
    const int rr = t - g * group_span;
    m = first_m + rr % gsize;
    n = rr / gsize;
}

__device__ __forceinline__ float gelu_erf(float x) {
    return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
            const __grid_constant__ CUtensorMap mapC, GemmParams p) {
    using Cfg = GemmCfg<BN>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ uint64_t full_bar[Cfg::STAGES], empty_bar[Cfg::STAGES];
    __shared__ uint64_t tfull_bar[2], tempty_bar[2], drain_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_flag;

    const uint32_t warp = warp_id(), lane = lane_id();
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);

    const int m_tiles = (p.M + kBM - 1) / kBM;
    const int n_tiles = p.N / BN;
    const int total = m_tiles * n_tiles;
    const int kblocks = p.K / kBK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull_bar[a], 1);
            mbar_init(&tempty_bar[a], 128);
        }
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(&tmem_base_sh, Cfg::TMEM_COLS);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_sh;
    const WaitCtl wc{&abort_flag, p.status, p.limit};
    if (!p.early_b) pdl_launch();

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer
        tma_prefetch_desc(&mapA);
        tma_prefetch_desc(&mapB);
        int s = 0;
        uint32_t ph = 0;
        long long issued = 0;
        bool ok = true;
        if (p.early_b) pdl_wait();
        for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
            int m, n;
            tile_coords(t, m_tiles, n_tiles, m, n);
            for (int kb = 0; kb < kblocks; ++kb) {
                if (!mbar_wait(&empty_bar[s], ph ^ 1u, wc, kSuspendNs)) { ok = false; break; }
                uint8_t* sa = smem + s * Cfg::STAGE_BYTES;
                mbar_arrive_expect_tx(&full_bar[s], Cfg::STAGE_BYTES);
                tma_load_3d(sa, &mapA, &full_bar[s], kb * kBK, m * kBM, 0);
                tma_load_3d(sa + Cfg::A_BYTES, &mapB, &full_bar[s], kb * kBK, n * BN, 0);
                ++issued;
                if (++s == Cfg::STAGES) { s = 0; ph ^= 1u; }
            }
        }
        if (!ok) {
            // Let every load already issued land before the CTA can exit.
            for (long long q = issued - 1; q >= 0 && q >= issued - Cfg::STAGES; --q)
                mbar_wait_drain(&full_bar[q % Cfg::STAGES], static_cast<uint32_t>((q / Cfg::STAGES) & 1),
                                p.limit, p.status);
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer
        int s = 0;
        uint32_t ph = 0;
        int it = 0;
        bool ok = true;
        // no bounded wait runs while the kernel that writes A does: its time is not this one's
        if (p.early_b) pdl_wait();
        for (int t = blockIdx.x; t < total && ok; t += gridDim.x, ++it) {
            const int acc = it & 1;
            const uint32_t aph = (it >> 1) & 1;
            if (!mbar_wait(&tempty_bar[acc], aph ^ 1u, wc, kSuspendNs)) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * BN;
            for (int kb = 0; kb < kblocks; ++kb) {
                if (!mbar_wait(&full_bar[s], ph, wc, kSuspendNs)) { ok = false; break; }
                tc_fence_after();
                const uint32_t a_addr = smem_u32(smem + s * Cfg::STAGE_BYTES);
                const uint32_t b_addr = a_addr + Cfg::A_BYTES;
#pragma unroll
                for (int k = 0; k < kBK / 16; ++k) {
                    const uint64_t ad = smem_desc_sw128(a_addr + k * 32, 16, 1024);
                    const uint64_t bd = smem_desc_sw128(b_addr + k * 32, 16, 1024);
                    umma_bf16(d_tmem, ad, bd, Cfg::IDESC, (kb | k) != 0);
                }
                umma_commit(&empty_bar[s]);
                if (++s == Cfg::STAGES) { s = 0; ph ^= 1u; }
            }
            if (!ok) break;
            umma_commit(&tfull_bar[acc]);
        }
        umma_commit(&drain_bar);
        mbar_wait_drain(&drain_bar, 0, p.limit, p.status);
    } else if (warp >= 2) {
        // ---------------- epilogue: TMEM -> registers -> bias/GELU -> bf16 -> staging -> TMA store
        const int q = warp & 3;
        if (p.early_b) pdl_wait();   // C may be read by the kernels before
        const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
        uint8_t* staging = smem + Cfg::OFF_STAGING + q * 2 * 4096;
        if (lane == 0) tma_prefetch_desc(&mapC);
        int it = 0;
        int nst = 0;   // stores issued by this warp (staging buffer = nst & 1)
        for (int t = blockIdx.x; t < total; t += gridDim.x, ++it) {
            const int acc = it & 1;
            const uint32_t aph = (it >> 1) & 1;
            if (!mbar_wait_warp(&tfull_bar[acc], aph, wc, kSuspendNs)) break;
            tc_fence_after();
            int m, n;
            tile_coords(t, m_tiles, n_tiles, m, n);
#pragma unroll 1
            for (int cg = 0; cg < BN / 64; ++cg, ++nst) {
                uint8_t* buf = staging + (nst & 1) * 4096;
                // the store issued from this buffer two groups ago has finished reading it
                if (lane == 0) bulk_wait_read<1>();
                __syncwarp();
#pragma unroll 1
                for (int hh = 0; hh < 2; ++hh) {
                    const int c = cg * 2 + hh;
                    uint32_t r[32];
                    tmem_ld32(lane_addr + acc * BN + c * 32, r);
                    tmem_wait_ld();
                    float v[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
                    if (p.bias != nullptr) {
                        const bf16* bp = p.bias + n * BN + c * 32;
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] += __bfloat162float(bp[j]);
                    }
                    if (p.gelu) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = gelu_erf(v[j]);
                    }
                    // row `lane` of the staging tile: 16-byte chunk k of the row at k ^ (lane & 7)
                    uint8_t* row = buf + lane * 128;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        uint4 w;
                        w.x = pack_bf16x2(v[8 * j + 0], v[8 * j + 1]);
                        w.y = pack_bf16x2(v[8 * j + 2], v[8 * j + 3]);
                        w.z = pack_bf16x2(v[8 * j + 4], v[8 * j + 5]);
                        w.w = pack_bf16x2(v[8 * j + 6], v[8 * j + 7]);
                        const int k = hh * 4 + j;
                        *reinterpret_cast<uint4*>(row + ((k ^ (lane & 7)) << 4)) = w;
                    }
                }
                fence_proxy_async_smem();
                __syncwarp();
                // rows past M are clipped by the tensor store
                if (lane == 0) {
                    tma_store_3d(&mapC, buf, n * BN + cg * 64, m * kBM + q * 32, 0);
                    bulk_commit();
                }
            }
            tc_fence_before();
            mbar_arrive(&tempty_bar[acc]);
        }
        if (lane == 0) bulk_wait_all();
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
    }
}

// One 128 x BN tile per cluster of S CTAs; CTA r accumulates its share of the K
// blocks in TMEM, leaves the fp32 partial tile in its shared memory, and after
// a cluster barrier adds the S partials (in rank order) of every S-th group of
// 512 elements, applies the epilogue and stores.  Bound by the latency of its
// few K blocks: the second product's CTAs start while the first one drains and
// fetch their first weights before its output is complete.
template <int BN>
__global__ void __launch_bounds__(kThreads)
gemm_split_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, GemmParams p) {
    using Cfg = SplitCfg<BN>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ uint64_t full_bar[Cfg::STAGES], empty_bar[Cfg::STAGES], acc_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_flag;

    const uint32_t warp = warp_id(), lane = lane_id();
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    const int S = cluster_size(), rank = cluster_rank();
    const int tile = static_cast<int>(blockIdx.x) / S;
    const int n_tiles = p.N / BN;
    const int m = tile / n_tiles, n = tile - m * n_tiles;
    const int kblocks = p.K / kBK;
    const int k0 = static_cast<int>(static_cast<long long>(kblocks) * rank / S);
    const int nk = static_cast<int>(static_cast<long long>(kblocks) * (rank + 1) / S) - k0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&acc_bar, 1);
        abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(&tmem_base_sh, BN);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;
    const WaitCtl wc{&abort_flag, p.status, p.limit};
    if (!p.early_b) pdl_launch();

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer; B (the weights) of the first stages goes out
        // ahead of the wait for the kernel that writes A
        tma_prefetch_desc(&mapA);
        tma_prefetch_desc(&mapB);
        const int pre = min(nk, Cfg::STAGES);
        for (int kb = 0; kb < pre; ++kb) {
            uint8_t* sa = smem + kb * Cfg::STAGE_BYTES;
            mbar_arrive_expect_tx(&full_bar[kb], Cfg::STAGE_BYTES);
            tma_load_3d(sa + Cfg::A_BYTES, &mapB, &full_bar[kb], (k0 + kb) * kBK, n * BN, 0);
        }
        if (p.early_b) pdl_wait();
        for (int kb = 0; kb < pre; ++kb)
            tma_load_3d(smem + kb * Cfg::STAGE_BYTES, &mapA, &full_bar[kb], (k0 + kb) * kBK, m * kBM, 0);
        int issued = pre;
        bool ok = true;
        for (int kb = pre; kb < nk; ++kb) {
            const int s = kb % Cfg::STAGES;
            if (!mbar_wait(&empty_bar[s], ((kb / Cfg::STAGES) & 1) ^ 1u, wc, kSuspendNs)) { ok = false; break; }
            uint8_t* sa = smem + s * Cfg::STAGE_BYTES;
            mbar_arrive_expect_tx(&full_bar[s], Cfg::STAGE_BYTES);
            tma_load_3d(sa, &mapA, &full_bar[s], (k0 + kb) * kBK, m * kBM, 0);
            tma_load_3d(sa + Cfg::A_BYTES, &mapB, &full_bar[s], (k0 + kb) * kBK, n * BN, 0);
            ++issued;
        }
        (void)ok;
        // every load lands before the ring is reused for the partial tile
        for (int q = issued - 1; q >= 0 && q >= issued - Cfg::STAGES; --q)
            mbar_wait_drain(&full_bar[q % Cfg::STAGES], (q / Cfg::STAGES) & 1, p.limit, p.status);
    } else if (warp == 1) {
        // ---------------- MMA issuer (whole warp; the elected lane issues).  The wait for
        // the kernel that writes A comes first: its time is not on the bounded waits' budget
        if (p.early_b) pdl_wait();
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % Cfg::STAGES;
            if (!mbar_wait_warp(&full_bar[s], (kb / Cfg::STAGES) & 1, wc, kSuspendNs)) break;
            tc_fence_after();
            const uint32_t a_addr = smem_u32(smem + s * Cfg::STAGE_BYTES);
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < kBK / 16; ++k)
                    umma_bf16(tmem, smem_desc_sw128(a_addr + k * 32, 16, 1024),
                              smem_desc_sw128(a_addr + Cfg::A_BYTES + k * 32, 16, 1024), Cfg::IDESC, (kb | k) != 0);
                umma_commit(&empty_bar[s]);
            }
            __syncwarp();
        }
        if (elect_one()) {
            umma_commit(&acc_bar);
            mbar_wait_drain(&acc_bar, 0, p.limit, p.status);
        }
        __syncwarp();
    } else if (p.early_b) {
        pdl_wait();   // C may be read by the kernels before
    }
    // the loads have landed and the MMAs are complete: the ring is free
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const int rows = min(kBM, p.M - m * kBM);
    float* part = reinterpret_cast<float*>(smem);
    if (warp >= 2) {
        const int q = warp & 3, r = q * 32 + lane;
        const uint32_t lane_addr = tmem + (static_cast<uint32_t>(q * 32) << 16);
        if (q * 32 < rows) {
#pragma unroll 1
            for (int c = 0; c < BN; c += 16) {
                uint32_t v[16];
                tmem_ld16(lane_addr + c, v);
                tmem_wait_ld();
                float4* dst = reinterpret_cast<float4*>(part + r * Cfg::PITCH + c);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    dst[j] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                         __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
            }
        }
        tc_fence_before();
    }
    cluster_sync();
    if (warp >= 2) {
        constexpr int kQuads = BN / 4;
        const int t = (warp - 2) * 32 + lane;
        const uint32_t own = smem_u32(part);
        for (int e = rank * 128 + t; e < rows * kQuads; e += S * 128) {
            const int r = e / kQuads, c = (e % kQuads) * 4;
            const uint32_t at = own + (r * Cfg::PITCH + c) * 4;
            float4 v = dsmem_ld_f4(cluster_map(at, 0));
            for (int k = 1; k < S; ++k) {
                const float4 w = dsmem_ld_f4(cluster_map(at, k));
                v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
            }
            if (p.bias != nullptr) {
                const uint2 b = __ldg(reinterpret_cast<const uint2*>(p.bias + n * BN + c));
                v.x += __uint_as_float(b.x << 16); v.y += __uint_as_float(b.x & 0xffff0000u);
                v.z += __uint_as_float(b.y << 16); v.w += __uint_as_float(b.y & 0xffff0000u);
            }
            if (p.gelu) {
                v.x = gelu_erf(v.x); v.y = gelu_erf(v.y); v.z = gelu_erf(v.z); v.w = gelu_erf(v.w);
            }
            *reinterpret_cast<uint2*>(p.C + static_cast<long long>(m * kBM + r) * p.N + n * BN + c) =
                make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
        }
    }
    cluster_sync();   // the peers have read this CTA's partial tile
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, BN);
    }
}

GemmParams gemm_params(const GemmProblem& p, const KernelEnv& env) {
    GemmParams gp;
    gp.C = static_cast<bf16*>(p.C);
    gp.bias = static_cast<const bf16*>(p.bias);
    gp.M = p.M; gp.N = p.N; gp.K = p.K;
    gp.gelu = p.gelu;
    gp.early_b = p.after_gemm;
    gp.status = env.status; gp.limit = env.limit;
    return gp;
}

// Launches with the optional attributes: a cluster of `cluster` CTAs, and ahead
// of the end of the stream's previous kernel (programmatic dependent launch).
template <class... Params, class... Args>
cudaError_t launch_ex(void (*kernel)(Params...), int grid, int smem, int cluster, bool early, cudaStream_t stream,
                      Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (early) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Clusters of s split CTAs of 128 x BN tiles for which the device has room at one CTA
// an SM (a cluster has to find it in one GPC); 0 if it cannot say.
template <int BN>
int split_clusters(int s) {
    using Cfg = SplitCfg<BN>;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(s);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {static_cast<unsigned>(s), 1, 1};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (ensure_smem_attr(reinterpret_cast<const void*>(gemm_split_kernel<BN>), Cfg::SMEM) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, gemm_split_kernel<BN>, &cfg) == cudaSuccess)
        return n;
    cudaGetLastError();
    return 0;
}

// SMs of the current device and those counts, asked for by its first problem.
struct Room {
    int sms, bn128[kMaxSplit + 1], bn64[kMaxSplit + 1];
};
const Room& device_room() {
    constexpr int kMaxDevices = 128;
    static Room rooms[kMaxDevices + 1];   // the last: no device known, one SM and no cluster
    static std::once_flag once[kMaxDevices + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = kMaxDevices;
    Room& r = rooms[dev];
    std::call_once(once[dev], [&r, dev] {
        r.sms = dev < kMaxDevices ? device_sm_count() : 1;
        for (int s = 2; s <= kMaxSplit && dev < kMaxDevices; ++s) {
            r.bn128[s] = split_clusters<128>(s);
            r.bn64[s] = 2 * split_clusters<64>(s);   // two share an SM, which the count leaves out
        }
    });
    return r;
}

template <int BN>
cudaError_t launch_split(const GemmProblem& p, int split, const KernelEnv& env, const char** err) {
    using Cfg = SplitCfg<BN>;
    cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(gemm_split_kernel<BN>), Cfg::SMEM);
    if (e != cudaSuccess) { *err = "cudaFuncSetAttribute(gemm split)"; return e; }
    CUtensorMap ma, mb;
    if (make_tmap_bf16_3d(&ma, p.A, p.K, p.M, 1, kBK, kBM) != 0) { *err = "tensor map A"; return cudaErrorInvalidValue; }
    if (make_tmap_bf16_3d(&mb, p.B, p.K, p.N, 1, kBK, BN) != 0) { *err = "tensor map B"; return cudaErrorInvalidValue; }
    const int tiles = (p.M + kBM - 1) / kBM * (p.N / BN);
    e = launch_ex(gemm_split_kernel<BN>, tiles * split, Cfg::SMEM, split, p.after_gemm != 0, env.stream, ma, mb,
                  gemm_params(p, env));
    if (e != cudaSuccess) *err = "gemm split launch";
    return e;
}

template <int BN>
cudaError_t launch_bn(const GemmProblem& p, const KernelEnv& env, const char** err) {
    using Cfg = GemmCfg<BN>;
    {
        cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(gemm_kernel<BN>), Cfg::SMEM);
        if (e != cudaSuccess) { *err = "cudaFuncSetAttribute(gemm)"; return e; }
    }
    CUtensorMap ma, mb, mc;
    if (make_tmap_bf16_3d(&ma, p.A, p.K, p.M, 1, kBK, kBM) != 0) { *err = "tensor map A"; return cudaErrorInvalidValue; }
    if (make_tmap_bf16_3d(&mb, p.B, p.K, p.N, 1, kBK, BN) != 0) { *err = "tensor map B"; return cudaErrorInvalidValue; }
    if (make_tmap_bf16_3d(&mc, p.C, p.N, p.M, 1, 64, 32) != 0) { *err = "tensor map C"; return cudaErrorInvalidValue; }
    const GemmParams gp = gemm_params(p, env);
    const long long tiles = static_cast<long long>((p.M + kBM - 1) / kBM) * (p.N / BN);
    int grid = device_room().sms;
    if (tiles < grid) grid = static_cast<int>(tiles);
    cudaError_t e = launch_ex(gemm_kernel<BN>, grid, Cfg::SMEM, 1, p.after_gemm != 0, env.stream, ma, mb, mc, gp);
    if (e != cudaSuccess) *err = "gemm launch";
    return e;
}

// Tile width and K split for a problem (split = 0: the persistent kernel).
// Estimated SM cycles of a K block (64) of a 128 x BN tile: 600, 400 and 300 at
// BN = 256, 128, 64 (tensor time 512, 256 and 192; the operand bytes an SM takes
// from L2, 48, 32 and 24 KB, hold the narrow tiles); tiles go in whole waves.
// A split tile's CTAs run together (BN = 64: two per SM share it) and pay the
// exchange of partial sums, about 3000 cycles.  A split is taken only where the device
// holds all its clusters at once: with 48 clusters of three where 46 find room, 1024
// rows of 768 x 3072 took 38 us, with 48 pairs 29 (64 rows of 2560 x 9728: 42 and 31,
// 500 rows of 1536 x 6144: 50 and 38).  Measured (us for both MLP
// products, 256-wide tiles on one CTA per tile -> this choice): 2560 x 9728 at
// 64 rows 84 -> 31, 256 rows 87 -> 46, 777 rows 103 -> 85 (its down-projection
// has 70 tiles of 256 columns for 152 SMs, 140 of 128); 1024 x 4096 at 64 rows
// 41 -> 19.  With the narrow tiles' tensor time alone in the estimate, 4096 rows
// of 3072 x 12288 took 128-wide tiles and went from 421 to 499.
struct GemmShape {
    int bn, split;
};
GemmShape pick_shape(int M, int N, int K, const Room& room) {
    const int sms = room.sms;
    const long long mt = (M + kBM - 1) / kBM, kb = K / kBK;
    GemmShape best{64, 0};
    long long cost = -1;
    for (int bn = 256; bn >= 64; bn /= 2) {
        if (N % bn != 0) continue;
        const long long tiles = mt * (N / bn), per = bn == 256 ? 600 : (bn == 128 ? 400 : 300);
        const long long c = (tiles + sms - 1) / sms * kb * per;
        if (cost < 0 || c < cost) {
            cost = c;
            best = {bn, 0};
        }
        if (bn == 256) continue;
        const long long slots = bn == 64 ? 2 * sms : sms;
        for (int s = 2; s <= kMaxSplit; ++s) {
            if (tiles * s > slots || kb < 4 * s) continue;
            const long long both = tiles * s > sms ? 2 : 1;   // CTAs on the fullest SM
            const long long cs = (kb + s - 1) / s * per * both + 3000;
            if (cs < cost && tiles <= (bn == 128 ? room.bn128[s] : room.bn64[s])) {
                cost = cs;
                best = {bn, s};
            }
        }
    }
    return best;
}

}  // namespace

cudaError_t launch_gemm(const GemmProblem& p, const KernelEnv& env, const char** err) {
    const GemmShape g = pick_shape(p.M, p.N, p.K, device_room());
    if (g.split > 0) return g.bn == 128 ? launch_split<128>(p, g.split, env, err) : launch_split<64>(p, g.split, env, err);
    switch (g.bn) {
        case 256: return launch_bn<256>(p, env, err);
        case 128: return launch_bn<128>(p, env, err);
        case 64: return launch_bn<64>(p, env, err);
        default: *err = "gemm: unsupported tile width"; return cudaErrorInvalidValue;
    }
}

}  // namespace sas
