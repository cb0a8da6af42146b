// The decode step's list kernels on candidates and lists that a test makes up: what a
// score kernel leaves behind when a summary load gives up.  Built by
// tests/test_gpu_decode_lists.py against libsas.so (tensor maps).
#include "../../paper_2609_13141_gb300/csrc/k_decode.cu"

// of this library's own kernels: libsas.so has another instance of the CUDA runtime
namespace sas {
cudaError_t ensure_smem_attr(const void* func, size_t bytes, bool, bool big_clusters) {
    cudaError_t e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
    if (e == cudaSuccess && big_clusters)
        e = cudaFuncSetAttribute(func, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}
int device_sm_count() {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, 0);
    return n;
}
}  // namespace sas

namespace {

__global__ void __launch_bounds__(sas::kScoreThreads) select_kernel(sas::DecodeArgs a, const uint32_t* key,
                                                                    const int32_t* blk, int M, int radix) {
    __shared__ __align__(16) uint32_t keys[2048];
    __shared__ int32_t idx[2048];
    __shared__ int hist[4096], scan[32], bc[4];
    for (int i = threadIdx.x; i < 2048; i += sas::kScoreThreads) {
        keys[i] = i < M ? key[i] : 0u;
        idx[i] = i < M ? blk[i] : -1;
    }
    __syncthreads();
    if (radix) sas::select_candidates(a, 0, M, keys, idx, hist, scan, bc);
    else sas::select_by_rank(a, 0, M, keys, idx, scan);
}

}  // namespace

// Top-K of M <= 2048 candidates (radix = 0: M <= 256) of one group into list[64], *list_n and sel_idx[K].
extern "C" int decode_lists_select(const uint32_t* key, const int32_t* blk, int M, int K, int radix, int32_t* list,
                                   int32_t* list_n, int32_t* sel_idx) {
    if (M < K || K < 1 || K > 64 || M > (radix ? 2048 : sas::kRankMax)) return -1;
    sas::DecodeArgs a{};
    a.topk = K; a.list = list; a.list_n = list_n; a.sel_idx = sel_idx;
    select_kernel<<<1, sas::kScoreThreads>>>(a, key, blk, M, radix);
    return static_cast<int>(cudaDeviceSynchronize());
}

// Attention of one sequence of n tokens and one KV head over the list given.
extern "C" int decode_lists_attend(const void* q, void* K_cache, void* V_cache, const int32_t* table, const int32_t* n,
                                   int max_blocks, int pages, int G, int d, int topk, int32_t* list, int32_t* list_n,
                                   void* O, float* LSE, float* part, int part_floats, int* counters, int* status) {
    sas::DecodeArgs a{};
    a.B = 1; a.Hq = G; a.Hkv = 1; a.G = G; a.d = d; a.d_sel = d; a.topk = topk;
    a.max_blocks = max_blocks; a.num_pages = pages; a.dense = 0;
    a.sm_scale = 1.f / sqrtf(static_cast<float>(d));
    sas::decode_attn_split(topk + 1, d, false, 1, G, sas::device_sm_count(), &a.nsplit_a, &a.bpc, &a.nst, &a.cluster);
    if (sas::decode_part_floats(a) > static_cast<size_t>(part_floats)) return -1;
    a.q = q; a.K_cache = K_cache; a.V_cache = V_cache; a.block_table = table; a.seq_lens = n;
    a.list = list; a.list_n = list_n; a.O = O; a.LSE = LSE; a.part = part; a.cnt_sel = counters; a.cnt_attn = counters + 1;
    const sas::KernelEnv env{nullptr, status, 4000000000LL};
    cudaError_t e = sas::decode_prepare(a);
    if (e == cudaSuccess) e = sas::launch_decode_attn(a, env);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    return static_cast<int>(e);
}
