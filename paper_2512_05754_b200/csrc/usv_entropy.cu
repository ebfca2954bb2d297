// Entropy-aware scheduler inputs (Sec. 3.4 of the USV paper).
//
//   marginal_tc_kernel    Eq. 16: abar[b,j] = 1/(H N) sum_h sum_i A(h,i,j) for the block-masked
//                         attention of Eq. 5 (usv_entropy_tc.cu).
//   entropy_kernel        Eq. 17: h[b] = -(1/log N) sum_j abar log abar.
//   usv_allocate_sparsity Eq. 18-19 on the host: w = (1-h)^gamma, rho_l = clip(rho_bar w_l / mean w).
//
// This sits beside the hot path: a per-layer statistic the scheduler reads between steps.
#include <math.h>

#include "usv_entropy.cuh"

namespace usv {

// one CTA per batch element
__global__ void __launch_bounds__(1024) entropy_kernel(const float* __restrict__ marg, int N, float* __restrict__ h) {
    dep_sync();
    __shared__ float red[32];
    const float* m = marg + (int64_t)blockIdx.x * N;
    float s = 0.f;
    for (int j0 = threadIdx.x; j0 < N; j0 += 8 * 1024) {   // eight loads on their way at a time
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = j0 + i * 1024 < N ? m[j0 + i * 1024] : 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (v[i] > 0.f) s -= v[i] * logf(v[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = red[threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) h[blockIdx.x] = N > 1 ? s / logf((float)N) : 0.f;
    }
}

}  // namespace usv

static int attn_entropy_impl(int B, int H, int N, int d, const void* q, const usv_strides* sq,
                             const void* k, const usv_strides* sk, const int32_t* sel,
                             const int32_t* k_per_head, int kmax, const float* lse, float scale,
                             float* key_marginal, float* entropy, void* ws, size_t ws_bytes, void* stream) {
    using namespace usv;
    if (B <= 0 || H <= 0 || N <= 0) return fail(USV_ERR_INVALID_ARG, "attn_entropy: B,H,N must be positive");
    if (d != 64 && d != 128) return fail(USV_ERR_UNSUPPORTED, "attn_entropy: d=%d (need 64 or 128)", d);
    if (H > USV_MAX_HEADS) return fail(USV_ERR_UNSUPPORTED, "attn_entropy: H > %d", USV_MAX_HEADS);
    int rc;
    if ((rc = check_view("q", q, sq, d)) != USV_OK) return rc;
    if ((rc = check_view("k", k, sk, d)) != USV_OK) return rc;
    if (sel == nullptr || k_per_head == nullptr || lse == nullptr || key_marginal == nullptr || entropy == nullptr)
        return fail(USV_ERR_INVALID_ARG, "attn_entropy: null pointer");
    if (!(scale >= 0.f)) return fail(USV_ERR_INVALID_ARG, "attn_entropy: scale must be >= 0");
    const int NB = ceil_div(N, USV_BLOCK);
    MargArgs a;
    int kmx = 0;
    for (int h = 0; h < H; ++h) {
        if (k_per_head[h] < 1 || k_per_head[h] > NB)
            return fail(USV_ERR_INVALID_ARG, "attn_entropy: k_per_head[%d]=%d outside [1,%d]", h, k_per_head[h], NB);
        a.k_per_head[h] = k_per_head[h];
        kmx = k_per_head[h] > kmx ? k_per_head[h] : kmx;
    }
    if (kmax < kmx) return fail(USV_ERR_INVALID_ARG, "attn_entropy: kmax=%d < max k=%d", kmax, kmx);
    const int64_t grid = (int64_t)B * H * NB;
    if (grid > 2147483647LL) return fail(USV_ERR_UNSUPPORTED, "attn_entropy: too many query blocks");
    a.q = static_cast<const __nv_bfloat16*>(q);
    a.k = static_cast<const __nv_bfloat16*>(k);
    a.sq = *sq; a.sk = *sk;
    a.sel = sel; a.lse = lse; a.marg = key_marginal;
    a.status = static_cast<unsigned int*>(ws);
    a.B = B; a.H = H; a.N = N; a.NB = NB; a.kmax = kmax;
    const float sc = scale == 0.f ? 1.0f / sqrtf((float)d) : scale;
    a.scale_log2 = sc * 1.4426950408889634f;
    a.inv_hn = 1.0f / ((float)H * (float)N);
    a.pairs = nullptr;
    a.lists = nullptr;
    a.list_batch = 0;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemsetAsync(key_marginal, 0, (size_t)B * N * sizeof(float), st);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "attn_entropy: memset: %s", cudaGetErrorString(e));
    int sms;
    if ((rc = sm_count(&sms)) != USV_OK) return rc;
    if (ws != nullptr && ws_bytes > WS_HEADER && marginal_planned(a, sms) && ws_bytes >= WS_HEADER + pair_plan_bytes(B, H, NB, k_per_head) &&
        (rc = launch_marginal_plan(a, static_cast<char*>(ws) + WS_HEADER, st)) != USV_OK)
        return rc;
    if ((rc = launch_marginal_tc(a, d, st)) != USV_OK) return rc;
    launch_dep_smem(entropy_kernel, dim3(B), dim3(1024), 0, st, key_marginal, N, entropy);
    USV_CHECK_LAUNCH("entropy_kernel");
    return USV_OK;
}

extern "C" int usv_attn_entropy(int B, int H, int N, int d, const void* q, const usv_strides* sq,
                                const void* k, const usv_strides* sk, const int32_t* sel,
                                const int32_t* k_per_head, int kmax, const float* lse, float scale,
                                float* key_marginal, float* entropy, void* ws, void* stream) {
    return attn_entropy_impl(B, H, N, d, q, sq, k, sk, sel, k_per_head, kmax, lse, scale, key_marginal, entropy, ws, 0, stream);
}

extern "C" size_t usv_attn_entropy_workspace(int B, int H, int N, int kmax) {
    using namespace usv;
    if (B <= 0 || H <= 0 || N <= 0 || H > USV_MAX_HEADS) return WS_HEADER;
    return WS_HEADER + marginal_plan_bytes(B, H, ceil_div(N, USV_BLOCK), kmax);
}

extern "C" size_t usv_attn_entropy_lists_workspace(int B, int H, int N, const int32_t* k_per_head) {
    using namespace usv;
    MargArgs a;
    int sms;
    if (B <= 0 || H <= 0 || N <= 0 || H > USV_MAX_HEADS || k_per_head == nullptr || sm_count(&sms) != USV_OK) return WS_HEADER;
    a.B = B; a.H = H; a.N = N; a.NB = ceil_div(N, USV_BLOCK);
    for (int h = 0; h < H; ++h) {
        if (k_per_head[h] < 1 || k_per_head[h] > a.NB) return WS_HEADER;   // (refused by the call)
        a.k_per_head[h] = k_per_head[h];
    }
    return WS_HEADER + (marginal_planned(a, sms) ? pair_plan_bytes(B, H, a.NB, k_per_head) : 0);
}

extern "C" int usv_attn_entropy_ws(int B, int H, int N, int d, const void* q, const usv_strides* sq,
                                   const void* k, const usv_strides* sk, const int32_t* sel,
                                   const int32_t* k_per_head, int kmax, const float* lse, float scale,
                                   float* key_marginal, float* entropy, void* ws, size_t ws_bytes, void* stream) {
    return attn_entropy_impl(B, H, N, d, q, sq, k, sk, sel, k_per_head, kmax, lse, scale, key_marginal, entropy, ws, ws_bytes, stream);
}

extern "C" int usv_allocate_sparsity(int L, const float* entropy, float gamma, float rho_bar, float rho_min,
                                     float rho_max, float* rho) {
    using namespace usv;
    if (L <= 0 || entropy == nullptr || rho == nullptr) return fail(USV_ERR_INVALID_ARG, "allocate_sparsity: bad L or null pointer");
    if (!(gamma >= 1.f)) return fail(USV_ERR_INVALID_ARG, "allocate_sparsity: gamma must be >= 1");
    if (!(rho_min <= rho_max)) return fail(USV_ERR_INVALID_ARG, "allocate_sparsity: rho_min > rho_max");
    double mean = 0.0;
    for (int l = 0; l < L; ++l) {
        if (!(entropy[l] >= 0.f && entropy[l] <= 1.f))
            return fail(USV_ERR_INVALID_ARG, "allocate_sparsity: entropy[%d]=%g outside [0,1]", l, (double)entropy[l]);
        mean += pow(1.0 - (double)entropy[l], (double)gamma);
    }
    mean /= (double)L;
    for (int l = 0; l < L; ++l) {
        // all layers at entropy 1 (mean 0): no layer is favoured, every one keeps the base ratio
        const double w = mean > 0.0 ? pow(1.0 - (double)entropy[l], (double)gamma) / mean : 1.0;
        const double r = (double)rho_bar * w;
        rho[l] = (float)(r < rho_min ? rho_min : (r > rho_max ? rho_max : r));
    }
    return USV_OK;
}
