// Coarse stage of the key-block selection: block pooling (HBM stream) and block scores.
//
//   pool_kernel   : one CTA per (tensor, b, h, four blocks); 16-byte loads, the next block in
//                   flight while the current one is reduced (fp32 tree), mean over the VALID
//                   rows of a block.  It also writes the three bf16 planes
//                   (mean = hi + mid + lo) that the tensor-core score kernel multiplies, so the
//                   fp32 means are not read back for a separate split pass.
//   scores_cluster_kernel : pooling and scores of short sequences in one launch.
//   scores_small_kernel : the scores of small calls, fp32 CUDA cores (both head widths).
//   scores_kernel : fp32 CUDA-core NT GEMM per (b,h), 64x64 output tile, 4x4 per thread, for the entry
//                   point without caller scratch, which has no room for the planes.
#include "usv_scores.cuh"

namespace usv {

struct PoolArgs {
    const __nv_bfloat16* x[2];
    int64_t sb[2], sh[2], sn[2];
    int N[2], NB[2];
    float* out[2];  // [B,H,NB,d]
    int H;
    // for the tensor-core score kernel: bf16 planes [3][B*H][NB_pad][d] per tensor
    // (NULL: not wanted); rows NB .. NB_pad - 1 are written as zero
    __nv_bfloat16* planes[2];
    int NB_pad[2];
    int span;           // consecutive blocks per CTA
};

// D = head dim (64 or 128).  Threads: 128.  A row of D bf16 is D/8 uint4; TPR threads per row.
// A CTA pools `span` consecutive blocks of one (tensor, b, h); the loads of the next block are issued
// before the current one is reduced, so that the CTA always has a block in flight.  Up to four blocks
// where there are enough of them to fill the GPU, fewer (and more CTAs) for small calls.
constexpr int POOL_SPAN = 4;
static int pool_span(int64_t blocks, int sms) {
    const int64_t s = blocks / (10 * sms);   // ten CTAs per SM
    return s < 1 ? 1 : (s < POOL_SPAN ? (int)s : POOL_SPAN);
}

template <int D>
__global__ void __launch_bounds__(128) pool_kernel(const PoolArgs a) {
    dep_sync();
    constexpr int TPR = D / 8;          // 16 (d=128) or 8 (d=64)
    constexpr int RPI = 128 / TPR;      // rows per iteration: 8 or 16
    constexpr int ITERS = USV_BLOCK / RPI;
    const int which = blockIdx.z;
    const int NB = a.NB[which];
    const int I0 = blockIdx.x * a.span;
    if (I0 >= NB) return;
    const int I1 = min(I0 + a.span, NB);
    const int bh = blockIdx.y;
    const int b = bh / a.H, h = bh % a.H;
    const int N = a.N[which];
    const int col = threadIdx.x % TPR, rg = threadIdx.x / TPR;
    const __nv_bfloat16* base =
        a.x[which] + b * a.sb[which] + h * a.sh[which] + (int64_t)col * 8;
    const int64_t sn = a.sn[which];
    __shared__ float red[2][RPI][D + 4];

    auto load_block = [&](int I, uint4* v) {
        const int row0 = I * USV_BLOCK;
        const int nvalid = min(USV_BLOCK, N - row0);
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            const int r = it * RPI + rg;
            v[it] = make_uint4(0, 0, 0, 0);
            if (r < nvalid) v[it] = __ldg(reinterpret_cast<const uint4*>(base + (row0 + r) * sn));
        }
    };
    uint4 v[ITERS], vn[ITERS];
    load_block(I0, v);
    for (int I = I0; I < I1; ++I) {
        if (I + 1 < I1) load_block(I + 1, vn);
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            float f[8];
            bf16x8_to_float(v[it], f);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] += f[e];
        }
        float (*rd)[D + 4] = red[(I - I0) & 1];   // two buffers: one barrier per block is enough
#pragma unroll
        for (int e = 0; e < 8; ++e) rd[rg][col * 8 + e] = acc[e];
        __syncthreads();
        if (threadIdx.x < D) {
            const int nvalid = min(USV_BLOCK, N - I * USV_BLOCK);
            float s = 0.f;
#pragma unroll
            for (int g = 0; g < RPI; ++g) s += rd[g][threadIdx.x];
            const float mean = s / (float)nvalid;
            a.out[which][((int64_t)bh * NB + I) * D + threadIdx.x] = mean;
            if (a.planes[which] != nullptr) {
                const int64_t plane = (int64_t)gridDim.y * a.NB_pad[which] * D;
                __nv_bfloat16* dst = a.planes[which] + ((int64_t)bh * a.NB_pad[which] + I) * D + threadIdx.x;
                float rem = mean;
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    const __nv_bfloat16 hp = __float2bfloat16_rn(rem);
                    dst[p * plane] = hp;
                    rem -= __bfloat162float(hp);
                }
            }
        }
#pragma unroll
        for (int it = 0; it < ITERS; ++it) v[it] = vn[it];
    }
    // the CTA that pooled the last block also clears the padding rows of the planes
    if (I1 == NB && a.planes[which] != nullptr && threadIdx.x < D) {
        const int64_t plane = (int64_t)gridDim.y * a.NB_pad[which] * D;
        for (int I = NB; I < a.NB_pad[which]; ++I) {
            __nv_bfloat16* dst = a.planes[which] + ((int64_t)bh * a.NB_pad[which] + I) * D + threadIdx.x;
#pragma unroll
            for (int p = 0; p < 3; ++p) dst[p * plane] = __float2bfloat16_rn(0.f);
        }
    }
}

// scores[bh, I, J] = scale * sum_e qbar[bh,I,e] * kbar[bh,J,e]
// CTA: 256 threads, 64x64 tile; smem tiles stored e-major so that the inner product reads
// float4 along the tile row/column.
__global__ void __launch_bounds__(256) scores_kernel(const float* __restrict__ qbar,
                                                     const float* __restrict__ kbar,
                                                     float* __restrict__ scores, int NBq, int NBk,
                                                     int d, float scale) {
    dep_sync();
    constexpr int TM = 64, TN = 64, TK = 32;
    __shared__ __align__(16) float As[TK][TM + 4];
    __shared__ __align__(16) float Bs[TK][TN + 4];
    const int bh = blockIdx.z;
    const int i0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
    const float* A = qbar + (int64_t)bh * NBq * d;
    const float* Bm = kbar + (int64_t)bh * NBk * d;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < d; k0 += TK) {
        // 64 rows x 32 floats = 512 float4; 256 threads -> 2 each
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int idx = threadIdx.x + t * 256;
            const int r = idx / 8, c4 = idx % 8;
            float4 va = make_float4(0, 0, 0, 0), vb = va;
            if (i0 + r < NBq)
                va = *reinterpret_cast<const float4*>(A + (int64_t)(i0 + r) * d + k0 + c4 * 4);
            if (j0 + r < NBk)
                vb = *reinterpret_cast<const float4*>(Bm + (int64_t)(j0 + r) * d + k0 + c4 * 4);
            As[c4 * 4 + 0][r] = va.x; As[c4 * 4 + 1][r] = va.y;
            As[c4 * 4 + 2][r] = va.z; As[c4 * 4 + 3][r] = va.w;
            Bs[c4 * 4 + 0][r] = vb.x; Bs[c4 * 4 + 1][r] = vb.y;
            Bs[c4 * 4 + 2][r] = vb.z; Bs[c4 * 4 + 3][r] = vb.w;
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < TK; ++e) {
            const float4 av = *reinterpret_cast<const float4*>(&As[e][ty * 4]);
            const float4 bv = *reinterpret_cast<const float4*>(&Bs[e][tx * 4]);
            const float ar[4] = {av.x, av.y, av.z, av.w};
            const float br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
        }
        __syncthreads();
    }
    float* out = scores + (int64_t)bh * NBq * NBk;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int I = i0 + ty * 4 + i;
        if (I >= NBq) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int J = j0 + tx * 4 + j;
            if (J < NBk) out[(int64_t)I * NBk + J] = acc[i][j] * scale;
        }
    }
}

// The same product for small calls: 32 x 32 output tiles, 64 features of both operands in shared memory
// after one round of loads, 2 x 2 outputs a thread, features in ascending order as above.  (All 128
// features at once need 34 KB, and with that another split of the SM's memory than pool_kernel has.)
constexpr int SCT = 32;

template <int D>
__global__ void __launch_bounds__(256) scores_small_kernel(const float* __restrict__ qbar, const float* __restrict__ kbar,
                                                           float* __restrict__ scores, int NBq, int NBk, float scale) {
    dep_sync();
    constexpr int TK = 64;
    __shared__ __align__(16) float As[SCT][TK + 4];
    __shared__ __align__(16) float Bs[SCT][TK + 4];
    const int bh = blockIdx.z;
    const int i0 = blockIdx.y * SCT, j0 = blockIdx.x * SCT;
    const float4* A = reinterpret_cast<const float4*>(qbar + (int64_t)bh * NBq * D);
    const float4* Bm = reinterpret_cast<const float4*>(kbar + (int64_t)bh * NBk * D);
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    constexpr int L = SCT * TK / 4 / 256;   // 16-byte loads per thread, operand and round
    float4 va[D / TK][L], vb[D / TK][L];
#pragma unroll
    for (int k = 0; k < D / TK; ++k)
#pragma unroll
        for (int l = 0; l < L; ++l) {
            const int r = ty + 16 * l, c = k * (TK / 4) + tx;
            va[k][l] = i0 + r < NBq ? A[(int64_t)(i0 + r) * (D / 4) + c] : make_float4(0, 0, 0, 0);
            vb[k][l] = j0 + r < NBk ? Bm[(int64_t)(j0 + r) * (D / 4) + c] : make_float4(0, 0, 0, 0);
        }
    float acc[2][2] = {};
#pragma unroll
    for (int k = 0; k < D / TK; ++k) {
        if (k > 0) __syncthreads();
#pragma unroll
        for (int l = 0; l < L; ++l) {
            *reinterpret_cast<float4*>(&As[ty + 16 * l][tx * 4]) = va[k][l];
            *reinterpret_cast<float4*>(&Bs[ty + 16 * l][tx * 4]) = vb[k][l];
        }
        __syncthreads();
#pragma unroll 8
        for (int e = 0; e < TK; e += 4) {
            float4 av[2], bv[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                av[i] = *reinterpret_cast<const float4*>(&As[ty + 16 * i][e]);
                bv[i] = *reinterpret_cast<const float4*>(&Bs[tx + 16 * i][e]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    acc[i][j] = fmaf(av[i].w, bv[j].w, fmaf(av[i].z, bv[j].z, fmaf(av[i].y, bv[j].y, fmaf(av[i].x, bv[j].x, acc[i][j]))));
        }
    }
    float* out = scores + (int64_t)bh * NBq * NBk;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int I = i0 + ty + 16 * i, J = j0 + tx + 16 * j;
            if (I < NBq && J < NBk) out[(int64_t)I * NBk + J] = acc[i][j] * scale;
        }
}

// Pooling and scores of short sequences in one kernel: a cluster of CLC CTAs per (b, h).  Each pools its share of the query and of
// the key blocks (sums in the order of pool_kernel), writes its key means into the shared memory of
// all of them, and after one cluster barrier computes its query rows of scores (features in ascending order, as above).  Two
// launches, a round trip of the means through the L2 and the wait between them are saved.
constexpr int CLC = 8, CL_MAX = 48;   // CTAs of a cluster; blocks of the longest sequence

template <int D, int G>
constexpr size_t cluster_smem() {     // key means, the CTA's query means, partial sums of two rounds of blocks
    return (size_t)(CL_MAX + CL_MAX / CLC) * (D + 4) * 4 + 2 * (size_t)G * (128 / (D / 8)) * (D + 4) * 4;
}

// G groups of 128 threads, each with a block at a time; PER CTAs an SM
template <int D, int G, int PER>
__global__ void __launch_bounds__(128 * G, PER) __cluster_dims__(CLC, 1, 1) scores_cluster_kernel(const PoolArgs a, float* __restrict__ scores, float scale) {
    extern __shared__ __align__(16) float s_mem[];
    constexpr int LD = D + 4, TPR = D / 8, RPI = 128 / TPR, ITERS = USV_BLOCK / RPI;
    float* s_k = s_mem;                          // [CL_MAX][LD]
    float* s_q = s_k + CL_MAX * LD;              // [CL_MAX / CLC][LD]
    float* s_red = s_q + CL_MAX / CLC * LD;      // [2 buffers][G blocks][RPI][LD]
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // (waited for before anything is written to a neighbour)
    dep_sync();
    const int rank = blockIdx.x, bh = blockIdx.y;
    const int b = bh / a.H, h = bh % a.H;
    const int half = threadIdx.x >> 7, tid = threadIdx.x & 127;
    const int col = tid % TPR, rg = tid / TPR;
    const int per_q = (a.NB[0] + CLC - 1) / CLC, per_k = (a.NB[1] + CLC - 1) / CLC;
    const int nq = max(0, min(per_q, a.NB[0] - rank * per_q)), nk = max(0, min(per_k, a.NB[1] - rank * per_k));
    const int n = nk + nq;                       // the CTA's blocks, keys first
    auto load = [&](int i, uint4* v) {
        const int which = i < nk ? 1 : 0, I = i < nk ? rank * per_k + i : rank * per_q + i - nk;
        const __nv_bfloat16* base = a.x[which] + b * a.sb[which] + h * a.sh[which] + (int64_t)col * 8;
        const int nvalid = i < n ? min(USV_BLOCK, a.N[which] - I * USV_BLOCK) : 0;
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            const int r = it * RPI + rg;
            v[it] = r < nvalid ? __ldg(reinterpret_cast<const uint4*>(base + (int64_t)(I * USV_BLOCK + r) * a.sn[which])) : make_uint4(0, 0, 0, 0);
        }
    };
    uint4 v[ITERS], vn[ITERS];
    load(half, v);
    bool first = true;
    int buf = 0;
    for (int i0 = 0; i0 < n; i0 += G, buf ^= 1) {
        const int i = i0 + half;
        if (i0 + G < n) load(i + G, vn);
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            float f[8];
            bf16x8_to_float(v[it], f);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] += f[e];
        }
        float* rd = s_red + (buf * G + half) * RPI * LD;   // two buffers: one barrier a round is enough
#pragma unroll
        for (int e = 0; e < 8; ++e) rd[rg * LD + col * 8 + e] = acc[e];
        __syncthreads();
        if (first) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        first = false;
        if (tid < D && i < n) {
            const int which = i < nk ? 1 : 0, I = i < nk ? rank * per_k + i : rank * per_q + i - nk;
            const int nvalid = min(USV_BLOCK, a.N[which] - I * USV_BLOCK);
            float s = 0.f;
#pragma unroll
            for (int g = 0; g < RPI; ++g) s += rd[g * LD + tid];
            const float mean = s / (float)nvalid;
            if (which == 0) {
                s_q[(i - nk) * LD + tid] = mean;
            } else {
                const uint32_t at = (uint32_t)__cvta_generic_to_shared(s_k + I * LD + tid);
#pragma unroll
                for (int c = 0; c < CLC; ++c) {
                    uint32_t to;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(at), "r"(c));
                    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to), "f"(mean) : "memory");
                }
            }
        }
#pragma unroll
        for (int it = 0; it < ITERS; ++it) v[it] = vn[it];
    }
    if (first) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    const int NBk = a.NB[1];
    float* out = scores + ((int64_t)bh * a.NB[0] + rank * per_q) * NBk;
    for (int i = threadIdx.x; i < nq * NBk; i += 128 * G) {
        const int I = i / NBk, J = i - I * NBk;
        const float4* x = reinterpret_cast<const float4*>(s_q + I * LD);
        const float4* y = reinterpret_cast<const float4*>(s_k + J * LD);
        float acc = 0.f;
#pragma unroll 8
        for (int e = 0; e < D / 4; ++e) {
            const float4 av = x[e], bv = y[e];
            acc = fmaf(av.w, bv.w, fmaf(av.z, bv.z, fmaf(av.y, bv.y, fmaf(av.x, bv.x, acc))));
        }
        out[i] = acc * scale;
    }
}

template <int D, int G, int PER>
static int launch_scores_cluster(const PoolArgs& a, int BH, float* scores, float scale, cudaStream_t st) {
    constexpr size_t smem = cluster_smem<D, G>();
    cudaError_t e = cudaFuncSetAttribute(scores_cluster_kernel<D, G, PER>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "block_scores: smem attribute: %s", cudaGetErrorString(e));
    launch_dep_smem(scores_cluster_kernel<D, G, PER>, dim3(CLC, BH), dim3(128 * G), smem, st, a, scores, scale);
    USV_CHECK_LAUNCH("scores_cluster_kernel");
    return USV_OK;
}

// Calls that are better off with it, as groups of 128 threads a CTA (0: none): a cluster has an eighth of a (b, h)'s blocks a CTA,
// so sequences are short, and its CTAs are resident together.  Whole calls, us, two kernels / this one: d = 64, 2 heads x 16 blocks
// 5.4 / 3.0, 12 x 32 5.3 / 5.0, 12 x 48 6.1 / 7.1, 24 x 16 5.3 / 3.8, 40 x 16 5.8 / 5.2; d = 128, 2 x 16 5.4 / 3.7, 12 x 32 6.6 / 5.3,
// 12 x 48 8.2 / 7.0, 12 x 64 8.0 / 9.0, 24 x 16 7.0 / 5.0, 24 x 32 7.6 / 7.5, 40 x 16 8.0 / 5.7, 40 x 32 9.1 / 9.9, 80 x 16 9.0 / 10.4.
static int cluster_groups(int BH, int NBq, int NBk, int d, int sms) {
    const int ctas = BH * CLC, nb = NBq > NBk ? NBq : NBk;
    if (ctas <= sms && nb <= (d == 128 ? CL_MAX : 32)) return 4;
    if (ctas <= 2 * sms && nb <= (d == 128 ? 16 : 32)) return 4;
    return ctas <= (d == 128 ? 3 : 4) * sms && nb <= 16 ? 2 : 0;
}

// The small form takes calls of at most this many 32 x 32 tiles.  Whole calls, us, with the tensor-core kernel / with
// this one: d = 64, 12 heads x 32 blocks (12 tiles) 9.9 / 4.9, 24 x 64 (96) 11.7 / 7.2, 4 x 256 (256) 10.1 / 6.8, 2 x 512 (512)
// 10.2 / 8.8, 12 x 220 (588) 13.6 / 12.4, 3 x 512 (768) 11.1 / 11.2; d = 128, in that order, 15.1 / 6.4, 18.6 / 10.8, 16.2 / 9.9,
// 16.2 / 13.5, 25.2 / 19.5, 18.0 / 18.6.
constexpr int64_t SMALL_TILES = 700;
static int64_t small_tiles(int BH, int NBq, int NBk) { return (int64_t)BH * ceil_div(NBq, SCT) * ceil_div(NBk, SCT); }

}  // namespace usv

extern "C" size_t usv_block_scores_workspace(int B, int H, int Nq, int Nk, int d) {
    if (B <= 0 || H <= 0 || Nq <= 0 || Nk <= 0 || d <= 0) return 0;
    const size_t nbq = usv::ceil_div(Nq, USV_BLOCK), nbk = usv::ceil_div(Nk, USV_BLOCK);
    // header, pooled means of q and k, the bf16 planes of the tensor-core scores kernel (small calls at d = 64
    // never had them, and do not run it)
    const bool planes = d == 128 || (d == 64 && usv::small_tiles(B * H, (int)nbq, (int)nbk) > usv::SMALL_TILES);
    return usv::WS_HEADER + usv::align_up((size_t)B * H * nbq * d * sizeof(float), 256) +
           usv::align_up((size_t)B * H * nbk * d * sizeof(float), 256) +
           (planes ? usv::scores_tc_bytes(B * H, (int)nbq, (int)nbk, d) : 0);
}

extern "C" int usv_block_scores(int B, int H, int Nq, int Nk, int d, const void* q,
                                const usv_strides* sq, const void* k, const usv_strides* sk,
                                float* scores, void* ws, size_t ws_bytes, void* stream) {
    using namespace usv;
    if (B <= 0 || H <= 0 || Nq <= 0 || Nk <= 0)
        return fail(USV_ERR_INVALID_ARG, "block_scores: B,H,Nq,Nk must be positive");
    if (d != 64 && d != 128) return fail(USV_ERR_UNSUPPORTED, "block_scores: d=%d (need 64 or 128)", d);
    if ((int64_t)B * H > 65535) return fail(USV_ERR_UNSUPPORTED, "block_scores: B*H > 65535");
    int rc;
    if ((rc = check_view("q", q, sq, d)) != USV_OK) return rc;
    if ((rc = check_view("k", k, sk, d)) != USV_OK) return rc;
    if (scores == nullptr || ws == nullptr) return fail(USV_ERR_INVALID_ARG, "block_scores: null scores/ws");
    if (!aligned16(scores) || !aligned16(ws))
        return fail(USV_ERR_UNSUPPORTED, "block_scores: scores/ws not 16-byte aligned");
    if (ws_bytes < usv_block_scores_workspace(B, H, Nq, Nk, d))
        return fail(USV_ERR_WORKSPACE, "block_scores: workspace %zu < %zu", ws_bytes,
                    usv_block_scores_workspace(B, H, Nq, Nk, d));
    const int NBq = ceil_div(Nq, USV_BLOCK), NBk = ceil_div(Nk, USV_BLOCK);
    float* qbar = reinterpret_cast<float*>(static_cast<char*>(ws) + WS_HEADER);
    float* kbar = reinterpret_cast<float*>(static_cast<char*>(ws) + WS_HEADER +
                                           align_up((size_t)B * H * NBq * d * sizeof(float), 256));
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    PoolArgs a;
    a.x[0] = static_cast<const __nv_bfloat16*>(q);
    a.x[1] = static_cast<const __nv_bfloat16*>(k);
    a.sb[0] = sq->sb; a.sh[0] = sq->sh; a.sn[0] = sq->sn;
    a.sb[1] = sk->sb; a.sh[1] = sk->sh; a.sn[1] = sk->sn;
    a.N[0] = Nq; a.N[1] = Nk; a.NB[0] = NBq; a.NB[1] = NBk;
    a.out[0] = qbar; a.out[1] = kbar;
    a.H = H;
    a.planes[0] = a.planes[1] = nullptr;
    a.NB_pad[0] = a.NB_pad[1] = 0;
    void* tc_mem = reinterpret_cast<char*>(kbar) + align_up((size_t)B * H * NBk * d * sizeof(float), 256);
    const int64_t tiles = small_tiles(B * H, NBq, NBk);
    const bool small = tiles <= SMALL_TILES;
    if (!small) scores_tc_planes(tc_mem, B * H, NBq, NBk, d, &a.planes[0], &a.planes[1], &a.NB_pad[0], &a.NB_pad[1]);
    int sms;
    if ((rc = sm_count(&sms)) != USV_OK) return rc;
    a.span = pool_span((int64_t)B * H * (NBq + NBk), sms);
    const float sc = 1.0f / sqrtf((float)d);
    const int groups = small ? cluster_groups(B * H, NBq, NBk, d, sms) : 0;
    if (groups == 2)
        return d == 128 ? launch_scores_cluster<128, 2, 2>(a, B * H, scores, sc, st) : launch_scores_cluster<64, 2, 2>(a, B * H, scores, sc, st);
    if (groups == 4 && d == 64) return launch_scores_cluster<64, 4, 2>(a, B * H, scores, sc, st);
    if (groups == 4)
        return B * H * CLC <= sms ? launch_scores_cluster<128, 4, 1>(a, B * H, scores, sc, st) : launch_scores_cluster<128, 4, 2>(a, B * H, scores, sc, st);
    dim3 pg(ceil_div(NBq > NBk ? NBq : NBk, a.span), B * H, 2);
    if (d == 128) launch_dep(pool_kernel<128>, dim3(pg), dim3(128), 0, st, a);
    else launch_dep(pool_kernel<64>, dim3(pg), dim3(128), 0, st, a);
    USV_CHECK_LAUNCH("pool_kernel");

    if (small) {
        dim3 tg(ceil_div(NBk, SCT), ceil_div(NBq, SCT), B * H);
        if (d == 128) launch_dep(scores_small_kernel<128>, tg, dim3(256), 0, st, qbar, kbar, scores, NBq, NBk, sc);
        else launch_dep(scores_small_kernel<64>, tg, dim3(256), 0, st, qbar, kbar, scores, NBq, NBk, sc);
        USV_CHECK_LAUNCH("scores_small_kernel");
        return USV_OK;
    }
    return launch_scores_tc(scores, qbar, kbar, B * H, NBq, NBk, d, sc, tc_mem, static_cast<unsigned int*>(ws), st);
}

// ------------------------------------------------------------------------------------------
// Variant without caller scratch: the pooled means go to a fixed array inside the library image.
// For callers that may neither allocate device memory nor lend a buffer (allocator-frozen
// sections of a host framework, plugins that only receive tensors, fixed-budget loops).

namespace usv {

static __device__ __align__(256) unsigned char g_noalloc_scratch[USV_NOALLOC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
static void* g_noalloc_ptr[kMaxDevices] = {};  // device address of the array, per device

// In host code `g_noalloc_scratch` is only a handle for the runtime, not an address a kernel
// can use; the real per-device address has to be asked for once, with that device current.
static int noalloc_scratch(void** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "block_scores_noalloc: cudaGetDevice: %s", cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return fail(USV_ERR_UNSUPPORTED, "block_scores_noalloc: device %d out of range", dev);
    void* p = __atomic_load_n(&g_noalloc_ptr[dev], __ATOMIC_ACQUIRE);
    if (p == nullptr) {
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || p == nullptr)
            return fail(USV_ERR_CUDA, "block_scores_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
        __atomic_store_n(&g_noalloc_ptr[dev], p, __ATOMIC_RELEASE);  // same value from any thread
    }
    *out = p;
    return USV_OK;
}

}  // namespace usv

extern "C" int usv_block_scores_noalloc(int B, int H, int Nq, int Nk, int d, const void* q,
                                        const usv_strides* sq, const void* k,
                                        const usv_strides* sk, float* scores, void* stream) {
    using namespace usv;
    if (B <= 0 || H <= 0 || Nq <= 0 || Nk <= 0)
        return fail(USV_ERR_INVALID_ARG, "block_scores_noalloc: B,H,Nq,Nk must be positive");
    if (d != 64 && d != 128) return fail(USV_ERR_UNSUPPORTED, "block_scores_noalloc: d=%d (need 64 or 128)", d);
    if ((int64_t)B * H > 65535) return fail(USV_ERR_UNSUPPORTED, "block_scores_noalloc: B*H > 65535");
    int rc;
    if ((rc = check_view("q", q, sq, d)) != USV_OK) return rc;
    if ((rc = check_view("k", k, sk, d)) != USV_OK) return rc;
    if (scores == nullptr) return fail(USV_ERR_INVALID_ARG, "block_scores_noalloc: null scores");
    if (!aligned16(scores)) return fail(USV_ERR_UNSUPPORTED, "block_scores_noalloc: scores not 16-byte aligned");
    const size_t need = align_up((size_t)B * H * ceil_div(Nq, USV_BLOCK) * d * sizeof(float), 256) +
                        align_up((size_t)B * H * ceil_div(Nk, USV_BLOCK) * d * sizeof(float), 256);
    if (need > (size_t)USV_NOALLOC_SCRATCH_BYTES)
        return fail(USV_ERR_WORKSPACE,
                    "block_scores_noalloc: needs %zu bytes of scratch, the built-in array holds %u; "
                    "use usv_block_scores with a caller workspace for this size",
                    need, (unsigned)USV_NOALLOC_SCRATCH_BYTES);
    void* scratch = nullptr;
    if ((rc = noalloc_scratch(&scratch)) != USV_OK) return rc;

    const int NBq = ceil_div(Nq, USV_BLOCK), NBk = ceil_div(Nk, USV_BLOCK);
    float* qbar = static_cast<float*>(scratch);
    float* kbar = reinterpret_cast<float*>(static_cast<char*>(scratch) +
                                           align_up((size_t)B * H * NBq * d * sizeof(float), 256));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PoolArgs a;
    a.x[0] = static_cast<const __nv_bfloat16*>(q);
    a.x[1] = static_cast<const __nv_bfloat16*>(k);
    a.sb[0] = sq->sb; a.sh[0] = sq->sh; a.sn[0] = sq->sn;
    a.sb[1] = sk->sb; a.sh[1] = sk->sh; a.sn[1] = sk->sn;
    a.N[0] = Nq; a.N[1] = Nk; a.NB[0] = NBq; a.NB[1] = NBk;
    a.out[0] = qbar; a.out[1] = kbar;
    a.H = H;
    a.planes[0] = a.planes[1] = nullptr;
    a.NB_pad[0] = a.NB_pad[1] = 0;
    int sms;
    if ((rc = sm_count(&sms)) != USV_OK) return rc;
    a.span = pool_span((int64_t)B * H * (NBq + NBk), sms);
    dim3 pg(ceil_div(NBq > NBk ? NBq : NBk, a.span), B * H, 2);
    if (d == 128) pool_kernel<128><<<pg, 128, 0, st>>>(a);
    else pool_kernel<64><<<pg, 128, 0, st>>>(a);
    USV_CHECK_LAUNCH("pool_kernel (noalloc)");
    dim3 sg(ceil_div(NBk, 64), ceil_div(NBq, 64), B * H);
    scores_kernel<<<sg, 256, 0, st>>>(qbar, kbar, scores, NBq, NBk, d, 1.0f / sqrtf((float)d));
    USV_CHECK_LAUNCH("scores_kernel (noalloc)");
    return USV_OK;
}
