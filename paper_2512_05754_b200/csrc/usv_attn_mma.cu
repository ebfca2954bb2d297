// Block-sparse attention forward, legacy tensor-core path (mma.sync m16n8k16, bf16).
//
// The faster path for small calls (usv_attn_api.cu says where the line lies), the exact recomputation
// of the query blocks the tcgen05 kernel reports, the path beyond its longest sequence, and an
// on-device cross-check of it.  One CTA (4 warps) per (b, h, query block); each warp owns 16
// query rows.  Selected K/V blocks stream through a double-buffered cp.async pipeline; S = QK^T
// and O += PV run on mma.sync with the softmax kept in registers (fp32, base-2 exponentials).
#include "usv_mma_sync.cuh"

namespace usv {

// Weights of a 64-key tile from its logits, relative to ms (rows g and g + 8 of the warp): pf gets them as bf16, in the layout
// of an A operand, and add(nt, r, e, w) sees the sum of the unrounded pair of 8-key piece nt and row r, and the rounded pair.
template <typename Add>
__device__ __forceinline__ void tile_weights(const float (&s)[8][4], float c, const float (&ms)[2], uint32_t (&pf)[4][4], Add add) {
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float e0 = exp2f(fmaf(s[nt][2 * r], c, -ms[r]));
            const float e1 = exp2f(fmaf(s[nt][2 * r + 1], c, -ms[r]));
            const uint32_t w = pack_bf16x2(e0, e1);
            pf[nt >> 1][(nt & 1) * 2 + r] = w;
            add(nt, r, e0 + e1, w);
        }
}
__device__ __forceinline__ float sum_bf16x2(uint32_t w) { return __uint_as_float(w << 16) + __uint_as_float(w & 0xffff0000u); }

// Q fragments of the warp's 16 rows, and the logits of one K tile
template <int D>
__device__ __forceinline__ void load_q_frags(uint32_t (&qf)[D / 16][4], const __nv_bfloat16* Qs, int warp, int lane) {
    constexpr int LD = MmaSmem<D>::LD;
    const __nv_bfloat16* qrow = Qs + (warp * 16 + (lane >> 2)) * LD + 2 * (lane & 3);
#pragma unroll
    for (int kt = 0; kt < D / 16; ++kt) {
        qf[kt][0] = *reinterpret_cast<const uint32_t*>(qrow + kt * 16);
        qf[kt][1] = *reinterpret_cast<const uint32_t*>(qrow + 8 * LD + kt * 16);
        qf[kt][2] = *reinterpret_cast<const uint32_t*>(qrow + kt * 16 + 8);
        qf[kt][3] = *reinterpret_cast<const uint32_t*>(qrow + 8 * LD + kt * 16 + 8);
    }
}
// s: 16 x 64 logits, keys from nvalid on -inf; mx: the maxima of rows g and g + 8
template <int D>
__device__ __forceinline__ void tile_logits(float (&s)[8][4], float (&mx)[2], const uint32_t (&qf)[D / 16][4], const __nv_bfloat16* Kt,
                                            int nvalid, int lane) {
    constexpr int LD = MmaSmem<D>::LD;
    const int g = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
        const __nv_bfloat16* krow = Kt + (nt * 8 + g) * LD + 2 * tig;
#pragma unroll
        for (int kt = 0; kt < D / 16; ++kt) {
            const uint32_t b0 = *reinterpret_cast<const uint32_t*>(krow + kt * 16);
            const uint32_t b1 = *reinterpret_cast<const uint32_t*>(krow + kt * 16 + 8);
            mma_bf16_16816(s[nt], qf[kt], b0, b1);
        }
    }
    if (nvalid < USV_BLOCK) {
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const int col = nt * 8 + 2 * tig;
            if (col >= nvalid) s[nt][0] = s[nt][2] = -INFINITY;
            if (col + 1 >= nvalid) s[nt][1] = s[nt][3] = -INFINITY;
        }
    }
    mx[0] = mx[1] = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        mx[0] = fmaxf(mx[0], fmaxf(s[nt][0], s[nt][1]));
        mx[1] = fmaxf(mx[1], fmaxf(s[nt][2], s[nt][3]));
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
    }
}
// The running maximum m of a row of scaled (base-2) logits past a tile whose maximum is mx * c: returns the factor for what was
// summed so far; ms is what the tile's weights are relative to.
__device__ __forceinline__ float next_max(float& m, float mx, float c, float& ms) {
    const float mnew = fmaxf(m, mx * c);
    ms = mnew == -INFINITY ? 0.f : mnew;
    const float alpha = exp2f(m - ms);
    m = mnew;
    return alpha;
}

// G groups of 4 warps share a query block: group i takes the entries i, i + G, ... of its list, and the groups' results, each
// relative to its own row maxima, are put together at the end.  (Each group's weights are rounded to bf16 relative to maxima of its
// own: results differ from those of one group by that rounding, and are no further from fp64.  Lists of 5 to 10 entries of white
// noise: 2.1e-4 to 3.5e-4 relative, 2.2e-4 to 3.7e-4 with one group, 3.0e-4 to 4.3e-4 on the tcgen05 kernel.)
// NBUF: K/V tiles a group has room for.
template <int D, int G, int NBUF>
__device__ __forceinline__ void attn_mma_block(const AttnArgs& a, const int work, unsigned char* smem_raw) {
    constexpr int LD = MmaSmem<D>::LD;
    constexpr int TILE = MmaSmem<D>::TILE;
    constexpr int NT = D / 8;   // n-tiles of the output
    const int grp = G == 1 ? 0 : threadIdx.x >> 7;
    __nv_bfloat16* Qs = reinterpret_cast<__nv_bfloat16*>(smem_raw);
    __nv_bfloat16* Ks = Qs + TILE + grp * (2 * NBUF * TILE);
    __nv_bfloat16* Vs = Ks + NBUF * TILE;
    auto group_sync = [&] {
        if (G == 1) __syncthreads();
        else asm volatile("barrier.sync %0, 128;" ::"r"(grp + 1) : "memory");
    };

    const int I = work % a.NB;
    const int bh_ord = work / a.NB;
    const int b = bh_ord / a.H;
    const int h = a.head_order[bh_ord % a.H];
    const int kh = a.k_per_head[h];
    const int N = a.N;
    const int32_t* sel = a.sel + (((int64_t)b * a.H + h) * a.NB + I) * a.kmax;

    const __nv_bfloat16* Q = a.q + b * a.sq.sb + h * a.sq.sh;
    const __nv_bfloat16* K = a.k + b * a.sk.sb + h * a.sk.sh;
    const __nv_bfloat16* V = a.v + b * a.sv.sb + h * a.sv.sh;

    const int warp = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;

    // first valid entry of the selection
    int t = grp;
    while (t < kh && sel[t] < 0) t += G;

    load_tile<D, G>(Qs, Q, a.sq.sn, I * USV_BLOCK, N);
    if (t < kh) {
        load_tile<D>(Ks, K, a.sk.sn, sel[t] * USV_BLOCK, N);
        load_tile<D>(Vs, V, a.sv.sn, sel[t] * USV_BLOCK, N);
    }
    cp_async_commit();

    uint32_t qf[D / 16][4];
    float o[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
    float m[2] = {-INFINITY, -INFINITY};  // running max of the scaled (base-2) logits, rows g, g+8
    float l[2] = {0.f, 0.f};              // this thread's share of the running denominators
    // The same sums taken over the bf16-rounded weights that feed the P.V product: normalising
    // by them makes the applied weights sum to one exactly, so the rounding of a dominant
    // weight cancels instead of scaling the whole row.
    float lr[2] = {0.f, 0.f};
    const float c = a.scale_log2;

    int buf = 0;
    bool first = true;
    if (G > 1) {   // the Q tile came through all groups
        cp_async_wait_all();
        __syncthreads();
    }
    while (t < kh) {
        const int J = sel[t];
        int tn = t + G;
        while (tn < kh && sel[tn] < 0) tn += G;

        cp_async_wait_all();
        group_sync();  // tile t is visible; every warp has left the tile of the step before
        if (NBUF == 2 && tn < kh) {
            load_tile<D>(Ks + (buf ^ 1) * TILE, K, a.sk.sn, sel[tn] * USV_BLOCK, N);
            load_tile<D>(Vs + (buf ^ 1) * TILE, V, a.sv.sn, sel[tn] * USV_BLOCK, N);
        }
        cp_async_commit();

        if (first) load_q_frags<D>(qf, Qs, warp, lane);
        first = false;

        const __nv_bfloat16* Vt = Vs + buf * TILE;
        float s[8][4], mx[2], alpha[2], ms[2];
        tile_logits<D>(s, mx, qf, Ks + buf * TILE, N - J * USV_BLOCK, lane);
        // online softmax (rows g -> elements 0,1; row g+8 -> elements 2,3)
#pragma unroll
        for (int r = 0; r < 2; ++r) alpha[r] = next_max(m[r], mx[r], c, ms[r]);
        uint32_t pf[4][4];
        tile_weights(s, c, ms, pf, [&](int nt, int r, float e, uint32_t w) {
            l[r] = nt == 0 ? fmaf(l[r], alpha[r], e) : l[r] + e;
            lr[r] = nt == 0 ? fmaf(lr[r], alpha[r], sum_bf16x2(w)) : lr[r] + sum_bf16x2(w);
        });
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            o[n][0] *= alpha[0];
            o[n][1] *= alpha[0];
            o[n][2] *= alpha[1];
            o[n][3] *= alpha[1];
        }
        // O += P V
#pragma unroll
        for (int kt = 0; kt < 4; ++kt) {
            const __nv_bfloat16* vrow = Vt + (kt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * LD +
                                        (lane >> 4) * 8;
#pragma unroll
            for (int n2 = 0; n2 < NT / 2; ++n2) {
                uint32_t bfr[4];
                ldmatrix_x4_trans(bfr, vrow + n2 * 16);
                mma_bf16_16816(o[2 * n2], pf[kt], bfr[0], bfr[1]);
                mma_bf16_16816(o[2 * n2 + 1], pf[kt], bfr[2], bfr[3]);
            }
        }
        if (NBUF == 2) buf ^= 1;   // (with one tile there is no next one)
        t = tn;
    }
    cp_async_wait_all();

    // finish the denominators across the quad, normalise, store
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
        lr[r] += __shfl_xor_sync(0xffffffffu, lr[r], 1);
        lr[r] += __shfl_xor_sync(0xffffffffu, lr[r], 2);
    }
    if constexpr (G > 1) {
        // each group's rows of O where its tiles were, its maxima and sums behind all tiles; then a thread puts 8 columns
        // of a row together
        static_assert(64 * (D + 8) * 4 <= 2 * TILE * 2, "a group's rows of O fit where a K and a V tile were");
        constexpr int OLD = D + 8;
        float* stat = reinterpret_cast<float*>(Qs + TILE + G * (2 * NBUF * TILE));   // [G][3][64]
        auto rows_of = [&](int i) { return reinterpret_cast<float*>(Qs + TILE + i * (2 * NBUF * TILE)); };
        group_sync();   // every warp of the group has left its tiles
        float* mine = rows_of(grp) + (warp * 16 + g) * OLD + 2 * tig;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            *reinterpret_cast<float2*>(mine + n * 8) = make_float2(o[n][0], o[n][1]);
            *reinterpret_cast<float2*>(mine + 8 * OLD + n * 8) = make_float2(o[n][2], o[n][3]);
        }
        if (tig == 0) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float* st = stat + grp * 192 + warp * 16 + g + 8 * r;
                st[0] = m[r];
                st[64] = l[r];
                st[128] = lr[r];
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < USV_BLOCK * (D / 8); i += 128 * G) {
            const int rr = i / (D / 8), cc = i % (D / 8) * 8, row = I * USV_BLOCK + rr;
            if (row >= N) continue;
            float mx = -INFINITY;
#pragma unroll
            for (int q = 0; q < G; ++q) mx = fmaxf(mx, stat[q * 192 + rr]);
            const float ms = mx == -INFINITY ? 0.f : mx;
            float ls = 0.f, ln = 0.f, y[8] = {};
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const float w = exp2f(stat[q * 192 + rr] - ms);
                ls += w * stat[q * 192 + 64 + rr];
                ln += w * stat[q * 192 + 128 + rr];
                const float4* x = reinterpret_cast<const float4*>(rows_of(q) + rr * OLD + cc);
                const float4 u = x[0], v = x[1];
                y[0] += w * u.x; y[1] += w * u.y; y[2] += w * u.z; y[3] += w * u.w;
                y[4] += w * v.x; y[5] += w * v.y; y[6] += w * v.z; y[7] += w * v.w;
            }
            const float inv = ln > 0.f ? 1.f / ln : 0.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) y[e] *= inv;
            const int64_t at = ((int64_t)b * a.H + h) * N + row;
            if (a.lse != nullptr && cc == 0) a.lse[at] = ls > 0.f ? (mx + log2f(ls)) * 0.69314718055994531f : 0.f;
            if (a.o_f32 != nullptr) {
                float4* dst = reinterpret_cast<float4*>(a.o_f32 + at * D + cc);
                dst[0] = make_float4(y[0], y[1], y[2], y[3]);
                dst[1] = make_float4(y[4], y[5], y[6], y[7]);
            }
            *reinterpret_cast<uint4*>(a.o + b * a.so.sb + h * a.so.sh + (int64_t)row * a.so.sn + cc) = float8_to_bf16x8(y);
        }
        return;
    }
    const float inv[2] = {lr[0] > 0.f ? 1.f / lr[0] : 0.f, lr[1] > 0.f ? 1.f / lr[1] : 0.f};
    const int row_g[2] = {I * USV_BLOCK + warp * 16 + g, I * USV_BLOCK + warp * 16 + g + 8};

    if (a.lse != nullptr && tig == 0) {
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (row_g[r] < N)
                a.lse[((int64_t)b * a.H + h) * N + row_g[r]] =
                    l[r] > 0.f ? (m[r] + log2f(l[r])) * 0.69314718055994531f : 0.f;
    }
    if (a.o_f32 != nullptr) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (row_g[r] >= N) continue;
            float* dst = a.o_f32 + (((int64_t)b * a.H + h) * N + row_g[r]) * D + 2 * tig;
#pragma unroll
            for (int n = 0; n < NT; ++n)
                *reinterpret_cast<float2*>(dst + n * 8) =
                    make_float2(o[n][2 * r] * inv[r], o[n][2 * r + 1] * inv[r]);
        }
    }
    // bf16 output through this warp's own rows of the (now idle) Q tile for 16-byte stores
    __syncthreads();  // all warps are done reading Q fragments and K/V tiles
    __nv_bfloat16* stage = Qs + (warp * 16) * LD;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
        *reinterpret_cast<uint32_t*>(stage + g * LD + n * 8 + 2 * tig) =
            pack_bf16x2(o[n][0] * inv[0], o[n][1] * inv[0]);
        *reinterpret_cast<uint32_t*>(stage + (g + 8) * LD + n * 8 + 2 * tig) =
            pack_bf16x2(o[n][2] * inv[1], o[n][3] * inv[1]);
    }
    __syncwarp();
    __nv_bfloat16* O = a.o + b * a.so.sb + h * a.so.sh;
    constexpr int VPR = D / 8;
    for (int idx = lane; idx < 16 * VPR; idx += 32) {
        const int r = idx / VPR, cc = idx % VPR;
        const int row = I * USV_BLOCK + warp * 16 + r;
        if (row < N)
            *reinterpret_cast<uint4*>(O + (int64_t)row * a.so.sn + cc * 8) =
                *reinterpret_cast<const uint4*>(stage + r * LD + cc * 8);
    }
}

// One CTA per query block, or a fixed grid whose CTAs walk a device-side work list or take every gridDim-th
// block's flag.
template <int D, bool FLAGS>
__global__ void __launch_bounds__(128) attn_mma_kernel(const AttnArgs a) {
    dep_sync();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (FLAGS) {
        const int blocks = a.B * a.H * a.NB;
        if (blockIdx.x == 0) {   // how many there are
            __shared__ int s_count;
            if (threadIdx.x == 0) s_count = 0;
            __syncthreads();
            int count = 0;
#pragma unroll 4
            for (int i = threadIdx.x; i < blocks / 8; i += 128) {
                const uint4 f = reinterpret_cast<const uint4*>(a.work_flags)[i];
                const uint32_t w[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) count += ((w[e] & 0xffffu) != 0) + ((w[e] >> 16) != 0);
            }
            if (threadIdx.x < blocks % 8) count += a.work_flags[blocks / 8 * 8 + threadIdx.x] != 0;
            if (count) atomicAdd(&s_count, count);
            __syncthreads();
            if (threadIdx.x == 0) *a.fallback_count = s_count;
        }
        const int stride = gridDim.x;
        for (int i0 = blockIdx.x; i0 < blocks; i0 += 128 * stride) {
            const int64_t mine = i0 + (int64_t)threadIdx.x * stride;
            if (!__syncthreads_or(mine < blocks && a.work_flags[mine] != 0)) continue;
            for (int64_t i = i0; i < blocks && i < i0 + 128 * (int64_t)stride; i += stride)
                if (a.work_flags[i] != 0) {
                    attn_mma_block<D, 1, 2>(a, (int)i, smem_raw);
                    __syncthreads();
                }
        }
        return;
    }
    if (a.work_list == nullptr) {
        // the words behind the sticky status word (fallback count, work counter, ...) start at zero
        if (blockIdx.x == 0 && threadIdx.x < (WS_HEADER - 4) / 4) a.status[1 + threadIdx.x] = 0u;
        attn_mma_block<D, 1, 2>(a, blockIdx.x, smem_raw);
        return;
    }
    const int n = *a.work_count;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        attn_mma_block<D, 1, 2>(a, a.work_list[i], smem_raw);
        __syncthreads();
    }
}

// One CTA per query block, G groups, lists of five to ten blocks.  A call of few blocks takes as long as one walk over a list:
// loads, two short chains of MMAs and the softmax between them, 1.3 us a key block at D = 64; G of them run side by side.
template <int D, int G, int NBUF>
__global__ void __launch_bounds__(128 * G) attn_split_kernel(const AttnArgs a) {
    dep_sync();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (blockIdx.x == 0 && threadIdx.x < (WS_HEADER - 4) / 4) a.status[1 + threadIdx.x] = 0u;   // (as attn_mma_kernel does)
    attn_mma_block<D, G, NBUF>(a, blockIdx.x, smem_raw);
}

int launch_attn_split(const AttnArgs& a, cudaStream_t st) {
    constexpr int D = 64, G = 4, NBUF = 2;
    constexpr size_t smem = (size_t)MmaSmem<D>::TILE * (1 + 2 * G * NBUF) * sizeof(__nv_bfloat16) + G * 192 * sizeof(float);
    static_assert(smem <= 232448, "shared memory budget");
    cudaError_t e = cudaFuncSetAttribute(attn_split_kernel<D, G, NBUF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "sparse_attn: smem attribute: %s", cudaGetErrorString(e));
    launch_dep_smem(attn_split_kernel<D, G, NBUF>, dim3((unsigned)(a.B * a.H * a.NB)), dim3(128 * G), smem, st, a);
    USV_CHECK_LAUNCH("attn_split_kernel");
    return USV_OK;
}

// Lists of up to four blocks where every query block has an SM to itself, one CTA per query block, four groups of 4 warps: group
// i loads entry i and takes its logits and, when the four maxima of a row are known, its weights, which every group
// then multiplies with a quarter of V's columns.  Maxima, sums and products come in the order of the list, so the result is that
// of attn_mma_block bit for bit.  Bound: the chain launch, loads, MMAs and the softmax between them, and 0.85 us an entry for its
// MMAs.  Calls at D = 64, us, one group / groups with maxima of their own / this kernel: 32 blocks, keep 4 8.3 / 7.3 / 7.0; 128, keep
// 2 7.0 / 5.8 / 5.2, keep 4 10.7 / 7.4 / 7.1; 40, keep 3 7.3 / 6.45 / 6.15.  (Several rounds of four entries, with all groups waiting for
// one another in each, take longer than groups of their own: 128 blocks, keep 8 11.9 / 9.9.)
template <int D, bool LSE>
struct FourSmem {
    static constexpr int TILE = MmaSmem<D>::TILE, G = 4;
    static constexpr size_t TILES = (size_t)TILE * (1 + 2 * G) * sizeof(__nv_bfloat16);   // Q, K and V; P takes the place of K
    static constexpr size_t MAXIMA = G * USV_BLOCK * sizeof(float);
    static constexpr size_t SUMS = LSE ? (size_t)G * 8 * USV_BLOCK * 4 * sizeof(float) : 0;   // unrounded pairs, for the log-sum-exp
    // More than half of an SM's, so that no two CTAs share one while others idle (a layer of 8 heads x 15 blocks 14.5 us with 85 KB, 12.2
    // so: CTAs may start where the kernel before has already left).
    static constexpr size_t ALONE = 118 * 1024;
    static constexpr size_t BYTES = TILES + MAXIMA + SUMS > ALONE ? TILES + MAXIMA + SUMS : ALONE;
};

template <int D, bool LSE>
__global__ void __launch_bounds__(512) attn_four_kernel(const AttnArgs a) {
    dep_sync();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using F = FourSmem<D, LSE>;
    constexpr int LD = MmaSmem<D>::LD, TILE = F::TILE, G = F::G;
    constexpr int NC = D / G / 8;   // n-tiles of the output a group has
    static_assert(NC == 2, "one ldmatrix of V per k-step");
    if (blockIdx.x == 0 && threadIdx.x < (WS_HEADER - 4) / 4) a.status[1 + threadIdx.x] = 0u;   // (as attn_mma_kernel does)
    __nv_bfloat16* Qs = reinterpret_cast<__nv_bfloat16*>(smem_raw);
    auto k_tile = [&](int grp) { return Qs + TILE * (1 + 2 * grp); };   // V behind it
    float* s_max = reinterpret_cast<float*>(smem_raw + F::TILES);                 // [G][64]
    float* s_sum = reinterpret_cast<float*>(smem_raw + F::TILES + F::MAXIMA);     // [G][8][64][4]

    const int I = blockIdx.x % a.NB, bh_ord = blockIdx.x / a.NB;
    const int b = bh_ord / a.H, h = a.head_order[bh_ord % a.H];
    const int kh = a.k_per_head[h], N = a.N;
    const int32_t* sel = a.sel + (((int64_t)b * a.H + h) * a.NB + I) * a.kmax;
    const __nv_bfloat16* K = a.k + b * a.sk.sb + h * a.sk.sh;
    const __nv_bfloat16* V = a.v + b * a.sv.sb + h * a.sv.sh;
    const int grp = threadIdx.x >> 7, warp = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;

    // the group's entry: the grp-th of the valid ones
    const int e_lane = lane < kh ? sel[lane] : -1;
    const unsigned valid = __ballot_sync(0xffffffffu, e_lane >= 0);
    const int entries = __popc(valid);   // at most G
    const unsigned here = __ballot_sync(0xffffffffu, e_lane >= 0 && __popc(valid & ((1u << lane) - 1u)) == grp);
    const int J = __shfl_sync(0xffffffffu, e_lane, here ? __ffs(here) - 1 : 0);
    load_tile<D, G>(Qs, a.q + b * a.sq.sb + h * a.sq.sh, a.sq.sn, I * USV_BLOCK, N);
    if (grp < entries) load_tile<D>(k_tile(grp), K, a.sk.sn, J * USV_BLOCK, N);
    cp_async_commit();
    if (grp < entries) load_tile<D>(k_tile(grp) + TILE, V, a.sv.sn, J * USV_BLOCK, N);
    cp_async_commit();
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");   // Q and K
    __syncthreads();

    uint32_t qf[D / 16][4];
    float o[NC][4] = {};
    float m[2] = {-INFINITY, -INFINITY};   // (as in attn_mma_block)
    // Of the sums over a row's weights each group takes one: of the rounded ones of rows g (0) and g + 8 (1), of the others (2, 3).
    const int own = grp & 1;
    float sum = 0.f;
    const float c = a.scale_log2;
    const int row = warp * 16 + g;
    load_q_frags<D>(qf, Qs, warp, lane);
    float s[8][4];
    if (grp < entries) {
        float mx[2];
        tile_logits<D>(s, mx, qf, k_tile(grp), N - J * USV_BLOCK, lane);
        if (tig < 2) s_max[grp * USV_BLOCK + row + 8 * tig] = tig ? mx[1] : mx[0];
    }
    __syncthreads();
    float ms[2] = {-INFINITY, -INFINITY};   // the running maxima at the group's entry
#pragma unroll
    for (int t = 0; t < G; ++t)
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (t <= grp && t < entries) ms[r] = fmaxf(ms[r], s_max[t * USV_BLOCK + row + 8 * r] * c);
#pragma unroll
    for (int r = 0; r < 2; ++r) ms[r] = ms[r] == -INFINITY ? 0.f : ms[r];
    if (grp < entries) {
        uint32_t pf[4][4];
        float* sums = s_sum + grp * (8 * USV_BLOCK * 4) + row * 4 + tig;
        tile_weights(s, c, ms, pf, [&](int nt, int r, float e, uint32_t) {
            if (LSE) sums[nt * (USV_BLOCK * 4) + r * 32] = e;
        });
        __nv_bfloat16* P = k_tile(grp) + row * LD + 2 * tig;   // (nobody reads the K tile any more)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
            for (int r = 0; r < 2; ++r)
                *reinterpret_cast<uint32_t*>(P + 8 * r * LD + nt * 8) = pf[nt >> 1][(nt & 1) * 2 + r];
    }
    cp_async_wait_all();   // V
    __syncthreads();
#pragma unroll 4
    for (int t = 0; t < entries; ++t) {
        float alpha[2], at;   // (taken here and not for all entries beforehand: the layer of 2 x 16 blocks 12.05 us, 12.45 so)
#pragma unroll
        for (int r = 0; r < 2; ++r) alpha[r] = next_max(m[r], s_max[t * USV_BLOCK + row + 8 * r], c, at);
        const __nv_bfloat16* prow = k_tile(t) + (warp * 16 + (lane & 15)) * LD + (lane >> 4) * 8;
        const __nv_bfloat16* vrow = k_tile(t) + TILE + (lane & 15) * LD + grp * (8 * NC) + (lane >> 4) * 8;
#pragma unroll
        for (int i = 0; i < NC; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[i][e] *= alpha[e >> 1];
#pragma unroll
        for (int kt = 0; kt < 4; ++kt) {
            uint32_t pf[4], bfr[4];
            ldmatrix_x4(pf, prow + kt * 16);
            ldmatrix_x4_trans(bfr, vrow + kt * 16 * LD);
            mma_bf16_16816(o[0], pf, bfr[0], bfr[1]);
            mma_bf16_16816(o[1], pf, bfr[2], bfr[3]);
            if (grp < 2) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {   // 8-key piece 2 kt + e
                    const float w = sum_bf16x2(own ? pf[2 * e + 1] : pf[2 * e]);
                    sum = kt == 0 && e == 0 ? fmaf(sum, own ? alpha[1] : alpha[0], w) : sum + w;
                }
            }
        }
        if (LSE && grp >= 2) {
            const float* sums = s_sum + t * (8 * USV_BLOCK * 4) + (row + 8 * own) * 4 + tig;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                const float e = sums[nt * (USV_BLOCK * 4)];
                sum = nt == 0 ? fmaf(sum, own ? alpha[1] : alpha[0], e) : sum + e;
            }
        }
    }

    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    if (tig == 0 && grp < 2) s_max[grp * USV_BLOCK + row] = sum;   // (nobody reads the maxima any more)
    if (LSE && tig == 0 && grp >= 2) {
        const int at = I * USV_BLOCK + row + 8 * own;
        if (at < N) a.lse[((int64_t)b * a.H + h) * N + at] = sum > 0.f ? ((own ? m[1] : m[0]) + log2f(sum)) * 0.69314718055994531f : 0.f;
    }
    __syncthreads();
    // the group's columns, the bf16 ones through the (now idle) Q tile for 16-byte stores
    __nv_bfloat16* stage = Qs + warp * 16 * LD + grp * (8 * NC);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const float lr = s_max[r * USV_BLOCK + row], inv = lr > 0.f ? 1.f / lr : 0.f;
        const int at = I * USV_BLOCK + row + 8 * r;
        const int64_t at_bh = ((int64_t)b * a.H + h) * N + at;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const float y0 = o[i][2 * r] * inv, y1 = o[i][2 * r + 1] * inv;
            if (a.o_f32 != nullptr && at < N)
                *reinterpret_cast<float2*>(a.o_f32 + at_bh * D + grp * (8 * NC) + i * 8 + 2 * tig) = make_float2(y0, y1);
            *reinterpret_cast<uint32_t*>(stage + (g + 8 * r) * LD + i * 8 + 2 * tig) = pack_bf16x2(y0, y1);
        }
    }
    __syncwarp();
    const int out_row = I * USV_BLOCK + warp * 16 + (lane >> 1);
    if (out_row < N)
        *reinterpret_cast<uint4*>(a.o + b * a.so.sb + h * a.so.sh + (int64_t)out_row * a.so.sn + grp * (8 * NC) + (lane & 1) * 8) =
            *reinterpret_cast<const uint4*>(stage + (lane >> 1) * LD + (lane & 1) * 8);
}

template <int D, bool LSE>
static int launch_four(const AttnArgs& a, cudaStream_t st) {
    constexpr size_t smem = FourSmem<D, LSE>::BYTES;
    static_assert(smem <= 232448, "shared memory budget");
    cudaError_t e = cudaFuncSetAttribute(attn_four_kernel<D, LSE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "sparse_attn: smem attribute: %s", cudaGetErrorString(e));
    launch_dep_smem(attn_four_kernel<D, LSE>, dim3((unsigned)(a.B * a.H * a.NB)), dim3(512), smem, st, a);
    USV_CHECK_LAUNCH("attn_four_kernel");
    return USV_OK;
}

int launch_attn_four(const AttnArgs& a, cudaStream_t st) {
    return a.lse != nullptr ? launch_four<64, true>(a, st) : launch_four<64, false>(a, st);
}

// Lists of one block: nothing follows the first K and V tile, and without a second buffer twice as many CTAs share an SM.
template <int D>
__global__ void __launch_bounds__(128, 4) attn_one_kernel(const AttnArgs a) {
    dep_sync();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (blockIdx.x == 0 && threadIdx.x < (WS_HEADER - 4) / 4) a.status[1 + threadIdx.x] = 0u;   // (as attn_mma_kernel does)
    attn_mma_block<D, 1, 1>(a, blockIdx.x, smem_raw);
}

int launch_attn_one(const AttnArgs& a, cudaStream_t st) {
    constexpr size_t smem = (size_t)MmaSmem<64>::TILE * 3 * sizeof(__nv_bfloat16);
    static_assert(smem <= 48 * 1024, "no attribute needed");
    const int64_t blocks = (int64_t)a.B * a.H * a.NB;
    if (blocks > 2147483647LL) return fail(USV_ERR_UNSUPPORTED, "sparse_attn: too many query blocks");
    launch_dep_smem(attn_one_kernel<64>, dim3((unsigned)blocks), dim3(128), smem, st, a);
    USV_CHECK_LAUNCH("attn_one_kernel");
    return USV_OK;
}

int launch_attn_mma(const AttnArgs& a, int d, cudaStream_t st) {
    int64_t grid = (int64_t)a.B * a.H * a.NB;
    if (grid > 2147483647LL) return fail(USV_ERR_UNSUPPORTED, "sparse_attn: too many query blocks");
    if ((a.work_list != nullptr || a.work_flags != nullptr) && grid > 296) grid = 296;
    auto launch = [&](auto kernel, size_t smem) {
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        launch_dep_smem(kernel, dim3((unsigned)grid), dim3(128), smem, st, a);
    };
    const bool flags = a.work_flags != nullptr;
    if (d == 128) launch(flags ? attn_mma_kernel<128, true> : attn_mma_kernel<128, false>, MmaSmem<128>::BYTES);
    else launch(flags ? attn_mma_kernel<64, true> : attn_mma_kernel<64, false>, MmaSmem<64>::BYTES);
    USV_CHECK_LAUNCH("attn_mma_kernel");
    return USV_OK;
}

}  // namespace usv
