// Token merge / unmerge (Sec. 3.3 of the USV paper).
//
//   desc_kernel        Eq. 7-8   head-averaged, unit-normalised key descriptors (HBM stream)
//                                and the ascending list of source tokens of the partition (Eq. 6)
//   (usv_match_tc.cu)  Eq. 8-9   cosine of every source against every destination of its batch
//                                element with a fused row arg-max, on the tensor cores
//   match_local_kernel           the same inside a window of partition blocks (fp32 CUDA cores)
//   plan_select_kernel Eq. 10         radix-select of the r-th most confident source
//   plan_assign_kernel Eq. 11, 14     ordered compaction, dst_of / pos
//                                and the lists of merged sources per destination (Eq. 12)
//   plan_held_kernel             both in one launch, by source counts
//   merge_kernel       Eq. 13-14 warp-per-row gather + mean, 16-byte accesses
//   unmerge_kernel     Eq. 15    warp-per-row gather copy, 16-byte accesses
#include <cuda_fp16.h>
#include <math.h>

#include "usv_match.cuh"

namespace usv {

// ---------------------------------------------------------------------------- descriptors
// HBM stream, one warp per token.  DM/8 lanes cover one head's row with 16-byte loads; 32/(DM/8) heads
// are read in parallel and combined with shuffles.  Besides the fp32 descriptors the warp writes what
// it has at hand without another pass: the tokens of the sources by rank, and for the tensor-core
// matcher (m.a_h != NULL) the fp16 rows of sources and destinations.  (Kernels of their own for those
// took 17 us at 32 760 tokens, 86 us at 2 x 118 800.  One warp per partition block, which could also
// compare sources with their destination, left too few loads in flight: 432 us at 2 x 118 800, 270 us
// this way.)  It also clears what later kernels count in: `zero` (zero_words words), exact_count.
template <int DM>
__global__ void __launch_bounds__(256) desc_kernel(const __nv_bfloat16* __restrict__ metric,
                                                   float* __restrict__ mhat, int Hm,
                                                   int32_t* __restrict__ src_idx, int32_t* __restrict__ zero,
                                                   int64_t zero_words, const MatchTcArgs m) {
    dep_sync();
    constexpr int LPH = DM / 8;    // lanes per head row
    constexpr int HPW = 32 / LPH;  // heads handled at once
    if (blockIdx.y == 0) {
        for (int64_t w = (int64_t)blockIdx.x * 256 + threadIdx.x; w < zero_words; w += (int64_t)gridDim.x * 256) zero[w] = 0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && m.a_h != nullptr) m.exact_count[blockIdx.y] = 0;
    const int b = blockIdx.y, n = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int chunk = lane % LPH, hsub = lane / LPH;
    if (n >= m.N) {
        // the rows that pad sources and destinations to multiples of 128
        const int i = n - m.N, pa = m.nA_pad - m.nA;
        if (m.a_h == nullptr || i >= pa + m.nB_pad - m.p.nB || hsub != 0) return;
        uint16_t* row = i < pa ? m.a_h + ((int64_t)b * m.nA_pad + m.nA + i) * DM
                               : m.b_h + ((int64_t)b * m.nB_pad + m.p.nB + i - pa) * DM;
        *reinterpret_cast<uint4*>(row + chunk * 8) = make_uint4(0, 0, 0, 0);
        return;
    }
    const int64_t tok = (int64_t)b * m.N + n;
    const __nv_bfloat16* src = metric + tok * Hm * DM + chunk * 8;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int h = hsub; h < Hm; h += HPW) {
        float f[8];
        bf16x8_to_float(__ldg(reinterpret_cast<const uint4*>(src + (int64_t)h * DM)), f);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] += f[e];
    }
#pragma unroll
    for (int o = LPH; o < 32; o <<= 1)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    float n2 = 0.f;
    const float invH = 1.0f / (float)Hm;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        acc[e] *= invH;
        n2 = fmaf(acc[e], acc[e], n2);
    }
#pragma unroll
    for (int o = 1; o < LPH; o <<= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
    const float inv = 1.0f / fmaxf(sqrtf(n2), 1e-12f);
    if (hsub != 0) return;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] *= inv;
    float* dst = mhat + tok * DM + chunk * 8;
    *reinterpret_cast<float4*>(dst) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    *reinterpret_cast<float4*>(dst + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
    int at;
    const bool is_dst = m.p.place(n, at);
    if (!is_dst && b == 0 && lane == 0) src_idx[at] = n;
    if (m.a_h == nullptr) return;
    uint16_t* row = is_dst ? m.b_h + ((int64_t)b * m.nB_pad + at) * DM : m.a_h + ((int64_t)b * m.nA_pad + at) * DM;
    struct alignas(16) { __half2 h[4]; } out;
#pragma unroll
    for (int e = 0; e < 4; ++e) out.h[e] = __floats2half2_rn(acc[2 * e], acc[2 * e + 1]);
    *reinterpret_cast<decltype(out)*>(row + chunk * 8) = out;
}

// ---------------------------------------------------------------------------- block scan (1024)
__device__ __forceinline__ int block_scan_1024(int v, int* scratch, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int incl = warp_incl_scan(v);
    if (lane == 31) scratch[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int w = scratch[lane];
        const int wi = warp_incl_scan(w);
        scratch[lane] = wi - w;
        if (lane == 31) scratch[32] = wi;
    }
    __syncthreads();
    const int res = scratch[warp] + incl - v;
    *total = scratch[32];
    __syncthreads();
    return res;
}

// ---------------------------------------------------------------------------- merged-source lists
// The sources merged into every destination, built by one atomic per source while the plan is
// written: the first SLOTS of a destination (in order of arrival, merge_kernel sorts them) sit in a
// 32-byte row of their own, further ones hang on a chain.  Counting, scanning and filling a CSR
// took three more kernels (13 us at 32 760 tokens, launches included) and left merge_kernel one
// more dependent load per row.
struct MergeLists {
    static constexpr int SLOTS = 8;
    int nB;              // destinations per batch element
    int32_t* cnt;        // [B,nB] sources of the destination, starts at zero
    int32_t* head;       // [B,nB] 1 + the last source chained (0: none), starts at zero
    int32_t* slots;      // [B,nB,SLOTS]
    int32_t* next;       // [B,N]  1 + the source chained before this one (0: none)
    int32_t* row_src;    // [B,nU] source token of every unmerged row
    int32_t* dst_copy;   // [B,N]  copy of dst_of inside a plan cache (NULL: not wanted)
    // source token n of batch element b (its tokens begin at token0) -> destination ordinal o; an ordinal that
    // does not exist (a stored plan of something else) writes nothing
    __device__ void push(int b, int o, int64_t token0, int n) const {
        if ((unsigned)o >= (unsigned)nB) return;
        const int64_t dst = (int64_t)b * nB + o;
        const int at = atomicAdd(cnt + dst, 1);
        if (at < SLOTS) slots[dst * SLOTS + at] = n;
        else next[token0 + n] = atomicExch(head + dst, n + 1);
    }
};

// ---------------------------------------------------------------------------- plan
// One CTA (1024 threads) per batch element.  Radix-select of the r-th largest u, then an ordered
// pass that marks the merged sources (ties to the lowest source index) and writes dst_of / pos.
// Key T of the r-th most confident source and the number of sources equal to T that still merge
// (Eq. 10 with ties to the lowest index), for 0 < r < nA.  One CTA per batch element.
// The first HELD * 1024 keys stay in registers over the four passes, each of which would wait for the L2 again (13.5 -> 8 us at
// 20 691 sources, when this kernel still took them; see plan_held_kernel for the counts that it is left with).
template <int HELD>
__global__ void __launch_bounds__(1024) plan_select_kernel(int nA, int r, const float* __restrict__ u_s,
                                                           int2* __restrict__ tsel) {
    dep_sync();
    __shared__ int hist[256];
    __shared__ uint32_t s_prefix;
    __shared__ int s_remaining;
    const int b = blockIdx.x;
    const float* u = u_s + (int64_t)b * nA;
    uint32_t held[HELD];
#pragma unroll
    for (int i = 0; i < HELD; ++i) {
        const int a = threadIdx.x + 1024 * i;
        held[i] = a < nA ? float_key(u[a]) : 0u;
    }
    if (threadIdx.x == 0) {
        s_prefix = 0;
        s_remaining = r;
    }
    __syncthreads();
    for (int shift = 24; shift >= 0; shift -= 8) {
        if (threadIdx.x < 256) hist[threadIdx.x] = 0;
        __syncthreads();
        const uint32_t prefix = s_prefix;
        const uint32_t mask = shift == 24 ? 0u : (0xffffffffu << (shift + 8));
#pragma unroll
        for (int i = 0; i < HELD; ++i)
            if (threadIdx.x + 1024 * i < nA && (held[i] & mask) == prefix) atomicAdd(&hist[(held[i] >> shift) & 255], 1);
        for (int a = threadIdx.x + 1024 * HELD; a < nA; a += 1024) {
            const uint32_t key = float_key(u[a]);
            if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255], 1);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            const int remaining = s_remaining;
            int local[8], sum = 0;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                local[t] = hist[255 - (lane * 8 + t)];
                sum += local[t];
            }
            const int incl = warp_incl_scan(sum);
            int before = incl - sum;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                if (before < remaining && remaining <= before + local[t]) {
                    s_prefix = prefix | ((uint32_t)(255 - (lane * 8 + t)) << shift);
                    s_remaining = remaining - before;
                }
                before += local[t];
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) tsel[b] = make_int2((int)s_prefix, s_remaining);
}

// Sum over the CTA of one int per thread (1024 threads); `scratch` holds >= 33 ints.
__device__ __forceinline__ int block_sum_1024(int v, int* scratch) {
    int tot;
    block_scan_1024(v, scratch, &tot);
    return tot;
}

// dst_of / pos of the sources (ordered compaction of the unmerged ones, Eq. 11 and 14) and of the
// destinations.  CTA (c, b) owns the sources [1024 c, 1024 c + 1024) of batch element b; what
// it needs to know of the sources before its own (how many are above T, how many equal T) it
// counts itself, so the CTAs are independent.
__global__ void __launch_bounds__(1024) plan_assign_kernel(Part p, int N, int nA, int r, uint32_t T_imm, int need_imm,
                                                           const int2* __restrict__ tsel,
                                                           const int32_t* __restrict__ src_idx,
                                                           const int32_t* __restrict__ jstar_s,
                                                           const float* __restrict__ u_s,
                                                           int32_t* __restrict__ dst_of,
                                                           int32_t* __restrict__ pos,
                                                           float* __restrict__ u_out,
                                                           int32_t* __restrict__ jstar_out,
                                                           const MergeLists lists) {
    dep_sync();
    __shared__ int scratch[33];
    const int b = blockIdx.y;
    const float* u = u_s + (int64_t)b * nA;
    const int32_t* js = jstar_s + (int64_t)b * nA;
    int32_t* d_of = dst_of + (int64_t)b * N;
    int32_t* ps = pos + (int64_t)b * N;
    const int nU = nA - r;
    const uint32_t T = tsel != nullptr ? (uint32_t)tsel[b].x : T_imm;
    const int need_eq = tsel != nullptr ? tsel[b].y : need_imm;
    const int a0 = blockIdx.x * 1024;
    if (a0 < nA) {
        int gt_b = 0, eq_b = 0;
        if (r > 0 && r < nA) {   // otherwise every source, or none, merges: ranks follow from the index
            for (int a = threadIdx.x; a < a0; a += 1024) {
                const uint32_t key = float_key(u[a]);
                gt_b += key > T ? 1 : 0;
                eq_b += key == T ? 1 : 0;
            }
            gt_b = block_sum_1024(gt_b, scratch);
            eq_b = block_sum_1024(eq_b, scratch);
        } else if (r == nA) {
            gt_b = a0;
        }
        const int un_b = a0 - gt_b - min(eq_b, need_eq);   // unmerged sources before this CTA's
        const int a = a0 + threadIdx.x;
        const bool in = a < nA;
        const float ua = in ? u[a] : 0.f;
        const uint32_t key = in ? float_key(ua) : 0u;
        const int is_gt = (in && r > 0 && key > T) ? 1 : 0;
        const int is_eq = (in && r > 0 && key == T) ? 1 : 0;
        int tot;
        const int eq_rank = eq_b + block_scan_1024(is_eq, scratch, &tot);
        const int merged = is_gt | (is_eq && eq_rank < need_eq);
        const int un = (in && !merged) ? 1 : 0;
        const int un_rank = un_b + block_scan_1024(un, scratch, &tot);
        if (in) {
            const int n = src_idx[a];
            const int j = js[a];
            if (merged) {
                const int o = p.ord(j);
                d_of[n] = j;
                ps[n] = nU + o;
                lists.push(b, o, (int64_t)b * N, n);
            } else {
                d_of[n] = -1;
                ps[n] = un_rank;
                lists.row_src[(int64_t)b * nU + un_rank] = n;
            }
            if (u_out) u_out[(int64_t)b * N + n] = ua;
            if (jstar_out) jstar_out[(int64_t)b * N + n] = j;
        }
    }
    const int o = blockIdx.x * 1024 + threadIdx.x;
    if (o < p.nB) {
        const int n = p.dst_token(o);
        d_of[n] = -1;
        ps[n] = nU + o;
        if (u_out) u_out[(int64_t)b * N + n] = __int_as_float(0x7fc00000);
        if (jstar_out) jstar_out[(int64_t)b * N + n] = -1;
    }
}

// Both steps in one launch: the CTA, or the cluster of eight, of a batch element holds every key in registers, a warp 32 * PER
// consecutive ones, so that the ranks among the unmerged sources follow from ballots and sums over warps and CTAs.  Every CTA counts
// digits in its own shared memory, and one cluster barrier a pass later adds up all counts.  Bound: the chain of a launch, reads
// and barriers, and beyond about 50 000 sources the scattered stores and atomics of eight SMs.  Whole merges with two kernels /
// with this one, us.  One CTA: 96 sources 17.2 / 15.6, 2 x 1024 20.7 / 17.1, 840 with a matching of all destinations 46.5 / 42.5, 2880 20.6 /
// 18.8, but 4500 25.3 / 26.9, 7500 29.0 / 32.2.  Eight: 1024 20.4 / 24.0, 10 140 38.0 / 38.5, 15 210 44.9 / 41.8, 2 x 16 380 119.9 / 116.9,
// 4 x 24 570 181 / 176, 37 800 71.4 / 68.1, 65 480 136 / 123, 2 x 59 400 189 / 182, 2 x 88 440 216 / 191.
template <int CL, int PER>
__global__ void __launch_bounds__(1024) __cluster_dims__(CL, 1, 1)
plan_held_kernel(Part p, int N, int nA, int r, const int32_t* __restrict__ src_idx, const int32_t* __restrict__ jstar_s,
                 const float* __restrict__ u_s, int32_t* __restrict__ dst_of, int32_t* __restrict__ pos,
                 float* __restrict__ u_out, int32_t* __restrict__ jstar_out, const MergeLists lists) {
    __shared__ __align__(16) int s_hist[4][256];          // one a pass: peers may still read the one before
    __shared__ uint32_t s_prefix, s_total, s_warp[32];   // s_warp, s_total: (keys above T) << 16 | keys equal to T
    __shared__ int s_remaining;
    (&s_hist[0][0])[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        s_prefix = 0;
        s_remaining = r;
    }
    dep_sync();
    const int rank = blockIdx.x, b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float* u = u_s + (int64_t)b * nA;
    const int32_t* js = jstar_s + (int64_t)b * nA;
    int32_t* d_of = dst_of + (int64_t)b * N;
    int32_t* ps = pos + (int64_t)b * N;
    const int nU = nA - r;
    const int first = (rank * 32 + warp) * 32 * PER + lane;   // element i of the thread: first + 32 i
    constexpr int AHEAD = CL == 1 ? PER : 1;   // sources and destinations read before they are needed
    uint32_t key[PER];
    int src[AHEAD], to[AHEAD];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int a = first + 32 * i;
        const bool in = a < nA;
        key[i] = in ? float_key(u[a]) : 0u;
        if (CL == 1) {
            src[i] = in ? src_idx[a] : 0;
            to[i] = in ? js[a] : 0;
        }
    }
    for (int o = rank * 1024 + threadIdx.x; o < p.nB; o += CL * 1024) {
        const int n = p.dst_token(o);
        d_of[n] = -1;
        ps[n] = nU + o;
        if (u_out) u_out[(int64_t)b * N + n] = __int_as_float(0x7fc00000);
        if (jstar_out) jstar_out[(int64_t)b * N + n] = -1;
    }
    auto peer = [](const void* at, int cta) {
        uint32_t to;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"((uint32_t)__cvta_generic_to_shared(at)), "r"(cta));
        return to;
    };
    __syncthreads();
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        const uint32_t prefix = s_prefix, mask = pass == 0 ? 0u : (0xffffffffu << (shift + 8));
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (first + 32 * i < nA && (key[i] & mask) == prefix) atomicAdd(&s_hist[pass][(key[i] >> shift) & 255], 1);
        if (CL > 1) {
            __syncwarp();
            asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        } else {
            __syncthreads();
        }
        if (warp == 0) {
            const int remaining = s_remaining;
            int local[8] = {0, 0, 0, 0, 0, 0, 0, 0}, sum = 0;   // bins 248 - 8 lane and up, of all CTAs
#pragma unroll
            for (int c = 0; c < CL; ++c) {
                int v[8];
                const int* at = &s_hist[pass][248 - 8 * lane];
                if (CL > 1) {
                    const uint32_t far = peer(at, c);
                    asm volatile("ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(far) : "memory");
                    asm volatile("ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(far + 16) : "memory");
                }
#pragma unroll
                for (int t = 0; t < 8; ++t) local[t] += CL > 1 ? v[t] : at[t];
            }
#pragma unroll
            for (int t = 0; t < 8; ++t) sum += local[t];
            int before = warp_incl_scan(sum) - sum;
#pragma unroll
            for (int t = 7; t >= 0; --t) {
                if (before < remaining && remaining <= before + local[t]) {
                    s_prefix = prefix | ((uint32_t)(248 - 8 * lane + t) << shift);
                    s_remaining = remaining - before;
                }
                before += local[t];
            }
        }
        __syncthreads();
    }
    const uint32_t T = s_prefix;
    const int need_eq = s_remaining;
    uint32_t gt[PER], eq[PER];
    int n_gt = 0, n_eq = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const bool in = first + 32 * i < nA;
        gt[i] = __ballot_sync(0xffffffffu, in && key[i] > T);
        eq[i] = __ballot_sync(0xffffffffu, in && key[i] == T);
        n_gt += __popc(gt[i]);
        n_eq += __popc(eq[i]);
    }
    if (lane == 0) s_warp[warp] = (uint32_t)n_gt << 16 | (uint32_t)n_eq;
    __syncthreads();
    const uint32_t mine = s_warp[lane];
    const uint32_t ahead = __reduce_add_sync(0xffffffffu, lane < warp ? mine : 0u);
    int gt_b = (int)(ahead >> 16), eq_b = (int)(ahead & 0xffffu);
    if (CL > 1) {   // what the CTAs before hold
        const uint32_t total = __reduce_add_sync(0xffffffffu, mine);
        if (threadIdx.x == 0) s_total = total;
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        uint32_t other = 0;
        if (lane < rank) asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(other) : "r"(peer(&s_total, lane)) : "memory");
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // (nobody leaves while a peer may read)
        gt_b += (int)__reduce_add_sync(0xffffffffu, other >> 16);
        eq_b += (int)__reduce_add_sync(0xffffffffu, other & 0xffffu);
    }
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int a = first + 32 * i;
        const int g = gt_b + __popc(gt[i] & below), e = eq_b + __popc(eq[i] & below);
        gt_b += __popc(gt[i]);
        eq_b += __popc(eq[i]);
        if (a >= nA) continue;
        const int n = CL == 1 ? src[CL == 1 ? i : 0] : src_idx[a], j = CL == 1 ? to[CL == 1 ? i : 0] : js[a];
        if (key[i] > T || (key[i] == T && e < need_eq)) {
            const int o = p.ord(j);
            d_of[n] = j;
            ps[n] = nU + o;
            lists.push(b, o, (int64_t)b * N, n);
        } else {
            const int un_rank = a - g - min(e, need_eq);
            d_of[n] = -1;
            ps[n] = un_rank;
            lists.row_src[(int64_t)b * nU + un_rank] = n;
        }
        if (u_out) u_out[(int64_t)b * N + n] = u[a];
        if (jstar_out) jstar_out[(int64_t)b * N + n] = j;
    }
    if (CL > 1) {
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// The same lists from a stored plan.  cnt and head start at zero.
__global__ void __launch_bounds__(256) plan_lists_kernel(Part p, int N, int nU,
                                                         const int32_t* __restrict__ dst_of,
                                                         const int32_t* __restrict__ pos,
                                                         const MergeLists lists) {
    dep_sync();
    const int b = blockIdx.y;
    const int n = blockIdx.x * 256 + threadIdx.x;
    if (n >= N) return;
    const int j = dst_of[(int64_t)b * N + n];
    if (lists.dst_copy != nullptr) lists.dst_copy[(int64_t)b * N + n] = j;
    if (j >= 0) lists.push(b, p.ord(j), (int64_t)b * N, n);
    else if (!p.is_dst(n)) lists.row_src[(int64_t)b * nU + pos[(int64_t)b * N + n]] = n;
}

// Exclusive scan of cnt[b,:] -> off[b,0..nB], cursor[b,:] = off[b,:nB] (unmerge map).  CTA (c, b) owns the
// rows [1024 c, 1024 c + 1024) and sums the counts before its own itself.
__global__ void __launch_bounds__(1024) row_scan_kernel(int nB, const int32_t* __restrict__ cnt,
                                                        int32_t* __restrict__ off,
                                                        int32_t* __restrict__ cursor) {
    dep_sync();
    __shared__ int scratch[33];
    const int b = blockIdx.y;
    const int o0 = blockIdx.x * 1024;
    int before = 0;
    for (int o = threadIdx.x; o < o0; o += 1024) before += cnt[(int64_t)b * nB + o];
    int tot;
    block_scan_1024(before, scratch, &tot);
    const int base = tot;
    const int o = o0 + threadIdx.x;
    const int c = o < nB ? cnt[(int64_t)b * nB + o] : 0;
    const int e = base + block_scan_1024(c, scratch, &tot);
    if (o < nB) {
        off[(int64_t)b * (nB + 1) + o] = e;
        cursor[(int64_t)b * nB + o] = e;
    }
    if (o0 + 1024 >= nB && threadIdx.x == 0) off[(int64_t)b * (nB + 1) + nB] = base + tot;
}

// ---------------------------------------------------------------------------- local matching
// The other reading of Sec. 3.3 (matching kept inside neighbouring 3D blocks): Eq. 8-9 with the
// arg-max over the destinations of the partition blocks within (wt, wh, ww) blocks of the
// source's own block; a later destination wins only when strictly better.  One warp per source, 32
// candidates in ascending order at a time: the lanes split the descriptors, all candidates' rows are
// requested before any is used, and the 32 sums over lanes are taken together (at every step a lane
// hands half of its candidates over: 31 shuffles, where one candidate after the other takes 160), which
// leaves candidate l in lane l.  Rows of three destinations (the window reaches one block along x) are asked for from one address a
// row, 30 candidates at a time.  Bound: the L1's data pipe, which the shuffles go through too (71 % busy), and the latency behind it
// (half of a warp's wait is for loads, issue slots are 56 % busy; a third of the adds and shuffles less changed nothing).  2 x 16 380 sources, 27 candidates of 128: 73 -> 41 us (46 us without the bound on registers).
// A CTA goes through neighbouring sources, whose windows share most of their rows in L1, where there are several waves of
// them.  Whole merges, us, one source a warp / rows of three and several sources: 2 x 16 380 122 / 120, 4 x 24 570 196 / 181, 65 480
// 144 / 136, 8 x 17 550 239 / 224.  OWN: a window of the own block alone has one candidate and needs no registers for 32: 2 x 16 380
// 63.6 / 57.0, 37 800 78.5 / 71.6, 2 x 59 400 222 / 189, 138 000 206 / 165.
template <int DM, bool OWN>
__global__ void __launch_bounds__(256, OWN ? 6 : 3) match_local_kernel(const float* __restrict__ mhat, Part p, int N, int nA,
                                                          int wt, int wh, int ww,
                                                          const int32_t* __restrict__ src_idx,
                                                          int32_t* __restrict__ jstar_s, float* __restrict__ u_s) {
    dep_sync();
    constexpr int V = DM / 32;   // floats per lane
    struct alignas(4 * V) Vec { float f[V]; };
    const int per = (nA + (int)gridDim.x - 1) / (int)gridDim.x;   // consecutive sources of the CTA
    const int end = min(nA, ((int)blockIdx.x + 1) * per);
    int a = blockIdx.x * per + (threadIdx.x >> 5);
    if (a >= end) return;
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const float* mb = mhat + (int64_t)b * N * DM + lane * V;
    const int nBt = p.nB / (p.nHy * p.nWx);
    int i = src_idx[a];
    Vec mi = *reinterpret_cast<const Vec*>(mb + (int64_t)i * DM);
    for (; a < end; a += 8) {
        int t, y, x;
        p.coords(i, t, y, x);
        const int bt = p.dst.quot(t), by = p.dsh.quot(y), bx = p.dsw.quot(x);
        const int t0 = max(bt - wt, 0), y0 = max(by - wh, 0), x0 = max(bx - ww, 0);
        const int ny = min(by + wh, p.nHy - 1) - y0 + 1, nx = min(bx + ww, p.nWx - 1) - x0 + 1;
        const int64_t count = (int64_t)(min(bt + wt, nBt - 1) - t0 + 1) * ny * nx;   // (the block's own destination is among them)
        float best = -INFINITY;
        int jbest = ((bt * p.st) * p.Hh + by * p.sh) * p.W + bx * p.sw;   // no comparable cosine (NaN in the metric): its own block
        if (OWN || count == 1) {   // the window is its own block: one cosine, its products added in the same order
            const Vec mj = *reinterpret_cast<const Vec*>(mb + (int64_t)jbest * DM);
            float c = 0.f;
#pragma unroll
            for (int e = 0; e < V; ++e) c = fmaf(mi.f[e], mj.f[e], c);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            if (c > best) best = c;
        }
        const bool rows3 = nx == 3;   // rows of three: their candidates follow from one address a row
        const int step = rows3 ? 30 : 32, dx = p.sw * 32;
        for (int64_t k0 = 0; !OWN && k0 < count && count > 1; k0 += step) {
            const int n = (int)min((int64_t)step, count - k0);
            const int k = (int)k0 + min(lane, n - 1);
            const int row = k / nx, ct = row / ny;
            const int jk = (((t0 + ct) * p.st) * p.Hh + (y0 + row - ct * ny) * p.sh) * p.W + (x0 + k - row * nx) * p.sw;
            float c[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) c[q] = 0.f;
            if (rows3) {
#pragma unroll
                for (int q0 = 0; q0 < 30; q0 += 9) {
                    if (q0 >= n) continue;
                    Vec mj[9];
#pragma unroll
                    for (int q = 0; q < 9 && q0 + q < 30; q += 3) {
                        const Vec* at = reinterpret_cast<const Vec*>(mb + (int64_t)__shfl_sync(0xffffffffu, jk, min(q0 + q, n - 3)) * DM);   // (past n: the last row again)
                        mj[q] = at[0];
                        mj[q + 1] = at[dx];
                        mj[q + 2] = at[2 * dx];
                    }
#pragma unroll
                    for (int q = 0; q < 9 && q0 + q < 30; ++q)
#pragma unroll
                        for (int e = 0; e < V; ++e) c[q0 + q] = fmaf(mi.f[e], mj[q].f[e], c[q0 + q]);
                }
            } else {
#pragma unroll
                for (int q0 = 0; q0 < 32; q0 += 8) {
                    if (q0 >= n) continue;
                    Vec mj[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        mj[q] = *reinterpret_cast<const Vec*>(mb + (int64_t)__shfl_sync(0xffffffffu, jk, q0 + q) * DM);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
#pragma unroll
                        for (int e = 0; e < V; ++e) c[q0 + q] = fmaf(mi.f[e], mj[q].f[e], c[q0 + q]);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const bool up = lane & o;
#pragma unroll
                for (int q = 0; q < o; ++q) {
                    const float give = up ? c[q] : c[q + o], keep = up ? c[q + o] : c[q];
                    c[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            }
            const uint32_t key = lane < n && c[0] > -INFINITY ? float_key(c[0]) : 0u;   // NaN never wins
            const uint32_t top = __reduce_max_sync(0xffffffffu, key);
            const int w = __ffs(__ballot_sync(0xffffffffu, key == top)) - 1;
            const float cw = __shfl_sync(0xffffffffu, c[0], w);
            const int jw = __shfl_sync(0xffffffffu, jk, w);
            if (top != 0 && cw > best) { best = cw; jbest = jw; }
        }
        if (lane == 0) {
            jstar_s[(int64_t)b * nA + a] = jbest;
            u_s[(int64_t)b * nA + a] = best;
        }
        if (a + 8 >= end) return;
        i = src_idx[a + 8];
        mi = *reinterpret_cast<const Vec*>(mb + (int64_t)i * DM);
    }
}

// ---------------------------------------------------------------------------- merge
// Sum of rows (fp32, in the order they are added) at two 16-byte chunks per lane, c0 and c0 + 32 of nvec.
struct RowSum {
    static constexpr int ROWS = 4;   // in flight
    const __nv_bfloat16* xb;
    int C, c0, nvec;
    float acc[2][8];
    __device__ RowSum(const __nv_bfloat16* xb_, int C_, int c0_, int nvec_) : xb(xb_), C(C_), c0(c0_), nvec(nvec_) {
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[0][e] = acc[1][e] = -0.f;   // (-0 + x is x for every x)
    }
    // the rows of the tokens in lanes 0 .. n - 1 (whole warp)
    __device__ void add_rows(int tok, int n) {
        for (int s = 0; s < n; s += ROWS) {
            uint4 w[ROWS][2];
#pragma unroll
            for (int q = 0; q < ROWS; ++q)
                if (s + q < n) {
                    const uint4* src = reinterpret_cast<const uint4*>(xb + (int64_t)__shfl_sync(0xffffffffu, tok, s + q) * C);
#pragma unroll
                    for (int g = 0; g < 2; ++g)
                        w[q][g] = c0 + g * 32 < nvec ? __ldg(src + c0 + g * 32) : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
            for (int q = 0; q < ROWS; ++q)
                if (s + q < n) {
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        float f[8];
                        bf16x8_to_float(w[q][g], f);
#pragma unroll
                        for (int e = 0; e < 8; ++e) acc[g][e] += f[e];
                    }
                }
        }
    }
    __device__ void store(uint4* dst, float inv) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            if (c0 + g * 32 >= nvec) continue;
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[g][e] *= inv;
            dst[c0 + g * 32] = float8_to_bf16x8(acc[g]);
        }
    }
};

// A destination with more than 31 sources (flat regions of a picture give dozens to thousands), apart from the
// kernel so that its registers are not the kernel's.  Two ways to the sources in ascending order: the chain,
// collected into registers and ranked; or a pass over dst_of, 512 tokens at a time, for
// every 64 chunks of the row.  A step of the chain and of the pass both wait for the L2 once, but a pass fetches
// more: the chain is taken where it is shorter than twice the steps of all passes.  Either way 32 sources at a
// time go to the sum.  id: the first sources, in lanes 0 .. SLOTS - 1.
// Calls of a stored plan, us, list sorted in place by selection / dst_of walked 32 tokens at a time / this: 32 760
// tokens of 3 KB, longest list 46 128 / 904 / 107, 111 263 / 977 / 193, 410 946 / 2029 / 675, 4095 10 515 / 12 490 / 4616;
// 118 800 tokens of 6 KB, 56 378 / 6665 / 319, 223 1087 / 7019 / 748, 2930 12 970 / 22 250 / 7570.
__device__ __noinline__ void merge_long_row(const MergeLists& lists, const int32_t* dst_of, const __nv_bfloat16* xb, int N, int C,
                                            int b, int j, int64_t od, int len, int id, uint4* dst, float inv) {
    constexpr int CHAINED = 256, R = CHAINED / 32;
    const int lane = threadIdx.x & 31, nvec = C / 8;
    const bool chained = len <= CHAINED && (int64_t)(len - MergeLists::SLOTS) * 256 < (int64_t)((nvec + 63) / 64) * N;
    int ids[R], rank[R];   // source s in lane s % 32, register s / 32
    if (chained) {
        const int32_t* next = lists.next + (int64_t)b * N;
#pragma unroll
        for (int h = 0; h < R; ++h) { ids[h] = 0x7fffffff; rank[h] = 0; }
        if (lane < MergeLists::SLOTS) ids[0] = id;
        int n = lists.head[od];
#pragma unroll
        for (int h = 0; h < R; ++h)
            for (int q = h == 0 ? MergeLists::SLOTS : 0; q < 32 && 32 * h + q < len; ++q) {
                if (lane == q) ids[h] = n - 1;
                n = next[n - 1];
            }
#pragma unroll
        for (int g = 0; g < R; ++g)
            for (int q = 0; q < 32 && 32 * g + q < len; ++q) {
                const int other = __shfl_sync(0xffffffffu, ids[g], q);
#pragma unroll
                for (int h = 0; h < R; ++h) rank[h] += other < ids[h] ? 1 : 0;   // (empty places: rank len)
            }
    }
    for (int cb = 0; cb < nvec; cb += 64) {
        RowSum sum(xb, C, cb + lane, nvec);
        int tok = j, n = 1;    // tokens in lanes 0 .. n - 1 wait to be added: the destination, then the sources
        if (chained) {
            for (int s = 0; s < len; ++s) {
                int v = -1;
#pragma unroll
                for (int h = 0; h < R; ++h) v = rank[h] == s ? ids[h] : v;
                v = __reduce_max_sync(0xffffffffu, v);
                if (lane == n) tok = v;
                if (++n == 32) {
                    sum.add_rows(tok, 32);
                    n = 0;
                }
            }
        } else {
            for (int n0 = 0; n0 < N; n0 += 512) {
                uint32_t hits = 0;   // bit u: token n0 + 32 u + lane
#pragma unroll
                for (int u = 0; u < 16; ++u)
                    if (n0 + 32 * u + lane < N && dst_of[n0 + 32 * u + lane] == j) hits |= 1u << u;
                uint32_t any = __reduce_or_sync(0xffffffffu, hits);
                for (; any; any &= any - 1) {
                    const int u = __ffs(any) - 1;
                    for (unsigned found = __ballot_sync(0xffffffffu, (hits >> u) & 1u); found; found &= found - 1) {
                        if (lane == n) tok = n0 + 32 * u + __ffs(found) - 1;
                        if (++n == 32) {
                            sum.add_rows(tok, 32);
                            n = 0;
                        }
                    }
                }
            }
        }
        sum.add_rows(tok, n);
        sum.store(dst, inv);
    }
}

// HBM stream, one warp per output row.  Rows [0,nU) copy an unmerged source; rows [nU, nU+nB) hold a
// destination averaged with its merged sources, summed in ascending source index (fp32).  Most
// destinations have no more than two sources: their rows and the destination's are requested
// together, G 16-byte chunks a lane each, before any is used, and only one chunk's sums are live at a
// time.  Longer lists take RowSum::ROWS rows of two chunks at a time.  The destinations come first: a row with a
// long list takes several times a copy's time, and at the end of the grid it is all that runs.  Four
// warps a CTA, so that one long row keeps few others' registers.  Calls of a stored plan, us (256 threads,
// copies first, two rows at a time before; x the copy bandwidth of the device): 2 x 118 800 rows of 6 KB, a
// quarter merged: 393 -> 378 (1.03); 2 x 32 760 rows of 3 KB, 40 % merged: 62 -> 53 (0.93); 28 101 rows
// of 3 KB, blocks of 2 x 2, a quarter merged, up to ten sources a row: 42.6 -> 27.3 (0.85); 32 760 rows,
// blocks of 2 x 2 x 2, 40 %: 48 -> 29.  ROWS = 3 or 5, 6 or 8 CTAs an SM: within 5 % either way.
// Warps that stay and walk 1 KB segments, looking the next one's lists up ahead, were slower (96 us
// where 65).
__global__ void __launch_bounds__(128, 7) merge_kernel(Part p, int B, int N, int C, int nU, int Nm,
                                                       const __nv_bfloat16* __restrict__ x,
                                                       const MergeLists lists,
                                                       const int32_t* __restrict__ dst_of,
                                                       __nv_bfloat16* __restrict__ out) {
    dep_sync();
    const int64_t w = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (w >= (int64_t)B * Nm) return;
    const int lane = threadIdx.x & 31;
    // the destinations of all batch elements first, the plain copies last
    const bool is_copy = w >= (int64_t)B * p.nB;
    const int64_t wi = is_copy ? w - (int64_t)B * p.nB : w;
    const int per = is_copy ? nU : p.nB;
    const int b = B == 1 ? 0 : (wi >> 32 ? (int)(wi / per) : (int)((uint32_t)wi / (uint32_t)per));   // (64-bit division: 0.2 us)
    const int row = (int)(wi - (int64_t)b * per) + (is_copy ? 0 : nU);
    const int64_t gw = (int64_t)b * Nm + row;
    const __nv_bfloat16* xb = x + (int64_t)b * N * C;
    auto row_of = [&](int tok) { return reinterpret_cast<const uint4*>(xb + (int64_t)tok * C); };
    uint4* dst = reinterpret_cast<uint4*>(out + gw * C);
    const int nvec = C / 8;
    int len = 0, j, id = 0;
    const int64_t od = (int64_t)b * p.nB + row - nU;
    if (row < nU) {
        j = lists.row_src[(int64_t)b * nU + row];
    } else {
        j = p.dst_token(row - nU);
        len = lists.cnt[od];
        if (lane < MergeLists::SLOTS) id = lists.slots[od * MergeLists::SLOTS + lane];   // (asked for beside the count)
    }
    const uint4* srcj = row_of(j);
    if (len == 0) {
        for (int c = lane; c < nvec; c += 32) dst[c] = __ldg(srcj + c);
        return;
    }
    const float inv = 1.0f / (float)(len + 1);
    constexpr int G = 3;
    if (len <= 2) {
        int i0 = __shfl_sync(0xffffffffu, id, 0), i1 = len == 2 ? __shfl_sync(0xffffffffu, id, 1) : i0;
        const uint4 *src0 = row_of(min(i0, i1)), *src1 = row_of(max(i0, i1));
        for (int c0 = lane; c0 < nvec; c0 += 32 * G) {
            uint4 v[G], va[G], vb[G];
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (c0 + g * 32 < nvec) v[g] = __ldg(srcj + c0 + g * 32);
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (c0 + g * 32 < nvec) va[g] = __ldg(src0 + c0 + g * 32);
            if (len == 2) {
#pragma unroll
                for (int g = 0; g < G; ++g)
                    if (c0 + g * 32 < nvec) vb[g] = __ldg(src1 + c0 + g * 32);
            }
#pragma unroll
            for (int g = 0; g < G; ++g) {
                float acc[8], f[8];
                bf16x8_to_float(v[g], acc);
                bf16x8_to_float(va[g], f);
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] += f[e];
                if (len == 2) {
                    bf16x8_to_float(vb[g], f);
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[e] += f[e];
                }
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] *= inv;
                if (c0 + g * 32 < nvec) dst[c0 + g * 32] = float8_to_bf16x8(acc);
            }
        }
        return;
    }
    if (len > 31) {
        merge_long_row(lists, dst_of + (int64_t)b * N, xb, N, C, b, j, od, len, id, dst, inv);
        return;
    }
    // Lane 0 holds the destination's token, lane s + 1 the s-th smallest source.
    int myid = j;
    if (len > MergeLists::SLOTS) {
        int n = lists.head[od];
        for (int s = MergeLists::SLOTS; s < len; ++s) {
            if (lane == s) id = n - 1;
            n = lists.next[(int64_t)b * N + n - 1];
        }
    }
    if (lane >= len) id = 0x7fffffff;
    int rank = 0;
    for (int s = 0; s < len; ++s) rank += __shfl_sync(0xffffffffu, id, s) < id ? 1 : 0;
    // ids are distinct, so the ranks of the valid lanes are a permutation of 0..len-1
    for (int s = 0; s < len; ++s) {
        const int oid = __shfl_sync(0xffffffffu, id, s);
        const int orank = __shfl_sync(0xffffffffu, rank, s);
        if (orank + 1 == lane) myid = oid;
    }
    for (int cb = 0; cb < nvec; cb += 64) {   // (whole warps: the lanes hand the rows round)
        RowSum sum(xb, C, cb + lane, nvec);
        sum.add_rows(myid, len + 1);
        sum.store(dst, inv);
    }
}

static int launch_merge(const Part& p, int B, int N, int C, int nU, int Nm, const void* x, const MergeLists& lists,
                        const int32_t* dst_of, void* out, cudaStream_t st) {
    launch_dep(merge_kernel, dim3((unsigned)(((int64_t)B * Nm + 3) / 4)), dim3(128), 0, st, p, B, N, C, nU, Nm,
               static_cast<const __nv_bfloat16*>(x), lists, dst_of, static_cast<__nv_bfloat16*>(out));
    USV_CHECK_LAUNCH("merge_kernel");
    return USV_OK;
}

// ---------------------------------------------------------------------------- unmerge
__global__ void __launch_bounds__(256) unmerge_kernel(int N, int Nm, int C,
                                                      const __nv_bfloat16* __restrict__ ym,
                                                      const int32_t* __restrict__ pos,
                                                      __nv_bfloat16* __restrict__ y, int64_t rows) {
    dep_sync();
    const int64_t gw = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (gw >= rows) return;
    const int lane = threadIdx.x & 31;
    const int b = (int)(gw / N);
    const int pr = pos[gw];
    const uint4* src = reinterpret_cast<const uint4*>(ym + ((int64_t)b * Nm + pr) * C);
    uint4* dst = reinterpret_cast<uint4*>(y + gw * C);
    const int nvec = C / 8;
    for (int c = lane; c < nvec; c += 32) dst[c] = __ldg(src + c);
}

// ---------------------------------------------------------------------------- unmerge map
// Inverse of pos: for every merged row the original tokens that read it back (counting sort by
// merged row; the order inside a row is irrelevant, every token of a row receives the same values).
__global__ void __launch_bounds__(256) inv_count_kernel(int N, int Nm, const int32_t* __restrict__ pos,
                                                        int32_t* __restrict__ cnt) {
    dep_sync();
    const int b = blockIdx.y;
    const int n = blockIdx.x * 256 + threadIdx.x;
    if (n >= N) return;
    const int m = pos[(int64_t)b * N + n];
    if (m >= 0 && m < Nm) atomicAdd(&cnt[(int64_t)b * Nm + m], 1);
}

__global__ void __launch_bounds__(256) inv_fill_kernel(int N, int Nm, const int32_t* __restrict__ pos,
                                                       int32_t* __restrict__ cursor, int32_t* __restrict__ inv_idx) {
    dep_sync();
    const int b = blockIdx.y;
    const int n = blockIdx.x * 256 + threadIdx.x;
    if (n >= N) return;
    const int m = pos[(int64_t)b * N + n];
    if (m >= 0 && m < Nm) inv_idx[(int64_t)b * N + atomicAdd(&cursor[(int64_t)b * Nm + m], 1)] = n;
}

// ---------------------------------------------------------------------------- host side
struct MergeWs {
    size_t mhat, src_idx, jstar_s, u_s, row_src, cnt, head, slots, next, status, tsel, split, total;
};

static MergeWs merge_layout(int B, int N, int dm, int nA, int nB) {
    MergeWs w;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
    w.status = take(WS_HEADER);                                 // workspace header: word 0 = device status word
    w.mhat = take((size_t)B * N * (dm > 0 ? dm : 1) * sizeof(float));
    w.src_idx = take((size_t)nA * 4);
    w.jstar_s = take((size_t)B * nA * 4);
    w.u_s = take((size_t)B * nA * 4);
    w.row_src = take((size_t)B * nA * 4);
    w.cnt = take((size_t)B * nB * 4);                           // cnt and head are adjacent: cleared together
    w.head = take((size_t)B * nB * 4);
    w.slots = take((size_t)B * nB * MergeLists::SLOTS * 4);
    w.next = take((size_t)B * N * 4);
    w.tsel = take((size_t)B * sizeof(int2));                    // selection threshold per batch element
    w.split = take(dm == 128 || dm == 64 ? match_tc_bytes(B, N, dm) : 0);   // scratch of the tensor-core matcher
    w.total = o;
    return w;
}

}  // namespace usv

extern "C" size_t usv_token_merge_workspace(int B, int N, int C, int Hm, int dm) {
    (void)C; (void)Hm;
    if (B <= 0 || N <= 0) return 0;
    // sized for the worst partition (every token but one is a source / a destination)
    return usv::merge_layout(B, N, dm, N, N).total;
}

// win: NULL = arg-max over every destination of the batch element (Eq. 8-9 as printed); else the
// (wt, wh, ww) block window of the local reading.
static int token_merge_impl(int B, int N, int C, const void* x, int Hm, int dm,
                            const void* metric, int T, int Hh, int W, int st, int sh, int sw,
                            int r, void* x_merged, int32_t* dst_of, int32_t* pos, float* u_out,
                            int32_t* jstar_out, void* ws, size_t ws_bytes, void* stream, const int* win) {
    using namespace usv;
    if (win != nullptr && (win[0] < 0 || win[1] < 0 || win[2] < 0))
        return fail(USV_ERR_INVALID_ARG, "token_merge: window (%d,%d,%d) must not be negative", win[0], win[1], win[2]);
    if (B <= 0 || N <= 0 || C <= 0) return fail(USV_ERR_INVALID_ARG, "token_merge: B,N,C must be positive");
    if (T <= 0 || Hh <= 0 || W <= 0 || (int64_t)T * Hh * W != N)
        return fail(USV_ERR_INVALID_ARG, "token_merge: T*Hh*W = %lld != N = %d", (long long)T * Hh * W, N);
    if (st <= 0 || sh <= 0 || sw <= 0) return fail(USV_ERR_INVALID_ARG, "token_merge: partition sizes must be positive");
    if (C % 8) return fail(USV_ERR_UNSUPPORTED, "token_merge: C=%d not a multiple of 8", C);
    if (x == nullptr || x_merged == nullptr || dst_of == nullptr || pos == nullptr || ws == nullptr)
        return fail(USV_ERR_INVALID_ARG, "token_merge: null pointer");
    if (!aligned16(x) || !aligned16(x_merged) || !aligned16(ws))
        return fail(USV_ERR_UNSUPPORTED, "token_merge: x/x_merged/ws not 16-byte aligned");
    const Part p(T, Hh, W, st, sh, sw);
    const int nA = N - p.nB;
    if (r < 0 || r > nA) return fail(USV_ERR_INVALID_ARG, "token_merge: r=%d outside [0,%d] (number of sources)", r, nA);
    if (metric != nullptr) {
        if (dm != 64 && dm != 128) return fail(USV_ERR_UNSUPPORTED, "token_merge: dm=%d (need 64 or 128)", dm);
        if (Hm <= 0) return fail(USV_ERR_INVALID_ARG, "token_merge: Hm must be positive");
        if (!aligned16(metric)) return fail(USV_ERR_UNSUPPORTED, "token_merge: metric not 16-byte aligned");
    }
    if ((int64_t)B > 65535) return fail(USV_ERR_UNSUPPORTED, "token_merge: B > 65535");
    if (ws_bytes < usv_token_merge_workspace(B, N, C, Hm, dm))
        return fail(USV_ERR_WORKSPACE, "token_merge: workspace %zu < %zu", ws_bytes,
                    usv_token_merge_workspace(B, N, C, Hm, dm));
    const MergeWs L = merge_layout(B, N, dm, nA, p.nB);
    char* base = static_cast<char*>(ws);
    float* mhat = reinterpret_cast<float*>(base + L.mhat);
    int32_t* src_idx = reinterpret_cast<int32_t*>(base + L.src_idx);
    int32_t* jstar_s = reinterpret_cast<int32_t*>(base + L.jstar_s);
    float* u_s = reinterpret_cast<float*>(base + L.u_s);
    const MergeLists lists = {p.nB, reinterpret_cast<int32_t*>(base + L.cnt), reinterpret_cast<int32_t*>(base + L.head),
                              reinterpret_cast<int32_t*>(base + L.slots), reinterpret_cast<int32_t*>(base + L.next),
                              reinterpret_cast<int32_t*>(base + L.row_src), nullptr};
    const size_t zero_bytes = L.slots - L.cnt;   // cnt and head
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int nU = nA - r, Nm = N - r;

    if (metric != nullptr) {
        MatchTcArgs m = {};
        m.p = p; m.B = B; m.N = N; m.nA = nA;
        int rc = USV_OK;
        if (nA > 0 && win == nullptr)
            rc = match_tc_args(m, dm, src_idx, jstar_s, u_s, base + L.split, reinterpret_cast<unsigned int*>(base + L.status));
        if (rc != USV_OK) return rc;
        // one warp per token, and one per padding row
        const dim3 dg(ceil_div(m.a_h != nullptr ? m.nA_pad + m.nB_pad : N, 8), B);
        if (dm == 128) launch_dep(desc_kernel<128>, dg, dim3(256), 0, s, static_cast<const __nv_bfloat16*>(metric), mhat, Hm, src_idx, lists.cnt, (int64_t)(zero_bytes / 4), m);
        else launch_dep(desc_kernel<64>, dg, dim3(256), 0, s, static_cast<const __nv_bfloat16*>(metric), mhat, Hm, src_idx, lists.cnt, (int64_t)(zero_bytes / 4), m);
        USV_CHECK_LAUNCH("desc_kernel");
        if (nA > 0) {
            if (win != nullptr) {
                int sms;   // one wave of CTAs (their launch bounds) from two waves of single sources on
                if (int e = sm_count(&sms); e != USV_OK) return e;
                const bool own = win[0] == 0 && win[1] == 0 && win[2] == 0;
                const int groups = ceil_div(nA, 8), wave = std::max(1, (own ? 6 : 3) * sms / B);
                dim3 lg(groups > 2 * wave ? wave : groups, B);
                auto match = [&](auto kernel) {
                    launch_dep(kernel, lg, dim3(256), 0, s, mhat, p, N, nA, win[0], win[1], win[2], src_idx, jstar_s, u_s);
                };
                if (dm == 128) own ? match(match_local_kernel<128, true>) : match(match_local_kernel<128, false>);
                else own ? match(match_local_kernel<64, true>) : match(match_local_kernel<64, false>);
                USV_CHECK_LAUNCH("match_local_kernel");
            } else {
                // tensor cores: fp16 cosines propose, fp32 decides (usv_match_tc.cu)
                rc = launch_match_tc(mhat, m, dm, s);
                if (rc != USV_OK) return rc;
            }
        }
        auto held = [&](auto kernel, int ctas) {   // (see plan_held_kernel for where the lines are)
            launch_dep(kernel, dim3(ctas, B), dim3(1024), 0, s, p, N, nA, r, src_idx, jstar_s, u_s, dst_of, pos, u_out, jstar_out, lists);
        };
        if (r > 0 && r < nA && (nA <= 3 * 1024 || (nA > 12 * 1024 && nA <= 16 * 8 * 1024))) {
            const int per = ceil_div(nA, nA <= 3 * 1024 ? 1024 : 8 * 1024);
            if (nA <= 3 * 1024) per == 1 ? held(plan_held_kernel<1, 1>, 1) : per == 2 ? held(plan_held_kernel<1, 2>, 1) : held(plan_held_kernel<1, 3>, 1);
            else if (per <= 2) held(plan_held_kernel<8, 2>, 8);
            else if (per <= 3) held(plan_held_kernel<8, 3>, 8);
            else if (per <= 4) held(plan_held_kernel<8, 4>, 8);
            else if (per <= 5) held(plan_held_kernel<8, 5>, 8);
            else if (per <= 6) held(plan_held_kernel<8, 6>, 8);
            else if (per <= 8) held(plan_held_kernel<8, 8>, 8);
            else if (per <= 11) held(plan_held_kernel<8, 11>, 8);
            else held(plan_held_kernel<8, 16>, 8);
            USV_CHECK_LAUNCH("plan_held_kernel");
            return launch_merge(p, B, N, C, nU, Nm, x, lists, dst_of, x_merged, s);
        }
        const int2* tsel = nullptr;
        if (r > 0 && r < nA) {
            int2* tsel_w = reinterpret_cast<int2*>(base + L.tsel);
            if (nA <= 4 * 1024) launch_dep(plan_select_kernel<4>, dim3(B), dim3(1024), 0, s, nA, r, u_s, tsel_w);
            else if (nA <= 12 * 1024) launch_dep(plan_select_kernel<12>, dim3(B), dim3(1024), 0, s, nA, r, u_s, tsel_w);
            else launch_dep(plan_select_kernel<24>, dim3(B), dim3(1024), 0, s, nA, r, u_s, tsel_w);
            USV_CHECK_LAUNCH("plan_select_kernel");
            tsel = tsel_w;
        }
        // r = nA: every key is above 0; r = 0: no key is above or equal to the largest one
        dim3 pg(ceil_div(nA > p.nB ? nA : p.nB, 1024), B);
        launch_dep(plan_assign_kernel, dim3(pg), dim3(1024), 0, s, p, N, nA, r, r == nA ? 0u : 0xffffffffu, 0, tsel, src_idx, jstar_s, u_s,
                                               dst_of, pos, u_out, jstar_out, lists);
        USV_CHECK_LAUNCH("plan_assign_kernel");
    } else {
        cudaError_t e = cudaMemsetAsync(lists.cnt, 0, zero_bytes, s);
        if (e != cudaSuccess) return fail(USV_ERR_CUDA, "token_merge: memset: %s", cudaGetErrorString(e));
        launch_dep(plan_lists_kernel, dim3(ceil_div(N, 256), B), dim3(256), 0, s, p, N, nU, dst_of, pos, lists);
        USV_CHECK_LAUNCH("plan_lists_kernel");
    }
    return launch_merge(p, B, N, C, nU, Nm, x, lists, dst_of, x_merged, s);
}

extern "C" int usv_token_unmerge(int B, int N, int Nm, int C, const void* y_merged,
                                 const int32_t* pos, void* y, void* stream) {
    using namespace usv;
    if (B <= 0 || N <= 0 || Nm <= 0 || C <= 0 || Nm > N)
        return fail(USV_ERR_INVALID_ARG, "token_unmerge: need B,N,Nm,C > 0 and Nm <= N");
    if (C % 8) return fail(USV_ERR_UNSUPPORTED, "token_unmerge: C=%d not a multiple of 8", C);
    if (y_merged == nullptr || pos == nullptr || y == nullptr)
        return fail(USV_ERR_INVALID_ARG, "token_unmerge: null pointer");
    if (!aligned16(y_merged) || !aligned16(y))
        return fail(USV_ERR_UNSUPPORTED, "token_unmerge: y_merged/y not 16-byte aligned");
    const int64_t rows = (int64_t)B * N;
    launch_dep(unmerge_kernel, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, static_cast<cudaStream_t>(stream), 
        N, Nm, C, static_cast<const __nv_bfloat16*>(y_merged), pos,
        static_cast<__nv_bfloat16*>(y), rows);
    USV_CHECK_LAUNCH("unmerge_kernel");
    return USV_OK;
}

// ---------------------------------------------------------------------------- stored plan
// What merge_kernel needs of a plan, kept by the caller beside dst_of / pos so that applying the
// plan to further tensors is the streaming kernel alone: cnt | head | row_src | next | dst_copy |
// slots (SLOTS times the size), each B * (N + 1) ints.
namespace usv {
static size_t cache_stride(int B, int N) { return align_up((size_t)B * ((size_t)N + 1) * sizeof(int32_t), 256); }
static MergeLists cache_lists(void* cache, int B, int N, int nB) {
    char* base = static_cast<char*>(cache);
    const size_t cs = cache_stride(B, N);
    auto at = [&](int i) { return reinterpret_cast<int32_t*>(base + i * cs); };
    return {nB, at(0), at(1), at(5), at(3), at(2), at(4)};
}

static int fill_part(Part& p, int N, int T, int Hh, int W, int st, int sh, int sw, const char* who) {
    if (T <= 0 || Hh <= 0 || W <= 0 || (int64_t)T * Hh * W != N)
        return fail(USV_ERR_INVALID_ARG, "%s: T*Hh*W = %lld != N = %d", who, (long long)T * Hh * W, N);
    if (st <= 0 || sh <= 0 || sw <= 0) return fail(USV_ERR_INVALID_ARG, "%s: partition sizes must be positive", who);
    p = Part(T, Hh, W, st, sh, sw);
    return USV_OK;
}
}  // namespace usv

extern "C" size_t usv_merge_plan_cache_bytes(int B, int N) {
    if (B <= 0 || N <= 0) return 0;
    return (5 + usv::MergeLists::SLOTS) * usv::cache_stride(B, N);
}

extern "C" int usv_merge_plan_cache(int B, int N, int T, int Hh, int W, int st, int sh, int sw, int r,
                                    const int32_t* dst_of, const int32_t* pos, void* cache, size_t cache_bytes,
                                    void* stream) {
    using namespace usv;
    if (B <= 0 || N <= 0) return fail(USV_ERR_INVALID_ARG, "merge_plan_cache: B,N must be positive");
    if (B > 65535) return fail(USV_ERR_UNSUPPORTED, "merge_plan_cache: B > 65535");
    Part p;
    int rc = fill_part(p, N, T, Hh, W, st, sh, sw, "merge_plan_cache");
    if (rc != USV_OK) return rc;
    const int nA = N - p.nB;
    if (r < 0 || r > nA) return fail(USV_ERR_INVALID_ARG, "merge_plan_cache: r=%d outside [0,%d]", r, nA);
    if (dst_of == nullptr || pos == nullptr || cache == nullptr) return fail(USV_ERR_INVALID_ARG, "merge_plan_cache: null pointer");
    if (!aligned16(cache)) return fail(USV_ERR_UNSUPPORTED, "merge_plan_cache: cache not 16-byte aligned");
    if (cache_bytes < usv_merge_plan_cache_bytes(B, N))
        return fail(USV_ERR_WORKSPACE, "merge_plan_cache: cache %zu < %zu", cache_bytes, usv_merge_plan_cache_bytes(B, N));
    const MergeLists lists = cache_lists(cache, B, N, p.nB);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemsetAsync(lists.cnt, 0, 2 * cache_stride(B, N), s);   // cnt and head
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "merge_plan_cache: memset: %s", cudaGetErrorString(e));
    launch_dep(plan_lists_kernel, dim3(ceil_div(N, 256), B), dim3(256), 0, s, p, N, nA - r, dst_of, pos, lists);
    USV_CHECK_LAUNCH("plan_lists_kernel");
    return USV_OK;
}

extern "C" int usv_token_merge_apply(int B, int N, int C, const void* x, int T, int Hh, int W, int st, int sh,
                                     int sw, int r, void* cache, void* x_merged, void* stream) {
    using namespace usv;
    if (B <= 0 || N <= 0 || C <= 0) return fail(USV_ERR_INVALID_ARG, "token_merge_apply: B,N,C must be positive");
    if (C % 8) return fail(USV_ERR_UNSUPPORTED, "token_merge_apply: C=%d not a multiple of 8", C);
    Part p;
    int rc = fill_part(p, N, T, Hh, W, st, sh, sw, "token_merge_apply");
    if (rc != USV_OK) return rc;
    const int nA = N - p.nB;
    if (r < 0 || r > nA) return fail(USV_ERR_INVALID_ARG, "token_merge_apply: r=%d outside [0,%d]", r, nA);
    if (x == nullptr || cache == nullptr || x_merged == nullptr) return fail(USV_ERR_INVALID_ARG, "token_merge_apply: null pointer");
    if (!aligned16(x) || !aligned16(x_merged) || !aligned16(cache))
        return fail(USV_ERR_UNSUPPORTED, "token_merge_apply: x/x_merged/cache not 16-byte aligned");
    const MergeLists lists = cache_lists(cache, B, N, p.nB);
    const int Nm = N - r;
    return launch_merge(p, B, N, C, nA - r, Nm, x, lists, lists.dst_copy, x_merged,
                        static_cast<cudaStream_t>(stream));
}

extern "C" size_t usv_unmerge_map_workspace(int B, int Nm) {
    if (B <= 0 || Nm <= 0) return 0;
    return usv::WS_HEADER + 2 * usv::align_up((size_t)B * Nm * sizeof(int32_t), 256);
}

extern "C" int usv_unmerge_map(int B, int N, int Nm, const int32_t* pos, int32_t* inv_off, int32_t* inv_idx,
                               void* ws, size_t ws_bytes, void* stream) {
    using namespace usv;
    if (B <= 0 || N <= 0 || Nm <= 0 || Nm > N) return fail(USV_ERR_INVALID_ARG, "unmerge_map: need B,N,Nm > 0 and Nm <= N");
    if (pos == nullptr || inv_off == nullptr || inv_idx == nullptr || ws == nullptr)
        return fail(USV_ERR_INVALID_ARG, "unmerge_map: null pointer");
    if (B > 65535) return fail(USV_ERR_UNSUPPORTED, "unmerge_map: B > 65535");
    if (ws_bytes < usv_unmerge_map_workspace(B, Nm))
        return fail(USV_ERR_WORKSPACE, "unmerge_map: workspace %zu < %zu", ws_bytes, usv_unmerge_map_workspace(B, Nm));
    int32_t* cnt = reinterpret_cast<int32_t*>(static_cast<char*>(ws) + WS_HEADER);
    int32_t* cursor = reinterpret_cast<int32_t*>(static_cast<char*>(ws) + WS_HEADER + align_up((size_t)B * Nm * 4, 256));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemsetAsync(cnt, 0, (size_t)B * Nm * 4, s);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "unmerge_map: memset: %s", cudaGetErrorString(e));
    dim3 tg(ceil_div(N, 256), B);
    launch_dep(inv_count_kernel, dim3(tg), dim3(256), 0, s, N, Nm, pos, cnt);
    USV_CHECK_LAUNCH("inv_count_kernel");
    launch_dep(row_scan_kernel, dim3(dim3(ceil_div(Nm, 1024), B)), dim3(1024), 0, s, Nm, cnt, inv_off, cursor);
    USV_CHECK_LAUNCH("row_scan_kernel");
    launch_dep(inv_fill_kernel, dim3(tg), dim3(256), 0, s, N, Nm, pos, cursor, inv_idx);
    USV_CHECK_LAUNCH("inv_fill_kernel");
    return USV_OK;
}

extern "C" int usv_token_merge(int B, int N, int C, const void* x, int Hm, int dm,
                               const void* metric, int T, int Hh, int W, int st, int sh, int sw,
                               int r, void* x_merged, int32_t* dst_of, int32_t* pos, float* u_out,
                               int32_t* jstar_out, void* ws, size_t ws_bytes, void* stream) {
    return token_merge_impl(B, N, C, x, Hm, dm, metric, T, Hh, W, st, sh, sw, r, x_merged, dst_of, pos, u_out,
                            jstar_out, ws, ws_bytes, stream, nullptr);
}

extern "C" int usv_token_merge_local(int B, int N, int C, const void* x, int Hm, int dm,
                                     const void* metric, int T, int Hh, int W, int st, int sh, int sw,
                                     int wt, int wh, int ww, int r, void* x_merged, int32_t* dst_of,
                                     int32_t* pos, float* u_out, int32_t* jstar_out, void* ws,
                                     size_t ws_bytes, void* stream) {
    const int win[3] = {wt, wh, ww};
    return token_merge_impl(B, N, C, x, Hm, dm, metric, T, Hh, W, st, sh, sw, r, x_merged, dst_of, pos, u_out,
                            jstar_out, ws, ws_bytes, stream, win);
}
