// Attention of the heads that keep every key block, on pairs of SMs (tcgen05 cta_group::2), head width 128.
//
// Same formulation, roles and arithmetic as attn_pair_kernel (usv_attn_pair.cu): 128 query rows a CTA, two key blocks a tile,
//
//     S[128 q x 128 keys]  = Q . K_tile^T      tcgen05.mma, A = Q in smem,        B = K in smem
//     O[128 q x 128]      += P . V_tile        tcgen05.mma, A = P (bf16) in TMEM, B = V in smem
//
// but the two CTAs of a cluster work on one item of FOUR consecutive query blocks and walk the same keys: one MMA of the
// leader computes 256 rows, and each CTA stages only its half of the B operands: the K rows of one of the tile's two key
// blocks, and one 64-column half of the V tile.  A tile's traffic through shared memory, which bounds the other kernel, falls
// from 160 to 96 KB per CTA (1280 -> 768 cycles beside 1024 of MMAs), and what comes out of the L2, 64 KB per tile and CTA
// there (10 TB/s over the chip), to 32 KB.  It pays only where all four query blocks want every key block: sparse lists of
// four blocks have a union of 1.8 times a list, of two 1.3 times.
//
// Every list is 0 .. NB - 1 (query blocks whose list has holes are left to the exact kernel), so there is no plan, no scout and no item ring: cluster c takes items c, c + clusters, ...
// Roles of a CTA: warps 0-15 softmax, 16-19 output, 20 Q and K producer, 21 P.V issuer, 22 V producer, 23 S issuer; the
// issuers of the second CTA have nothing to do.  Barriers the issuers wait on live in the leader (rank 0): the second CTA's
// TMA loads and softmax and output warps signal them there; what the issuers signal goes to both CTAs (tcgen05.commit with
// a CTA mask).  No load is multicast.  All waits are bounded, as there.
#include "usv_attn.cuh"
#include "usv_attn_softmax.cuh"

namespace usv {

namespace dn {

using namespace t5;

constexpr int D = 128;
constexpr int KT = 2 * USV_BLOCK;               // keys per tile = two key blocks
constexpr int NWG = 4;                          // softmax warpgroups
constexpr int SBUF = 3;                         // S/P buffers in TMEM
constexpr int KSTAGES = 4, VSTAGES = 4;         // stages of half a tile (16 KB); five and six change nothing
// Every POLY-th pair of exponentials goes to the FMA pipe (exp2_fma; the special-function unit is 77 % busy without).  12
// full heads of 20 280 tokens: none 1752 us, one in eight 1725, one in four 1746.
constexpr int POLY = 8;
constexpr int NSLOT = 4;                        // per-item row sums and references (see the softmax warps)
constexpr uint32_t HALF_BYTES = USV_BLOCK * D * 2;
constexpr uint32_t Q_BYTES = 2 * HALF_BYTES;

constexpr uint32_t SM_Q = 0;                                   // [d-half][128 rows][128 B]
constexpr uint32_t SM_K = SM_Q + Q_BYTES;                      // stage: [d-half][64 keys][128 B]
constexpr uint32_t SM_V = SM_K + KSTAGES * HALF_BYTES;         // stage: [128 keys][128 B], one d-half
constexpr uint32_t SM_BAR = SM_V + VSTAGES * HALF_BYTES;
enum { B_QFULL = 0, B_QFREE, B_KFULL, B_KEMPTY = B_KFULL + KSTAGES, B_VFULL = B_KEMPTY + KSTAGES, B_VEMPTY = B_VFULL + VSTAGES,
       B_SFULL = B_VEMPTY + VSTAGES, B_PFULL = B_SFULL + 2 * SBUF, B_PHALF = B_PFULL + 2 * SBUF, B_OFULL = B_PHALF + 2 * SBUF, B_OFREE, B_SUMS,
       B_REF = B_SUMS + NSLOT, B_COUNT = B_REF + 2 * NSLOT };
static_assert(B_COUNT <= 64, "barrier area");
constexpr uint32_t SM_MISC = SM_BAR + 8 * 64;                  // tmem base, abort flag
constexpr uint32_t SM_REFV = SM_MISC + 64;                     // float[NSLOT][128]: minus the softmax reference per row
constexpr uint32_t SM_SUM = SM_REFV + NSLOT * 128 * 4;         // float[NSLOT][NWG][128]: partial row sums
constexpr uint32_t SM_TOTAL = SM_SUM + NSLOT * NWG * 128 * 4;
constexpr size_t SMEM_BYTES = SM_TOTAL + 1024;                 // + slack for 1024-byte alignment
static_assert(SMEM_BYTES <= 232448, "shared memory budget");

// TMEM columns: O | S/P buffer 0 | S/P buffer 1 | S/P buffer 2
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t TO = 0, TS = 128;

constexpr int NSOFT = NWG * 128;
constexpr int NTHREADS = NSOFT + 128 + 128;
constexpr int W_EPI = NSOFT / 32, W_TMA = W_EPI + 4, W_MMA = W_EPI + 5, W_TMA_V = W_EPI + 6, W_MMA_S = W_EPI + 7;
constexpr int REG_LAUNCH = 80, REG_SOFT = 96, REG_EPI = 56, REG_SERVICE = 40;   // (setmaxnreg, as in usv_attn_pair.cu)
static_assert(16 * REG_SOFT + 4 * REG_EPI + 4 * REG_SERVICE <= 24 * REG_LAUNCH, "register pool of the CTA");

struct Maps {
    CUtensorMap q, k, v;
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of the leader's copy of a barrier
__device__ __forceinline__ uint32_t in_leader(uint32_t addr) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
    return r;
}
__device__ __forceinline__ void arrive_leader(uint32_t addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// A tile of this CTA's own memory; its bytes are counted by a barrier of the leader.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t leader_bar, int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(leader_bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// completion of the MMAs issued so far -> the barrier at this offset in both CTAs
__device__ __forceinline__ void commit_pair(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void umma2_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma2_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Items: (b, full head in order, four query blocks).  The full heads are the first a.full_heads of a.head_order.
__global__ void __launch_bounds__(NTHREADS, 1) __cluster_dims__(2, 1, 1)
attn_dense_kernel(const AttnArgs a, const __grid_constant__ Maps maps) {
    // the set-up touches shared and tensor memory only; dep_sync() follows it, with the columns allocated
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* sm = smem_raw + (base - raw);
    auto bar = [&](int i) { return base + SM_BAR + 8u * i; };
    volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(sm + SM_MISC);
    volatile int* s_abort = reinterpret_cast<volatile int*>(sm + SM_MISC + 4);
    int* s_flag = reinterpret_cast<int*>(sm + SM_MISC + 16);   // [NSLOT][2]: 1 + the last item in which this side was reported
    float* s_refv = reinterpret_cast<float*>(sm + SM_REFV);
    float* s_sum = reinterpret_cast<float*>(sm + SM_SUM);

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int NB = a.NB, N = a.N;
    const int T = (NB + 1) >> 1;                  // tiles an item
    const int NQ = (NB + 3) >> 2;                 // items per (b, h)
    const int items = a.B * a.full_heads * NQ;
    const int clusters = gridDim.x >> 1, first = blockIdx.x >> 1;
    // item w: its (b, h) and this CTA's first query block
    struct Item { int b, bh_ord, h, I; };
    auto item_of = [&](int w) {
        const int bf = w / NQ, b = bf / a.full_heads, f = bf - b * a.full_heads;
        return Item{b, b * a.H + f, a.head_order[f], 4 * (w - bf * NQ) + 2 * (int)rank};
    };

    // ---- set-up: barriers, TMEM
    if (threadIdx.x < B_COUNT) {
        const int i = threadIdx.x;
        uint32_t count = 1;                                           // Q, K/V stages, SFULL, OFULL
        if (i >= B_PFULL && i < B_PHALF + 2 * SBUF) count = 16;       // PFULL, PHALF: one per warp of a tile's two groups in either CTA
        if (i == B_OFREE) count = 8;                                  // one per output warp of either CTA
        if (i >= B_SUMS && i < B_SUMS + NSLOT) count = NSOFT / 32;
        if (i >= B_REF && i < B_REF + 2 * NSLOT) count = 2;           // the two warps of the owning group on a side
        mbar_init(bar(i), count);
        if (i == 0) *s_abort = 0;
        if (i < 2 * NSLOT) s_flag[i] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + SM_MISC), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    cluster_sync();    // the barriers of both CTAs are there
    fence_after();
    dep_sync();
    const uint32_t tmem = *s_tmem;

    if (warp == W_TMA) {
        // ===== Q and K producer (whole warp in the loop, one elected lane issues) ================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_SERVICE));
        int g = 0, n = 0;
        bool ok = true;
        for (int w = first; ok && w < items; w += clusters, ++n) {
            const Item it = item_of(w);
            for (int t = 0; t < T; ++t, ++g) {
                const int s = g % KSTAGES;
                if (!mbar_wait(bar(B_KEMPTY + s), ((g / KSTAGES) & 1) ^ 1, s_abort, a.status, 0x1)) { ok = false; break; }
                if (elect_one()) {
                    const uint32_t full = in_leader(bar(B_KFULL + s)), dst = base + SM_K + s * HALF_BYTES;
                    if (rank == 0) mbar_expect_tx(bar(B_KFULL + s), 2 * HALF_BYTES);
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf)   // key block 2t + rank; past the end: zeros, masked
                        tma_load_pair(dst + hf * 8192, &maps.k, full, hf * 64, (2 * t + (int)rank) * USV_BLOCK, it.h, it.b);
                }
                __syncwarp();
                // the Q rows follow the item's first K tile: their buffer comes free later than that stage does
                if (t == 0) {
                    if (n >= 1 && !mbar_wait(bar(B_QFREE), (n - 1) & 1, s_abort, a.status, 0x4000)) { ok = false; break; }
                    if (elect_one()) {
                        const uint32_t full = in_leader(bar(B_QFULL));
                        if (rank == 0) mbar_expect_tx(bar(B_QFULL), 2 * Q_BYTES);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            tma_load_pair(base + SM_Q + i * 8192, &maps.q, full, (i >> 1) * 64, (it.I + (i & 1)) * USV_BLOCK, it.h, it.b);
                    }
                    __syncwarp();
                }
            }
        }
    } else if (warp == W_TMA_V) {
        // ===== V producer ========================================================================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_SERVICE));
        int g = 0;
        bool ok = true;
        for (int w = first; ok && w < items; w += clusters) {
            const Item it = item_of(w);
            for (int t = 0; t < T; ++t, ++g) {
                const int s = g % VSTAGES;
                if (!mbar_wait(bar(B_VEMPTY + s), ((g / VSTAGES) & 1) ^ 1, s_abort, a.status, 0x2)) { ok = false; break; }
                if (elect_one()) {
                    const uint32_t full = in_leader(bar(B_VFULL + s)), dst = base + SM_V + s * HALF_BYTES;
                    if (rank == 0) mbar_expect_tx(bar(B_VFULL + s), 2 * HALF_BYTES);
#pragma unroll
                    for (int j = 0; j < 2; ++j)      // columns 64 rank .. of both key blocks
                        tma_load_pair(dst + j * 8192, &maps.v, full, (int)rank * 64, (2 * t + j) * USV_BLOCK, it.h, it.b);
                }
                __syncwarp();
            }
        }
    } else if (warp == W_MMA) {
        // ===== P.V issuer, TMEM owner ============================================================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_SERVICE));
        constexpr uint32_t IDESC_O = instr_desc(256, D, 0, 1);     // P (TMEM) x V (MN-major)
        const uint64_t vdesc0 = smem_desc(base + SM_V, HALF_BYTES, 1024);
        int g = 0, n = 0;
        bool ok = rank == 0;
        for (int w = first; ok && w < items; w += clusters, ++n) {
            for (int t = 0; t < T; ++t, ++g) {
                const int s = g % VSTAGES, b6 = g % (2 * SBUF);
                if (!mbar_wait(bar(B_VFULL + s), (g / VSTAGES) & 1, s_abort, a.status, 0x20)) { ok = false; break; }
                if (!mbar_wait(bar(B_PHALF + b6), (g / (2 * SBUF)) & 1, s_abort, a.status, 0x40)) { ok = false; break; }
                // the first P.V of an item overwrites O: the item before must have been read out
                if (t == 0 && n > 0 && !mbar_wait(bar(B_OFREE), (n - 1) & 1, s_abort, a.status, 0x2000)) { ok = false; break; }
                fence_after();
                const uint64_t vdesc = vdesc0 + ((s * HALF_BYTES) >> 4);
                const uint32_t pb = tmem + TS + (g % SBUF) * 128;   // P: 32 columns at the head of each 64-column half
                // keys ks * 16 ... of the tile: the first half of each block, then the second
                auto mma = [&](int ks) {
                    umma2_ts(tmem + TO, pb + (ks >> 2) * 64 + (ks & 3) * 8, vdesc + ((ks * 2048) >> 4), IDESC_O, (t > 0 || ks > 0));
                };
                if (elect_one()) {
                    mma(0); mma(1); mma(4); mma(5);
                }
                __syncwarp();
                if (!mbar_wait(bar(B_PFULL + b6), (g / (2 * SBUF)) & 1, s_abort, a.status, 0x40)) { ok = false; break; }
                fence_after();
                if (elect_one()) {
                    mma(2); mma(3); mma(6); mma(7);
                    commit_pair(bar(B_VEMPTY + s));      // V stage free; S buffer free for S(g + 3)
                    if (t == T - 1) commit_pair(bar(B_OFULL));
                }
                __syncwarp();
            }
        }
    } else if (warp == W_MMA_S) {
        // ===== S issuer ===========================================================================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_SERVICE));
        static_assert(VSTAGES >= SBUF, "the V stage barrier of tile g - 3 doubles as the hand-back of its S buffer");
        constexpr uint32_t IDESC_S = instr_desc(256, KT, 0, 0);    // Q (K-major) x K (K-major)
        const uint64_t qdesc = smem_desc(base + SM_Q, 16, 1024);
        const uint64_t kdesc0 = smem_desc(base + SM_K, 16, 1024);
        int g = 0, n = 0;
        bool ok = rank == 0;
        for (int w = first; ok && w < items; w += clusters, ++n) {
            if (!mbar_wait(bar(B_QFULL), n & 1, s_abort, a.status, 0x4)) break;
            for (int t = 0; t < T; ++t, ++g) {
                const int s = g % KSTAGES;
                if (!mbar_wait(bar(B_KFULL + s), (g / KSTAGES) & 1, s_abort, a.status, 0x8)) { ok = false; break; }
                // the buffer held P(g - 3): P.V(g - 3) must be complete
                if (g >= SBUF && !mbar_wait(bar(B_VEMPTY + (g - SBUF) % VSTAGES), ((g - SBUF) / VSTAGES) & 1, s_abort, a.status, 0x100)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint64_t kdesc = kdesc0 + ((s * HALF_BYTES) >> 4);
                const uint32_t d_s = tmem + TS + (g % SBUF) * 128;
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        umma2_ss(d_s, qdesc + (((ks >> 2) * 16384 + (ks & 3) * 32) >> 4), kdesc + (((ks >> 2) * 8192 + (ks & 3) * 32) >> 4),
                                 IDESC_S, ks > 0);
                    commit_pair(bar(B_SFULL + g % (2 * SBUF)));
                    commit_pair(bar(B_KEMPTY + s));
                    if (t == T - 1) commit_pair(bar(B_QFREE));
                }
                __syncwarp();
            }
        }
    } else if (warp >= W_EPI && warp < W_TMA) {
        // ===== output warps: thread e <-> TMEM lane e <-> query row e of this CTA ================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_EPI));
        const int e = threadIdx.x - NSOFT;
        const int side = e >> 6;
        const uint32_t lane_base = tmem + ((uint32_t)((warp - W_EPI) * 32) << 16);
        const uint32_t ofree = in_leader(bar(B_OFREE));
        int m = 0;
        for (int w = first; w < items; w += clusters, ++m) {
            const Item it = item_of(w);
            const int slot = m % NSLOT;
            const int iq = it.I + side, row = iq * USV_BLOCK + (e & 63);
            const bool live = row < N;
            // a list with holes (entries of -1) is not the full set: its query block goes to the exact kernel.  (64 threads read a list while
            // the item's tiles are computed.  Unrolled, the loop costs 1.5 % of a call, as it stands 0.4: 12 x 317 blocks 1701 us without, 1708.)
            bool hole = false;
            if (iq < NB) {
                const int32_t* list = a.sel + (((int64_t)it.b * a.H + it.h) * NB + iq) * a.kmax;
#pragma unroll 1
                for (int j = e & 63; j < NB; j += 64) hole |= (unsigned)__ldg(list + j) >= (unsigned)NB;
            }
            if (!mbar_wait(bar(B_SUMS + slot), (m / NSLOT) & 1, s_abort, a.status, 0x800)) break;
            float l = 0.f;
#pragma unroll
            for (int q = 0; q < NWG; ++q) l += s_sum[slot * (NWG * 128) + q * 128 + e];
            const float nref = s_refv[slot * 128 + e];
            const bool in_range = l > 7.9e-31f && l < 1.2e30f;   // ~[2^-100, 2^100]
            const float inv = l > 0.f ? 1.0f / l : 0.f;
            if (a.lse != nullptr && live)
                a.lse[((int64_t)it.b * a.H + it.h) * N + row] = (log2f(l) - nref) * 0.69314718055994531f;
            // so does a query block with a row out of range: the first of its threads to notice says so
            if ((hole || (live && !in_range)) && atomicExch(&s_flag[slot * 2 + side], m + 1) != m + 1)
                a.fallback_list[atomicAdd(a.fallback_count, 1)] = it.bh_ord * NB + iq;
            if (!mbar_wait(bar(B_OFULL), m & 1, s_abort, a.status, 0x200)) break;
            fence_after();
            float* o32 = (a.o_f32 != nullptr && live) ? a.o_f32 + (((int64_t)it.b * a.H + it.h) * N + row) * D : nullptr;
            __nv_bfloat16* O = a.o + it.b * a.so.sb + it.h * a.so.sh + (int64_t)row * a.so.sn;
#pragma unroll 1
            for (int qd = 0; qd < D / 32; ++qd) {
                uint32_t r0[32];
                tmem_ld32(lane_base + TO + qd * 32, r0);
                tmem_wait_ld();
                if (qd == D / 32 - 1) {
                    fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_leader(ofree);
                }
                if (o32 != nullptr) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        *reinterpret_cast<float4*>(o32 + qd * 32 + j * 4) =
                            make_float4(__uint_as_float(r0[4 * j]) * inv, __uint_as_float(r0[4 * j + 1]) * inv,
                                        __uint_as_float(r0[4 * j + 2]) * inv, __uint_as_float(r0[4 * j + 3]) * inv);
                }
                if (live) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        *reinterpret_cast<uint4*>(O + qd * 32 + 8 * i) =
                            make_uint4(pack_bf16x2(__uint_as_float(r0[8 * i]) * inv, __uint_as_float(r0[8 * i + 1]) * inv),
                                       pack_bf16x2(__uint_as_float(r0[8 * i + 2]) * inv, __uint_as_float(r0[8 * i + 3]) * inv),
                                       pack_bf16x2(__uint_as_float(r0[8 * i + 4]) * inv, __uint_as_float(r0[8 * i + 5]) * inv),
                                       pack_bf16x2(__uint_as_float(r0[8 * i + 6]) * inv, __uint_as_float(r0[8 * i + 7]) * inv));
                }
            }
        }
    } else if (warp < W_EPI) {
        // ===== softmax warpgroups ================================================================
        // Slot n % NSLOT of the sums and references is used again by item n + NSLOT.  With two tiles an item and more (attn_dense_heads
        // sees to that) every group has a tile in every item, and the first S tile of item n + 4 waits for the P.V of a tile three
        // before it, of item n + 2 at the earliest.  That was issued behind the first P.V of its item, which waits for
        // the output warps to have read item n + 1 (OFREE), and so item n.  (With one tile a group without it would
        // wait for nothing, and its arrival for item n + 4 could be counted for item n.)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REG_SOFT));
        const int grp = warp >> 2;                       // tiles of running parity grp >> 1, key block grp & 1
        const int tp = grp >> 1, hb = grp & 1;
        const int r = threadIdx.x & 127;                 // query row within the CTA, = TMEM lane
        const int side = r >> 6;
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + TS + hb * 64;
        const uint32_t pfull = in_leader(bar(B_PFULL)), phalf = in_leader(bar(B_PHALF));
        const float c = a.scale_log2;
        const uint64_t c2 = pack_f32x2(c, c);
        int g = 0, n = 0;       // running tile (first of the current item), running item
        bool ok = true;
        for (int w = first; ok && w < items; w += clusters, ++n) {
            const int slot = n % NSLOT;
            const uint32_t ref_bar = bar(B_REF + side * NSLOT + slot);
            float* refv = s_refv + slot * 128;
            float nref = 0.f;         // minus the softmax reference (base-2, scaled)
            bool have_ref = false;
            uint64_t lr2 = 0, nref2 = 0;
            for (int t = (tp - g) & 1; t < T; t += 2) {   // tiles of this item whose running index has parity tp
                const int gt = g + t;
                const int nv = N - (2 * t + hb) * USV_BLOCK;   // keys of the block with index < N
                const int b6 = gt % (2 * SBUF);
                const uint32_t sbase = lane_base + (gt % SBUF) * 128;
                if (!mbar_wait(bar(B_SFULL + b6), (gt / (2 * SBUF)) & 1, s_abort, a.status, 0x80)) { ok = false; break; }
                fence_after();
                if (!have_ref) {
                    if (t == 0 && hb == 0) {
                        // the row maximum over the first key block is the row's softmax reference
                        uint32_t m0[32], m1[32];
                        tmem_ld32(sbase, m0);
                        tmem_ld32(sbase + 32, m1);
                        tmem_wait_ld();
                        float mx = -INFINITY;
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            if (j < nv) mx = fmaxf(mx, __uint_as_float(m0[j]));
                            if (j + 32 < nv) mx = fmaxf(mx, __uint_as_float(m1[j]));
                        }
                        nref = mx == -INFINITY ? 0.f : -mx * c;
                        refv[r] = nref;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(ref_bar);
                    } else {
                        if (!mbar_wait(ref_bar, (n / NSLOT) & 1, s_abort, a.status, 0x400)) { ok = false; break; }
                        nref = refv[r];
                    }
                    nref2 = pack_f32x2(nref, nref);
                    have_ref = true;
                }
                // The weights (bf16 pairs) go back into the columns their logits came from: P takes the first 32 of the 64
                // columns.  Each half is handed over when it is there, so that P.V starts half a softmax earlier.
                auto hand_over = [&](uint32_t at) {
                    tmem_wait_st();
                    fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_leader(at + 8 * b6);
                };
                uint32_t pk[16];
                if (nv > 0) {
                    uint32_t sx[32];
                    tmem_ld32(sbase, sx);
                    tmem_wait_ld();
                    if (nv >= USV_BLOCK) weights32<false, SUM_ROUNDED, POLY>(sx, pk, c2, nref2, 0, nv, lr2);
                    else weights32<true, SUM_ROUNDED, POLY>(sx, pk, c2, nref2, 0, nv, lr2);
                    tmem_st16(sbase, pk);
                    uint32_t sy[32];
                    tmem_ld32(sbase + 32, sy);
                    hand_over(phalf);
                    tmem_wait_ld32(sy);
                    if (nv >= USV_BLOCK) weights32<false, SUM_ROUNDED, POLY>(sy, pk, c2, nref2, 32, nv, lr2);
                    else weights32<true, SUM_ROUNDED, POLY>(sy, pk, c2, nref2, 32, nv, lr2);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) pk[j] = 0u;
                    tmem_st16(sbase, pk);
                    hand_over(phalf);
                }
                tmem_st16(sbase + 16, pk);
                hand_over(pfull);
            }
            if (!ok) break;
            // placed by the parity of the tile within the item: the four partial sums are added in one order in every item
            float lr_lo, lr_hi;
            unpack_f32x2(lr2, lr_lo, lr_hi);
            s_sum[slot * (NWG * 128) + ((((tp - g) & 1) << 1) | hb) * 128 + r] = lr_lo + lr_hi;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_SUMS + slot));
            g += T;
        }
    }

    // ---- teardown
    fence_before();
    __syncthreads();
    if (*s_abort) {
        // give copies and MMAs that may still be in flight time to land before the CTA's
        // shared memory and TMEM are handed back
        const unsigned long long t0 = gtime();
        while (gtime() - t0 < 2000000ull) { }
        __syncthreads();
    }
    cluster_sync();    // nobody signals a CTA that has left
    if (warp == W_MMA) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

}  // namespace dn

// Clusters of the kernel that the device holds at once; 0 where it cannot run.
static int dense_clusters() {
    cudaLaunchConfig_t cfg = {};
    int sms = 0, n = 0;
    if (sm_count(&sms) != USV_OK) return 0;
    cfg.gridDim = dim3(sms & ~1);
    cfg.blockDim = dim3(dn::NTHREADS);
    cfg.dynamicSmemBytes = dn::SMEM_BYTES;
    if (cudaFuncSetAttribute(dn::attn_dense_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dn::SMEM_BYTES) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, dn::attn_dense_kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

// Calls whose heads are all full, beyond those without a plan, go here where waves of items take less time than on the paired kernel,
// whose items have two query blocks: a wave is a tenth shorter here, but the last one may be emptier, and an item has room for four
// query blocks however many are left for it.  us, pair kernel with a plan / this one, with the waves of either: 12 heads x 30 blocks 42.5 / 40.9
// (2 / 2), 24 x 28 48.2 / 45.4 (3 / 3), 1 x 140 62.6 / 58.2 (1 / 1), 24 x 53 131 / 119 (5 / 5), 12 x 101 254 / 229 (5 / 5), 12 x 317 1899 / 1687 (13 / 13),
// 1 x 1857 5671 / 5102 (7 / 7), 400 x 21 401 / 397 (30 / 33); but 8 x 73 74 / 91 (2 / 3), 16 x 53 79 / 88 (3 / 4), 40 x 21 46 / 52 (3 / 4), 240 x 10
// 63.4 / 65.5 (9 / 10), 400 x 17 289 / 291 (25 / 28), 600 x 14 276 / 289 (29 / 33), 900 x 9 258 / 267 (31 / 37).  Up to eight blocks what an item costs
// beside its tiles counts, and there are half as many here: 1000 x 3 88.5 / 64.6, 800 x 4 140 / 99, 2400 x 5 267 / 252, 600 x 6 123 / 117, 800 x 8 190 / 167.
// Two tiles an item are the least (see the softmax warps).
// Where other heads are sparse the two kernels run one after the other, and what the last, partly empty wave of
// this one leaves idle has to be won back: 16 heads x 317 blocks, four of them full (4.3 waves), 978 / 1007; 24 heads, six full
// (6.5 waves), 1435 / 1403; 48 x 122, twelve full (5.0 waves), 491 / 502.
int attn_dense_heads(const AttnArgs& a, int d, int sms) {
    int full = 0;
    while (full < a.H && a.k_per_head[a.head_order[full]] >= a.NB) ++full;
    if (full == 0 || d != dn::D || a.y != nullptr || a.NB < 3) return 0;
    const int64_t items = (int64_t)a.B * full * ((a.NB + 3) / 4), pairs = (int64_t)a.B * full * ((a.NB + 1) / 2);
    if (items > 1000000000LL) return 0;
    const int clusters = dense_clusters();
    if (clusters <= 0) return 0;
    const int64_t waves = (items + clusters - 1) / clusters;
    if (full == a.H) return a.NB <= 8 || 9 * waves < 10 * ((pairs + sms - 1) / sms) ? full : 0;
    return waves > 6 && 10 * items >= 9 * waves * clusters && 9 * waves * sms < 10 * pairs ? full : 0;
}

int launch_attn_dense(const AttnArgs& a, cudaStream_t st) {
    dn::Maps maps;
    int rc;
    if ((rc = t5::make_bhnd_map(&maps.q, a.q, a.sq, a.B, a.H, a.N, dn::D, "q")) != USV_OK) return rc;
    if ((rc = t5::make_bhnd_map(&maps.k, a.k, a.sk, a.B, a.H, a.N, dn::D, "k")) != USV_OK) return rc;
    if ((rc = t5::make_bhnd_map(&maps.v, a.v, a.sv, a.B, a.H, a.N, dn::D, "v")) != USV_OK) return rc;
    // (see launch_pair in usv_attn_pair.cu)
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, dn::attn_dense_kernel);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "sparse_attn: kernel attributes: %s", cudaGetErrorString(e));
    if (fa.numRegs * (dn::NTHREADS / 32) < 16 * dn::REG_SOFT + 4 * dn::REG_EPI + 4 * dn::REG_SERVICE)
        return fail(USV_ERR_UNSUPPORTED, "sparse_attn: kernel built with %d registers per thread, the roles need %d per lane",
                    fa.numRegs, 16 * dn::REG_SOFT + 4 * dn::REG_EPI + 4 * dn::REG_SERVICE);
    const int most = dense_clusters();
    if (most <= 0) return fail(USV_ERR_CUDA, "sparse_attn: no room for a cluster");
    const int64_t items = (int64_t)a.B * a.full_heads * ((a.NB + 3) / 4);
    const int clusters = items < most ? (int)items : most;
    launch_dep(dn::attn_dense_kernel, dim3(2 * clusters), dim3(dn::NTHREADS), dn::SMEM_BYTES, st, a, maps);
    USV_CHECK_LAUNCH("attn_dense_kernel");
    return USV_OK;
}

}  // namespace usv
