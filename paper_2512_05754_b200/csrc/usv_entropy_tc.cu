// Key marginal of the block-masked attention (Sec. 3.4, Eq. 16) on the 5th-generation tensor
// cores, head width D = 64 or 128.
//
//     abar[b,j] = 1/(H N) sum_h sum_i A(h,i,j),   A(h,i,j) = exp(scale <q_i,k_j> - lse_i)
//
// with lse_i the log-sum-exp the attention forward wrote.  Only the logits are needed, and the
// sum runs over the queries, so the product is taken transposed: one CTA per (b, h, two
// consecutive query blocks, in large calls two with overlapping lists; one in small calls) walks the union of the two
// lists two key blocks at a time and computes
//
//     S^T[128 keys x 128 queries] = K_tile . Q^T      tcgen05.mma, A = K tile in smem, B = Q in smem
//
// into one of two 128-column TMEM buffers.  Keys live on TMEM lanes: thread r of a warpgroup owns
// key r of the tile and one warpgroup serves each query block: it exponentiates the 64 logits of
// its side and adds their sum to abar with one atomic per key and tile; it skips a key block that
// its side did not select.  (With one query block a CTA each warpgroup takes half of the 64 logits.)  The log-sum-exps of the CTA's 128 queries lie in shared memory, where a
// warp's lanes read the same four at a time (a broadcast), so that no thread has to hold 64 of them and twice as
// many warps fit.  (As one more K = 16 step of the product, split into three bf16 terms, they cost nothing, but the
// tensor cores cut the sum off: entropies of 24 heads x 128 blocks were off by 2.1e-7 where they are off by
// 9e-8 now, and the call took 385 -> 367 us at D = 64, 437 -> 415 at D = 128, 512 blocks, keep 52.)
//
// Bounds at D = 128: 128 x 128 exponentials a tile are 1024 cycles at 16 a clock, less what one side
// skips; the tile's traffic through shared memory (32 KB in by TMA, 64 KB out to the MMAs) is
// 768, and 128 broadcasts of four log-sum-exps.  With one query block a CTA the traffic was 640 cycles for half as many exponentials.
// Measured with the entropy (us; one query block a CTA at D = 128, mma.sync at D = 64, before): 12 heads x 512
// blocks of random keys, keep 52, D = 128: 607 -> 437, D = 64: 1324 -> 385; 8 x 1182, keep 60, D = 128: 924 -> 820,
// D = 64: 2274 -> 690.
//
// The union is built as a list in shared memory (two bitmaps over the key blocks, compacted by one warp), or copied from
// the pairing plan of a large call.
// CTAs that run at the same time start at different entries of it, those near their own query blocks:
// their atomic adds would otherwise meet on the same keys.  A launch covers a window of 16 384 key blocks.
// Two CTAs share an SM and fill each other's gaps.  Warp 8 is the TMA producer, warp 9 the MMA
// issuer and TMEM owner.  All waits are bounded; a role that gives up raises the CTA's abort flag and
// the others follow.
#include "usv_attn.cuh"
#include "usv_entropy.cuh"
#include "usv_tcgen05.cuh"

namespace usv {

namespace et {

using namespace t5;

constexpr int KT = 2 * USV_BLOCK;               // keys per tile = two key blocks
constexpr int QT = 2 * USV_BLOCK;               // queries per CTA = two query blocks
constexpr int NBUF = 2;                         // S^T buffers of 128 columns
constexpr int WINDOW = 1 << 14;                 // key blocks a launch covers (16-bit list entries)
constexpr int64_t PLAN_MIN_WORK = 500000;       // kept key blocks over all query blocks

template <int D>
struct Cfg {
    static constexpr int NH = D / 64;                   // column halves of a tile
    static constexpr int KSTAGES = D == 64 ? 4 : 2;
    // every POLY-th pair of exponentials goes to the FMA pipe (12 heads at D = 128 / 24 at D = 64, 512 blocks of
    // video, keep 52, with the log-sum-exp inside the product: none 448 / 822 us, one in eight 439 / 820, in five
    // 439 / 775, in four 439 / 813)
    static constexpr int POLY = D == 64 ? 5 : 4;
    static constexpr uint32_t TILE_BYTES = KT * D * 2;  // [d-half][128 rows][128 B], for K and Q alike
    static constexpr uint32_t SM_Q = 0;
    static constexpr uint32_t SM_K = SM_Q + TILE_BYTES;
    static constexpr uint32_t SM_LSE = SM_K + KSTAGES * TILE_BYTES;    // float[QT]: minus the base-2 log-sum-exp
    static constexpr uint32_t SM_BAR = SM_LSE + QT * 4;
    static constexpr uint32_t SM_MISC = SM_BAR + 8 * 16;               // tmem base, abort flag, union size
    static constexpr uint32_t SM_LIST = SM_MISC + 64;                  // union: (key block - window) << 2 | in-A | in-B << 1
    enum { B_QFULL = 0, B_KFULL, B_KEMPTY = B_KFULL + KSTAGES, B_SFULL = B_KEMPTY + KSTAGES,
           B_SFREE = B_SFULL + NBUF, B_COUNT = B_SFREE + NBUF };
    static_assert(B_COUNT <= 16, "barrier area");
    static_assert(2 * (WINDOW / 32) * 4 <= KSTAGES * TILE_BYTES, "the bitmaps lie in the K stages");
    static size_t smem_bytes(int entries) { return SM_LIST + 2 * (size_t)entries + 1024; }   // + slack for alignment
};

constexpr uint32_t TMEM_COLS = NBUF * QT;
constexpr int NCONS = 256;                      // consumer threads: one warpgroup per query block
constexpr int NTHREADS = NCONS + 64;
constexpr int W_TMA = NCONS / 32, W_MMA = NCONS / 32 + 1;

struct Maps {
    CUtensorMap q, k;
};

// weights of two logits; pair i of a row, every POLY-th one on the FMA pipe
template <int POLY>
__device__ __forceinline__ uint64_t weight2(int i, uint32_t a, uint32_t b, uint64_t c2, uint64_t nl2) {
    const uint64_t x2 = fma_f32x2(pack_f32x2(__uint_as_float(a), __uint_as_float(b)), c2, nl2);
    float p0, p1;
    if (POLY && i % (POLY ? POLY : 1) == POLY - 1) {
        exp2_fma(x2, p0, p1);
    } else {
        float x0, x1;
        unpack_f32x2(x2, x0, x1);
        p0 = ex2(x0);
        p1 = ex2(x1);
    }
    return pack_f32x2(p0, p1);
}

// PER: query blocks a CTA; PLANNED: which two, and their union, come from a pairing plan
template <int D, int PER, bool PLANNED>
__global__ void __launch_bounds__(NTHREADS, 2)
marginal_tc_kernel(const MargArgs a, int w0, const __grid_constant__ Maps maps) {
    using F = Cfg<D>;
    constexpr int KSTAGES = F::KSTAGES;
    constexpr uint32_t TILE_BYTES = F::TILE_BYTES;
    // the set-up touches shared and tensor memory only; dep_sync() follows it, with the columns allocated
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* sm = smem_raw + (base - raw);
    auto bar = [&](int i) { return base + F::SM_BAR + 8u * i; };
    volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(sm + F::SM_MISC);
    volatile int* s_abort = reinterpret_cast<volatile int*>(sm + F::SM_MISC + 4);
    volatile int* s_union = reinterpret_cast<volatile int*>(sm + F::SM_MISC + 8);   // entries, first one taken
    uint32_t* s_bits = reinterpret_cast<uint32_t*>(sm + F::SM_K);
    uint16_t* s_list = reinterpret_cast<uint16_t*>(sm + F::SM_LIST);

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int N = a.N, NB = a.NB;
    const int NP = (NB + PER - 1) / PER, words = (min(NB - w0, WINDOW) + 31) >> 5;   // key blocks [w0, w0 + 32 words)
    const int bh = blockIdx.x / NP;
    const int b = bh / a.H, h = bh % a.H;
    const int kh = a.k_per_head[h];

    if (threadIdx.x < F::B_COUNT) {
        const int i = threadIdx.x;
        mbar_init(bar(i), (i >= F::B_SFREE && i < F::B_SFREE + NBUF) ? NCONS / 32 : 1);
        if (i == 0) { *s_abort = 0; s_union[1] = 0; }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; !PLANNED && i < 2 * words; i += NTHREADS) s_bits[i] = 0;
    if (warp == W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + F::SM_MISC), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    dep_sync();
    const uint32_t tmem = *s_tmem;

    // the CTA's query blocks, the second one -1 or NB where there is none
    const int2 blk = PLANNED ? a.pairs[blockIdx.x] : make_int2(PER * (blockIdx.x % NP), PER * (blockIdx.x % NP) + 1);
    const int I = blk.x, last = min(I + PER, NB);   // (without a plan the CTA has blocks [I, last))

    // ---- the query rows on their way, the lists as bitmaps, the log-sum-exps
    if (warp == W_TMA && elect_one()) {
        const int hq = a.sq.sh ? h : 0, bq = a.sq.sb ? b : 0;
        mbar_expect_tx(bar(F::B_QFULL), TILE_BYTES / 2 * PER);
#pragma unroll
        for (int hf = 0; hf < F::NH; ++hf)
#pragma unroll
            for (int p = 0; p < PER; ++p)
                tma_load_4d(base + F::SM_Q + hf * 16384 + p * 8192, &maps.q, bar(F::B_QFULL), hf * 64,
                            (p == 0 ? I : (blk.y < 0 ? NB : blk.y)) * USV_BLOCK, hq, bq);   // (rows past the end: zeros)
    }
    for (int i = threadIdx.x; !PLANNED && i < PER * kh; i += NTHREADS) {
        const int side = i >= kh;
        if (I + side >= last) continue;
        const int e = a.sel[((int64_t)bh * NB + I + side) * a.kmax + (i - side * kh)];
        if (e >= w0 && e < NB && e - w0 < WINDOW) atomicOr(&s_bits[side * words + ((e - w0) >> 5)], 1u << (e & 31));
    }
    if (threadIdx.x < USV_BLOCK * PER) {
        // a query at or beyond N counts nothing
        const int row = (threadIdx.x < USV_BLOCK ? I : blk.y) * USV_BLOCK + (threadIdx.x & (USV_BLOCK - 1));
        reinterpret_cast<float*>(sm + F::SM_LSE)[threadIdx.x] =
            row >= 0 && row < N ? -a.lse[(int64_t)bh * N + row] * 1.4426950408889634f : -INFINITY;
    }
    if (PLANNED) {
        const int* pl = a.lists + b * a.list_batch + a.list_off[h] + (int64_t)(blockIdx.x % NP) * list_stride(kh, NB);
        const int n = __ldg(pl);
        int before = 0;   // entries below the CTA's own block
        for (int i = threadIdx.x; i < n; i += NTHREADS) {
            const int e = __ldg(pl + 1 + i);
            s_list[i] = (uint16_t)e;
            before += (e >> 2) < I;
        }
        before = __reduce_add_sync(0xffffffffu, before);
        if (lane == 0 && before) atomicAdd(const_cast<int*>(s_union + 1), before);
        if (threadIdx.x == 0) s_union[0] = n;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (!PLANNED && warp == 0) {
        int n = 0;
        for (int i0 = 0; i0 < words; i0 += 32) {
            const int i = i0 + lane;
            const uint32_t ba = i < words ? s_bits[i] : 0, bb = i < words ? s_bits[words + i] : 0;
            uint32_t m = ba | bb;
            const int incl = warp_incl_scan(__popc(m));
            int at = n + incl - __popc(m);
            if (i == (I - w0) >> 5) s_union[1] = at;
            for (; m; m &= m - 1) {
                const int bit = __ffs(m) - 1;
                s_list[at++] = (uint16_t)((i * 32 + bit) << 2 | ((ba >> bit) & 1u) | ((bb >> bit) & 1u) << 1);
            }
            n += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) s_union[0] = n;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the K stages go to the TMA
    }
    if (!PLANNED) __syncthreads();
    const int nU = s_union[0], T = (nU + 1) >> 1;   // tiles of two key blocks
    const int first = s_union[1] < nU ? s_union[1] : 0;
    // n-th entry from `first` on, around the end; 0 (no side) behind the last one
    auto entry = [&](int n) -> int {
        const int i = first + n;
        return n < nU ? s_list[i < nU ? i : i - nU] : 0;
    };

    if (warp == W_TMA) {
        // ===== producer: the key tiles =============================================================
        const int hk = a.sk.sh ? h : 0, bk = a.sk.sb ? b : 0;
        for (int t = 0; t < T; ++t) {
            const int s = t % KSTAGES;
            const int J0 = w0 + (entry(2 * t) >> 2), J1 = w0 + (entry(2 * t + 1) >> 2);   // odd tail: any tile, not counted
            if (!mbar_wait(bar(F::B_KEMPTY + s), ((t / KSTAGES) & 1) ^ 1, s_abort, a.status, 0x1000000u)) break;
            const uint32_t dst = base + F::SM_K + s * TILE_BYTES;
            if (elect_one()) {
                mbar_expect_tx(bar(F::B_KFULL + s), TILE_BYTES);
#pragma unroll
                for (int hf = 0; hf < F::NH; ++hf) {
                    tma_load_4d(dst + hf * 16384, &maps.k, bar(F::B_KFULL + s), hf * 64, J0 * USV_BLOCK, hk, bk);
                    tma_load_4d(dst + hf * 16384 + 8192, &maps.k, bar(F::B_KFULL + s), hf * 64, J1 * USV_BLOCK, hk, bk);
                }
            }
            __syncwarp();
        }
    } else if (warp == W_MMA) {
        // ===== MMA issuer ==========================================================================
        constexpr uint32_t IDESC = instr_desc(128, USV_BLOCK * PER, 0, 0);    // K tile (K-major) x Q (K-major)
        const uint64_t kdesc0 = smem_desc(base + F::SM_K, 16, 1024);
        const uint64_t qdesc0 = smem_desc(base + F::SM_Q, 16, 1024);
        bool ok = mbar_wait(bar(F::B_QFULL), 0, s_abort, a.status, 0x2000000u);
        for (int t = 0; ok && t < T; ++t) {
            const int s = t % KSTAGES;
            const int bf = t % NBUF;
            if (!mbar_wait(bar(F::B_KFULL + s), (t / KSTAGES) & 1, s_abort, a.status, 0x4000000u)) break;
            if (t >= NBUF && !mbar_wait(bar(F::B_SFREE + bf), ((t / NBUF) - 1) & 1, s_abort, a.status, 0x8000000u)) break;
            fence_after();
            const uint64_t kdesc = kdesc0 + ((s * TILE_BYTES) >> 4);
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const uint32_t off = ((ks >> 2) * 16384 + (ks & 3) * 32) >> 4;
                    umma_ss(tmem + bf * QT, kdesc + off, qdesc0 + off, IDESC, ks > 0);
                }
                umma_commit(bar(F::B_SFULL + bf));
                umma_commit(bar(F::B_KEMPTY + s));
            }
            __syncwarp();
        }
    } else {
        // ===== consumers: thread r of a group <-> TMEM lane r <-> key r of the tile =================
        const int grp = warp >> 2;                      // the warpgroup's query block, or (PER = 1) its half of the queries
        const int side = PER == 2 ? grp : 0;
        const int r = threadIdx.x & 127;
        const int second = r >> 6;                      // which key block of the tile (uniform per warp)
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + grp * (32 * PER);
        const uint64_t c2 = both(a.scale_log2);
        const ulonglong2* nl2 = reinterpret_cast<const ulonglong2*>(sm + F::SM_LSE) + grp * (8 * PER);
        float* marg = a.marg + (int64_t)b * N;
        for (int t = 0; t < T; ++t) {
            const int bf = t % NBUF;
            const int e = entry(2 * t + second);
            const bool mine = (e >> side) & 1;
            if (!mbar_wait(bar(F::B_SFULL + bf), (t / NBUF) & 1, s_abort, a.status, 0x10000000u)) break;
            if (!mine) {
                if (lane == 0) mbar_arrive(bar(F::B_SFREE + bf));
                continue;
            }
            fence_after();
            uint32_t sx[32 * PER];
#pragma unroll
            for (int p = 0; p < PER; ++p) tmem_ld32(lane_base + bf * QT + p * 32, sx + p * 32);
            tmem_wait_ld();
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(F::B_SFREE + bf));   // the logits are in registers
            uint64_t acc[2] = {0, 0};
#pragma unroll
            for (int i = 0; i < 16 * PER; i += 2) {
                const ulonglong2 n = nl2[i / 2];
                uint64_t& to = acc[PER == 2 ? i / 16 : (i / 2) & 1];
                to = add_f32x2(to, weight2<F::POLY>(i, sx[2 * i], sx[2 * i + 1], c2, n.x));
                to = add_f32x2(to, weight2<F::POLY>(i + 1, sx[2 * i + 2], sx[2 * i + 3], c2, n.y));
            }
            float x, y;
            unpack_f32x2(add_f32x2(acc[0], acc[1]), x, y);
            const int j = (w0 + (e >> 2)) * USV_BLOCK + (r & 63);
            if (j < N) atomicAdd(marg + j, (x + y) * a.inv_hn);
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
    if (warp == W_MMA) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

template <int D, int PER, bool PLANNED>
static int launch(const MargArgs& a, cudaStream_t st) {
    Maps maps;
    int rc;
    if ((rc = make_bhnd_map(&maps.q, a.q, a.sq, a.B, a.H, a.N, D, "q")) != USV_OK) return rc;
    if ((rc = make_bhnd_map(&maps.k, a.k, a.sk, a.B, a.H, a.N, D, "k")) != USV_OK) return rc;
    const int64_t grid = (int64_t)a.B * a.H * ((a.NB + PER - 1) / PER);
    int kmx = 0;
    for (int h = 0; h < a.H; ++h) kmx = a.k_per_head[h] > kmx ? a.k_per_head[h] : kmx;
    const int widest = a.NB < WINDOW ? a.NB : WINDOW;
    const size_t smem = Cfg<D>::smem_bytes(widest < 2 * kmx ? widest : 2 * kmx);
    // (the limit is the function's, not the call's: always the most any call needs, for calls from several threads)
    cudaError_t e = cudaFuncSetAttribute(marginal_tc_kernel<D, PER, PLANNED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Cfg<D>::smem_bytes(WINDOW));
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "attn_entropy: smem attribute: %s", cudaGetErrorString(e));
    for (int w0 = 0; w0 < a.NB; w0 += WINDOW) {
        launch_dep_smem(marginal_tc_kernel<D, PER, PLANNED>, dim3((unsigned)grid), dim3(NTHREADS), smem, st, a, w0, maps);
        USV_CHECK_LAUNCH("marginal_tc_kernel");
    }
    return USV_OK;
}

}  // namespace et

static bool marginal_single(const MargArgs& a, int sms) {
    // One query block a CTA where all of them are resident together (two CTAs an SM): such a call takes as long as one walk
    // over a list, and a union is longer than a list.  So too, up to twice as many, where lists are long and hold so little
    // of the sequence that neighbours need not share much.  Marginal + entropy, us, two blocks a CTA / one, D = 128 (D = 64),
    // random lists: 2 x 16 blocks, keep 4 12.4 / 10.4 (12.3 / 10.4); 200, keep 100 59.2 / 47.8 (54.5 / 45.1); 2 x 160, keep 16
    // 22.4 / 21.3 (20.1 / 20.1), keep 32 34.8 / 31.0 (31.1 / 29.4); 12 x 32, keep 7 13.8 / 15.2 (13.0 / 14.4); 8 x 48, keep 16
    // 20.6 / 20.8 (19.8 / 19.6); 12 x 64, keep 16 29.8 / 32.6 (27.9 / 30.5).
    int kmx = 0;
    for (int h = 0; h < a.H; ++h) kmx = a.k_per_head[h] > kmx ? a.k_per_head[h] : kmx;
    const int64_t blocks = (int64_t)a.B * a.H * a.NB;
    return blocks <= 2 * sms || (blocks <= 4 * sms && kmx >= 16 && 4 * kmx <= a.NB);
}

// The plan costs 8 to 20 us (40 where the blocks are ordered first) and takes a quarter of the tiles away: the union of two
// paired lists is 1.28 to 1.35 times a list, that of neighbours in index 1.9 times.  Marginal + entropy of video inputs, us,
// neighbours / paired: 12 heads x 122 blocks, keep 13 48 / 58; 12 x 317, keep 39 226 / 220; 12 x 512, keep 52 496 / 493;
// 24 x 512 at D = 64 786 / 750; 40 x 1182, keep 60 5074 / 4405; 12 x 3023, keep 152 10 093 / 8139.  Long lists overlap
// anyway: 12 x 512, keep 180 1573 / 1578; 16 x 317, keep 317, 80, 32 and 16 851 / 838.
bool marginal_planned(const MargArgs& a, int sms) {
    int64_t kept = 0;
    int heads = 0;
    for (int h = 0; h < a.H; ++h)
        if (a.k_per_head[h] < a.NB) {
            kept += a.k_per_head[h];
            ++heads;
        }
    return a.NB <= PLAN_MAX_NB && !marginal_single(a, sms) && (int64_t)a.B * a.NB * kept >= et::PLAN_MIN_WORK &&
           4 * kept <= (int64_t)heads * a.NB;
}

size_t marginal_plan_bytes(int B, int H, int NB, int kmax) {
    const int k = kmax < 1 ? 1 : (kmax > NB ? NB : kmax);
    if (NB > PLAN_MAX_NB || (int64_t)B * H * NB * k < et::PLAN_MIN_WORK) return 0;   // (see marginal_planned)
    int32_t kk[USV_MAX_HEADS];
    for (int h = 0; h < H; ++h) kk[h] = k;
    return pair_plan_bytes(B, H, NB, kk);
}

int launch_marginal_plan(MargArgs& a, void* mem, cudaStream_t st) {
    AttnArgs p = {};
    p.sel = a.sel;
    p.status = a.status;
    p.B = a.B; p.H = a.H; p.N = a.N; p.NB = a.NB; p.kmax = a.kmax;
    for (int h = 0; h < a.H; ++h) p.k_per_head[h] = a.k_per_head[h];
    const int rc = launch_pair_plan(p, mem, st);
    if (rc != USV_OK) return rc;
    a.pairs = p.pairs;
    a.lists = p.lists;
    a.list_batch = p.list_batch;
    for (int h = 0; h < a.H; ++h) a.list_off[h] = p.list_off[h];
    return USV_OK;
}

int launch_marginal_tc(const MargArgs& a, int d, cudaStream_t st) {
    int rc, sms;
    if ((rc = sm_count(&sms)) != USV_OK) return rc;
    if (a.pairs != nullptr) return d == 64 ? et::launch<64, 2, true>(a, st) : et::launch<128, 2, true>(a, st);
    const bool one = marginal_single(a, sms);
    if (d == 64) return one ? et::launch<64, 1, false>(a, st) : et::launch<64, 2, false>(a, st);
    return one ? et::launch<128, 1, false>(a, st) : et::launch<128, 2, false>(a, st);
}

}  // namespace usv
