// Pairing plan of the block-sparse attention kernel.
//
// The tcgen05 kernel computes two query blocks per work item over the UNION of their key-block
// lists, so it pays for every key block only one of the two selected.  Which blocks are paired is
// free: this file chooses, per (batch, head), a pairing with large list overlaps.
//
// pair_plan_kernel works inside chunks of 128 query blocks: bitmaps, all-pairs overlaps, a greedy
// matching, the union lists.  Small calls are cut into chunks in index order.  In long sequences a
// block's best partner usually lies more than a chunk away (the same place in a neighbouring
// frame), so the blocks are first put in an order that brings similar lists together: by the minimum
// of a hash over the list, which two lists share with the probability of their overlap over
// their union (Broder, "On the resemblance and containment of documents", 1997).  The first pass keeps
// what its first two rounds match; the blocks left go through a second pass in the order of a second
// hash.  Unions, and with them the attention kernel's time, shrink: 40 heads x 1182 blocks, keep 60,
// 5650 -> 5380 us; 12 x 3023, keep 152, 11.9 -> 10.8 ms.
//   plan_keys_kernel   both sort keys of every block's list (one warp per block)
//   plan_sort_kernel   the blocks of a head in the order of either key
//
// The result only affects speed: any pairing gives the same attention output.
#include "usv_attn.cuh"
#include "usv_tcgen05.cuh"

namespace usv {

namespace plan {

constexpr int ORDER_MIN_NB = 400;                 // four chunks and more
constexpr int64_t ORDER_MIN_WORK = 1000000;       // kept key blocks over all query blocks (see plan_ordered)
constexpr int ROUNDS_FIRST = 2;   // rounds of the first of two passes
constexpr int ROUNDS = 5;      // upper limit; the matching stops as soon as a round finds nothing new
constexpr int CH = 128;        // query blocks per chunk
constexpr int THREADS = 4 * CH;
// bitmap row pitch in 32-bit words: whole slabs, and 4 x odd (consecutive rows start in different banks)
__host__ __device__ inline int plan_pitch(int nwords) { return (nwords + 7) / 8 * 8 + 4; }
constexpr uint32_t SLAB = CH * 128;   // 128 key blocks of every row of the chunk, one byte each, 128-byte swizzle
constexpr int OVP = CH + 8;     // row pitch of the overlap matrix (uint16): rows start 4 banks apart
static_assert(CH * OVP * 2 <= 3 * SLAB, "the overlaps take the place of the slabs");

// How the query blocks of a head get into chunks, and what the two passes share.
struct Order {
    const uint16_t* by_rank;   // [2][B*H][NB] blocks in the order of either key
    uint8_t* taken;            // [B*H][NB] written by the first pass: 1 = paired
    int* count;                // [B*H] pairs written so far (starts at zero)
    int pass;                  // 0: one pass in index order (the rest unused); 1, 2: first and second of two
};

__device__ __forceinline__ uint32_t mix12(uint32_t x, uint32_t a, uint32_t b) {   // a bijection of 0 .. 4095
    x = (x * a) & 4095u;
    x ^= x >> 7;
    x = (x * b) & 4095u;
    return x ^ (x >> 5);
}

// keys [2][B*H][NB]: (smallest hash of the list's blocks, 12 bits | a second one, 8 bits | block, 12 bits).
// Also clears what pair_plan_kernel counts in.
__global__ void __launch_bounds__(256) plan_keys_kernel(const AttnArgs a, uint32_t* __restrict__ keys, int* __restrict__ count) {
    dep_sync();
    const int NB = a.NB;
    const int64_t rows = (int64_t)a.B * a.H * NB;
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (t < a.B * a.H) count[t] = 0;
    const int64_t row = t >> 5;
    if (row >= rows) return;
    const int lane = threadIdx.x & 31;
    const int bh = (int)(row / NB), I = (int)(row - (int64_t)bh * NB);
    const int kh = a.k_per_head[bh % a.H];
    const int32_t* sel = a.sel + row * a.kmax;
    uint32_t m0 = 0x0fff0fffu, m1 = 0x0fff0fffu;   // two 16-bit minima each
#pragma unroll 4
    for (int i = lane; i < kh; i += 32) {
        const uint32_t J = (uint32_t)sel[i];
        if (J < (uint32_t)NB) {
            m0 = __vminu2(m0, mix12(J, 2909, 1597) | (mix12(J, 1709, 3037) << 16));
            m1 = __vminu2(m1, mix12(J, 3461, 2273) | (mix12(J, 1181, 3701) << 16));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m0 = __vminu2(m0, __shfl_xor_sync(0xffffffffu, m0, o));
        m1 = __vminu2(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    }
    if (lane == 0) {
        keys[row] = (m0 & 0xffffu) << 20 | min(m0 >> 16, 255u) << 12 | (uint32_t)I;
        keys[rows + row] = (m1 & 0xffffu) << 20 | min(m1 >> 16, 255u) << 12 | (uint32_t)I;
    }
}

// by_rank [2][B*H][NB]: the blocks of one (b, h) in the order of one of its keys.  Bitonic sort of 4096
// keys by one CTA, four consecutive ones per thread: exchanges stay in registers, in the warp
// (shuffles), or go through shared memory.  (Gathering equal hashes and ranking inside each group took
// 7 to 59 us, the most where hashes are popular; this 6 to 10 us.)
__global__ void __launch_bounds__(1024) plan_sort_kernel(int NB, const uint32_t* __restrict__ keys, uint16_t* __restrict__ by_rank) {
    dep_sync();
    __shared__ uint4 s_x[2][1024];
    const int64_t base = (int64_t)blockIdx.x * NB;
    const int t = threadIdx.x;
    uint32_t x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = 4 * t + q < NB ? keys[base + 4 * t + q] : 0xffffffffu;
    int buf = 0;
#pragma unroll
    for (int k = 2; k <= 4096; k <<= 1) {
        if (k >> 1 >= NB) break;   // (places from NB on hold the largest key: already in order)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j < 4) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if ((q & j) == 0) {
                        const uint32_t lo = min(x[q], x[q ^ j]), hi = max(x[q], x[q ^ j]);
                        const bool up = ((4 * t + q) & k) == 0;
                        x[q] = up ? lo : hi;
                        x[q ^ j] = up ? hi : lo;
                    }
            } else {
                const bool take_min = ((4 * t & k) == 0) == ((4 * t & j) == 0);
                uint32_t y[4];
                if (j < 128) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) y[q] = __shfl_xor_sync(0xffffffffu, x[q], j / 4);
                } else {
                    s_x[buf][t] = make_uint4(x[0], x[1], x[2], x[3]);
                    __syncthreads();
                    const uint4 v = s_x[buf][t ^ (j / 4)];
                    y[0] = v.x; y[1] = v.y; y[2] = v.z; y[3] = v.w;
                    buf ^= 1;   // (two buffers: one barrier per exchange is enough)
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) x[q] = take_min ? min(x[q], y[q]) : max(x[q], y[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (4 * t + q < NB) by_rank[base + 4 * t + q] = (uint16_t)(x[q] & 4095u);
}

// The ascending union of two bitmaps over the key blocks, each entry flagged with the row(s) it is from (bitsB NULL: one row);
// a warp's work.  out[0]: number of entries.
__device__ __forceinline__ void write_union(const uint32_t* bitsA, const uint32_t* bitsB, int nwords, int* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    int running = 0;
    for (int w0 = 0; w0 < nwords; w0 += 32) {
        const int w = w0 + lane;
        const uint32_t ba = w < nwords ? bitsA[w] : 0u;
        const uint32_t bb = (w < nwords && bitsB != nullptr) ? bitsB[w] : 0u;
        uint32_t u = ba | bb;
        const int incl = warp_incl_scan(__popc(u));
        int off = running + incl - __popc(u);
        while (u) {
            const int bit = __ffs(u) - 1;
            u &= u - 1;
            out[1 + off++] = ((w * 32 + bit) << 2) | ((ba >> bit) & 1u) | (((bb >> bit) & 1u) << 1);
        }
        running += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) out[0] = running;
}

// One CTA per chunk of CH query blocks of one (batch, head).
//   1. bitmaps of the chunk's selection rows (shared memory)
//   2. overlap |sel(I) & sel(J)| of every two blocks of the chunk
//   3. rounds of "mutual best free partner" (larger overlap first, then the lower block) until a
//      round matches nobody; what is left is paired in index order, an odd block out stays single
//   4. the pairs ordered by their lower block -> pairs[chunk * CH / 2 ...]
//   5. ascending union of the two rows of every pair, each entry flagged with the side(s) that
//      selected it (one warp per pair)
__global__ void __launch_bounds__(THREADS, 2)
pair_plan_kernel(const AttnArgs a, int2* __restrict__ pairs, int* __restrict__ lists, const Order ord, int nbuf) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = t5::smem_u32(smem_raw), slabs = (raw + 1023u) & ~1023u;
    // overlaps [CH][OVP] (rows 16-byte aligned), in the place of the nbuf slabs they come from; bitmaps [CH][pitch]
    uint16_t* ov = reinterpret_cast<uint16_t*>(smem_raw + (slabs - raw));
    uint32_t* bm = reinterpret_cast<uint32_t*>(smem_raw + (slabs - raw) + nbuf * SLAB);
    __shared__ __align__(8) unsigned long long s_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ int s_blk[CH];               // the chunk's query blocks
    __shared__ int s_scan[THREADS / 32 + 1], s_base;
    __shared__ int16_t partner[CH];
    __shared__ int16_t best[CH];
    __shared__ int16_t order[CH];           // ranks -> blocks (singles, then lower blocks of the pairs)
    __shared__ uint32_t freebits[CH / 32];  // bit set while the block is unmatched
    __shared__ int s_new[2], s_count;       // s_new: one flag per round parity (reset while the other is read)
    const int NB = a.NB;
    const int NP = (NB + 1) >> 1;
    const int nwords = (NB + 31) >> 5;
    const int pitch = plan_pitch(nwords);
    const int bh = blockIdx.y;
    const int b = bh / a.H, h = bh % a.H;
    const int kh = a.k_per_head[h];
    const int I0 = blockIdx.x * CH;
    int nI = min(CH, NB - I0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int2* out_pairs = pairs + (int64_t)bh * NP;
    const int npairs = (nI + 1) >> 1;
    const int lstride = (int)list_stride(kh, NB);
    int* out_lists = lists + b * a.list_batch + a.list_off[h];

    // The attention kernel may start once the columns are allocated (see dep_sync()), and not before this kernel does:
    // its CTAs, already resident, would leave room for one CTA of this kernel an SM instead of two (D = 64, 12 heads x 256
    // blocks, keep 26: 134 us a call, 138 with the wait behind the signal).
    dep_wait();
    const bool full = kh >= NB;   // every list is the full set but for holes: no overlaps to compute
    if (warp == 0 && !full) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(t5::smem_u32(&s_tmem)), "r"(128u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        t5::mbar_init(t5::smem_u32(&s_bar), 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    t5::fence_before();
    __syncthreads();
    t5::fence_after();
    dep_launch();
    const uint32_t tmem = full ? 0 : s_tmem;
    auto release = [&] {
        if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128u) : "memory");
    };
    // the words behind the sticky status word (fallback count, work counter, ...) start at zero
    if (a.work_counter != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < (WS_HEADER - 4) / 4) a.status[1 + threadIdx.x] = 0u;

    if (full) {
        if (ord.pass == 2 || a.full_heads > 0) return;   // (done by the first pass, or not wanted)
        out_pairs += blockIdx.x * (CH / 2);
        out_lists += (int64_t)blockIdx.x * (CH / 2) * lstride;
        // every list is the full set unless it has holes: pairing is arbitrary and every key block belongs to both sides
        for (int p = threadIdx.x; p < npairs; p += THREADS)
            out_pairs[p] = make_int2(I0 + 2 * p, 2 * p + 1 < nI ? I0 + 2 * p + 1 : -1);
        // pairs warp, warp + 16, ...: their rows are read together (one pair after the other 8 heads x 101 blocks took 7 us longer)
        constexpr int WARPS = THREADS / 32, P = CH / 2 / WARPS;
        const int32_t* rows = a.sel + ((int64_t)bh * NB + I0 + 2 * warp) * a.kmax;
        auto row = [&](int i, int side) { return rows + (int64_t)(2 * WARPS * i + side) * a.kmax; };
        auto in = [&](int i, int side) { return 2 * (warp + WARPS * i) + side < nI; };
        bool hole[P] = {};
#pragma unroll 2
        for (int j = lane; j < NB; j += 32) {
            int at[P][2];
#pragma unroll
            for (int i = 0; i < P; ++i)
#pragma unroll
                for (int side = 0; side < 2; ++side) at[i][side] = in(i, side) ? __ldg(row(i, side) + j) : 0;
#pragma unroll
            for (int i = 0; i < P; ++i) {
                hole[i] |= (unsigned)at[i][0] >= (unsigned)NB || (unsigned)at[i][1] >= (unsigned)NB;
                if (in(i, 0)) out_lists[(int64_t)(warp + WARPS * i) * lstride + 1 + j] = (j << 2) | (in(i, 1) ? 3 : 1);
            }
        }
        uint32_t* mine = bm + 2 * warp * pitch;
#pragma unroll 1
        for (int i = 0; i < P && in(i, 0); ++i) {
            int* out = out_lists + (int64_t)(warp + WARPS * i) * lstride;
            if (lane == 0) out[0] = NB;
            bool any = false;
#pragma unroll
            for (int q = 0; q < P; ++q) any = q == i ? hole[q] : any;
            if (!__any_sync(0xffffffffu, any)) continue;
            for (int w = lane; w < 2 * pitch; w += 32) mine[w] = 0u;
            __syncwarp();
            for (int j = lane; j < NB; j += 32) {
                const unsigned ja = __ldg(row(i, 0) + j), jb = in(i, 1) ? __ldg(row(i, 1) + j) : -1;
                if (ja < (unsigned)NB) atomicOr(&mine[ja >> 5], 1u << (ja & 31));
                if (jb < (unsigned)NB) atomicOr(&mine[pitch + (jb >> 5)], 1u << (jb & 31));
            }
            __syncwarp();
            write_union(mine, mine + pitch, nwords, out);
            __syncwarp();
        }
        return;
    }

    // the chunk's query blocks
    if (ord.pass == 2) {
        // blocks the first pass left, in the order of the second key: the CTA finds its own 128 of them
        const uint16_t* order = ord.by_rank + ((int64_t)gridDim.y + bh) * NB;
        const uint8_t* taken = ord.taken + (int64_t)bh * NB;
        const int per = (NB + THREADS - 1) / THREADS, r0 = threadIdx.x * per;   // per <= 8
        uint32_t free = 0;
        for (int i = 0; i < per; ++i)
            if (r0 + i < NB && !taken[order[r0 + i]]) free |= 1u << i;
        const int incl = warp_incl_scan(__popc(free));
        if (lane == 31) s_scan[warp + 1] = incl;
        __syncthreads();
        if (threadIdx.x == 0) {
            s_scan[0] = 0;
            for (int w = 0; w < THREADS / 32; ++w) s_scan[w + 1] += s_scan[w];
        }
        __syncthreads();
        int at = s_scan[warp] + incl - __popc(free) - I0;
        for (int i = 0; i < per; ++i)
            if ((free >> i) & 1u) {
                if (at >= 0 && at < CH) s_blk[at] = order[r0 + i];
                ++at;
            }
        nI = min(CH, s_scan[THREADS / 32] - I0);
        if (nI <= 0) {         // uniform
            release();
            return;
        }
    } else if (threadIdx.x < nI) {
        s_blk[threadIdx.x] = ord.pass == 1 ? ord.by_rank[(int64_t)bh * NB + I0 + threadIdx.x] : I0 + threadIdx.x;
    }

    // 1. bitmaps
    for (int i = threadIdx.x; i < CH * pitch; i += THREADS) bm[i] = 0u;
    __syncthreads();
    {
        // eight rows a warp, their loads in flight together
        constexpr int R = CH / (THREADS / 32);
        const int32_t* src[R];
#pragma unroll
        for (int r = 0; r < R; ++r)
            src[r] = warp * R + r < nI ? a.sel + ((int64_t)bh * NB + s_blk[warp * R + r]) * a.kmax : nullptr;
        uint32_t* rows = bm + warp * R * pitch;
#pragma unroll 2
        for (int i = lane; i < kh; i += 32) {
            int J[R];
#pragma unroll
            for (int r = 0; r < R; ++r) J[r] = src[r] != nullptr ? src[r][i] : -1;
#pragma unroll
            for (int r = 0; r < R; ++r)
                if ((unsigned)J[r] < (unsigned)NB) atomicOr(&rows[r * pitch + (J[r] >> 5)], 1u << (J[r] & 31));
        }
    }
    if (threadIdx.x < CH) partner[threadIdx.x] = -1;
    if (threadIdx.x < CH / 32) {
        const int first = threadIdx.x * 32;
        freebits[threadIdx.x] = first >= nI ? 0u : (nI - first >= 32 ? 0xffffffffu : (1u << (nI - first)) - 1u);
    }
    __syncthreads();

    // 2. overlaps of every two blocks of the chunk: the product of the 0/1 matrix of the rows with its own
    // transpose.  The bits become bytes (e4m3 2^-9: products of 2^-18 add up exactly) in slabs of 128 key
    // blocks, as many at a time as there is room for, which the tensor cores multiply.  (128 rows of
    // 3023 key blocks took 62 k cycles with AND + popcount; the single-bit mma.sync is no faster.)
    const int nsl = (nwords + 3) >> 2;
    bool ok = true;
    int steps = 0;
    for (int s0 = 0; s0 < nsl; s0 += nbuf, ++steps) {
        const int n = min(nbuf, nsl - s0);
        if (steps > 0) ok = t5::mbar_wait(t5::smem_u32(&s_bar), (steps - 1) & 1, &s_abort, a.status, 0x20000000u) && ok;
        const int row = threadIdx.x & (CH - 1), word = threadIdx.x / CH;   // 4 words of every row and slab
        for (int sl = 0; sl < n; ++sl) {
            const uint32_t w = bm[row * pitch + (s0 + sl) * 4 + word];
            unsigned char* line = reinterpret_cast<unsigned char*>(ov) + sl * SLAB + row * 128;
            auto spread = [&](int nibble) { return (((w >> (4 * nibble)) & 15u) * 0x00204081u) & 0x01010101u; };
#pragma unroll
            for (int c = 0; c < 2; ++c)
                *reinterpret_cast<uint4*>(line + (((2 * word + c) ^ (row & 7)) << 4)) =
                    make_uint4(spread(4 * c), spread(4 * c + 1), spread(4 * c + 2), spread(4 * c + 3));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (warp == 0) {
            if (t5::elect_one()) {
                t5::fence_after();
                for (int sl = 0; sl < n; ++sl) {
                    const uint64_t desc = t5::smem_desc(slabs + sl * SLAB, 16, 1024);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        t5::umma_ss_f8(tmem, desc + ks * 2, desc + ks * 2, t5::instr_desc_e4m3(CH, CH), s0 + sl > 0 || ks > 0);
                }
                t5::umma_commit(t5::smem_u32(&s_bar));
            }
            __syncwarp();
        }
    }
    ok = t5::mbar_wait(t5::smem_u32(&s_bar), (steps - 1) & 1, &s_abort, a.status, 0x20000000u) && ok;
    t5::fence_after();
    __syncthreads();   // the slabs are free
    {
        // warp w: TMEM lanes (rows) of quarter w & 3, columns 32 (w >> 2) ...
        uint32_t d[32];
        t5::tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * 32, d);
        t5::tmem_wait_ld();
        uint4* out = reinterpret_cast<uint4*>(ov + ((warp & 3) * 32 + lane) * OVP + (warp >> 2) * 32);
        auto count = [&](int i) { return ok ? (uint32_t)(__uint_as_float(d[i]) * 262144.0f) : 0u; };   // (a wait that gave up: any pairing will do)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            out[q] = make_uint4(count(8 * q) | count(8 * q + 1) << 16, count(8 * q + 2) | count(8 * q + 3) << 16,
                                count(8 * q + 4) | count(8 * q + 5) << 16, count(8 * q + 6) | count(8 * q + 7) << 16);
    }
    t5::fence_before();
    __syncthreads();
    t5::fence_after();
    release();

    // 3. matching: four threads per block, each scans a quarter of the chunk (four 16-byte loads);
    // key = overlap << 8 | (CH - 1 - j): the largest key is the largest overlap, then the lowest block
    {
        const int i = threadIdx.x >> 2, quarter = threadIdx.x & 3;
        const int j0 = quarter * (CH / 4);
        const uint4* row = reinterpret_cast<const uint4*>(ov + i * OVP + j0);
        const int rounds = ord.pass == 1 ? ROUNDS_FIRST : ROUNDS;
        for (int r = 0; r < rounds; ++r) {
            if (threadIdx.x == 0) s_new[r & 1] = 0;
            uint32_t bk = 0;
            if (i < nI && ((freebits[i >> 5] >> (i & 31)) & 1u)) {
                uint32_t mask = freebits[j0 >> 5];
                if (i >= j0 && i < j0 + CH / 4) mask &= ~(1u << (i - j0));
#pragma unroll
                for (int u = 0; u < CH / 32; ++u) {
                    const uint4 v = row[u];
                    const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int c = u * 8 + e;
                        const uint32_t o = (wv[e >> 1] >> ((e & 1) * 16)) & 0xffffu;
                        const uint32_t key = ((o + 1u) << 8) | (uint32_t)(CH - 1 - (j0 + c));
                        bk = max(bk, ((mask >> c) & 1u) ? key : 0u);
                    }
                }
            }
            bk = max(bk, __shfl_xor_sync(0xffffffffu, bk, 1));
            bk = max(bk, __shfl_xor_sync(0xffffffffu, bk, 2));
            if (quarter == 0) best[i] = bk ? (int16_t)(CH - 1 - (int)(bk & 0xffu)) : (int16_t)-1;
            __syncthreads();
            if (threadIdx.x < nI) {
                const int me = threadIdx.x, j = best[me];
                if (j > me && best[j] == me) {
                    partner[me] = (int16_t)j;
                    partner[j] = (int16_t)me;
                    atomicAnd(&freebits[me >> 5], ~(1u << (me & 31)));
                    atomicAnd(&freebits[j >> 5], ~(1u << (j & 31)));
                    s_new[r & 1] = 1;
                }
            }
            __syncthreads();
            if (!s_new[r & 1]) break;
        }
    }
    // blocks still single are paired in index order; 4. then the pairs are ordered by their lower
    // block (warp 0: two ordered compactions over the chunk)
    if (warp == 0) {
        int run = 0;
#pragma unroll
        for (int c = 0; c < CH / 32; ++c) {
            const int i = c * 32 + lane;
            const bool single = ord.pass != 1 && i < nI && partner[i] < 0;
            const unsigned m = __ballot_sync(0xffffffffu, single);
            if (single) order[run + __popc(m & ((1u << lane) - 1u))] = (int16_t)i;
            run += __popc(m);
        }
        __syncwarp();
        for (int q = lane; 2 * q + 1 < run; q += 32) {
            const int x = order[2 * q], y = order[2 * q + 1];
            partner[x] = (int16_t)y;
            partner[y] = (int16_t)x;
        }
        __syncwarp();
        run = 0;
#pragma unroll
        for (int c = 0; c < CH / 32; ++c) {
            const int i = c * 32 + lane;
            const bool low = i < nI && (partner[i] < 0 ? ord.pass != 1 : partner[i] > i);
            const unsigned m = __ballot_sync(0xffffffffu, low);
            if (low) order[run + __popc(m & ((1u << lane) - 1u))] = (int16_t)i;
            run += __popc(m);
        }
        // where the pairs go: a chunk in index order has its place, the others take the next one free
        if (lane == 0) {
            s_count = run;
            s_base = ord.pass == 0 ? blockIdx.x * (CH / 2) : atomicAdd(ord.count + bh, run);
        }
    }
    if (ord.pass == 1 && threadIdx.x < nI) ord.taken[(int64_t)bh * NB + s_blk[threadIdx.x]] = partner[threadIdx.x] >= 0;
    __syncthreads();
    out_pairs += s_base;
    out_lists += (int64_t)s_base * lstride;
    for (int p = threadIdx.x; p < s_count; p += THREADS) {
        const int i = order[p];
        out_pairs[p] = make_int2(s_blk[i], partner[i] >= 0 ? s_blk[partner[i]] : -1);
    }
    // 5. union lists
    for (int p = warp; p < s_count; p += THREADS / 32) {
        const int i = order[p], j = partner[i];
        write_union(bm + i * pitch, j >= 0 ? bm + j * pitch : nullptr, nwords, out_lists + (int64_t)p * lstride);
    }
}

// Slabs that fit beside the bitmaps when two CTAs share an SM, at least the room of the overlaps.
static int plan_slabs(int NB) {
    const int nwords = (NB + 31) >> 5;
    const int most = (112 * 1024 - CH * plan_pitch(nwords) * 4) / (int)SLAB, need = (nwords + 3) / 4;
    return most < 3 || need < 3 ? 3 : (need < most ? need : most);
}
static size_t plan_smem(int NB) {
    return 1024 + (size_t)plan_slabs(NB) * SLAB + (size_t)CH * plan_pitch((NB + 31) >> 5) * sizeof(uint32_t);
}

// The most that any call needs: what is left to the slabs when two CTAs share an SM, or three slabs beside the
// bitmaps of the longest rows (4096 key blocks).
constexpr int MAX_PITCH = 4096 / 32 + 4;
constexpr size_t MOST_SMEM = 1024 + (3 * SLAB + CH * MAX_PITCH * 4 > 112 * 1024 ? 3 * SLAB + CH * MAX_PITCH * 4 : 112 * 1024);

// Ordering the blocks first saves 3 to 9 % of the attention kernel, which takes 1.5 to 2 ns per query block
// and key block it keeps, and costs three more launches.  Layers, index order / list order: 12 heads x
// 512 blocks, keep 52 (0.32 M kept): 877 / 879 us; 24 x 512 at d = 64 (0.64 M): 1181 / 1179 us; 40 x 1182,
// keep 60 (2.8 M): 7.43 / 7.30 ms; 12 x 3023, keep 152 (5.5 M): 14.16 / 13.43 ms.
static bool plan_ordered(const AttnArgs& a) {
    int64_t kept = 0;
    for (int h = 0; h < a.H; ++h)
        if (a.k_per_head[h] < a.NB) kept += a.k_per_head[h];
    return a.NB >= ORDER_MIN_NB && (int64_t)a.B * a.NB * kept >= ORDER_MIN_WORK;
}

}  // namespace plan

static size_t pairs_bytes(int B, int H, int NB) {
    return align_up((size_t)B * H * ((size_t)(NB + 1) / 2) * sizeof(int2), 256);
}
static int64_t lists_ints_per_batch(int H, int NB, const int32_t* k_per_head) {
    int64_t n = 0;
    for (int h = 0; h < H; ++h) n += ((int64_t)(NB + 1) / 2) * list_stride(k_per_head[h], NB);
    return n;
}

// pairs | lists | keys [2] | by_rank [2] | taken | count
struct PlanLayout {
    size_t lists, keys, by_rank, taken, count, total;
    PlanLayout(int B, int H, int NB, const int32_t* k_per_head) {
        const size_t rows = (size_t)B * H * NB;
        lists = pairs_bytes(B, H, NB);
        keys = lists + align_up((size_t)B * lists_ints_per_batch(H, NB, k_per_head) * sizeof(int), 256);
        by_rank = keys + align_up(2 * rows * sizeof(uint32_t), 256);
        taken = by_rank + align_up(2 * rows * sizeof(uint16_t), 256);
        count = taken + align_up(rows, 256);
        total = count + align_up((size_t)B * H * sizeof(int), 256);
    }
};

size_t pair_plan_bytes(int B, int H, int NB, const int32_t* k_per_head) { return PlanLayout(B, H, NB, k_per_head).total; }

int launch_pair_plan(AttnArgs& a, void* mem, cudaStream_t st) {
    const int NP = (a.NB + 1) / 2, BH = a.B * a.H;
    char* base = static_cast<char*>(mem);
    const PlanLayout L(a.B, a.H, a.NB, a.k_per_head);
    int2* pairs = reinterpret_cast<int2*>(base);
    int* lists = reinterpret_cast<int*>(base + L.lists);
    a.pairs = pairs;
    a.lists = lists;
    int64_t off = 0;
    for (int h = 0; h < a.H; ++h) {
        a.list_off[h] = off;
        off += (int64_t)NP * list_stride(a.k_per_head[h], a.NB);
    }
    a.list_batch = off;
    const size_t smem = plan::plan_smem(a.NB);
    const int nbuf = plan::plan_slabs(a.NB);
    // (the limit is the function's, not the call's: always the most any call needs, for calls from several threads)
    cudaError_t e = cudaFuncSetAttribute(plan::pair_plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan::MOST_SMEM);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "sparse_attn: plan smem attribute: %s", cudaGetErrorString(e));
    const dim3 grid((a.NB + plan::CH - 1) / plan::CH, BH);
    plan::Order ord = {nullptr, nullptr, nullptr, 0};
    if (plan::plan_ordered(a)) {
        uint32_t* keys = reinterpret_cast<uint32_t*>(base + L.keys);
        uint16_t* by_rank = reinterpret_cast<uint16_t*>(base + L.by_rank);
        ord = {by_rank, reinterpret_cast<uint8_t*>(base + L.taken), reinterpret_cast<int*>(base + L.count), 1};
        const int64_t rows = (int64_t)BH * a.NB;
        launch_dep_smem(plan::plan_keys_kernel, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, st, a, keys, ord.count);
        USV_CHECK_LAUNCH("plan_keys_kernel");
        launch_dep_smem(plan::plan_sort_kernel, dim3(2 * BH), dim3(1024), 0, st, a.NB, keys, by_rank);
        USV_CHECK_LAUNCH("plan_sort_kernel");
        launch_dep_smem(plan::pair_plan_kernel, grid, dim3(plan::THREADS), smem, st, a, pairs, lists, ord, nbuf);
        USV_CHECK_LAUNCH("pair_plan_kernel (first pass)");
        ord.pass = 2;
    }
    launch_dep_smem(plan::pair_plan_kernel, grid, dim3(plan::THREADS), smem, st, a, pairs, lists, ord, nbuf);
    USV_CHECK_LAUNCH("pair_plan_kernel");
    return USV_OK;
}

}  // namespace usv
