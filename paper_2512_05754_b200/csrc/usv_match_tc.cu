// Bipartite matching of token merge (Sec. 3.3, Eq. 8-9) on the tensor cores: for every source
// token the destination with the largest cosine, ties to the lowest destination.
//
// The cosines decide an integer (the arg-max) that is compared with an fp64 evaluation.  All
// N_src x N_dst cosines are computed ONCE, from fp16 roundings of the fp32 unit descriptors of DM = 64
// or 128 features (DM / 16 tcgen05.mma, M = 128 sources, N = 128 destinations, K = 16, per 128 x 128
// tile, fp32 accumulation), which are not exact but carry a rigorous bound: every component is off by at most
// 2^-11 relative, so a cosine of two unit vectors is off by at most sum|a_i b_i| (2^-10 + 2^-22)
// <= 2^-10, plus ~1e-6 of accumulation: EPS = 1e-3.  The true best destination of a source
// therefore has an approximate cosine within 2 EPS of the approximate row maximum.  Each source keeps
// its largest approximate cosines (eight per half of the destination tiles); if the last kept one lies
// below (max - 2 EPS) the true arg-max is among the others, and they are re-evaluated in fp32 (exactly what an fp32 pass over the whole
// row would have chosen among them: ties to the lowest destination).  A source with a full list of
// destinations inside the window (duplicates, near-duplicates) is handed to a plain fp32 scan of
// all its destinations.  The result is the fp32 arg-max for every source, whatever the data.
//
// 20 691 sources against 7410 destinations at DM = 64: 852 us on fp32 CUDA cores, 101 us here (all
// kernels of this file).
//
//   (usv_merge.cu)      desc_kernel writes the fp16 rows, sources (by rank) and destinations (by
//                       ordinal) apart, zero-padded to multiples of 128 rows
//   match_tc_kernel     one CTA per 128 sources and part of the destinations: the sources sit in TMEM as the A operand, the
//                       destination rows stream through shared memory (TMA, 4 stages); warp 8 =
//                       TMA producer, warps 9-10 = MMA issuers on alternate tiles, warps 0-3 / 4-7 =
//                       two groups of one thread per source row, reading the 128 x 128 tiles of even /
//                       odd index out of TMEM (three accumulator tiles in rotation) and keeping the eight best (value,
//                       destination) inside the window of their running maximum, ascending destinations
//   recheck_kernel      per source: the candidates of all parts inside the window in fp32 -> j*, u; sources
//                       with a full window are listed
//   match_exact_kernel  fp32 scan of every destination for the listed sources (normally none; tiles where they are many)
#include <cuda_fp16.h>

#include "usv_match.cuh"
#include "usv_tcgen05.cuh"

namespace usv {

namespace mt {

using namespace t5;

constexpr int STAGES = 4;
constexpr int NBUF = 3;                                 // accumulator tiles in TMEM: the hand-over of a tile between
                                                        // MMA issuer and epilogue takes longer than its MMAs
constexpr int W_PROD = 8, W_MMA0 = 9;                   // warps 0-7: two epilogue warpgroups
constexpr int NCAND = 8;                                // best approximate cosines kept per source and tile parity
constexpr float EPS = 1.0e-3f;                          // bound on |approximate - exact cosine| (see above)
constexpr uint32_t SM_SCR = 0;                          // float[32][256]: a chunk of one row per epilogue thread
constexpr uint32_t SM_FLOOR = SM_SCR + 32 * 256 * 4;     // float[128]: floor per source row
constexpr uint32_t SM_BAR = SM_FLOOR + 128 * 4;
enum { B_AFULL = 0, B_BFULL = 1, B_BEMPTY = B_BFULL + STAGES, B_DFULL = B_BEMPTY + STAGES, B_DFREE = B_DFULL + 2 * NBUF,
       B_COUNT = B_DFREE + 2 * NBUF };
static_assert(B_COUNT <= 32, "barrier area");
constexpr uint32_t SM_MISC = SM_BAR + 8 * 32;
constexpr uint32_t SM_B = (SM_MISC + 64 + 1023) / 1024 * 1024;   // STAGES tiles of fp16 rows, [d-half][128 rows][128 B]
template <int DM>
constexpr uint32_t STAGE_BYTES = 128 * DM * 2;          // 32 or 16 KB
template <int DM>
constexpr size_t SMEM_BYTES = SM_B + STAGES * STAGE_BYTES<DM> + 1024;
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t TA = 0, TD = 128;                    // A rows (fp16) at 0; D buffers at 128, 256 and 384
static_assert(TD + NBUF * 128 <= TMEM_COLS, "TMEM budget");

// DM / 32 consecutive floats per lane of a warp that holds one descriptor row
template <int V>
struct alignas(V * 4) Floats { float v[V]; };

template <int V>
__device__ __forceinline__ float dot(const Floats<V>& x, const Floats<V>& y) {
    float acc = x.v[V - 1] * y.v[V - 1];
#pragma unroll
    for (int e = V - 2; e >= 0; --e) acc = fmaf(x.v[e], y.v[e], acc);
    return acc;
}

struct Maps {
    CUtensorMap b_h;
};

// maximum of three fp32 values given as bit patterns (one instruction on this architecture)
__device__ __forceinline__ float max3(uint32_t a, uint32_t b, uint32_t c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(__uint_as_float(a)), "f"(__uint_as_float(b)), "f"(__uint_as_float(c)));
    return d;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}

template <int DM>
__global__ void __launch_bounds__(352, 1)
match_tc_kernel(const MatchTcArgs m, const __grid_constant__ Maps maps) {
    // the set-up touches shared and tensor memory only; dep_sync() follows it, with the columns allocated
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* sm = smem_raw + (base - raw);
    auto bar = [&](int i) { return base + SM_BAR + 8u * i; };
    volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(sm + SM_MISC);
    volatile int* s_abort = reinterpret_cast<volatile int*>(sm + SM_MISC + 4);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int b = blockIdx.y;
    const int a0 = blockIdx.x * 128;
    // destination tiles [t_lo, t_lo + T), walked in the same order by every CTA (walking them in rotated
    // orders, so that the CTAs ask for different L2 lines, was slower)
    const int t_all = m.nB_pad / 128, t_per = (t_all + m.parts - 1) / m.parts;
    const int t_lo = min(t_all, (int)blockIdx.z * t_per), T = min(t_per, t_all - t_lo);

    if (threadIdx.x == 0) {
        mbar_init(bar(B_AFULL), 4);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar(B_BFULL + s), 1);
            mbar_init(bar(B_BEMPTY + s), 1);
        }
        // Tile t uses accumulator t mod NBUF but the barriers t mod (2 NBUF): consecutive uses of an
        // accumulator belong to different issuer warps and epilogue groups (t and t + NBUF differ in
        // parity), and a waiter must see every phase of the barrier it waits on.
        for (int s = 0; s < 2 * NBUF; ++s) {
            mbar_init(bar(B_DFULL + s), 1);
            mbar_init(bar(B_DFREE + s), 4);
        }
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(base + SM_MISC), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    dep_sync();
    const uint32_t tmem = *s_tmem;

    if (warp == W_PROD) {
        // ===== TMA producer: destination rows =====
        const int row0 = b * m.nB_pad + t_lo * 128;
        for (int t = 0; t < T; ++t) {
            const int s = t % STAGES;
            const uint32_t ph = (t / STAGES) & 1;
            if (!mbar_wait(bar(B_BEMPTY + s), ph ^ 1, s_abort, m.status, 0x10000)) break;
            const uint32_t dst = base + SM_B + s * STAGE_BYTES<DM>;
            if (elect_one()) {
                mbar_expect_tx(bar(B_BFULL + s), STAGE_BYTES<DM>);
#pragma unroll
                for (int hf = 0; hf < DM / 64; ++hf)
                    tma_load_2d(dst + hf * 16384, &maps.b_h, bar(B_BFULL + s), hf * 64, row0 + t * 128);
            }
            __syncwarp();
        }
    } else if (warp == W_MMA0 || warp == W_MMA0 + 1) {
        // ===== two MMA issuers: warp 5 takes the even tiles, warp 6 the odd ones (each tile has its
        // own B stage and accumulator tile), so that one warp's barrier waits fall under the other's MMAs =====
        constexpr uint32_t IDESC = instr_desc_f16(128, 128, 0, 0);   // fp16 A (TMEM) x fp16 B (K-major) -> fp32
        const uint64_t bdesc0 = smem_desc(base + SM_B, 16, 1024);
        bool ok = mbar_wait(bar(B_AFULL), 0, s_abort, m.status, 0x20000);
        for (int t = warp - W_MMA0; ok && t < T; t += 2) {
            const int s = t % STAGES;
            const uint32_t ph = (t / STAGES) & 1;
            const int buf = t % NBUF;
            if (!mbar_wait_spin(bar(B_BFULL + s), ph, s_abort, m.status, 0x40000)) break;
            if (t >= NBUF && !mbar_wait_spin(bar(B_DFREE + (t - NBUF) % (2 * NBUF)), ((t - NBUF) / (2 * NBUF)) & 1, s_abort, m.status, 0x80000)) break;
            fence_after();
            const uint64_t bd = bdesc0 + ((s * STAGE_BYTES<DM>) >> 4);
            const uint32_t d = tmem + TD + buf * 128;
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < DM / 16; ++ks)
                    umma_ts(d, tmem + TA + ks * 8, bd + (((ks >> 2) * 16384 + (ks & 3) * 32) >> 4), IDESC, ks > 0);
                umma_commit(bar(B_BEMPTY + s));
                umma_commit(bar(B_DFULL + t % (2 * NBUF)));
            }
            __syncwarp();
        }
    } else {
        // ===== two warpgroups, one thread per source row in each: group e reads the tiles of parity e
        // (accumulator tile t mod NBUF) and keeps its own candidates; the two lists meet in recheck_kernel =====
        const int eg = warp >> 2;           // 0: even tiles, 1: odd tiles
        const int r = threadIdx.x & 127;    // TMEM lane = source row of the CTA
        const int a = a0 + r;
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        if (eg == 0) {
            const int64_t row = (int64_t)b * m.nA_pad + a;    // padded: always in range
            const uint4* ph = reinterpret_cast<const uint4*>(m.a_h + row * DM);
#pragma unroll
            for (int c4 = 0; c4 < DM / 32; ++c4) {
                uint32_t q[16];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 v = __ldg(ph + c4 * 4 + i);
                    q[4 * i] = v.x; q[4 * i + 1] = v.y; q[4 * i + 2] = v.z; q[4 * i + 3] = v.w;
                }
                tmem_st16(lane_base + TA + c4 * 16, q);
            }
            tmem_wait_st();
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_AFULL));
        }
        // The NCAND largest approximate cosines so far (registers), descending; equal values keep
        // the order of their destinations (ascending), so the lowest destination of a tie stands
        // first.  vmax / vlast mirror the first and the last entry.
        float cval[NCAND];
        int cidx[NCAND];
#pragma unroll
        for (int c = 0; c < NCAND; ++c) { cval[c] = -INFINITY; cidx[c] = 0; }
        float vmax = -INFINITY, vlast = -INFINITY;
        // A lower bound on the row's approximate maximum, known before the first tile: the cosine of
        // the fp16 rows of the source and of the destination of its own partition block, less
        // the accumulation error.  Video tokens mostly match a neighbour, so the bound is usually
        // close to the maximum and the window is narrow from the first tile on.  (Any value that cannot
        // exceed the approximate maximum is a valid floor; a poor one only costs time.)  Group 1
        // works it out while group 0 fills the A operand.
        float* s_floor = reinterpret_cast<float*>(sm + SM_FLOOR);
        if (eg == 1) {
            float c0 = 0.f, c1 = 0.f;
            if (a < m.nA) {
                const int own = m.p.ord(m.src_idx[a]);
                const uint4* px = reinterpret_cast<const uint4*>(m.a_h + ((int64_t)b * m.nA_pad + a) * DM);
                const uint4* py = reinterpret_cast<const uint4*>(m.b_h + ((int64_t)b * m.nB_pad + own) * DM);
#pragma unroll 4
                for (int i = 0; i < DM / 8; ++i) {
                    const uint4 xv = __ldg(px + i), yv = __ldg(py + i);
                    const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w}, yw[4] = {yv.x, yv.y, yv.z, yv.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 fx = __half22float2(*reinterpret_cast<const __half2*>(xw + e));
                        const float2 fy = __half22float2(*reinterpret_cast<const __half2*>(yw + e));
                        c0 = fmaf(fx.x, fy.x, c0);
                        c1 = fmaf(fx.y, fy.y, c1);
                    }
                }
            }
            s_floor[r] = c0 + c1 - 1e-5f;   // (sums of 128 products of unit vectors, two orders: 2e-6 apart at most)
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const float floor_v = s_floor[r];
        bool ok = true;
        for (int t = eg; t < T; t += 2) {
            const int buf = t % NBUF;
            if (!mbar_wait_spin(bar(B_DFULL + t % (2 * NBUF)), (t / (2 * NBUF)) & 1, s_abort, m.status, 0x100000)) { ok = false; break; }
            fence_after();
            const int nvalid = m.p.nB - (t_lo + t) * 128;   // destinations of this tile that exist
            // the whole 128-column row in one go (four loads in flight, one wait), then the buffer goes back
            uint32_t sr[128];
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) tmem_ld32(lane_base + TD + buf * 128 + ch * 32, sr + ch * 32);
            tmem_wait_ld();
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_DFREE + t % (2 * NBUF)));
            // The four chunk maxima first (three-input maxima on sixteen independent chains), and
            // from them the tile's: most tiles lie below the window of the running maximum and are done
            // here.  (The maximum only grows, so a destination below the window can never matter.)
            float cm[4];
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
                if (nvalid < (ch + 1) * 32) {   // only the chunks of the last tile that reach past the end (uniform)
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (ch * 32 + j >= nvalid) sr[ch * 32 + j] = 0xff800000u;   // -inf: a destination that does not exist
                }
                float c0 = max3(sr[ch * 32], sr[ch * 32 + 1], sr[ch * 32 + 2]);
                float c1 = max3(sr[ch * 32 + 3], sr[ch * 32 + 4], sr[ch * 32 + 5]);
                float c2 = max3(sr[ch * 32 + 6], sr[ch * 32 + 7], sr[ch * 32 + 8]);
                float c3 = max3(sr[ch * 32 + 9], sr[ch * 32 + 10], sr[ch * 32 + 11]);
#pragma unroll
                for (int j = 12; j < 28; j += 8) {
                    c0 = max3(__float_as_uint(c0), sr[ch * 32 + j], sr[ch * 32 + j + 1]);
                    c1 = max3(__float_as_uint(c1), sr[ch * 32 + j + 2], sr[ch * 32 + j + 3]);
                    c2 = max3(__float_as_uint(c2), sr[ch * 32 + j + 4], sr[ch * 32 + j + 5]);
                    c3 = max3(__float_as_uint(c3), sr[ch * 32 + j + 6], sr[ch * 32 + j + 7]);
                }
                c0 = max3(__float_as_uint(c0), sr[ch * 32 + 28], sr[ch * 32 + 29]);
                c1 = max3(__float_as_uint(c1), sr[ch * 32 + 30], sr[ch * 32 + 31]);
                cm[ch] = fmaxf(fmaxf(c0, c1), fmaxf(c2, c3));
            }
            const float tm = fmaxf(fmaxf(cm[0], cm[1]), fmaxf(cm[2], cm[3]));
            if (tm >= fmaxf(vmax, floor_v) - 2.0f * EPS && tm > vlast) {
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) {
                    const float thr = fmaxf(vmax, floor_v) - 2.0f * EPS;
                    if (cm[ch] >= thr && cm[ch] > vlast) {
                        // Rare.  The chunk is parked in shared memory and a bit mask marks the elements
                        // inside the window as it stands; only those are read back and inserted (one
                        // short rolled loop: unrolled over the register elements the insertion is
                        // tens of KB of code, and the kernel then waits on instruction fetch).
                        float* scr = reinterpret_cast<float*>(sm + SM_SCR) + (threadIdx.x & 255);
                        uint32_t mask = 0;
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const float v = __uint_as_float(sr[ch * 32 + j]);
                            scr[j * 256] = v;
                            if (v >= thr && v > vlast) mask |= 1u << j;
                        }
#pragma unroll 1
                        while (mask != 0) {
                            const int j = __ffs(mask) - 1;
                            mask &= mask - 1;
                            const float v = scr[j * 256];
                            if (v >= fmaxf(vmax, floor_v) - 2.0f * EPS && v > vlast) {
                                const int idx = (t_lo + t) * 128 + ch * 32 + j;
                                // descending cosine, then ascending destination: the entries the
                                // new one beats move down one place, the last one drops out
                                bool placed = false;
#pragma unroll
                                for (int pos = NCAND - 1; pos > 0; --pos) {
                                    const bool up = v > cval[pos - 1] || (v == cval[pos - 1] && idx < cidx[pos - 1]);
                                    if (!placed) {
                                        cval[pos] = up ? cval[pos - 1] : v;
                                        cidx[pos] = up ? cidx[pos - 1] : idx;
                                    }
                                    placed |= !up;
                                }
                                if (!placed) { cval[0] = v; cidx[0] = idx; }
                                vmax = cval[0];
                                vlast = cval[NCAND - 1];
                            }
                        }
                    }
                }
            }
        }
        if (ok && a < m.nA) {
            const int64_t g4 = ((((int64_t)b * m.nA + a) * m.parts + blockIdx.z) * 2 + eg) * NCAND;
#pragma unroll
            for (int c = 0; c < NCAND; ++c) {
                m.cand_v[g4 + c] = cval[c];
                m.cand_i[g4 + c] = cidx[c];
            }
        }
    }

    fence_before();
    __syncthreads();
    if (*s_abort) {
        const unsigned long long t0 = gtime();
        while (gtime() - t0 < 2000000ull) { }
        __syncthreads();
    }
    if (warp == W_MMA0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// fp32 cosines that decide.  DM = 128: a warp holds both rows, four products a lane, then a
// butterfly.  DM = 64: every lane works through a whole destination row of its own, in ascending
// feature order.  (Each width keeps one order of summation wherever a cosine is decided, so that the
// same pair always gives the same value.)
__device__ __forceinline__ float warp_cosine(const Floats<4>& x, const Floats<4>& y) {
    float acc = dot<4>(x, y);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}
__device__ __forceinline__ float lane_cosine64(const float* __restrict__ x, const float* __restrict__ y) {
    float acc = 0.f;
#pragma unroll 4
    for (int e = 0; e < 64; e += 4) {
        const float4 xv = __ldg(reinterpret_cast<const float4*>(x + e)), yv = __ldg(reinterpret_cast<const float4*>(y + e));
        acc = fmaf(xv.w, yv.w, fmaf(xv.z, yv.z, fmaf(xv.y, yv.y, fmaf(xv.x, yv.x, acc))));
    }
    return acc;
}

// One warp per source: the candidates inside the window (approximate cosine >= max - 2 EPS) are
// re-evaluated in fp32; the largest wins, equal values go to the lowest destination.  A source whose
// last kept candidate is still inside the window may have more destinations in it than were kept: it is
// appended to the list of the exact scan.  Lane c holds candidates c and c + 32 of the two lists per part
// (even and odd destination tiles), each complete for its tiles unless its last entry is still inside the
// window.
template <int DM>
__global__ void __launch_bounds__(256)
recheck_kernel(const float* __restrict__ mhat, MatchTcArgs m) {
    dep_sync();
    static_assert(NCAND == 8, "four lists a warp");
    const int64_t gw = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (gw >= (int64_t)m.B * m.nA) return;
    const int b = (int)(gw / m.nA), a = (int)(gw % m.nA);
    const int src = m.src_idx[a];
    const int total = m.parts * 2 * NCAND;
    float v[2];
    int id[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int c = g * 32 + lane;
        v[g] = c < total ? m.cand_v[gw * total + c] : -INFINITY;
        id[g] = c < total ? m.cand_i[gw * total + c] : 0x7fffffff;
    }
    float top = fmaxf(v[0], v[1]);
#pragma unroll
    for (int o = NCAND; o < 32; o <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    const float window = __shfl_sync(0xffffffffu, top, 0) - 2.0f * EPS;   // (a list's first entry is its largest)
    unsigned in[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) in[g] = __ballot_sync(0xffffffffu, v[g] >= window);   // (never true for -inf entries)
    if ((in[0] | in[1]) & 0x80808080u) {
        if (lane == 0) {
            const int64_t w = (int64_t)b * m.nA + atomicAdd(m.exact_count + b, 1);
            m.exact_list[w] = a;
            m.exact_done[w] = 0;
            m.exact_best[w] = 0ull;
        }
        return;
    }
    const float* M = mhat + (int64_t)b * m.N * DM;
    const float* X = M + (int64_t)src * DM;
    float best = -INFINITY;
    int bj = 0x7fffffff;
    if (DM == 128) {
        const Floats<4> x = *reinterpret_cast<const Floats<4>*>(X + lane * 4);
#pragma unroll
        for (int g = 0; g < 2; ++g)
            while (in[g]) {
                const int j = __shfl_sync(0xffffffffu, id[g], __ffs(in[g]) - 1);
                in[g] &= in[g] - 1;
                const float c = warp_cosine(x, *reinterpret_cast<const Floats<4>*>(M + (int64_t)m.p.dst_token(j) * DM + lane * 4));
                if (c > best || (c == best && j < bj)) { best = c; bj = j; }
            }
    } else {
#pragma unroll
        for (int g = 0; g < 2; ++g)
            if ((in[g] >> lane) & 1u) {
                const float c = lane_cosine64(X, M + (int64_t)m.p.dst_token(id[g]) * DM);
                if (c > best || (c == best && id[g] < bj)) { best = c; bj = id[g]; }
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            if (ob > best || (ob == best && oj < bj)) { best = ob; bj = oj; }
        }
    }
    if (lane == 0) {
        m.jstar_s[gw] = m.p.dst_token(bj == 0x7fffffff ? 0 : bj);   // (no comparable cosine, NaN in the metric: any destination)
        m.u_s[gw] = best;
    }
}

// fp32 scan of every destination for the listed sources (normally few or none): the same summation order per cosine
// as recheck_kernel.  blockIdx.y = batch element.  The best (cosine, lowest destination) of a work unit goes into
// the source's slot with one 64-bit atomic maximum (order-preserving key of the cosine above, complement of the
// destination below); whoever finishes a source's last unit writes its result.
__device__ __forceinline__ unsigned long long exact_key(float cosine, int j) {
    return ((unsigned long long)float_key_any(cosine) << 32) | (0xffffffffu - (unsigned)j);
}
__device__ __forceinline__ void exact_finish(const MatchTcArgs& m, int b, int w, unsigned long long best, int units) {
    const int64_t at = (int64_t)b * m.nA + w;
    atomicMax(m.exact_best + at, best);
    __threadfence();
    if (atomicAdd(m.exact_done + at, 1) != units - 1) return;
    __threadfence();
    const unsigned long long key = atomicMax(m.exact_best + at, 0ull);
    const uint32_t fk = (uint32_t)(key >> 32);
    const uint32_t bits = (fk & 0x80000000u) ? (fk & 0x7fffffffu) : ~fk;    // inverse of float_key (NaN: -0)
    const int64_t g = (int64_t)b * m.nA + m.exact_list[at];
    m.jstar_s[g] = m.p.dst_token((int)(0xffffffffu - (uint32_t)key));
    m.u_s[g] = __uint_as_float(bits);
}

// Few listed sources.  Work unit = (source, chunk of 256 destinations); a warp takes four destinations at a time so
// that their loads overlap (DM = 64: one a lane).
constexpr int EX_CHUNK = 256;

template <int DM>
__device__ __forceinline__ void exact_rows(const float* __restrict__ M, const MatchTcArgs& m, int count) {
    __shared__ unsigned long long s_key[8];
    const int b = blockIdx.y;
    const int nchunks = (m.p.nB + EX_CHUNK - 1) / EX_CHUNK;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int64_t unit = blockIdx.x; unit < (int64_t)count * nchunks; unit += gridDim.x) {
        const int w = (int)(unit / nchunks), c = (int)(unit % nchunks);
        const float* X = M + (int64_t)m.src_idx[m.exact_list[(int64_t)b * m.nA + w]] * DM;
        unsigned long long best = 0ull;
        const int j0 = c * EX_CHUNK + warp * 32;
        if (DM == 64) {
            const int j = j0 + lane;
            if (j < m.p.nB) best = exact_key(lane_cosine64(X, M + (int64_t)m.p.dst_token(j) * DM), j);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
                best = other > best ? other : best;
            }
        } else {
            const Floats<4> x = *reinterpret_cast<const Floats<4>*>(X + lane * 4);
#pragma unroll 1
            for (int q = 0; q < 32; q += 4) {
                Floats<4> y[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int j = j0 + q + e;
                    y[e] = j < m.p.nB ? *reinterpret_cast<const Floats<4>*>(M + (int64_t)m.p.dst_token(j) * DM + lane * 4)
                                      : Floats<4>{};
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int j = j0 + q + e;
                    const float acc = warp_cosine(x, y[e]);
                    if (j < m.p.nB) {
                        const unsigned long long key = exact_key(acc, j);
                        best = key > best ? key : best;
                    }
                }
            }
        }
        if (lane == 0) s_key[warp] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long bb = s_key[0];
            for (int q = 1; q < 8; ++q) bb = s_key[q] > bb ? s_key[q] : bb;
            exact_finish(m, b, w, bb, nchunks);
        }
        __syncthreads();
    }
}

// Many listed sources at DM = 64 (flat regions of a picture: every destination is alike): tiles of 128 sources x 128
// destinations on the CUDA cores, 8 x 8 a thread, features in ascending order as in lane_cosine64.  Whole merges, us, all of it on
// CUDA cores / rows only / this: 2 x 20 280 tokens, 2730 destinations each, 40 flat regions with noise 687 / 7637 / 795;
// 20 280 tokens, 10 140 destinations 1602 / 10 339 / 788, two per cent of the picture flat 2007 / 1437 / 410.
constexpr int EX_TILE = 128;
constexpr int EX_MANY = 128;   // sources of a batch element from which on the tiles are faster

__device__ __forceinline__ void exact_tiles64(const float* __restrict__ M, const MatchTcArgs& m, int count) {
    constexpr int TK = 16;
    __shared__ __align__(16) float As[TK][EX_TILE + 4];
    __shared__ __align__(16) float Bs[TK][EX_TILE + 4];
    const int b = blockIdx.y;
    const int ntiles = (m.p.nB + EX_TILE - 1) / EX_TILE;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    for (int64_t unit = blockIdx.x; unit < (int64_t)((count + EX_TILE - 1) / EX_TILE) * ntiles; unit += gridDim.x) {
        const int w0 = (int)(unit / ntiles) * EX_TILE, j0 = (int)(unit % ntiles) * EX_TILE;
        // this thread stages 4 features of two rows of either operand
        const float *pa[2], *pb[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int r = (threadIdx.x >> 2) + 64 * t;   // rows past the end repeat the first one
            pa[t] = M + (int64_t)m.src_idx[m.exact_list[(int64_t)b * m.nA + (w0 + r < count ? w0 + r : w0)]] * 64 + (threadIdx.x & 3) * 4;
            pb[t] = M + (int64_t)m.p.dst_token(j0 + r < m.p.nB ? j0 + r : j0) * 64 + (threadIdx.x & 3) * 4;
        }
        float acc[8][8] = {};
#pragma unroll 1
        for (int k0 = 0; k0 < 64; k0 += TK) {
            float4 va[2], vb[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                va[t] = *reinterpret_cast<const float4*>(pa[t] + k0);
                vb[t] = *reinterpret_cast<const float4*>(pb[t] + k0);
            }
            __syncthreads();   // the tile before has been read
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int r = (threadIdx.x >> 2) + 64 * t, c = (threadIdx.x & 3) * 4;
                As[c][r] = va[t].x; As[c + 1][r] = va[t].y; As[c + 2][r] = va[t].z; As[c + 3][r] = va[t].w;
                Bs[c][r] = vb[t].x; Bs[c + 1][r] = vb[t].y; Bs[c + 2][r] = vb[t].z; Bs[c + 3][r] = vb[t].w;
            }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < TK; ++e) {
                float a[8], d[8];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    *reinterpret_cast<float4*>(a + 4 * h) = *reinterpret_cast<const float4*>(&As[e][ty * 4 + 64 * h]);
                    *reinterpret_cast<float4*>(d + 4 * h) = *reinterpret_cast<const float4*>(&Bs[e][tx * 4 + 64 * h]);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], d[j], acc[i][j]);
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int w = w0 + (i >> 2) * 64 + ty * 4 + (i & 3);
            uint32_t top = 0u;
            int at = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {   // (ascending destinations: the first of equal ones stays)
                const int dj = j0 + (j >> 2) * 64 + tx * 4 + (j & 3);
                const uint32_t key = dj < m.p.nB ? float_key_any(acc[i][j]) : 0u;
                if (key > top) { top = key; at = dj; }
            }
            unsigned long long best = top ? ((unsigned long long)top << 32) | (0xffffffffu - (unsigned)at) : 0ull;
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) {   // over the 16 threads of the row
                const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
                best = other > best ? other : best;
            }
            if (tx == 0 && w < count) exact_finish(m, b, w, best, ntiles);
        }
    }
}

template <int DM>
__global__ void __launch_bounds__(256)
match_exact_kernel(const float* __restrict__ mhat, MatchTcArgs m) {
    dep_sync();
    const int b = blockIdx.y, count = m.exact_count[b];
    const float* M = mhat + (int64_t)b * m.N * DM;
    if (DM == 64 && count >= EX_MANY) exact_tiles64(M, m, count);
    else if (count > 0) exact_rows<DM>(M, m, count);
}

static int make_rows_map(CUtensorMap* map, const void* ptr, int64_t rows, int DM, const char* name) {
    EncodeTiledFn fn = encode_fn();
    if (fn == nullptr) return fail(USV_ERR_CUDA, "token_merge: cuTensorMapEncodeTiled not available");
    cuuint64_t dims[2] = {(cuuint64_t)DM, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)DM * 2};
    cuuint32_t box[2] = {64, 128};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = encode_tiled(fn, map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(USV_ERR_CUDA, "token_merge: cuTensorMapEncodeTiled(%s) failed with %d", name, (int)r);
    return USV_OK;
}

}  // namespace mt

static inline int pad128(int n) { return (n + 127) / 128 * 128; }

static size_t rows_bytes(int B, int N, int dm) { return align_up((size_t)B * ((size_t)N + 256) * dm * sizeof(uint16_t), 256); }
// several parts for up to PARTS_MAX_SOURCES sources only
constexpr int64_t PARTS_MAX_SOURCES = 32768;
static size_t cand_bytes(int B, int N) {
    const int64_t n = (int64_t)B * N, few = n < PARTS_MAX_SOURCES ? n : PARTS_MAX_SOURCES;
    return align_up((size_t)(n > 4 * few ? n : 4 * few) * 2 * mt::NCAND * sizeof(float), 256);
}
// CTAs that share the destinations of 128 sources: one CTA an SM is resident, its start takes as long as
// eight destination tiles (sixteen gives the same times).  Whole merges, us, one part / as chosen: 4680
// tokens 59.7 / 50.5, 9600 55.3 / 50.1, 12 000 57.7 / 53.3, 28 101 (162 CTAs) 145.5 / 137, 39 000 (153 CTAs)
// 196 / 178.
static int match_parts(int B, int nA, int nB, int sms) {
    if ((int64_t)B * nA > PARTS_MAX_SOURCES) return 1;
    const int ctas = B * ceil_div(nA, 128), tiles = ceil_div(nB, 128);
    int best = 1, least = 0;
    for (int parts = 1; parts <= 4 && parts <= tiles; parts *= 2) {
        const int time = ceil_div(ctas * parts, sms) * (8 + ceil_div(tiles, parts));
        if (parts == 1 || time < least) { best = parts; least = time; }
    }
    return best;
}
static size_t list_bytes(int B, int N) { return align_up((size_t)B * N * sizeof(int), 256); }

size_t match_tc_bytes(int B, int N, int dm) {
    // fp16 rows | candidate values | candidate destinations | exact scan: list, unit counters, results, counts
    return rows_bytes(B, N, dm) + 2 * cand_bytes(B, N) + 4 * list_bytes(B, N) + align_up((size_t)B * sizeof(int), 256);
}

int match_tc_args(MatchTcArgs& m, int dm, const int32_t* src_idx, int32_t* jstar_s, float* u_s, void* mem,
                   unsigned int* status) {
    const int B = m.B, N = m.N;
    m.nA_pad = pad128(m.nA); m.nB_pad = pad128(m.p.nB);
    m.src_idx = src_idx; m.jstar_s = jstar_s; m.u_s = u_s; m.status = status;
    int sms;
    if (int rc = sm_count(&sms)) return rc;
    m.parts = match_parts(B, m.nA, m.p.nB, sms);
    char* at = static_cast<char*>(mem);
    auto take = [&](size_t bytes) { char* p = at; at += bytes; return p; };
    m.a_h = reinterpret_cast<uint16_t*>(take(rows_bytes(B, N, dm)));
    m.b_h = m.a_h + (size_t)B * m.nA_pad * dm;
    m.cand_v = reinterpret_cast<float*>(take(cand_bytes(B, N)));
    m.cand_i = reinterpret_cast<int*>(take(cand_bytes(B, N)));
    m.exact_list = reinterpret_cast<int*>(take(list_bytes(B, N)));
    m.exact_done = reinterpret_cast<int*>(take(list_bytes(B, N)));
    m.exact_best = reinterpret_cast<unsigned long long*>(take(2 * list_bytes(B, N)));
    m.exact_count = reinterpret_cast<int*>(take(align_up((size_t)B * sizeof(int), 256)));
    return USV_OK;
}

template <int dm>
static int launch_match(const float* mhat, const MatchTcArgs& m, cudaStream_t st) {
    mt::Maps maps;
    int rc;
    if ((rc = mt::make_rows_map(&maps.b_h, m.b_h, (int64_t)m.B * m.nB_pad, dm, "b_h")) != USV_OK) return rc;
    cudaError_t e = cudaFuncSetAttribute(mt::match_tc_kernel<dm>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mt::SMEM_BYTES<dm>);
    if (e != cudaSuccess) return fail(USV_ERR_CUDA, "token_merge: smem attribute: %s", cudaGetErrorString(e));
    dim3 grid(m.nA_pad / 128, m.B, m.parts);
    launch_dep(mt::match_tc_kernel<dm>, dim3(grid), dim3(352), mt::SMEM_BYTES<dm>, st, m, maps);
    USV_CHECK_LAUNCH("match_tc_kernel");
    const int64_t srcs = (int64_t)m.B * m.nA;
    launch_dep(mt::recheck_kernel<dm>, dim3((unsigned)((srcs + 7) / 8)), dim3(256), 0, st, mhat, m);
    USV_CHECK_LAUNCH("recheck_kernel");
    launch_dep(mt::match_exact_kernel<dm>, dim3(ceil_div(592, m.B), m.B), dim3(256), 0, st, mhat, m);
    USV_CHECK_LAUNCH("match_exact_kernel");
    return USV_OK;
}

int launch_match_tc(const float* mhat, const MatchTcArgs& m, int dm, cudaStream_t st) {
    return dm == 64 ? launch_match<64>(mhat, m, st) : launch_match<128>(mhat, m, st);
}

}  // namespace usv
