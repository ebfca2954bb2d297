// Top-k key-block selection: a row of scores in the registers of one warp (up to 544 scores) or of a few.
//
// The k-th largest score is bracketed by probes: two counts of the scores at or above a value per
// step.  The first two values come from the mean and spread of the row as if it were normal, the next
// from interpolation, until at most 32 scores lie between the probes on either side of k (two to four
// steps on video-like rows).  Those are ranked directly, and everything above the last one kept, with
// its equals up to its index, is written in ascending order: "k largest, ties to the lowest index".
// Where the probes make no headway (heavy tails), the next two come from the ranks of 32 scores of the row; rows
// where that does not help either (NaN, no spread, many equal scores at the cut) go on over order-preserving keys.
#include <math.h>

#include "usv_common.cuh"

namespace usv {

constexpr int SEL_MAX_NB = 8192;

struct SelHeads {
    int k[USV_MAX_HEADS];
    float z[2][USV_MAX_HEADS];   // where the first two probes lie, in standard deviations from the mean
};

constexpr int CANDS = 32;       // scores between the probes that are ranked directly (one per lane)
constexpr int MAX_STEPS = 10;   // of probes between values

// What the warps of a row share, and their sums over it.
template <int W>
struct RowShared {
    uint32_t key[CANDS];
    int n;
    int cnt[2][W];
    uint32_t ends[2][2][W];
    float sum[3][W];
};
template <int W>
__device__ __forceinline__ void row_sync() {
    if (W == 1) __syncwarp();
    else __syncthreads();
}
// sum of one int over the row; `turn` alternates between the calls (one barrier each)
template <int W>
__device__ __forceinline__ int row_total(RowShared<W>& s, int c, int w, int lane, int& turn) {
    c = __reduce_add_sync(0xffffffffu, c);
    if (W == 1) return c;
    if (lane == 0) s.cnt[turn][w] = c;
    __syncthreads();
    c = 0;
#pragma unroll
    for (int q = 0; q < W; ++q) c += s.cnt[turn][q];
    turn ^= 1;
    return c;
}
// exclusive sum over the lanes of the row, in index order
template <int W>
__device__ __forceinline__ int row_before(RowShared<W>& s, int c, int w, int lane, int& turn) {
    const int incl = warp_incl_scan(c);
    int b = incl - c;
    if (W > 1) {
        if (lane == 31) s.cnt[turn][w] = incl;
        __syncthreads();
        for (int q = 0; q < w; ++q) b += s.cnt[turn][q];
        turn ^= 1;
    }
    return b;
}

// Two probes three ranks of 32 scores of the row on either side of where the k-th should lie among them; the scores
// lie in [lo, hi), `need` of the n there are to be kept.  Of several warps the first one's lanes give the scores.
// False where they are too much alike.
template <int W>
__device__ __noinline__ bool sample_probes(RowShared<W>& s, float v, float lo, float hi, int need, int n, int w, int lane,
                                           int turn, float& t1, float& t2) {
    const bool in = v >= lo && v < hi && fabsf(v) <= 3.402823466e38f;
    const int m = __popc(__ballot_sync(0xffffffffu, in));
    int rank = 0;
    for (int q = 0; q < 32; ++q) {
        const float vq = __shfl_sync(0xffffffffu, in ? v : -INFINITY, q);
        rank += vq > v || (vq == v && q < lane) ? 1 : 0;
    }
    const int r = (int)((int64_t)need * m / n);
    const uint32_t b2 = __ballot_sync(0xffffffffu, in && rank == max(r - 3, 0)), b1 = __ballot_sync(0xffffffffu, in && rank == min(r + 3, m - 1));
    t2 = __shfl_sync(0xffffffffu, v, b2 ? __ffs(b2) - 1 : 0);
    t1 = __shfl_sync(0xffffffffu, v, b1 ? __ffs(b1) - 1 : 0);
    bool ok = m >= 8 && b1 && b2 && t1 > lo && t2 > t1 && t2 < hi;
    if (W > 1) {
        if (w == 0 && lane == 0) { s.sum[0][0] = t1; s.sum[1][0] = t2; s.ends[turn][0][0] = ok; }
        __syncthreads();
        t1 = s.sum[0][0];
        t2 = s.sum[1][0];
        ok = s.ends[turn][0][0];
        __syncthreads();
    }
    return ok;
}

// The search over keys, apart from the kernel so that its registers are not the kernel's.  [kl, kh] holds the key
// of the last score kept and n keys; c_hi keys lie above.  Returns bit i: the lane's i-th score is kept.  Two
// counts a step, at the thirds of the bracket; where a step leaves more than half of the keys the bracket is drawn in
// to the smallest and largest key inside it, until it holds one value or few enough to rank.
template <int W, int KPL>
__device__ __noinline__ uint64_t select_by_key(RowShared<W>& s, const float* buf, int NBk, int first, int k, uint32_t kl,
                                               uint32_t kh, int n, int c_hi, int w, int lane, int& turn) {
    uint32_t key[KPL];
#pragma unroll
    for (int i = 0; i < KPL; ++i) key[i] = first + i < NBk ? float_key_any(buf[lane * KPL + i]) : 0u;   // 0: below every key
    uint32_t T = 0;
    int need_eq = 0;
    bool stuck = true;
#pragma unroll 1
    for (;;) {
        if (stuck) {
            uint32_t mn = 0xffffffffu, mx = 0u;
#pragma unroll
            for (int i = 0; i < KPL; ++i)
                if (key[i] - kl <= kh - kl) {
                    mn = min(mn, key[i]);
                    mx = max(mx, key[i]);
                }
            mn = __reduce_min_sync(0xffffffffu, mn);
            mx = __reduce_max_sync(0xffffffffu, mx);
            if (W > 1) {
                if (lane == 0) { s.ends[turn][0][w] = mn; s.ends[turn][1][w] = mx; }
                __syncthreads();
#pragma unroll
                for (int q = 0; q < W; ++q) {
                    mn = min(mn, s.ends[turn][0][q]);
                    mx = max(mx, s.ends[turn][1][q]);
                }
                turn ^= 1;
            }
            kl = mn;
            kh = mx;
        }
        if (kl == kh) {   // one value: all n are equal
            T = kl;
            need_eq = k - c_hi;
            break;
        }
        if (n <= CANDS) break;
        const uint32_t third = (kh - kl) / 3, p1 = kl + third + 1, p2 = max(p1, kh - third);   // kl < p1 <= p2 <= kh
        int c = 0;
#pragma unroll
        for (int i = 0; i < KPL; ++i) {
            if (key[i] >= p1) c += 1;
            if (key[i] >= p2) c += 0x10000;
        }
        c = row_total<W>(s, c, w, lane, turn);
        const int c1 = c & 0xffff, c2 = c >> 16, was = n;
        if (c2 >= k) { kl = p2; n = c2 - c_hi; }
        else if (c1 >= k) { kl = p1; kh = p2 - 1; n = c1 - c2; c_hi = c2; }
        else { kh = p1 - 1; n += c_hi - c1; c_hi = c1; }
        stuck = 2 * n > was;
    }
    if (kl != kh) {
        // rank the few that are left: the (k - c_hi)-th largest is the last one kept
        const int need = k - c_hi;
#pragma unroll
        for (int i = 0; i < KPL; ++i)
            if (key[i] - kl <= kh - kl) s.key[atomicAdd(&s.n, 1)] = key[i];
        row_sync<W>();
        const uint32_t v = lane < n ? s.key[lane] : 0u;
        int above = 0, equal = 0;
        for (int q = 0; q < n; ++q) {
            const uint32_t vq = __shfl_sync(0xffffffffu, v, q);
            above += vq > v ? 1 : 0;
            equal += vq == v ? 1 : 0;
        }
        const int at = __ffs(__ballot_sync(0xffffffffu, lane < n && above < need && need <= above + equal)) - 1;
        T = __shfl_sync(0xffffffffu, v, at);
        need_eq = need - __shfl_sync(0xffffffffu, above, at);
    }
    int equal = 0;
#pragma unroll
    for (int i = 0; i < KPL; ++i) equal += key[i] == T ? 1 : 0;
    int seen = row_before<W>(s, equal, w, lane, turn);
    uint32_t take[2] = {0, 0};
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        if (key[i] > T || (key[i] == T && seen < need_eq)) take[i / 32] |= 1u << (i % 32);
        seen += key[i] == T ? 1 : 0;
    }
    return (uint64_t)take[1] << 32 | take[0];
}

// W warps per row (W = 1: eight rows a CTA, no barrier).  The row passes through shared memory: warp w
// gets the scores [w 32 KPL, ...) with coalesced asynchronous copies, and lane l of it takes KPL consecutive
// ones (KPL is odd: no bank conflicts), so that a lane's kept indices are consecutive in the output.
// Issue slots bound it.  40 heads x 1182 x 1182, keep 60: 113 us (316 us with the row striped over the
// lanes, a search bit by bit, and two ballots per 32 scores on the way out); 12 x 3023 x 3023, keep 152: 186 us
// (442 us with one CTA a row and radix passes in shared memory).  Rows of other kinds, us, the forms named last / this
// with the search bit by bit where the probes fail / as it stands: 24 x 512 x 512, keep 51, normal 25.5 / 15.1 / 15.8, two values
// 36.6 / 66.0 / 25.8, 0.6 % outliers 25.5 / 59.6 / 29.2, exp(3 normal) 23.0 / 35.7 / 29.9, all equal 11.9 / 49.6 / 21.2; 12 x 1900 x 1900,
// keep 190, normal 222 / 98 / 82, two values 266 / 420 / 141, outliers 222 / 415 / 172, all equal 132 / 323 / 120.
template <int W, int KPL>
__global__ void __launch_bounds__(W == 1 ? 256 : W * 32) select_kernel(const float* __restrict__ scores,
                                                                      int32_t* __restrict__ sel, int H, int NBq,
                                                                      int NBk, int kmax, const SelHeads heads,
                                                                      int64_t rows) {
    dep_sync();
    static_assert(KPL % 2 == 1 && KPL <= 64, "");
    constexpr int G = W == 1 ? 8 : 1;               // rows per CTA
    constexpr int SEG = 32 * KPL;                   // scores per warp
    extern __shared__ float s_rows[];               // [G or W warps][SEG]
    __shared__ RowShared<W> s_row[G];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = W == 1 ? warp : 0, w = W == 1 ? 0 : warp;
    RowShared<W>& s = s_row[g];
    const int64_t row = (int64_t)blockIdx.x * G + g;
    if (row >= rows) return;                         // (W = 1: a whole warp; W > 1: never)
    const int h = (int)((row / NBq) % H);
    const int k = heads.k[h];
    const int tid = w * 32 + lane;                   // thread of the row
    int32_t* out = sel + row * kmax;
    if (k >= NBk) {   // keep everything: no search (uniform over the row)
        for (int j = tid; j < NBk; j += W * 32) out[j] = j;
        for (int t = NBk + tid; t < kmax; t += W * 32) out[t] = -1;
        return;
    }
    const int j0 = w * SEG;
    float* buf = s_rows + warp * SEG;
    {
        const float* src = scores + row * NBk + j0 + lane;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(buf) + lane * 4;
        const int mine = NBk - j0 - lane;            // this lane copies the scores i * 32 < mine
#pragma unroll
        for (int i = 0; i < KPL; ++i) {
            if (i * 32 < mine) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + i * 128), "l"(src + i * 32) : "memory");
            else buf[i * 32 + lane] = -INFINITY;     // past the end: no probe counts it
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    for (int t = k + tid; t < kmax; t += W * 32) out[t] = -1;
    if (tid == 0) s.n = 0;
    row_sync<W>();
    float x[KPL];
#pragma unroll
    for (int i = 0; i < KPL; ++i) x[i] = buf[lane * KPL + i];
    const int first = j0 + lane * KPL;               // index of x[0]

    int turn = 0;

    // 1. mean and spread of the finite scores
    bool nan = false;
    float sum = 0.f, sq = 0.f, cnt = 0.f;
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        if (fabsf(x[i]) <= 3.402823466e38f) { sum += x[i]; sq = fmaf(x[i], x[i], sq); cnt += 1.f; }
        nan |= x[i] != x[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if (__any_sync(0xffffffffu, nan)) sum = __int_as_float(0x7fc00000);   // (reaches every warp of the row through the sum)
    if (W > 1) {
        if (lane == 0) { s.sum[0][w] = sum; s.sum[1][w] = sq; s.sum[2][w] = cnt; }
        __syncthreads();
        sum = sq = cnt = 0.f;
#pragma unroll
        for (int q = 0; q < W; ++q) { sum += s.sum[0][q]; sq += s.sum[1][q]; cnt += s.sum[2][q]; }
    }
    const float mean = sum / cnt;
    const float sd = sqrtf(fmaxf(sq / cnt - mean * mean, 0.f));
    float last_v = 0.f;     // the last score kept
    bool found = false;
    uint32_t kl = 1u, kh = 0xffffffffu;   // keys that the search may be left with (see select_by_key)
    int c_lo = NBk, c_hi = 0;
    if (sd > 0.f && sd < 1e30f && fabsf(mean) < 1e30f) {   // (uniform over the row)
        // 2. two probes a step, aimed at a few ranks on either side of k: first from the normal
        // distribution of that mean and spread, then by interpolation between the bracketing probes
        float lo = -INFINITY, hi = INFINITY;   // count(x >= lo) = c_lo >= k > c_hi = count(x >= hi)
        float t1 = fmaf(sd, heads.z[0][h], mean), t2 = fmaf(sd, heads.z[1][h], mean), reach = 0.5f * sd;
        int stalls = 0;
        bool sampled = false;
#pragma unroll 1
        for (int step = 0; step < MAX_STEPS; ++step) {
            int c = 0;
#pragma unroll
            for (int i = 0; i < KPL; ++i) {
                if (x[i] >= t1) c += 1;
                if (x[i] >= t2) c += 0x10000;
            }
            c = row_total<W>(s, c, w, lane, turn);
            const int c1 = c & 0xffff, c2 = c >> 16, was = c_lo - c_hi;
            if (c1 >= k) { lo = t1; c_lo = c1; } else { hi = t1; c_hi = c1; }
            if (c2 >= k) { lo = t2; c_lo = c2; } else if (c1 >= k) { hi = t2; c_hi = c2; }
            if (c_lo - c_hi <= CANDS && hi < INFINITY && lo > -INFINITY) { found = true; break; }
            if (step > 0 && 8 * (c_lo - c_hi) > 7 * was && ++stalls == 6) break;   // no headway
            if (stalls == 1 && !sampled) {
                if (!sample_probes<W>(s, buf[lane * KPL + KPL / 2], lo, hi, k - c_hi, c_lo - c_hi, w, lane, turn, t1, t2)) break;
                sampled = true;
            } else if (hi == INFINITY) {
                t1 = lo + reach;
                t2 = t1 + reach;
                reach *= 4.f;
            } else if (lo == -INFINITY) {
                t2 = hi - reach;
                t1 = t2 - reach;
                reach *= 4.f;
            } else {
                const float span = hi - lo, per = span / (float)(c_lo - c_hi);
                const float at = lo + per * (float)(c_lo - k);
                const float side = fmaxf(12.f * per, 0.02f * span);
                t1 = fmaxf(at - side, lo + 0.02f * span);
                t2 = fminf(at + side, hi - 0.02f * span);
                if (!(t1 > lo && t2 > t1 && t2 < hi)) break;   // the bracket has no room left
            }
        }
        if (found) {
            // 3. rank the few scores between the probes: the (k - c_hi)-th is the last one kept, unless
            // equal scores lie on both sides of the cut
            const int n = c_lo - c_hi, need = k - c_hi;
            uint32_t in[2] = {0, 0};
#pragma unroll
            for (int i = 0; i < KPL; ++i)
                if (x[i] >= lo && x[i] < hi) in[i / 32] |= 1u << (i % 32);
            if (in[0] | in[1]) {
                int at = atomicAdd(&s.n, __popc(in[0]) + __popc(in[1]));
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    for (uint32_t m = in[q]; m; m &= m - 1) s.key[at++] = __float_as_uint(buf[lane * KPL + q * 32 + __ffs(m) - 1]);
            }
            row_sync<W>();
            const float v = lane < n ? __uint_as_float(s.key[lane]) : 0.f;
            int above = 0, equal = 0;
            for (int q = 0; q < n; ++q) {
                const float vq = __shfl_sync(0xffffffffu, v, q);
                above += vq > v ? 1 : 0;
                equal += vq == v ? 1 : 0;
            }
            // (among equal scores exactly the last of the kept ones has above + equal == need, if they all are kept)
            const uint32_t at = __ballot_sync(0xffffffffu, lane < n && above + equal == need);
            found = at != 0;
            last_v = __shfl_sync(0xffffffffu, v, at ? __ffs(at) - 1 : 0);
            if (!found) {   // equal scores on both sides of the cut: the search over keys ranks them
                row_sync<W>();
                if (tid == 0) s.n = 0;
                row_sync<W>();
            }
        }
        if (lo > -INFINITY) kl = float_key(lo);
        if (hi < INFINITY) kh = float_key(hi) - 1u;
    }
    uint32_t take[2] = {0, 0};                        // bit i: x[i] is kept
    if (found) {
#pragma unroll
        for (int i = 0; i < KPL; ++i)
            if (x[i] >= last_v) take[i / 32] |= 1u << (i % 32);
    } else {
        const uint64_t t = select_by_key<W, KPL>(s, buf, NBk, first, k, kl, kh, c_lo - c_hi, c_hi, w, lane, turn);
        take[0] = (uint32_t)t;
        take[1] = (uint32_t)(t >> 32);
    }
    // 4. the kept indices in ascending order
    int at = row_before<W>(s, __popc(take[0]) + __popc(take[1]), w, lane, turn);
#pragma unroll
    for (int q = 0; q < 2; ++q)
        for (uint32_t m = take[q]; m; m &= m - 1) out[at++] = first + q * 32 + __ffs(m) - 1;
}

// Rows of at most 32 KPL scores (KPL = 1, 2), one warp each: every score is ranked against all the others, in a quarter of the
// instructions of the search above and without its chain of dependent steps, which a call of few rows waits for.
// Calls back to back, us, search / ranking: 384 rows of 32 3.2 / 1.7, 60 000 44.8 / 23.4, 684 of 57 3.5 / 2.8, 4560 of 57 4.9 / 5.2.
template <int KPL>
__global__ void __launch_bounds__(256) select_rank_kernel(const float* __restrict__ scores, int32_t* __restrict__ sel, int H,
                                                          int NBq, int NBk, int kmax, const SelHeads heads, int64_t rows) {
    dep_sync();
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= rows) return;
    const int k = min(heads.k[(row / NBq) % H], NBk);
    int32_t* out = sel + row * kmax;
    for (int t = k + lane; t < kmax; t += 32) out[t] = -1;
    if (k == NBk) {   // keep everything (uniform over the row)
#pragma unroll
        for (int i = 0; i < KPL; ++i)
            if (i * 32 + lane < NBk) out[i * 32 + lane] = i * 32 + lane;
        return;
    }
    uint32_t key[KPL];
    int rank[KPL];
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        const int j = i * 32 + lane;
        key[i] = j < NBk ? float_key_any(scores[row * NBk + j]) : 0u;   // 0: below every key
        rank[i] = 0;
    }
#pragma unroll 8
    for (int q = 0; q < 32; ++q) {
        const uint32_t before = q < lane ? 1u : 0u;   // of equal scores the one of the lower index comes first
#pragma unroll
        for (int p = 0; p < KPL; ++p) {
            const uint32_t other = __shfl_sync(0xffffffffu, key[p], q);
#pragma unroll
            for (int i = 0; i < KPL; ++i)
                if (p == i ? other + before > key[i] : (p < i ? other >= key[i] : other > key[i])) ++rank[i];
        }
    }
    int at = 0;
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        const bool kept = i * 32 + lane < NBk && rank[i] < k;
        const uint32_t m = __ballot_sync(0xffffffffu, kept);
        if (kept) out[at + __popc(m & ((1u << lane) - 1u))] = i * 32 + lane;
        at += __popc(m);
    }
}

template <int KPL>
static cudaError_t launch_rank(const float* scores, int32_t* sel, int H, int NBq, int NBk, int kmax, const SelHeads& heads,
                               int64_t rows, cudaStream_t st) {
    return launch_dep_smem(select_rank_kernel<KPL>, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, st, scores, sel, H, NBq, NBk, kmax,
                           heads, rows);
}

template <int W, int KPL>
static cudaError_t launch_select(const float* scores, int32_t* sel, int H, int NBq, int NBk, int kmax, const SelHeads& heads,
                                 int64_t rows, cudaStream_t st) {
    constexpr int WARPS = W == 1 ? 8 : W;
    constexpr size_t smem = (size_t)WARPS * 32 * KPL * sizeof(float);
    static_assert(smem <= 48 * 1024, "no attribute needed");
    return launch_dep_smem(select_kernel<W, KPL>, dim3((unsigned)(W == 1 ? (rows + 7) / 8 : rows)), dim3(WARPS * 32), smem, st,
                      scores, sel, H, NBq, NBk, kmax, heads, rows);
}

// Standard deviations above the mean at which a normal distribution has a share p (0 < p < 1) of its
// mass above: rational approximation 26.2.23 of Abramowitz and Stegun (error below 4.5e-4).
static float upper_quantile(float p) {
    const float q = p < 0.5f ? p : 1.f - p;
    const float t = sqrtf(-2.f * logf(q));
    const float z = t - (2.515517f + t * (0.802853f + t * 0.010328f)) /
                            (1.f + t * (1.432788f + t * (0.189269f + t * 0.001308f)));
    return p < 0.5f ? z : -z;
}

// Probes at a sixth of the smaller side (but at least 8 ranks) below and above rank k.
static void first_probes(SelHeads& heads, int h, int NBk) {
    const float n = (float)NBk, k = (float)heads.k[h];
    const float side = fmaxf(8.f, fminf(k, n - k) / 6.f);
    heads.z[0][h] = upper_quantile(fminf(k + side, n - 0.5f) / n);
    heads.z[1][h] = upper_quantile(fmaxf(k - side, 0.5f) / n);
}

}  // namespace usv

extern "C" int usv_select_blocks(int B, int H, int NBq, int NBk, const float* scores,
                                 const int32_t* k_per_head, int kmax, int32_t* sel, void* stream) {
    using namespace usv;
    if (B <= 0 || H <= 0 || NBq <= 0 || NBk <= 0)
        return fail(USV_ERR_INVALID_ARG, "select_blocks: B,H,NBq,NBk must be positive");
    if (H > USV_MAX_HEADS) return fail(USV_ERR_UNSUPPORTED, "select_blocks: H > %d", USV_MAX_HEADS);
    if (NBk > SEL_MAX_NB) return fail(USV_ERR_UNSUPPORTED, "select_blocks: NBk > %d", SEL_MAX_NB);
    if (scores == nullptr || sel == nullptr || k_per_head == nullptr)
        return fail(USV_ERR_INVALID_ARG, "select_blocks: null pointer");
    SelHeads heads;
    int kmx = 0;
    for (int h = 0; h < H; ++h) {
        if (k_per_head[h] < 1 || k_per_head[h] > NBk)
            return fail(USV_ERR_INVALID_ARG, "select_blocks: k_per_head[%d]=%d outside [1,%d]", h,
                        k_per_head[h], NBk);
        heads.k[h] = k_per_head[h];
        kmx = k_per_head[h] > kmx ? k_per_head[h] : kmx;
    }
    if (kmax < kmx) return fail(USV_ERR_INVALID_ARG, "select_blocks: kmax=%d < max k=%d", kmax, kmx);
    const int64_t rows = (int64_t)B * H * NBq;
    if (rows > 2147483647LL) return fail(USV_ERR_UNSUPPORTED, "select_blocks: too many rows");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    for (int h = 0; h < H; ++h) first_probes(heads, h, NBk);
#define USV_SEL(W, KPL) launch_select<W, KPL>(scores, sel, H, NBq, NBk, kmax, heads, rows, st)
    // The smallest form that holds the row; up to 64 scores they are ranked, where a call of 33 to 64 has few rows (see
    // select_rank_kernel).  One warp a row up to 544 scores (512 scores, 12 288 rows: 16.7 us,
    // 22.4 with two warps), then two: at 1182 scores and 47 280 rows two warps of 19 scores a lane take
    // 113 us and one warp of 37 119 us; at 3023 and 36 276 rows two warps take 186 us, four 239 us.
    if (NBk <= 32) launch_rank<1>(scores, sel, H, NBq, NBk, kmax, heads, rows, st);
    else if (NBk <= 64 && rows <= 1500) launch_rank<2>(scores, sel, H, NBq, NBk, kmax, heads, rows, st);
    else if (NBk <= 288) USV_SEL(1, 9);
    else if (NBk <= 352) USV_SEL(1, 11);
    else if (NBk <= 544) USV_SEL(1, 17);
    else if (NBk <= 832) USV_SEL(2, 13);
    else if (NBk <= 1088) USV_SEL(2, 17);
    else if (NBk <= 1216) USV_SEL(2, 19);
    else if (NBk <= 1472) USV_SEL(2, 23);
    else if (NBk <= 2112) USV_SEL(2, 33);
    else if (NBk <= 3136) USV_SEL(2, 49);
    else if (NBk <= 4224) USV_SEL(4, 33);
    else if (NBk <= 6272) USV_SEL(4, 49);
    else USV_SEL(8, 33);
#undef USV_SEL
    USV_CHECK_LAUNCH("select_kernel");
    return USV_OK;
}
