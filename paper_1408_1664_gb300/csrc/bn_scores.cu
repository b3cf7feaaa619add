// bn_scores.cu -- step 1 of Algorithm 1: BDeu local scores (Eq. 6).
//
// Scores by variable sets.  With a = ess / |X| for the |X| joint states of a
// set X of variables and T_a(N) = lgamma(a + N) - lgamma(a), let
//   H(X) = sum over the joint states x of X of T_a(N(x)).
// The BDeu score of node i with parents G uses alpha_jk = ess / (r_i q) over
// the states of G + {i} and alpha_j = ess / q over those of G, so
//   log B_i(G) = H(G + {i}) - H(G) + log rho(|G|),
// and the n K families need only the sets of at most d + 1 variables: a set
// of k + 1 variables serves k + 1 families and, as a parent set, n - k - 1
// more (n = 25, d = 8: 4.1 M sets against 31.8 M families).  H is summed
// exactly in 64-bit fixed point, so the difference is the integer that a
// family's own sum over its configurations gives.
//
// Sets are numbered by size, then colexicographically (small_subset_rank
// over the n variables).
#include "bn_device.cuh"
#include "bn_kernels.cuh"

#include <algorithm>
#include <cmath>

namespace bn {
namespace {

constexpr unsigned WARPMASK = 0xffffffffu;

// C(a, b) in global memory: lanes look up different entries, which the
// constant cache would serialise.
__device__ const BinomTable g_binom_scores = make_binom_table();
__device__ __forceinline__ uint32_t gbinom(int a, int b) { return g_binom_scores.v[a][b]; }

// Rank (colex) of mask x among the masks of its size.
__device__ __forceinline__ uint32_t colex_rank(uint32_t x)
{
    uint32_t r = 0;
    int t = 1;
    for (; x; x &= x - 1, ++t) r += gbinom(__ffs(x) - 1, t);
    return r;
}

// The set of number idx (size first) over nb variables and its size.
__device__ __forceinline__ uint32_t set_of(uint32_t idx, int nb, int* size)
{
    int k = 0;
    for (uint32_t c = gbinom(nb, 0); idx >= c; c = gbinom(nb, k)) {
        idx -= c;
        ++k;
    }
    *size = k;
    uint32_t x = 0;
    int c = nb - 1;
    for (int t = k; t >= 1; --t) {
        while (gbinom(c, t) > idx) --c;
        x |= 1u << c;
        idx -= gbinom(c, t);
        --c;
    }
    return x;
}

// Bit pattern of the double equal to the integer q >= 1, by integer
// operations only.
__device__ __forceinline__ long long double_bits(uint32_t q)
{
    const int e = 31 - __clz(q);
    return ((long long)(1023 + e) << 52) | (long long)(((uint64_t)q << (52 - e)) & ((1ull << 52) - 1));
}

// Row of the denominator D in the sorted table of denominators.  Positive
// doubles are ordered like their bit patterns, so the search compares
// integers: the FP64 pipe, narrow on this GPU, is not used.
__device__ __forceinline__ int find_row(const double* Dvals, int rows, uint32_t D)
{
    const long long key = double_bits(D);
    int lo = 0, hi = rows - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__double_as_longlong(Dvals[mid]) < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ long long warp_sum(long long x)
{
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(WARPMASK, x, o);
    return x;
}

}  // namespace

// Everything step 1 prepares before the sets, in one launch (a warp per work
// item, grid-stride):
//  * bit planes: planes[(v*rmax + x)*W + w] bit b <=> data[(64w + b)*n + v] == x,
//    one item per variable and 32 samples, packed by ballots;
//  * T[row*(m+1) + N] = [lgamma(alpha_row + N) - lgamma(alpha_row)] * scale
//    rounded to an integer (scale = 2^S): the fixed-point table;
//  * the rank tables of the 13-bit patterns (rank13 may be null);
//  * the per-node maxima, started at the lowest encoding, the job's error word
//    and step 5's accumulators (enc, err and acc may be null).
// In a batch group mj holds each job's own sample count and fxj its
// (scale, 1/scale): entries past the job's m stay 0 (no count reaches them).
__global__ void __launch_bounds__(256)
k_step1_prep(const uint8_t* __restrict__ data, int n, int m, int rmax, int W,
             uint64_t* __restrict__ planes, const int* __restrict__ mj,
             const double* __restrict__ alpha, int rows, long long* __restrict__ T, double scale,
             const double* __restrict__ fxj, uint16_t* __restrict__ rank13,
             unsigned long long* __restrict__ enc, int* __restrict__ err,
             unsigned long long* __restrict__ acc, size_t js)
{
    data = job_ptr(data, js);
    planes = job_ptr(planes, js);
    alpha = job_ptr(alpha, js);
    T = job_ptr(T, js);
    const int mown = mj ? *job_ptr(mj, js) : m;
    if (fxj) scale = job_ptr(fxj, js)[0];
    const int lane = threadIdx.x & 31;
    const int64_t nplane = (int64_t)n * 2 * W;
    const int64_t ntab = ((int64_t)rows * (m + 1) + 31) / 32;
    const int64_t nrank = rank13 ? 8192 / 32 : 0;
    const int64_t total = nplane + ntab + nrank + 1;
    const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; q < total; q += step) {
        if (q < ntab) {                             // the longest items first
            const int64_t t = q * 32 + lane;
            if (t < (int64_t)rows * (m + 1)) {
                const int row = (int)(t / (m + 1));
                const int N = (int)(t % (m + 1));
                const double a = alpha[row];
                T[t] = (N == 0 || N > mown) ? 0ll
                                            : __double2ll_rn((lgamma(a + (double)N) - lgamma(a)) * scale);
            }
        } else if (q < ntab + nplane) {
            const int64_t p = q - ntab;
            const int v = (int)(p % n), g = (int)(p / n);
            const int s = 32 * g + lane;
            const int val = s < mown ? (int)data[(size_t)s * n + v] : -1;
            uint32_t* half = reinterpret_cast<uint32_t*>(planes) + ((size_t)v * rmax * W) * 2 + g;
            for (int x = 0; x < rmax; ++x) {
                const uint32_t b = __ballot_sync(WARPMASK, val == x);
                if (lane == 0) half[(size_t)x * W * 2] = b;
            }
        } else if (q < ntab + nplane + nrank) {
            uint16_t* rk = job_ptr(rank13, js);
            const uint32_t L = (uint32_t)(q - ntab - nplane) * 32 + lane;
            uint32_t r = colex_rank(L);
            for (int k = 0; k < __popc(L); ++k) r += gbinom(13, k);
            rk[L] = (uint16_t)r;
            rk[8192 + r] = (uint16_t)L;
        } else {
            if (enc && lane < n) job_ptr(enc, js)[lane] = 0ull;
            if (acc)
                for (int t = lane; t < n * (n + 1); t += 32) job_ptr(acc, js)[t] = 0ull;
            // the error word and the counters of k_sweeps after it (256 bytes)
            if (err) reinterpret_cast<int2*>(job_ptr(err, js))[lane] = make_int2(0, 0);
        }
    }
}

// err |= 1 when some data value is not below its variable's arity.
__global__ void k_check_data(const uint8_t* __restrict__ data, const uint8_t* __restrict__ arity,
                             int n, int m, int* err)
{
    const int64_t total = (int64_t)n * m;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        if (data[t] >= arity[t % n]) atomicOr(err, 1);
    }
}

// Binary data, part 1: cnt[X] = the samples in which every variable of X is
// 1, the popcount of the AND of its value-1 planes; 2^lq lanes per set split
// the words.
__global__ void __launch_bounds__(256)
k_set_ones(int n, int m, int W, uint32_t nsets, int lq, const uint64_t* __restrict__ planes,
           const int* __restrict__ mj, uint32_t* __restrict__ cnt, size_t js)
{
    planes = job_ptr(planes, js);
    cnt = job_ptr(cnt, js);
    const int64_t gt = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool live = (gt >> lq) < (int64_t)nsets;
    const uint32_t idx = live ? (uint32_t)(gt >> lq) : nsets - 1;
    int k;
    const uint32_t X = set_of(idx, n, &k);
    uint32_t c = 0;
    for (int w = (int)(gt & ((1 << lq) - 1)); w < W; w += 1 << lq) {
        uint64_t M = ~0ull;
        for (uint32_t x = X; x; x &= x - 1) M &= planes[((size_t)(__ffs(x) - 1) * 2 + 1) * W + w];
        c += (uint32_t)__popcll(M);
    }
    for (int o = 1; o < (1 << lq); o <<= 1) c += __shfl_xor_sync(WARPMASK, c, o);
    if (k == 0) c = (uint32_t)(mj ? *job_ptr(mj, js) : m);
    if (live && (gt & ((1 << lq) - 1)) == 0) cnt[BN_AT(idx, 1, nsets)] = c;
}

// Binary data, part 2: H(X) from the all-ones counts of X's subsets.  The
// count of the joint state whose ones are exactly s is the alternating sum of
// cnt over the supersets of s inside X: one subtraction per state and
// variable (a downward Moebius transform of 2^k values), then a table lookup
// per state.  The samples are not touched, so the cost does not depend on m
// (n = 25, d = 8, m = 500: the scores 33.3 -> 4.8 ms, and with
// k_set_pairs 3.7).  Sets of at most 5 variables take a thread (32 registers; the
// states of a missing variable count 0 and add T[0] = 0), the first ns5 of
// them; larger ones (up to 10) a warp: the five lowest variables are the lane
// bits, the others 2^(k-5) registers.  What bounds it: the gathers of cnt and
// T (both L2-resident), and for k = 9 the 80 shuffles of the lane bits.
template <int RB>
__device__ __forceinline__ long long moebius_warp(uint32_t X, int lane,
                                                  const uint32_t* __restrict__ soff,
                                                  const uint32_t* __restrict__ cnt, uint32_t nsets,
                                                  const long long* __restrict__ Tk, int64_t* dbg)
{
    constexpr int R = 1 << RB;
    const int p0 = __popc(lane);
    uint32_t low = 0, rest = X;
    int pos = 1;
#pragma unroll
    for (int e = 0; e < 5; ++e) {
        const int c = __ffs(rest) - 1;
        rest &= rest - 1;
        if (lane >> e & 1) low += gbinom(c, pos++);
    }
    uint32_t hb[RB][RB], so[RB + 1], rr[R];
#pragma unroll
    for (int e = 0; e < RB; ++e) {
        const int c = __ffs(rest) - 1;
        rest &= rest - 1;
#pragma unroll
        for (int j = 0; j <= e; ++j) hb[e][j] = gbinom(c, p0 + j + 1);
    }
#pragma unroll
    for (int j = 0; j <= RB; ++j) so[j] = soff[p0 + j] + low;
    uint32_t v[R];
    rr[0] = 0;
    v[0] = cnt[BN_AT(so[0], 1, nsets)];
#pragma unroll
    for (int e = 0; e < RB; ++e)
#pragma unroll
        for (int r = 0; r < (1 << e); ++r) {
            int pc = 0;
#pragma unroll
            for (int b = 0; b < RB; ++b) pc += r >> b & 1;
            const int s = r | (1 << e);
            rr[s] = rr[r] + hb[e][pc];
            v[s] = cnt[BN_AT(so[pc + 1] + rr[s], 1, nsets)];
        }
#pragma unroll
    for (int b = 0; b < RB; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (!(r >> b & 1)) v[r] -= v[r | (1 << b)];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t y = __shfl_xor_sync(WARPMASK, v[r], o);
            v[r] -= (lane & o) ? 0u : y;
        }
    long long acc = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) acc += Tk[v[r]];
    if (dbg) {
#pragma unroll
        for (int r = 0; r < R; ++r) dbg[lane | (r << 5)] = v[r];
    }
    return warp_sum(acc);
}

constexpr int kMoebiusMax = 10;                     // variables of a set a warp holds
constexpr int kMoebiusRun = 4;                      // consecutive sets per warp

__global__ void __launch_bounds__(256)
k_set_moebius(int n, int m, uint32_t nsets, uint32_t ns5, uint32_t nall,
              const uint32_t* __restrict__ cnt, const double* __restrict__ Dvals, int rows,
              const long long* __restrict__ T, long long* __restrict__ H, int64_t* __restrict__ dbg,
              uint32_t dbg_set, size_t js)
{
    cnt = job_ptr(cnt, js);
    Dvals = job_ptr(Dvals, js);
    T = job_ptr(T, js);
    H = job_ptr(H, js);
    __shared__ uint32_t soff[16];
    if (threadIdx.x < 16) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= n; ++k) o += gbinom(n, k);
        soff[threadIdx.x] = o;
    }
    __syncthreads();
    const uint32_t nb5 = (ns5 + blockDim.x - 1) / blockDim.x;
    if (blockIdx.x < nb5) {
        const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
        if (idx >= ns5) return;
        int k;
        const uint32_t X = set_of(idx, n, &k);
        uint32_t bx[5][5];
        uint32_t rest = X;
#pragma unroll
        for (int e = 0; e < 5; ++e) {
            const int c = rest ? __ffs(rest) - 1 : 0;
            rest &= rest - 1;
#pragma unroll
            for (int j = 0; j <= e; ++j) bx[e][j] = gbinom(c, j + 1);
        }
        uint32_t rr[32], v[32];
        rr[0] = 0;
        v[0] = cnt[0];
#pragma unroll
        for (int e = 0; e < 5; ++e)
#pragma unroll
            for (int r = 0; r < (1 << e); ++r) {
                int pc = 0;
#pragma unroll
                for (int b = 0; b < 5; ++b) pc += r >> b & 1;
                const int s = r | (1 << e);
                rr[s] = rr[r] + bx[e][pc];
                v[s] = e < k ? cnt[BN_AT(soff[pc + 1] + rr[s], 1, nall)] : 0u;
            }
#pragma unroll
        for (int b = 0; b < 5; ++b)
#pragma unroll
            for (int r = 0; r < 32; ++r)
                if (!(r >> b & 1)) v[r] -= v[r | (1 << b)];
        const long long* Tk = T + (size_t)find_row(Dvals, rows, 1u << k) * (m + 1);
        long long acc = 0;
#pragma unroll
        for (int r = 0; r < 32; ++r)
            if (r < (1 << k)) acc += Tk[v[r]];
        H[BN_AT(idx, 1, nall)] = acc;
        if (dbg && idx == dbg_set) {
#pragma unroll
            for (int r = 0; r < 32; ++r)
                if (r < (1 << k)) dbg[r] = v[r];
        }
        return;
    }
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x - nb5) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    uint32_t idx = ns5 + warp * kMoebiusRun;
    if (idx >= nsets) return;
    const uint32_t end = min(nsets, idx + kMoebiusRun);
    int k;
    uint32_t X = set_of(idx, n, &k);
    const long long* Tk = T + (size_t)find_row(Dvals, rows, 1u << k) * (m + 1);
    for (;;) {
        int64_t* db = dbg && idx == dbg_set ? dbg : nullptr;
        long long h;
        switch (k) {
        case 6: h = moebius_warp<1>(X, lane, soff, cnt, nall, Tk, db); break;
        case 7: h = moebius_warp<2>(X, lane, soff, cnt, nall, Tk, db); break;
        case 8: h = moebius_warp<3>(X, lane, soff, cnt, nall, Tk, db); break;
        case 9: h = moebius_warp<4>(X, lane, soff, cnt, nall, Tk, db); break;
        default: h = moebius_warp<5>(X, lane, soff, cnt, nall, Tk, db); break;
        }
        if (lane == 0) H[BN_AT(idx, 1, nall)] = h;
        if (++idx >= end) break;
        if (X >> (n - k) == (1u << k) - 1u) {       // the last set of its size
            ++k;
            X = (1u << k) - 1u;
            Tk = T + (size_t)find_row(Dvals, rows, 1u << k) * (m + 1);
        } else {                                    // the next mask with k elements
            const uint32_t u = X & (0u - X), w = X + u;
            X = w | (((w ^ X) >> 2) >> (__ffs(u) - 1));
        }
    }
}

// The sets of b, b + 1 and b + 2 variables (b + 2 the largest size, b = 5 .. 8) from their
// bases: a warp takes the base Y (b variables, bits as in moebius_warp), then
// each variable c below all of Y, then each pair c0 < c1 below all of Y, so
// every set comes up once.  With v the counts of Y's joint states among the
// samples whose added variables are 1 (2^b counts gathered and transformed),
// the states with an added variable 0 are differences of such counts:
//   Y + c:        v_c, v - v_c
//   Y + c0 + c1:  v_01, v_1 - v_01, v_0 - v_01, v - v_0 - v_1 + v_01.
// That takes a quarter of the gathers and shuffles of 2^(b+2) counts; the
// table lookups, one per state, are the same.  The v_c stay in shared memory
// (16 bits: m < 65536).  Bases with many variables below them go first.  What
// bounds it: the L1 requests of the gathers (cnt: a line per lane; T: one per
// distinct count).  Scores, us, set by set -> from bases: n = 25, m = 500,
// d = 6 656 -> 427, d = 8 4826 -> 3699.  Four pairs at once measured 427
// against 519 with bases of 5 but 4998 against 4303 with bases of 7.
template <int RB>
__device__ __forceinline__ void pairs_warp(uint32_t Y, int b, int lane, const uint32_t* __restrict__ soff,
                                           const uint32_t* __restrict__ cnt, uint32_t nsets,
                                           const long long* __restrict__ T0, const long long* __restrict__ T1,
                                           const long long* __restrict__ T2, uint16_t* __restrict__ vc,
                                           long long* __restrict__ H, int64_t* __restrict__ dbg, uint32_t dbg_set)
{
    constexpr int R = 1 << RB;
    const int p0 = __popc(lane);
    // off[s][r]: index of this lane's subset of Y with s smaller variables
    // added, less the ranks of those
    uint32_t off[3][R];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        uint32_t low = 0, rest = Y, rr[R];
        int pos = 1 + s;
#pragma unroll
        for (int e = 0; e < 5; ++e) {
            const int c = __ffs(rest) - 1;
            rest &= rest - 1;
            if (lane >> e & 1) low += gbinom(c, pos++);
        }
        rr[0] = 0;
        off[s][0] = soff[p0 + s] + low;
#pragma unroll
        for (int e = 0; e < RB; ++e) {
            const int c = __ffs(rest) - 1;
            rest &= rest - 1;
#pragma unroll
            for (int r = 0; r < (1 << e); ++r) {
                int pc = 0;
#pragma unroll
                for (int q = 0; q < RB; ++q) pc += r >> q & 1;
                rr[r | 1 << e] = rr[r] + gbinom(c, p0 + pc + 1 + s);
                off[s][r | 1 << e] = soff[p0 + pc + 1 + s] + low + rr[r | 1 << e];
            }
        }
    }
    auto counts = [&](uint32_t (&v)[R], const uint32_t (&o)[R], uint32_t add) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = cnt[BN_AT(o[r] + add, 1, nsets)];
#pragma unroll
        for (int q = 0; q < RB; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (!(r >> q & 1)) v[r] -= v[r | (1 << q)];
#pragma unroll
        for (int w = 1; w < 32; w <<= 1)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const uint32_t y = __shfl_xor_sync(WARPMASK, v[r], w);
                v[r] -= (lane & w) ? 0u : y;
            }
    };
    auto leave = [&](uint32_t idx, long long acc) {
        acc = warp_sum(acc);
        if (lane == 0) H[BN_AT(idx, 1, nsets)] = acc;
    };
    const uint32_t i0 = __shfl_sync(WARPMASK, off[0][R - 1], 31), i1 = __shfl_sync(WARPMASK, off[1][R - 1], 31),
                   i2 = __shfl_sync(WARPMASK, off[2][R - 1], 31);
    const int nc = __ffs(Y) - 1;                    // the variables below Y
    uint32_t v[R];
    counts(v, off[0], 0u);
    long long acc = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        acc += T0[v[r]];
        if (dbg && i0 == dbg_set) dbg[lane | r << 5] = v[r];
    }
    leave(i0, acc);
    for (int c1 = 0; c1 < nc; ++c1) {
        uint32_t v1[R];
        counts(v1, off[1], (uint32_t)c1);
        acc = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            vc[(c1 * R + r) * 32 + lane] = (uint16_t)v1[r];
            acc += T1[v1[r]] + T1[v[r] - v1[r]];
            if (dbg && i1 + c1 == dbg_set) {
                dbg[(lane | r << 5) << 1 | 1] = v1[r];
                dbg[(lane | r << 5) << 1] = v[r] - v1[r];
            }
        }
        leave(i1 + c1, acc);
        const uint32_t rank1 = (uint32_t)c1 * (uint32_t)(c1 - 1) / 2;   // C(c1, 2)
        // several pairs at once while they cost few registers
        constexpr int U = R == 1 ? 4 : 1;
        for (int c = 0; c < c1; c += U) {
            uint32_t w[U][R];
#pragma unroll
            for (int u = 0; u < U; ++u) counts(w[u], off[2], rank1 + min(c + u, c1 - 1));
            long long a[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c0 = min(c + u, c1 - 1);
                a[u] = 0;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t v0 = vc[(c0 * R + r) * 32 + lane];     // this lane's own
                    const uint32_t n10 = v1[r] - w[u][r], n01 = v0 - w[u][r], n00 = v[r] - v1[r] - n01;
                    a[u] += T2[w[u][r]] + T2[n10] + T2[n01] + T2[n00];
                    if (dbg && i2 + rank1 + c0 == dbg_set) {
                        int64_t* o = dbg + ((lane | r << 5) << 2);
                        o[0] = n00;
                        o[1] = n01;
                        o[2] = n10;
                        o[3] = w[u][r];
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) a[u] = warp_sum(a[u]);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (lane == 0 && c + u < c1) H[BN_AT(i2 + rank1 + c + u, 1, nsets)] = a[u];
        }
    }
}

constexpr int kPairsMin = 7;                        // largest size from which bases take over
template <int RB>
__global__ void __launch_bounds__(256, RB < 3 ? 3 : 2)
k_set_pairs(int n, int m, int b, uint32_t nsets, uint32_t nbase, const uint32_t* __restrict__ cnt,
            const double* __restrict__ Dvals, int rows, const long long* __restrict__ T,
            long long* __restrict__ H, int64_t* __restrict__ dbg, uint32_t dbg_set, size_t js)
{
    cnt = job_ptr(cnt, js);
    Dvals = job_ptr(Dvals, js);
    T = job_ptr(T, js);
    H = job_ptr(H, js);
    __shared__ uint32_t soff[16];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (threadIdx.x < 16) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= n; ++k) o += gbinom(n, k);
        soff[threadIdx.x] = o;
    }
    __syncthreads();
    const uint32_t warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (warp >= nbase) return;
    int k;
    const uint32_t Y = set_of(soff[b] + (nbase - 1 - warp), n, &k);
    const int lane = threadIdx.x & 31;
    uint16_t* vc = reinterpret_cast<uint16_t*>(smem_raw) + ((size_t)(threadIdx.x >> 5) * (n - b) << b);
    const long long* T0 = T + (size_t)find_row(Dvals, rows, 1u << b) * (m + 1);
    const long long* T1 = T + (size_t)find_row(Dvals, rows, 2u << b) * (m + 1);
    const long long* T2 = T + (size_t)find_row(Dvals, rows, 4u << b) * (m + 1);
    pairs_warp<RB>(Y, b, lane, soff, cnt, nsets, T0, T1, T2, vc, H, dbg, dbg_set);
}

// One set's counts over the staged words [0, words) of every column, the
// samples from 4 * from on and below upto: lane gl of G.
template <int G>
__device__ __forceinline__ void count_states(const uint32_t* col, int mw, int from, int words, int upto,
                                             const uint32_t* ar, uint32_t X, uint32_t* h, int gl, uint32_t states)
{
    uint32_t q = 1;
    for (int w0 = gl; w0 < words; w0 += 4 * G) {
        uint32_t lo[4] = {0, 0, 0, 0}, hi[4] = {0, 0, 0, 0};
        q = 1;
        for (uint32_t x = X; x; x &= x - 1) {
            const int v = __ffs(x) - 1;
            const uint32_t* cv = col + v * mw;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int w = w0 + u * G;
                const uint32_t y = w < words ? cv[w] : 0u;
                lo[u] += (y & 0x00ff00ffu) * q;
                hi[u] += ((y >> 8) & 0x00ff00ffu) * q;
            }
            q *= ar[v];
        }
        // key < q unless a value is not below its arity (device data, which
        // k_check_data reports): such a sample is left out
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int s = 4 * (from + w0 + u * G);
            const uint32_t key[4] = {lo[u] & 0xffffu, hi[u] & 0xffffu, lo[u] >> 16, hi[u] >> 16};
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (s + b < upto && key[b] < q) atomicAdd(&h[BN_AT(key[b], 1, states)], 1u);
        }
    }
}

// Data of any arity: H(X) from a histogram of the samples' joint states in
// shared memory.  A block stages the whole data set once, transposed to
// columns of bytes (four samples per 32-bit word), and its groups of G
// threads (a warp, or the block for sets of more states) then take sets: the
// keys of four samples are two packed pairs of 16-bit mixed-radix numbers
// (at most 65536 states), one multiply-add per variable and pair, and every
// sample adds 1 to its state's counter.  The work per set is O(m k + states),
// against states * m / 64 popcounts per family before (n = 20, arity 3,
// d = 4, m = 1000).  Sets [s0, s1) in turn over the groups.
template <int G>
__global__ void __launch_bounds__(256)
k_set_hist(int n, int m, int mw, uint32_t s0, uint32_t s1, uint32_t states,
           const uint8_t* __restrict__ data, const uint8_t* __restrict__ arity,
           const int* __restrict__ mj, const double* __restrict__ Dvals, int rows,
           const long long* __restrict__ T, long long* __restrict__ H, int64_t* __restrict__ dbg,
           uint32_t dbg_set, size_t js)
{
    data = job_ptr(data, js);
    arity = job_ptr(arity, js);
    Dvals = job_ptr(Dvals, js);
    T = job_ptr(T, js);
    H = job_ptr(H, js);
    const int mown = mj ? *job_ptr(mj, js) : m;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t* col = reinterpret_cast<uint32_t*>(smem_raw);      // [n][mw]
    uint32_t* ar = col + (size_t)n * mw;
    uint32_t* hist = ar + 32;
    __shared__ long long part[8];
    const int words = (mown + 3) >> 2;
    for (int t = threadIdx.x; t < n * words; t += blockDim.x) {
        const int v = t % n, w = t / n;
        uint32_t x = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (4 * w + b < mown) x |= (uint32_t)data[(size_t)(4 * w + b) * n + v] << (8 * b);
        col[v * mw + w] = x;
    }
    if (threadIdx.x < n) ar[threadIdx.x] = arity[threadIdx.x];
    const int gl = threadIdx.x % G;                 // lane within the group
    const uint32_t grp = blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
    const uint32_t ngrp = gridDim.x * (blockDim.x / G);
    uint32_t* h = hist + (size_t)(threadIdx.x / G) * states;
    for (uint32_t c = gl; c < states; c += G) h[c] = 0u;
    __syncthreads();
    for (uint32_t idx = s0 + grp; idx < s1; idx += ngrp) {
        int k;
        const uint32_t X = set_of(idx, n, &k);
        count_states<G>(col, mw, 0, words, mown, ar, X, h, gl, states);
        uint32_t q = 1;
        for (uint32_t x = X; x; x &= x - 1) q *= ar[__ffs(x) - 1];
        if (G == 32) __syncwarp(); else __syncthreads();
        const long long* Tk = T + (size_t)find_row(Dvals, rows, q) * (m + 1);
        long long acc = 0;
        for (uint32_t c = gl; c < q; c += G) {
            const uint32_t N = h[c];
            acc += Tk[N];
            if (dbg && idx == dbg_set) dbg[c] = N;
            h[c] = 0u;
        }
        acc = warp_sum(acc);
        if (G == 32) {
            __syncwarp();
        } else {
            if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
            __syncthreads();
            acc = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) acc += part[w];
            __syncthreads();                        // part is reused
        }
        if (gl == 0) H[BN_AT(idx, 1, s1)] = acc;
    }
}

// The same for data that do not fit: they pass by in chunks of 4 cw samples, once
// for every round of R sets per group, while the groups' R histograms add up.
// Walking the states with the bit planes instead, as k_set_any does, takes
// states * m / 64 words of k ANDs, each with a division for its digit.  Scores,
// n = 20, arity 3, d = 4, m = 10000: walked 5.57 ms, in chunks 0.52; n = 22, d = 5
// 94 and 4.1.
template <int G>
__global__ void __launch_bounds__(256)
k_set_hist_chunks(int n, int m, int mw, int cw, int R, uint32_t s0, uint32_t s1, uint32_t states,
                  const uint8_t* __restrict__ data, const uint8_t* __restrict__ arity,
                  const int* __restrict__ mj, const double* __restrict__ Dvals, int rows,
                  const long long* __restrict__ T, long long* __restrict__ H, int64_t* __restrict__ dbg,
                  uint32_t dbg_set, size_t js)
{
    data = job_ptr(data, js);
    arity = job_ptr(arity, js);
    Dvals = job_ptr(Dvals, js);
    T = job_ptr(T, js);
    H = job_ptr(H, js);
    const int mown = mj ? *job_ptr(mj, js) : m;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t* col = reinterpret_cast<uint32_t*>(smem_raw);      // [n][mw]
    uint32_t* ar = col + (size_t)n * mw;
    __shared__ long long part[8];
    const int all = (mown + 3) >> 2;
    if (threadIdx.x < n) ar[threadIdx.x] = arity[threadIdx.x];
    const int gl = threadIdx.x % G;
    uint32_t* h = ar + 32 + (size_t)(threadIdx.x / G) * R * states;     // this group's histograms
    for (uint32_t c = gl; c < R * states; c += G) h[c] = 0u;
    const uint32_t per = blockDim.x / G * R;
    for (uint32_t b0 = s0 + blockIdx.x * per; b0 < s1; b0 += gridDim.x * per) {
        const uint32_t i0 = b0 + threadIdx.x / G * R, i1 = min(s1, i0 + R);
        int k;
        for (int from = 0; from < all; from += cw) {
            const int words = min(all - from, cw);
            __syncthreads();                        // the last chunk is counted, its histograms are read
            for (int t = threadIdx.x; t < n * words; t += blockDim.x) {
                const int v = t % n, w = t / n, s = 4 * (from + w);
                uint32_t x = 0;
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (s + b < mown) x |= (uint32_t)data[(size_t)(s + b) * n + v] << (8 * b);
                col[v * mw + w] = x;
            }
            __syncthreads();
            for (uint32_t idx = i0; idx < i1; ++idx)
                count_states<G>(col, mw, from, words, min(mown, 4 * (from + words)), ar, set_of(idx, n, &k),
                                h + (idx - i0) * states, gl, states);
        }
        __syncthreads();
        for (uint32_t idx = i0; idx < i1; ++idx) {
            uint32_t q = 1;
            for (uint32_t x = set_of(idx, n, &k); x; x &= x - 1) q *= ar[__ffs(x) - 1];
            const long long* Tk = T + (size_t)find_row(Dvals, rows, q) * (m + 1);
            uint32_t* hs = h + (idx - i0) * states;
            long long acc = 0;
            for (uint32_t c = gl; c < q; c += G) {
                const uint32_t N = hs[c];
                acc += Tk[N];
                if (dbg && idx == dbg_set) dbg[c] = N;
                hs[c] = 0u;
            }
            acc = warp_sum(acc);
            if (G > 32) {
                if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
                __syncthreads();
                acc = 0;
                for (int w = 0; w < (int)(blockDim.x >> 5); ++w) acc += part[w];
                __syncthreads();                    // part is reused
            }
            if (gl == 0) H[BN_AT(idx, 1, s1)] = acc;
        }
    }
}

// Any set: a warp walks the joint states and counts each with the AND of its
// bit planes, lanes over the words.  For sets of more than kBlockStates states.
__global__ void __launch_bounds__(256)
k_set_any(int n, int m, int W, int rmax, uint32_t s0, uint32_t s1,
          const uint8_t* __restrict__ arity, const uint64_t* __restrict__ planes,
          const int* __restrict__ mj, const double* __restrict__ Dvals, int rows,
          const long long* __restrict__ T, long long* __restrict__ H, int64_t* __restrict__ dbg,
          uint32_t dbg_set, size_t js)
{
    const int mown = mj ? *job_ptr(mj, js) : m;
    arity = job_ptr(arity, js);
    planes = job_ptr(planes, js);
    Dvals = job_ptr(Dvals, js);
    T = job_ptr(T, js);
    H = job_ptr(H, js);
    const int lane = threadIdx.x & 31;
    const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t idx = s0 + warp0; idx < s1; idx += nwarps) {
        int k;
        const uint32_t X = set_of(idx, n, &k);
        uint32_t states = 1;
        for (uint32_t x = X; x; x &= x - 1) states *= arity[__ffs(x) - 1];
        const long long* Tk = T + (size_t)find_row(Dvals, rows, states) * (m + 1);
        long long acc = 0;
        for (uint32_t c = 0; c < states; ++c) {
            uint32_t part = 0;
            for (int w = lane; w < W; w += 32) {
                uint64_t M = ~0ull;
                uint32_t cc = c;
                for (uint32_t x = X; x; x &= x - 1) {
                    const int v = __ffs(x) - 1;
                    const uint32_t r = arity[v], dg = cc % r;
                    cc /= r;
                    M &= planes[((size_t)v * rmax + dg) * W + w];
                }
                part += (uint32_t)__popcll(M);
            }
            // the empty set's one state holds every sample (its planes' AND would
            // count the padding of the last word too)
            const uint32_t N = k == 0 ? (uint32_t)mown : __reduce_add_sync(WARPMASK, part);
            if (lane == (int)(c & 31)) {
                acc += Tk[N];
                if (dbg && idx == dbg_set) dbg[c] = N;
            }
        }
        acc = warp_sum(acc);
        if (lane == 0) H[BN_AT(idx, 1, s1)] = acc;
    }
}

// The families' scores from the sets: log B_i(G) = (H(G + i) - H(G)) 2^-S +
// log rho(|G|) + log w_i(G), the parent masks, and the running maximum of each
// node (an order-preserving encoding, integer atomics: the result does not
// depend on the order of arrival).  A thread per family; the two gathers of
// H hit L2.
__global__ void __launch_bounds__(256)
k_family_scores(int n, int64_t K, const long long* __restrict__ H, uint32_t nsets,
                const double* __restrict__ log_rho, const double* __restrict__ log_w,
                uint32_t* __restrict__ masks, uint32_t* __restrict__ cmasks,
                double* __restrict__ logB, unsigned long long* __restrict__ enc, double tinv,
                const double* __restrict__ fxj, size_t js)
{
    H = job_ptr(H, js);
    if (log_rho) log_rho = job_ptr(log_rho, js);
    if (log_w) log_w = job_ptr(log_w, js);
    masks = job_ptr(masks, js);
    cmasks = job_ptr(cmasks, js);
    logB = job_ptr(logB, js);
    if (fxj) tinv = job_ptr(fxj, js)[1];
    __shared__ unsigned long long top[32];
    __shared__ uint32_t soff[34];
    if (threadIdx.x < 32) top[threadIdx.x] = 0ull;
    if (threadIdx.x < 34) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= n; ++k) o += gbinom(n, k);
        soff[threadIdx.x] = o;
    }
    __syncthreads();
    const int64_t total = (int64_t)n * K;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    // every lane of a warp runs every round (the maxima use warp shuffles)
    for (int64_t x0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; x0 < total; x0 += step) {
        const int64_t x = x0 + lane;
        unsigned long long e = 0ull;
        int i = -1;
        if (x < total) {
            i = (int)(x / K);
            int k;
            const uint32_t cm = set_of((uint32_t)(x % K), n - 1, &k);
            const uint32_t G = expand(cm, i);
            uint32_t rg = 0, rx = 0;
            int tg = 1, tx = 1;
            for (uint32_t y = G | (1u << i); y; y &= y - 1) {
                const int c = __ffs(y) - 1;
                rx += gbinom(c, tx++);
                if (c != i) rg += gbinom(c, tg++);
            }
            const long long dh = H[BN_AT(soff[k + 1] + rx, 1, nsets)] - H[BN_AT(soff[k] + rg, 1, nsets)];
            double b = (double)dh * tinv + (log_rho ? log_rho[k] : 0.0);
            if (log_w) b += log_w[x];
            const size_t xc = BN_AT(x, 1, (size_t)n * K);
            logB[xc] = b;
            masks[xc] = G;
            cmasks[xc] = cm;
            e = ord_enc(b);
        }
        if (enc) {
            const int i0 = __shfl_sync(WARPMASK, i, 0);
            if (__all_sync(WARPMASK, i == i0)) {
                for (int o = 16; o; o >>= 1) {
                    const unsigned long long y = __shfl_xor_sync(WARPMASK, e, o);
                    e = y > e ? y : e;
                }
                if (lane == 0) atomicMax(&top[i0], e);
            } else if (i >= 0) {
                atomicMax(&top[i], e);
            }
        }
    }
    __syncthreads();
    if (enc && threadIdx.x < n && top[threadIdx.x]) atomicMax(job_ptr(enc, js) + threadIdx.x, top[threadIdx.x]);
}

__device__ __forceinline__ void from_ln(double x, float& y) { y = (float)LogOps<float>::from_ln(x); }
__device__ __forceinline__ void from_ln(double x, double& y) { y = x; }
__device__ __forceinline__ void from_ln(double x, X64& y) { y = x_from_ln(x); }

// The shifted scores lbs = log B - c_i in the working precision and base
// (X64: B / exp(c_i)),
// the shifts cmax themselves (from their encodings), and, for the
// 13-dimension up-zeta tiles (tab not null), the same scores reordered by
// high and low part of the parent set (see k_reorder_up).
template <typename T>
__global__ void __launch_bounds__(256)
k_shift_scores(int n, int d, int64_t K, const double* __restrict__ logB,
               const unsigned long long* __restrict__ enc, const uint32_t* __restrict__ cmasks,
               double* __restrict__ cmax, T* __restrict__ lbs, T* __restrict__ tab, size_t js)
{
    logB = job_ptr(logB, js);
    enc = job_ptr(enc, js);
    cmasks = job_ptr(cmasks, js);
    cmax = job_ptr(cmax, js);
    lbs = job_ptr(lbs, js);
    __shared__ uint32_t off13[16], rowoff[32];      // the reordered table's columns and rows
    const int h = n - 14;
    if (tab) {
        tab = job_ptr(tab, js);
        if (threadIdx.x < 16) {
            uint32_t o = 0;
            for (int k = 0; k < (int)threadIdx.x && k <= 13; ++k) o += gbinom(13, k);
            off13[threadIdx.x] = o;
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            uint32_t o = 0;
            for (int k = 0; k < (int)threadIdx.x && k <= min(d, h); ++k)
                o += gbinom(h, k) * off13[min(d - k, 13) + 1];
            rowoff[threadIdx.x] = o;
        }
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x < n) cmax[threadIdx.x] = ord_dec(enc[threadIdx.x]);
    const int64_t total = (int64_t)n * K;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(x / K);
        T y;
        from_ln(logB[x] - ord_dec(enc[i]), y);
        lbs[x] = y;
        if (tab) {
            const uint32_t cm = cmasks[x];
            const uint32_t gl = cm & 8191u, gh = cm >> 13;
            const int kh = __popc(gh);
            const uint32_t col = off13[__popc(gl)] + colex_rank(gl);
            const uint32_t row = rowoff[kh] + colex_rank(gh) * off13[min(d - kh, 13) + 1];
            tab[BN_AT((size_t)i * K + row + col, 1, (size_t)n * K)] = y;
        }
    }
}

#ifndef BN_MEGA  // host launchers (bn_mega.cu includes only the device code)
#ifdef BN_CHECK_BOUNDS
BN_BOUNDS_READER(bounds_line_scores)
#endif
namespace {

int grid_for(int64_t work, int threads, int cap = 152 * 32)
{
    int64_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

uint64_t choose(int n, int k)
{
    if (k < 0 || k > n) return 0;
    uint64_t r = 1;
    for (int t = 1; t <= k; ++t) r = r * (uint64_t)(n - k + t) / (uint64_t)t;
    return r;
}

// Sets of fewer than k variables.
uint32_t sets_before(int n, int k)
{
    uint64_t s = 0;
    for (int j = 0; j < k && j <= n; ++j) s += choose(n, j);
    return (uint32_t)std::min<uint64_t>(s, 0xffffffffu);
}

// The kernels of a plan's sets: sizes [0, moebius), [moebius, warp) and
// [warp, block) by warp and block histograms over the whole data, [block,
// cwarp) and [cwarp, cblock) by the same over chunks of it, [cblock, end) by
// k_set_any.  A warp's histogram holds at most 1024 states (32 KB per block),
// a block's at most 16384 (64 KB), beside the staged data; at most 192 KB in
// all.  Chunks and the histograms of a round (R sets per group, as many as 32
// and 64 KB hold, at most 8) take 96 KB, two blocks per SM.
struct SetSplit {
    int moebius, warp, block, cwarp, cblock, end;
    int pairs;                                      // size of k_set_pairs' bases (0: not used)
    int mw;                                         // words of a staged column
    uint32_t wstates, bstates, cwstates, cbstates;
};
constexpr uint32_t kWarpStates = 1024, kBlockStates = 16384;
constexpr size_t kSetSmem = 192 * 1024, kChunkSmem = 96 * 1024;

size_t hist_bytes(const Plan& P, int mw, uint32_t states) { return 4 * ((size_t)P.n * mw + 32 + states); }

SetSplit split_sets(const Plan& P)
{
    SetSplit x{};
    x.end = std::min(P.d + 1, P.n) + 1;
    x.mw = ((P.m + 3) / 4) | 1;                     // odd: columns start in different banks
    x.moebius = P.allbin ? std::min(x.end, kMoebiusMax + 1) : 0;
    x.pairs = x.moebius - 1 >= kPairsMin && P.m < 65536 ? x.moebius - 3 : 0;
    x.warp = x.moebius;
    while (x.warp < x.end && P.states[x.warp] <= kWarpStates &&
           hist_bytes(P, x.mw, 8 * P.states[x.warp]) <= kSetSmem)
        x.wstates = P.states[x.warp++];
    x.block = x.warp;
    while (x.block < x.end && P.states[x.block] <= kBlockStates &&
           hist_bytes(P, x.mw, P.states[x.block]) <= kSetSmem)
        x.bstates = P.states[x.block++];
    x.cwarp = x.block;
    while (x.cwarp < x.end && P.states[x.cwarp] <= kWarpStates) x.cwstates = P.states[x.cwarp++];
    x.cblock = x.cwarp;
    while (x.cblock < x.end && P.states[x.cblock] <= kBlockStates) x.cbstates = P.states[x.cblock++];
    return x;
}

// The shape of a chunked launch: `groups` per block, sets of at most `states`.
struct ChunkShape {
    int R, cw, mw;                                  // sets per group and round; words of a chunk, of a column
    size_t bytes;
    ChunkShape(const Plan& P, int groups, uint32_t states)
    {
        const uint32_t most = groups > 1 ? kWarpStates : kBlockStates;
        R = (int)std::min<uint32_t>(8, std::max<uint32_t>(1, most / states));
        const size_t h = 4 * ((size_t)groups * R * states + 32);
        cw = (int)((kChunkSmem - h) / (4 * (size_t)P.n)) - 1;      // at least 255 words (n <= 32)
        mw = cw | 1;
        bytes = h + 4 * (size_t)P.n * mw;
    }
};

}  // namespace

uint32_t score_sets(const Plan& P) { return sets_before(P.n, std::min(P.d + 1, P.n) + 1); }

cudaError_t launch_step1_prep(const Plan& P, const uint8_t* data, uint64_t* planes,
                              const double* alpha, void* T, uint16_t* rank13,
                              unsigned long long* enc, int* err, unsigned long long* acc, cudaStream_t s,
                              const int* mj, const double* fxj)
{
    const int64_t items = (int64_t)P.n * 2 * P.W + ((int64_t)P.rows * (P.m + 1) + 31) / 32 +
                          (rank13 ? 256 : 0) + 1;
    return launch_or_record(KID_STEP1_PREP, k_step1_prep, dim3(grid_for(items, 8), P.nj), 256, 0, s, data,
                            P.n, P.m, P.rmax, P.W, planes, mj, alpha, P.rows, (long long*)T,
                            std::ldexp(1.0, P.fxs), fxj, rank13, enc, err, acc, P.js);
}

cudaError_t launch_check_data(const uint8_t* data, const uint8_t* arity, int n, int m,
                              int* err, cudaStream_t s)
{
    if ((int64_t)n * m == 0) return cudaSuccess;
    launch_or_record(KID_CHECK_DATA, k_check_data, grid_for((int64_t)n * m, 256), 256, 0, s, data, arity, n, m, err);
    return cudaGetLastError();
}

int fixed_shift(int m, double ess, const double* Dvals, int rows)
{
    double L = std::log1p((double)m);
    for (int r = 0; r < rows; ++r) {
        const double a = ess / Dvals[r];
        L = std::max(L, std::max(std::fabs(std::log(a)), std::log(a + (double)m)));
    }
    const double B = 2.0 * (double)m * L + 1.0;
    const int S = 61 - (int)std::ceil(std::log2(B));
    return std::min(52, std::max(8, S));
}

cudaError_t launch_set_scores(const Plan& P, const uint8_t* data, const uint8_t* arity,
                              const uint64_t* planes, const double* Dvals, const void* Tv,
                              const SetScratch& x, cudaStream_t s, const int* mj, int64_t* dbg,
                              uint32_t dbg_set)
{
    const long long* T = static_cast<const long long*>(Tv);
    const SetSplit z = split_sets(P);
    cudaError_t e = cudaSuccess;
    if (z.moebius > 0) {
        const uint32_t nsets = sets_before(P.n, z.moebius), ns5 = sets_before(P.n, std::min(z.moebius, 6));
        // lanes per set: up to 8 while the words last and the sets are few
        int lq = 0;
        while (lq < 3 && (2 << lq) <= P.W && ((int64_t)nsets << lq) < 152 * 1024) ++lq;
        e = launch_or_record(KID_SET_ONES, k_set_ones,
                             dim3((unsigned)((((int64_t)nsets << lq) + 255) / 256), P.nj), 256, 0, s, P.n,
                             P.m, P.W, nsets, lq, planes, mj, x.cnt, P.js);
        if (e != cudaSuccess) return e;
        // the sizes up to `own` set by set, the last three from their bases
        const int b = z.pairs;
        const uint32_t own = b ? sets_before(P.n, b) : nsets, own5 = std::min(ns5, own);
        const uint32_t warps = (own - own5 + kMoebiusRun - 1) / kMoebiusRun;
        e = launch_or_record(KID_SET_MOEBIUS, k_set_moebius, dim3((own5 + 255) / 256 + (warps + 7) / 8, P.nj),
                             256, 0, s, P.n, P.m, own, own5, nsets, x.cnt, Dvals, P.rows, T,
                             x.H, dbg, dbg_set, P.js);
        if (e != cudaSuccess) return e;
        if (b) {
            const uint32_t nbase = (uint32_t)choose(P.n, b);
            // neighbouring bases differ widely in work (the variables below them),
            // and a block holds its place until its slowest warp ends: two warps
            // a block (with 8, 13 of the 24 warps an SM has room for were at work).
            // Whole job, m = 500: n = 25, d = 8 10.95 -> 10.52 ms, n = 20 1.052 ->
            // 1.026 ms; d = 6 4.67 -> 4.65.  A recorded launch has blocks of 256 threads.
            const unsigned threads = recording() ? 256 : 64, per = threads / 32;
            const auto launch = [&](int kid, auto kernel) {
                return launch_or_record(kid, kernel, dim3((nbase + per - 1) / per, P.nj), threads,
                                        ((size_t)(P.n - b) * per << b) * 2, s, P.n, P.m, b, nsets, nbase, x.cnt,
                                        Dvals, P.rows, T, x.H, dbg, dbg_set, P.js);
            };
            e = b == 5   ? launch(KID_SET_PAIRS5, k_set_pairs<0>)
                : b == 6 ? launch(KID_SET_PAIRS6, k_set_pairs<1>)
                : b == 7 ? launch(KID_SET_PAIRS7, k_set_pairs<2>)
                         : launch(KID_SET_PAIRS8, k_set_pairs<3>);
            if (e != cudaSuccess) return e;
        }
    }
    if (z.warp > z.moebius) {
        const uint32_t s0 = sets_before(P.n, z.moebius), s1 = sets_before(P.n, z.warp);
        // about four sets per warp pay for staging the data
        const unsigned g = (unsigned)std::min<int64_t>(((int64_t)(s1 - s0) + 31) / 32,
                                                       std::max(1, 152 * 4 / P.nj));
        e = launch_or_record(KID_SET_HIST_WARP, k_set_hist<32>, dim3(g, P.nj), 256,
                             hist_bytes(P, z.mw, 8 * z.wstates), s, P.n, P.m, z.mw, s0, s1, z.wstates, data,
                             arity, mj, Dvals, P.rows, T, x.H, dbg, dbg_set, P.js);
        if (e != cudaSuccess) return e;
    }
    if (z.block > z.warp) {
        const uint32_t s0 = sets_before(P.n, z.warp), s1 = sets_before(P.n, z.block);
        const unsigned g = (unsigned)std::min<int64_t>(((int64_t)(s1 - s0) + 3) / 4,
                                                       std::max(1, 152 * 4 / P.nj));
        e = launch_or_record(KID_SET_HIST_BLOCK, k_set_hist<256>, dim3(g, P.nj), 256,
                             hist_bytes(P, z.mw, z.bstates), s, P.n, P.m, z.mw, s0, s1, z.bstates, data,
                             arity, mj, Dvals, P.rows, T, x.H, dbg, dbg_set, P.js);
        if (e != cudaSuccess) return e;
    }
    if (z.cwarp > z.block) {
        const uint32_t s0 = sets_before(P.n, z.block), s1 = sets_before(P.n, z.cwarp);
        const ChunkShape c(P, 8, z.cwstates);
        const unsigned g = (unsigned)std::min<int64_t>(((int64_t)(s1 - s0) + 8 * c.R - 1) / (8 * c.R),
                                                       std::max(1, 152 * 4 / P.nj));
        e = launch_or_record(KID_SET_HISTC_WARP, k_set_hist_chunks<32>, dim3(g, P.nj), 256, c.bytes, s, P.n, P.m, c.mw,
                             c.cw, c.R, s0, s1, z.cwstates, data, arity, mj, Dvals, P.rows, T, x.H, dbg, dbg_set,
                             P.js);
        if (e != cudaSuccess) return e;
    }
    if (z.cblock > z.cwarp) {
        const uint32_t s0 = sets_before(P.n, z.cwarp), s1 = sets_before(P.n, z.cblock);
        const ChunkShape c(P, 1, z.cbstates);
        const unsigned g = (unsigned)std::min<int64_t>(((int64_t)(s1 - s0) + c.R - 1) / c.R,
                                                       std::max(1, 152 * 4 / P.nj));
        e = launch_or_record(KID_SET_HISTC_BLOCK, k_set_hist_chunks<256>, dim3(g, P.nj), 256, c.bytes, s, P.n, P.m, c.mw,
                             c.cw, c.R, s0, s1, z.cbstates, data, arity, mj, Dvals, P.rows, T, x.H, dbg, dbg_set,
                             P.js);
        if (e != cudaSuccess) return e;
    }
    if (z.end > z.cblock) {
        const uint32_t s0 = sets_before(P.n, z.cblock), s1 = sets_before(P.n, z.end);
        e = launch_or_record(KID_SET_ANY, k_set_any, dim3(grid_for((int64_t)(s1 - s0), 8, 152 * 16), P.nj),
                             256, 0, s, P.n, P.m, P.W, P.rmax, s0, s1, arity, planes, mj, Dvals, P.rows, T,
                             x.H, dbg, dbg_set, P.js);
    }
    return e;
}

cudaError_t launch_scores(const Plan& P, const uint8_t* data, const uint8_t* arity,
                          const uint64_t* planes, const double* Dvals, const void* T,
                          const double* log_rho, const double* log_w, const SetScratch& x,
                          uint32_t* masks, uint32_t* cmasks, double* logB, cudaStream_t s,
                          const int* mj, const double* fxj)
{
    const cudaError_t e = launch_set_scores(P, data, arity, planes, Dvals, T, x, s, mj);
    if (e != cudaSuccess) return e;
    return launch_or_record(KID_FAMILIES, k_family_scores, dim3(grid_for((int64_t)P.n * P.K, 256, 152 * 16), P.nj),
                            256, 0, s, P.n, P.K, x.H, score_sets(P), log_rho, log_w, masks, cmasks, logB,
                            x.enc, std::ldexp(1.0, -P.fxs), fxj, P.js);
}

int scores_launches(const Plan& P)
{
    const SetSplit z = split_sets(P);
    return (z.moebius > 0 ? 2 : 0) + (z.pairs > 0) + (z.warp > z.moebius) + (z.block > z.warp) +
           (z.cwarp > z.block) + (z.cblock > z.cwarp) + (z.end > z.cblock) + 1;
}

int any_set_sizes(const Plan& P)
{
    const SetSplit z = split_sets(P);
    return z.end - z.cblock;
}

cudaError_t launch_shift_scores(const Plan& P, const double* logB, const unsigned long long* enc,
                                const uint32_t* cmasks, double* cmax, void* lbs, void* tab, cudaStream_t s)
{
    const dim3 grid(grid_for((int64_t)P.n * P.K, 256, 152 * 16), P.nj);
    if (P.lin)
        return launch_or_record(KID_SHIFT_X, k_shift_scores<X64>, grid, 256, 0, s, P.n, P.d, P.K, logB, enc,
                                cmasks, cmax, (X64*)lbs, (X64*)tab, P.js);
    if (P.prec == 0)
        return launch_or_record(KID_SHIFT_D, k_shift_scores<double>, grid, 256, 0, s, P.n, P.d, P.K, logB, enc,
                                cmasks, cmax, (double*)lbs, (double*)tab, P.js);
    return launch_or_record(KID_SHIFT_F, k_shift_scores<float>, grid, 256, 0, s, P.n, P.d, P.K, logB, enc,
                            cmasks, cmax, (float*)lbs, (float*)tab, P.js);
}

cudaError_t set_scores_attributes()
{
    cudaError_t e = allow_max_dynamic_smem(k_set_hist<32>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_set_hist_chunks<32>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_set_hist_chunks<256>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_set_pairs<0>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_set_pairs<1>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_set_pairs<2>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_set_pairs<3>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_set_hist<256>);
    return e;
}

#endif  // BN_MEGA

}  // namespace bn
