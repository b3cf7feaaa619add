// bn_tile13.cu -- register-blocked 13-dimension tiles for the two truncated
// zeta transforms (Eq. 7 / Algorithm 2 and Eq. 12 / Algorithm 3) when n >= 14.
//
// A tile is the 2^13 subsets that share their high bits.  256 threads hold 32
// values each.  A transform over the 13 tile dimensions runs in three
// register layouts (dims 8..12, dims 3..7, dims 0..2), exchanging through a
// swizzled shared-memory array between layouts, so every butterfly is a
// register operation.
//
// Arithmetic is exact to working precision without a log-sum-exp per
// butterfly.  Most tiles are summed in linear scale, in one or a few
// single-scale passes (Window).  The others first compute the max-plus
// transform m(L), the largest single term of every output (a max per
// butterfly), and hold each value as y(L) * 2^m(L) (e^m(L) in FP64): every
// partial sum at L is at most the final output, so y(L) <= 8192, and a
// butterfly adds its partner scaled by 2^(m(partner) - m(L)) <= 1 (m is
// monotone along the butterflies).  A term can only underflow there when it
// is below 2^-126 of the output it belongs to.  One exponential enters per
// input and per butterfly, one logarithm leaves per output.  FP64 avoids a
// full-precision exponential per butterfly: it holds each value as
// x(L) * e^(BW*e(L)) with the band e(L) = floor(m(L) / BW), BW = 600 nats, so
// x(L) lies in [1, e^BW * 8192); a butterfly adds a partner from the same
// band unchanged, one band lower times e^-BW, and drops partners two or more
// bands lower (below e^-BW * 2^-13 of the result: under one rounding unit).
#include "bn_device.cuh"
#include "bn_kernels.cuh"

#include <cmath>

namespace bn {
namespace {

constexpr int TB = 13;            // tile dimensions
constexpr int TN = 1 << TB;       // tile elements
constexpr int TT = 256;           // threads per tile
constexpr int TR = 32;            // values per thread
constexpr unsigned FULLMASK = 0xffffffffu;

// Band width (natural logs) and the factor one band down, FP64 only.
struct Band64 {
    static constexpr double width = 600.0;
    static __device__ __forceinline__ double down1() { return 2.6503965530043108e-261; }  // e^-600
};

// a*b + c in the value's own precision (no promotion to double).
__device__ __forceinline__ float madd(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double madd(double a, double b, double c) { return __fma_rn(a, b, c); }

// Shared-memory position of tile element e.  Flips bits 3,4 by bits 8,9 and
// bit 2 by bit 5, which makes all three layouts' accesses free of bank
// conflicts (32-bit accesses in layouts 1 and 2, 128-bit in layout 3).
__device__ __forceinline__ uint32_t swz(uint32_t e)
{
    return e ^ (((e >> 8) & 3u) << 3) ^ (((e >> 5) & 1u) << 2);
}

// Element held in register r by thread t.
__device__ __forceinline__ uint32_t el1(int r, int t) { return ((uint32_t)r << 8) | (uint32_t)t; }
__device__ __forceinline__ uint32_t el2(int r, int t)
{
    return ((uint32_t)t & 7u) | ((uint32_t)r << 3) | (((uint32_t)t >> 3) << 8);
}
__device__ __forceinline__ uint32_t el3(int r, int t)
{
    return ((uint32_t)r & 7u) | ((uint32_t)t << 3) | (((uint32_t)r >> 3) << 11);
}

// Butterflies over register bits [k0, k0+nk): UP adds a subset into its
// superset (upward zeta), DOWN adds a superset into its subset.
template <bool UP, typename T>
__device__ __forceinline__ void bfly_max(T (&v)[TR], int k0, int nk)
{
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (k < k0 || k >= k0 + nk) continue;
#pragma unroll
        for (int r = 0; r < TR; ++r) {
            if (r & (1 << k)) continue;
            const int s = r | (1 << k);
            if (UP) v[s] = v[s] > v[r] ? v[s] : v[r];
            else v[r] = v[r] > v[s] ? v[r] : v[s];
        }
    }
}

// 2^e for an integer e <= 0, built in the exponent bits (0 below 2^-126).
__device__ __forceinline__ float pow2i(int e)
{
    return __int_as_float(max(e + 127, 0) << 23);
}

// FP32 sum butterflies on values held relative to their own integer scales
// (the bits of `m` are ints: floor of the final max-plus transform): the
// partner is scaled by the exact power of two 2^(m(partner) - m(self)) <= 1.
template <bool UP>
__device__ __forceinline__ void bfly_pow2(float (&x)[TR], const float (&m)[TR], int k0, int nk)
{
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (k < k0 || k >= k0 + nk) continue;
#pragma unroll
        for (int r = 0; r < TR; ++r) {
            if (r & (1 << k)) continue;
            const int s = r | (1 << k);
            const int mr = __float_as_int(m[r]), ms = __float_as_int(m[s]);
            if (UP) x[s] = madd(x[r], pow2i(mr - ms), x[s]);
            else x[r] = madd(x[s], pow2i(ms - mr), x[r]);
        }
    }
}

// Sum butterflies with bands e (exact small integers held as T).  Three
// cases per thread: all its bands equal (plain adds); two adjacent bands
// (factor 1 or e^-BW, one fused multiply-add); otherwise the full rule
// (1, e^-BW, or 0 for partners two or more bands down).
template <bool UP, typename T>
__device__ __forceinline__ void bfly_sum(T (&x)[TR], const T (&e)[TR], int k0, int nk)
{
    T lo = e[0], hi = e[0];
#pragma unroll
    for (int r = 1; r < TR; ++r) {
        lo = e[r] < lo ? e[r] : lo;
        hi = e[r] > hi ? e[r] : hi;
    }
    const T gap = hi - lo;
    if (gap == T(0)) {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if (k < k0 || k >= k0 + nk) continue;
#pragma unroll
            for (int r = 0; r < TR; ++r) {
                if (r & (1 << k)) continue;
                const int s = r | (1 << k);
                if (UP) x[s] += x[r];
                else x[r] += x[s];
            }
        }
    } else if (gap == T(1)) {
        // partner bands differ by 0 or 1: factor 1 or e^-BW
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if (k < k0 || k >= k0 + nk) continue;
#pragma unroll
            for (int r = 0; r < TR; ++r) {
                if (r & (1 << k)) continue;
                const int s = r | (1 << k);
                if (UP) x[s] = madd(x[r], e[s] == e[r] ? T(1) : Band64::down1(), x[s]);
                else x[r] = madd(x[s], e[r] == e[s] ? T(1) : Band64::down1(), x[r]);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if (k < k0 || k >= k0 + nk) continue;
#pragma unroll
            for (int r = 0; r < TR; ++r) {
                if (r & (1 << k)) continue;
                const int s = r | (1 << k);
                const T dd = UP ? e[s] - e[r] : e[r] - e[s];
                const T f = dd == T(0) ? T(1) : (dd == T(1) ? Band64::down1() : T(0));
                if (UP) x[s] = madd(x[r], f, x[s]);
                else x[r] = madd(x[s], f, x[r]);
            }
        }
    }
}

template <bool UP>
__device__ __forceinline__ void sum_bfly(float (&x)[TR], const float (&m)[TR], int k0, int nk)
{
    bfly_pow2<UP>(x, m, k0, nk);
}
template <bool UP>
__device__ __forceinline__ void sum_bfly(double (&x)[TR], const double (&e)[TR], int k0, int nk)
{
    bfly_sum<UP>(x, e, k0, nk);
}
// Scale of an output from its max-plus value, the log that the scale stands
// for, and an output's log from its scaled value.  FP32: an integer (kept as
// the bits of a float); FP64: a band of BW nats.
__device__ __forceinline__ float scale_of(float m) { return __int_as_float(__float2int_rd(m)); }
__device__ __forceinline__ double scale_of(double m) { return floor(m / Band64::width); }
__device__ __forceinline__ float scale_base(float sc) { return (float)__float_as_int(sc); }
__device__ __forceinline__ double scale_base(double sc) { return Band64::width * sc; }
__device__ __forceinline__ float scaled_log(float y, float sc)
{
    return scale_base(sc) + LogOps<float>::lg(y);
}
__device__ __forceinline__ double scaled_log(double x, double e)
{
    return madd(Band64::width, e, LogOps<double>::lg(x));
}

// Online log-sum-exp step (branchless): (m, s) stands for m + lg(s).
template <typename T>
__device__ __forceinline__ void lse_online(T& m, T& s, T x)
{
    using Lg = LogOps<T>;
    const T mn = x > m ? x : m;
    if (mn == Lg::ninf()) return;
    s = s * Lg::ex(m - mn) + Lg::ex(x - mn);
    m = mn;
}

// a0 += b0 and a1 += b1 in one packed FP32 instruction (each lane rounds
// like a scalar add).
__device__ __forceinline__ void add_f32x2(float& a0, float& a1, float b0, float b1)
{
    unsigned long long ra, rb;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a0), "f"(a1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b0), "f"(b1));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(ra) : "l"(rb));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a0), "=f"(a1) : "l"(ra));
}

// Sum butterflies without bands (every value in one common scale).  In FP32
// a butterfly over register bit k >= 1 pairs registers r, r + 1 with s, s + 1:
// packed adds.
template <bool UP, typename T>
__device__ __forceinline__ void bfly_plain(T (&x)[TR], int k0, int nk)
{
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (k < k0 || k >= k0 + nk) continue;
        if constexpr (sizeof(T) == 4) {
            if (k >= 1) {
#pragma unroll
                for (int r = 0; r < TR; r += 2) {
                    if (r & (1 << k)) continue;
                    const int s = r | (1 << k);
                    if (UP) add_f32x2(x[s], x[s + 1], x[r], x[r + 1]);
                    else add_f32x2(x[r], x[r + 1], x[s], x[s + 1]);
                }
                continue;
            }
        }
#pragma unroll
        for (int r = 0; r < TR; ++r) {
            if (r & (1 << k)) continue;
            const int s = r | (1 << k);
            if (UP) x[s] += x[r];
            else x[r] += x[s];
        }
    }
}

// Single-scale windows for both zeta tiles.  Pass p scales the terms by
// s_p = M - top - p * win (M bounds every output from above) and writes the
// outputs whose scaled value is at least 2^lo (e^lo): terms flushed below the
// smallest normal number (2^-126; e^-708) number at most 8192, under 2^-113
// (e^-699) in total, which is below 2^-33 (e^-99) of such an output.  An
// output left over has scaled value below 2^lo in pass p, hence below 2^top
// in pass p + 1, so no term of it overflows there (2^128; e^709).
template <typename T> struct Window;
// gap: how far below a relevance cut an output is held (64 bits; 45 nats).
template <> struct Window<float> {                 // bits
    static constexpr float top = 126.0f, lo = -80.0f, win = 206.0f, gap = 64.0f;
    static constexpr int max_pass = 2;     // a third pass costs more than the exact path
};
template <> struct Window<double> {                // nats
    static constexpr double top = 700.0, lo = -600.0, win = 1300.0, gap = 45.0;
    static constexpr int max_pass = 3;
};

// Layout loads and stores through the swizzled array.
template <typename T> __device__ __forceinline__ void ld1(const T* a, T (&v)[TR], int t)
{
#pragma unroll
    for (int r = 0; r < TR; ++r) v[r] = a[swz(el1(r, t))];
}
template <typename T> __device__ __forceinline__ void st1(T* a, const T (&v)[TR], int t)
{
#pragma unroll
    for (int r = 0; r < TR; ++r) a[swz(el1(r, t))] = v[r];
}
template <typename T> __device__ __forceinline__ void ld2(const T* a, T (&v)[TR], int t)
{
#pragma unroll
    for (int r = 0; r < TR; ++r) v[r] = a[swz(el2(r, t))];
}
template <typename T> __device__ __forceinline__ void st2(T* a, const T (&v)[TR], int t)
{
#pragma unroll
    for (int r = 0; r < TR; ++r) a[swz(el2(r, t))] = v[r];
}
// Layout 3: thread t owns four runs of 8 consecutive elements.
template <typename T> __device__ __forceinline__ void ld3(const T* a, T (&v)[TR], int t)
{
#pragma unroll
    for (int r = 0; r < TR; ++r) v[r] = a[swz(el3(r, t))];
}
template <> __device__ __forceinline__ void ld3<float>(const float* a, float (&v)[TR], int t)
{
    const bool flip = (t >> 2) & 1;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const uint32_t base = swz(el3(8 * x, t)) & ~7u;
        float4 p = *reinterpret_cast<const float4*>(a + base);
        float4 q = *reinterpret_cast<const float4*>(a + base + 4);
        if (flip) { float4 w = p; p = q; q = w; }
        v[8 * x + 0] = p.x; v[8 * x + 1] = p.y; v[8 * x + 2] = p.z; v[8 * x + 3] = p.w;
        v[8 * x + 4] = q.x; v[8 * x + 5] = q.y; v[8 * x + 6] = q.z; v[8 * x + 7] = q.w;
    }
}
template <typename T> __device__ __forceinline__ void st3(T* a, const T (&v)[TR], int t)
{
#pragma unroll
    for (int r = 0; r < TR; ++r) a[swz(el3(r, t))] = v[r];
}
template <> __device__ __forceinline__ void st3<float>(float* a, const float (&v)[TR], int t)
{
    const bool flip = (t >> 2) & 1;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const uint32_t base = swz(el3(8 * x, t)) & ~7u;
        float4 p = make_float4(v[8 * x + 0], v[8 * x + 1], v[8 * x + 2], v[8 * x + 3]);
        float4 q = make_float4(v[8 * x + 4], v[8 * x + 5], v[8 * x + 6], v[8 * x + 7]);
        if (flip) { float4 w = p; p = q; q = w; }
        *reinterpret_cast<float4*>(a + base) = p;
        *reinterpret_cast<float4*>(a + base + 4) = q;
    }
}
// Layout-3 values to global memory: registers 8q..8q+7 of thread t are the
// consecutive elements el3(8q, t) .. el3(8q, t) + 7 (32-byte aligned).
__device__ __forceinline__ void st_out3(float* out, const float (&x)[TR], int t)
{
#pragma unroll
    for (int q = 0; q < TR / 8; ++q) {
        float4* p = reinterpret_cast<float4*>(out + el3(8 * q, t));
        p[0] = make_float4(x[8 * q], x[8 * q + 1], x[8 * q + 2], x[8 * q + 3]);
        p[1] = make_float4(x[8 * q + 4], x[8 * q + 5], x[8 * q + 6], x[8 * q + 7]);
    }
}
__device__ __forceinline__ void st_out3(double* out, const double (&x)[TR], int t)
{
#pragma unroll
    for (int q = 0; q < TR / 8; ++q) {
        double2* p = reinterpret_cast<double2*>(out + el3(8 * q, t));
#pragma unroll
        for (int k = 0; k < 4; ++k) p[k] = make_double2(x[8 * q + 2 * k], x[8 * q + 2 * k + 1]);
    }
}

// The exact sum pass after the max-plus pass.  On entry v holds m (layout
// 3); A1 holds the transform's inputs (for UP only the slots with at most d
// elements are inputs).  On exit v and sc hold, in layout 1, each output as
// scaled_log(v, sc): FP32 keeps y relative to 2^floor(m), FP64 keeps x in
// its band.  The scales replace the inputs in A1: every thread reads its
// layout-3 inputs and writes its layout-3 scales to the same slots.
template <bool UP, typename T>
__device__ __forceinline__ void sum_pass(T (&v)[TR], T (&sc)[TR], T* A1, T* A0, int t, int d)
{
    using Lg = LogOps<T>;
    T* E = A1;
    const int pt = __popc(t);             // |el3(r, t)| = |r| + |t| (disjoint bits)
#pragma unroll
    for (int r = 0; r < TR; ++r) sc[r] = scale_of(v[r]);
    ld3(A1, v, t);                        // inputs
    st3(E, sc, t);                        // scales, read again in layouts 2 and 1
#pragma unroll
    for (int r = 0; r < TR; ++r)
        v[r] = (!UP || __popc(r) + pt <= d) ? Lg::ex(v[r] - scale_base(sc[r])) : T(0);
    sum_bfly<UP>(v, sc, 0, 3);
    __syncthreads();
    st3(A0, v, t);
    __syncthreads();
    ld2(A0, v, t);
    ld2(E, sc, t);
    sum_bfly<UP>(v, sc, 0, 5);
    __syncthreads();
    st2(A0, v, t);
    __syncthreads();
    ld1(A0, v, t);
    ld1(E, sc, t);
    sum_bfly<UP>(v, sc, 0, 5);
}

// Binomial coefficients C(a, b), a < 32, in shared memory, stored for
// b <= a / 2 only (C(a, b) = C(a, a - b)).  Lanes look up different entries,
// which would serialise constant-cache reads; the table is copied from a
// global-memory image with coalesced loads.
__device__ const BinomTable g_binom_image = make_binom_table();
struct SBinom {
    uint32_t v[32][16];
};
__device__ __forceinline__ void fill_sbinom(SBinom& sb)
{
    for (int x = threadIdx.x; x < 32 * 16; x += blockDim.x) sb.v[x >> 4][x & 15] = g_binom_image.v[x >> 4][x & 15];
}
__device__ __forceinline__ uint32_t sb_binom(const SBinom& sb, int a, int b)
{
    if (b < 0 || b > a) return 0u;
    return sb.v[a][min(b, a - b)];
}
__device__ __forceinline__ uint32_t sb_unrank(const SBinom& sb, uint32_t r, int nb, int* kout)
{
    int k = 0;
    while (r >= sb_binom(sb, nb, k)) { r -= sb_binom(sb, nb, k); ++k; }
    uint32_t x = 0;
    int c = nb - 1;
    for (int t = k; t >= 1; --t) {
        while (sb_binom(sb, c, t) > r) --c;
        x |= 1u << c;
        r -= sb_binom(sb, c, t);
        --c;
    }
    if (kout) *kout = k;
    return x;
}


uint64_t binom_host(int n, int k)
{
    if (k < 0 || k > n) return 0;
    uint64_t r = 1;
    for (int t = 1; t <= k; ++t) r = r * (uint64_t)(n - k + t) / (uint64_t)t;
    return r;
}

// Low patterns with at most d of the 13 tile bits (the columns of a tile).
uint32_t num_small_subsets_host(int d)
{
    uint64_t c = 0;
    for (int k = 0; k <= d && k <= TB; ++k) c += binom_host(TB, k);
    return (uint32_t)c;
}


}  // namespace

// ===========================================================================
// Families reordered by (high part G_H, low part g_L) for the tile scatter:
// row = rank of G_H among the subsets of the h = n-14 high index bits with at
// most d elements, column = rank of g_L among the subsets of the 13 low bits
// with at most d - |G_H| elements.  Row r of size k holds C13(<= d-k)
// columns, so the table holds exactly the K families of the node.
// ===========================================================================
__device__ __forceinline__ uint32_t row_offset(int h, int d, int kh, uint32_t rank_in_class)
{
    uint32_t off = 0;
    for (int k = 0; k < kh; ++k) off += binom(h, k) * num_small_subsets(TB, d - k);
    return off + rank_in_class * num_small_subsets(TB, d - kh);
}

template <typename T>
__global__ void k_reorder_up(int n, int d, int64_t K, const T* __restrict__ lbs, T* __restrict__ tab,
                             size_t js, int nodes)
{
    lbs = job_ptr(lbs, js);
    tab = job_ptr(tab, js);
    const int h = n - 1 - TB;
    const int64_t total = (int64_t)nodes * K;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(x / K);
        uint32_t f = (uint32_t)(x % K);
        int k = 0;
        while (f >= binom(n - 1, k)) { f -= binom(n - 1, k); ++k; }
        const uint32_t cm = colex_unrank(f, k, n - 1);
        const uint32_t gl = cm & (TN - 1u), gh = cm >> TB;
        const int kh = __popc(gh);
        // colex rank of gh within its size class
        uint32_t rk = 0;
        int t = 1;
        for (uint32_t y = gh; y; y &= y - 1, ++t) rk += binom(__ffs(y) - 1, t);
        const uint32_t col = small_subset_rank(gl, TB);
        tab[(size_t)i * K + row_offset(h, d, kh, rk) + col] = lbs[x];
    }
}

// ===========================================================================
// Step 2 for n >= 14, part 1: the column sums of tile (i, H) of A_i,
//   C_H(G_L) = log sum of B_i(G_H + G_L) over G_H inside H, |G_H| <= d - |G_L|,
// for every low pattern G_L (13 bits) with at most d elements, in column
// order (by size, then colex).  They go to the first ncol slots of the
// tile's own slice of A, which part 2 reads and then overwrites.  Small
// shared memory and register use keep many blocks resident, which hides the
// latency of the gathers from the score table.
// ===========================================================================
template <typename T>
__global__ void __launch_bounds__(TT, sizeof(T) == 4 ? 4 : 2)
k_upzeta13_cols(int n, int d, int64_t K, const T* __restrict__ tab, T* __restrict__ A, size_t js)
{
    tab = job_ptr(tab, js);
    A = job_ptr(A, js);
    using Lg = LogOps<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* part = reinterpret_cast<T*>(smem_raw);            // 2 * 8 * 96 partial (max, sum) pairs
    SBinom* sb = reinterpret_cast<SBinom*>(part + 2 * 8 * 96);
    int* meta = reinterpret_cast<int*>(sb + 1);          // [0,32) row offsets, [32,64) list starts
    uint32_t* off13 = reinterpret_cast<uint32_t*>(meta + 64);   // 16 entries
    uint32_t* rowbase = off13 + 16;                      // up to nrow entries
    const uint32_t ncol = num_small_subsets(TB, d);
    const int h = n - 1 - TB;

    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int i = (int)(blockIdx.x >> h);
    const uint32_t H = blockIdx.x & ((1u << h) - 1u);
    const T* tb = tab + (size_t)i * K;
    T* out = A + ((size_t)i << (n - 1)) + ((size_t)H << TB);

    fill_sbinom(*sb);
    if (t < 16) {
        uint32_t o = 0;
        for (int k = 0; k < t && k <= TB; ++k) o += binom(TB, k);
        off13[t] = o;
    }
    __syncthreads();

    // --- rows whose high part lies inside H, in row order (by size, then
    //     colex): the k-element subsets of H in increasing mask order.  Entry
    //     p of the list is unranked among the subsets of H's hc positions,
    //     its positions are mapped onto the bits of H, and the row's offset in
    //     the node's table follows from its colex rank among all h-bit sets.
    const int hc = __popc(H);
    const int kmax = min(d, hc);
    if (t < 32) {
        // meta[32 + k]: first list entry of class k (entries of size k)
        meta[32 + t] = (int)num_small_subsets(hc, min(t, d + 1) - 1);
        // meta[k]: offset of the first class-k row in the node's table
        uint32_t o = 0;
        for (int k = 0; k < t && k <= min(d, h); ++k) o += binom(h, k) * off13[min(d - k, TB) + 1];
        meta[t] = (int)o;
    }
    __syncthreads();
    const int total = meta[32 + kmax + 1];
    for (int p = t; p < total; p += TT) {
        int k;
        const uint32_t loc = sb_unrank(*sb, (uint32_t)p, hc, &k);
        uint32_t rk = 0, hh = H;
        int q = 0, idx = 1;
        while (hh) {
            const int b = __ffs(hh) - 1;
            hh &= hh - 1;
            if (loc >> q & 1u) rk += sb_binom(*sb, b, idx++);
            ++q;
        }
        rowbase[p] = (uint32_t)meta[k] + rk * off13[min(d - k, TB) + 1];
    }
    __syncthreads();

    // --- per-column log-sum over the admissible rows, in a fixed order ------
    // Column c (low pattern of size j) takes the rows of size at most d - j,
    // i.e. the list prefix before the first row of size d - j + 1; a row of
    // size k holds the first W_k = off13[d - k + 1] columns.
    // Long columns (at most d - 2 low elements, many rows): warp w takes the
    // rows w, w + 8, ... and its lanes the columns of a 96-column block
    // (coalesced reads along the row); the eight warp partials are combined
    // in warp order.
    const uint32_t nlong = d >= 2 ? off13[min(d - 2, TB) + 1] : 0u;
    for (uint32_t cb = 0; cb < nlong; cb += 96) {
        T m[3], sm[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) { m[q] = Lg::ninf(); sm[q] = T(0); }
        // rows of size k hold W_k columns; only sizes with W_k > cb reach this block
        int kb = 0;
        while (kb < kmax && off13[min(d - kb - 1, TB) + 1] > cb) ++kb;
        const int pend = meta[32 + kb + 1];
        int k = 0;
        for (int p0 = warp; p0 < pend; p0 += 4 * (TT / 32)) {
            T x[4][3];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = p0 + u * (TT / 32);
                while (k < kb && p >= meta[32 + k + 1]) ++k;
                const uint32_t W = p < pend ? min(nlong, off13[min(d - k, TB) + 1]) : 0u;
                const T* src = tb + (p < pend ? rowbase[p] : 0u);
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const uint32_t c = cb + lane + 32 * q;
                    x[u][q] = c < W ? src[c] : Lg::ninf();
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < 3; ++q) lse_online(m[q], sm[q], x[u][q]);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            part[(warp * 96 + lane + 32 * q) * 2] = m[q];
            part[(warp * 96 + lane + 32 * q) * 2 + 1] = sm[q];
        }
        __syncthreads();
        if (t < 96 && cb + t < nlong) {
            T mx = Lg::ninf(), s2 = T(0);
#pragma unroll
            for (int w = 0; w < TT / 32; ++w) {
                const T mw = part[(w * 96 + t) * 2], sw = part[(w * 96 + t) * 2 + 1];
                const T mn = mw > mx ? mw : mx;
                if (mn != Lg::ninf()) {
                    s2 = s2 * Lg::ex(mx - mn) + sw * Lg::ex(mw - mn);
                    mx = mn;
                }
            }
            out[cb + t] = mx + Lg::lg(s2);
        }
        __syncthreads();
    }
    // Columns with d - 1 low elements: the row of the empty set and the
    // 1-element rows, 1 + hc of them; a thread per column.
    const uint32_t ncopy = off13[min(d, TB + 1)];     // first column with d low elements
    const int rmid = meta[32 + 2];
    for (uint32_t c = nlong + t; c < ncopy; c += TT) {
        T mx = Lg::ninf(), sm = T(0);
#pragma unroll 8
        for (int rp = 0; rp < rmid; ++rp) lse_online(mx, sm, tb[rowbase[rp] + c]);
        out[c] = mx + Lg::lg(sm);
    }
    // Columns with d low elements take the row of the empty set alone (offset 0).
    for (uint32_t c = ncopy + t; c < ncol; c += TT) out[c] = tb[c];
}

// Column sums by butterflies over the h high dimensions.  Blocks below
// nodes * ceil(ncb / CPB) take one node i and a run of CPB consecutive low
// columns c < ncb: the 2^h values B_i(G_H + G_L) of each column (zero where
// |G_H| > d - |G_L|) are gathered from the reordered table, the upward zeta
// over the subsets of every H follows in shared memory (h * 2^(h-1) steps
// per column, against sum_H C(|H|, <= d - |G_L|) terms summed directly: the
// better order once a column has many rows), and each C_H(G_L) goes to slot
// c of tile (i, H), the CPB columns of a run side by side.  The steps run
// three dimensions at a time in registers (eight values per thread), the
// columns held one after another in shared memory.
//
// Every output of a column lies between its H = {} value f(G_L) and its
// largest input plus log 2^h, so when that span is under one single-scale
// window (Window), the column's sums run in linear scale (an exponential per
// input, an addition per step, a logarithm per output; exact as in the
// tiles); otherwise every step is a log-sum-exp.
// The blocks after those copy the columns from ncb on, whose sums have a
// single row (the empty high set), a warp per tile.
//
// Value e = (column << hl) | H sits at colb_pos(e): bits 5..7 of e go into
// the bank bits so that the steps over dims 0..2 (lanes differ in bits 3..7),
// 3..5 (bits 0..2, 6, 7) and above (bits 0..4) have no bank conflict (8 and 4
// lanes per bank without it; 64 bits: bits 4..6, over the 16 bank pairs of
// half a warp), and the column goes there too: rows are read and outputs
// written by lanes with the column fastest, 32 / CPB rows a request.  The map
// is linear over XOR, so a thread finds its eight places with seven XORs.
// A thread per row, 4 to 8 scattered columns each, was bound by its requests
// of 32 sectors.  FP32 sums, us before -> after (the swizzle alone): n = 26
// d = 4 305 -> 213 (264), n = 25 d = 6 1257 -> 612 (1126), d = 8 2945 -> 1353
// (2627).  512 threads measured 573 and 1288 at d = 6 and 8, but 19 against 14
// at n = 20 and 91 against 63 in FP64 at n = 23.
constexpr int kColbThreads = 256;

template <int BYTES, int CPB>
__device__ __forceinline__ uint32_t colb_pos(uint32_t e, int hl)
{
    constexpr int lanes = BYTES == 4 ? 32 : 16;
    const uint32_t p = e ^ ((e >> hl) * (lanes / CPB));
    if constexpr (BYTES == 4) return p ^ ((e >> 5) & 7u) ^ (((e >> 6) & 3u) << 3);
    else return p ^ ((e >> 4) & 7u) ^ (((e >> 6) & 1u) << 3);
}

// The upward zeta of CPB columns of 2^h values each, three dimensions at a
// time; `first` maps a value as it is first read, `op` adds two (column last).
template <int CPB, typename T, typename FIRST, typename OP>
__device__ __forceinline__ void colb_steps(T* v, int h, FIRST first, OP op)
{
    for (int j0 = 0; j0 < h; j0 += 3) {
        const int nb = min(3, h - j0);
        const uint32_t lowm = (1u << j0) - 1u;
        const uint32_t groups = (uint32_t)CPB << (h - nb);
        const uint32_t s1 = colb_pos<sizeof(T), CPB>(1u << j0, h), s2 = colb_pos<sizeof(T), CPB>(2u << j0, h),
                       s4 = colb_pos<sizeof(T), CPB>(4u << j0, h);
        for (uint32_t g = threadIdx.x; g < groups; g += blockDim.x) {
            const uint32_t cc = g >> (h - nb);
            const uint32_t base = colb_pos<sizeof(T), CPB>(((g & ~lowm) << nb) | (g & lowm), h);
            T x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < (1 << nb)) x[q] = v[base ^ (q & 1 ? s1 : 0u) ^ (q & 2 ? s2 : 0u) ^ (q & 4 ? s4 : 0u)];
            if (j0 == 0) {
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < (1 << nb)) x[q] = first(x[q], cc);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                if (k >= nb) continue;
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < (1 << nb) && (q >> k & 1)) x[q] = op(x[q], x[q ^ (1 << k)], cc);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < (1 << nb)) v[base ^ (q & 1 ? s1 : 0u) ^ (q & 2 ? s2 : 0u) ^ (q & 4 ? s4 : 0u)] = x[q];
        }
        __syncthreads();
    }
}

// The chunks of a column (hc > 0): a cluster's 2^hc blocks hold one chunk of
// the top hc high bits each; the steps over those bits read the peers' values
// for the same low bits H, in the butterflies' order (so the sums equal the
// unchunked ones bit for bit).
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
template <typename T> __device__ __forceinline__ T peer_ld(const T* p, uint32_t rank)
{
    const uint32_t own = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t at;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(own), "r"(rank));
    if constexpr (sizeof(T) == 4) {
        uint32_t u;
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(u) : "r"(at));
        return __builtin_bit_cast(T, u);
    } else {
        unsigned long long u;
        asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(u) : "r"(at));
        return __builtin_bit_cast(T, u);
    }
}
template <typename T, typename OP>
__device__ __forceinline__ T chunk_sum(const T* p, uint32_t chunk, uint32_t cc, OP op)
{
    T x[8];
#pragma unroll
    for (uint32_t q = 0; q < 8; ++q)
        if ((q & ~chunk) == 0) x[q] = peer_ld(p, q);
#pragma unroll
    for (uint32_t b = 0; b < 3; ++b) {
        if (!(chunk >> b & 1)) continue;
#pragma unroll
        for (uint32_t q = 0; q < 8; ++q)
            if ((q >> b & 1) && (q & ~chunk) == 0) x[q] = op(x[q], x[q ^ (1u << b)], cc);
    }
    T y = x[0];
#pragma unroll
    for (uint32_t q = 1; q < 8; ++q)
        if (q == chunk) y = x[q];
    return y;
}

template <typename T, int CPB>
__global__ void __launch_bounds__(kColbThreads)
k_upzeta13_colb(int n, int d, int64_t K, const T* __restrict__ tab, T* __restrict__ A,
                size_t js, int nodes, uint32_t ncb, int hc)
{
    tab = job_ptr(tab, js);
    A = job_ptr(A, js);
    using Lg = LogOps<T>;
    using Wn = Window<T>;
    __shared__ SBinom sb;
    __shared__ uint32_t off13[16];
    __shared__ uint32_t rowoff_k[32];
    __shared__ T wred[kColbThreads / 32][CPB];                       // the warps' column maxima
    __shared__ T cmax_s[CPB], f0_s[CPB];             // a column's largest and H = {} value
    __shared__ T scale_s[CPB];                       // a column's linear scale
    __shared__ int lin_s[CPB], all_lin;              // columns within one window
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* v = reinterpret_cast<T*>(smem_raw);           // [column of the run][H]
    const int h = n - 1 - TB;
    // hc > 0: the top hc high bits are this block's chunk, fixed, and the
    // block's rank in its cluster
    const int hl = h - hc;
    const uint32_t H2 = 1u << hl;
    const uint32_t ncol = num_small_subsets(TB, d);
    const uint32_t nrun = (ncb + CPB - 1) / CPB;
    const uint32_t nbb = ((uint32_t)nodes * nrun) << hc;
    const size_t asize = (size_t)nodes << (n - 1);
    if (blockIdx.x >= nbb) {                         // copies: a warp per tile
        const uint32_t tile = (blockIdx.x - nbb) * (blockDim.x >> 5) + (threadIdx.x >> 5);
        if (tile >= ((uint32_t)nodes << h)) return;
        const T* tb = tab + (size_t)(tile >> h) * K;
        T* out = A + BN_AT((size_t)tile << TB, TN, asize);
        for (uint32_t c = ncb + (threadIdx.x & 31); c < ncol; c += 32) out[c] = tb[BN_AT(c, 1, K)];
        return;
    }
    fill_sbinom(sb);
    if (threadIdx.x < 16) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= TB; ++k) o += binom(TB, k);
        off13[threadIdx.x] = o;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= min(d, h); ++k)
            o += binom(h, k) * off13[min(d - k, TB) + 1];
        rowoff_k[threadIdx.x] = o;
    }
    __syncthreads();
    const uint32_t chunk = blockIdx.x & ((1u << hc) - 1u);
    const int i = (int)((blockIdx.x >> hc) / nrun);
    const uint32_t c0 = ((blockIdx.x >> hc) % nrun) * CPB;
    const uint32_t Hc = chunk << hl;                 // the chunk's high bits
    const T* tb = tab + (size_t)i * K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t cc = lane & (CPB - 1), c = c0 + cc;   // this lane's column
    int kl = 0;                                      // its low elements (-1: none)
    while (kl < TB && off13[kl + 1] <= c) ++kl;
    if (c >= ncb) kl = -1;
    const int kl0 = __shfl_sync(FULLMASK, kl, 0);
    T mx = Lg::ninf();
    for (uint32_t Hb = warp * 32; Hb < H2; Hb += blockDim.x) {
        const uint32_t Hf = Hc | Hb | lane;
        const int kh = __popc(Hf);
        uint32_t row = 0;                            // the row of G_H in the node's table
        if (kh <= d - kl0) {                         // some column reads it
            int t = 1;                               // colex rank of Hf among kh-subsets
            for (uint32_t x = Hf; x; x &= x - 1, ++t) row += sb_binom(sb, __ffs(x) - 1, t);
            row = rowoff_k[kh] + row * off13[min(d - kh, TB) + 1];
        }
#pragma unroll
        for (int j = 0; j < CPB; ++j) {
            const uint32_t src = j * (32 / CPB) + lane / CPB, H = Hb | src;
            const uint32_t rj = __shfl_sync(FULLMASK, row, src);
            const bool in = kl >= 0 && __popc(Hc | H) <= d - kl;
            const T val = in ? tb[BN_AT(rj + c, 1, K)] : Lg::ninf();
            v[colb_pos<sizeof(T), CPB>((cc << hl) | H, hl)] = val;
            mx = val > mx ? val : mx;
        }
    }
    for (int o = 16; o >= CPB; o >>= 1) {
        const T y = __shfl_xor_sync(FULLMASK, mx, o);
        mx = y > mx ? y : mx;
    }
    if (lane < CPB) wred[warp][lane] = mx;
    __syncthreads();
    if (threadIdx.x < CPB) {
        T m = wred[0][threadIdx.x];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = wred[w][threadIdx.x] > m ? wred[w][threadIdx.x] : m;
        cmax_s[threadIdx.x] = m;
        f0_s[threadIdx.x] = v[colb_pos<sizeof(T), CPB>(threadIdx.x << hl, hl)];
    }
    if (hc) cluster_sync();
    else __syncthreads();
    if (threadIdx.x == 0) {
        // a column's outputs lie in [f(G_L), its largest input + log 2^h]
        const T hb = sizeof(T) == 4 ? T(h) : T(h) * T(0.69314718055994530942);
        int all = 1;
        for (uint32_t q = 0; q < CPB; ++q) {
            T m = cmax_s[q], f = f0_s[q];
            if (hc) {
                f = peer_ld(f0_s + q, 0);
                for (uint32_t p = 0; p < (1u << hc); ++p) {
                    const T x = peer_ld(cmax_s + q, p);
                    m = x > m ? x : m;
                }
            }
            const T top = m + hb;
            scale_s[q] = top - Wn::top;
            lin_s[q] = c0 + q >= ncb || top - f < Wn::win;
            all &= lin_s[q];
        }
        all_lin = all;
    }
    __syncthreads();
    if (all_lin)
        colb_steps<CPB>(v, hl, [&](T x, uint32_t cc) { return Lg::ex(x - scale_s[cc]); },
                   [](T a, T b, uint32_t) { return a + b; });
    else
        colb_steps<CPB>(v, hl, [&](T x, uint32_t cc) { return lin_s[cc] ? Lg::ex(x - scale_s[cc]) : x; },
                   [&](T a, T b, uint32_t cc) { return lin_s[cc] ? a + b : Lg::lse(a, b); });
    if (hc) cluster_sync();                          // the peers' steps are done
    T* Ai = A + ((size_t)i << (n - 1));
    if (c < ncb) {
        for (uint32_t H = warp * (32 / CPB) + lane / CPB; H < H2; H += (32 / CPB) * (blockDim.x >> 5)) {
            const T* at = v + colb_pos<sizeof(T), CPB>((cc << hl) | H, hl);
            const T x = hc ? chunk_sum(at, chunk, cc, [&](T a, T b, uint32_t q) { return lin_s[q] ? a + b : Lg::lse(a, b); })
                           : *at;
            Ai[BN_AT(((size_t)(Hc | H) << TB) + c, 1, (size_t)1 << (n - 1))] = lin_s[cc] ? scale_s[cc] + Lg::lg(x) : x;
        }
    }
    if (hc) cluster_sync();                          // no peer reads this block's values any more
}

// Part 1 with one warp per tile: each warp enumerates its tile's rows into
// its own list and sums the columns lane by lane (consecutive columns:
// coalesced reads of a row); no block barrier after the tables are filled.
// Columns with d low elements are copies, those with d - 1 take the 1 + |H|
// rows of at most one high element, the others every row of size at most
// d - |G_L|.
template <typename T>
__global__ void __launch_bounds__(256)
k_upzeta13_colw(int n, int d, int64_t K, const T* __restrict__ tab, T* __restrict__ A, size_t js,
                int nodes)
{
    tab = job_ptr(tab, js);
    A = job_ptr(A, js);
    __shared__ SBinom sb;
    __shared__ uint32_t off13[16];
    __shared__ uint32_t rowoff_k[32];            // offset of the first size-k row in a node's table
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int h = n - 1 - TB;
    const uint32_t nrow = num_small_subsets(h, d);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* rowbase = reinterpret_cast<uint32_t*>(smem_raw) + (size_t)warp * nrow;
    fill_sbinom(sb);
    if (threadIdx.x < 16) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= TB; ++k) o += binom(TB, k);
        off13[threadIdx.x] = o;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= min(d, h); ++k)
            o += binom(h, k) * off13[min(d - k, TB) + 1];
        rowoff_k[threadIdx.x] = o;
    }
    __syncthreads();
    const uint32_t ncol = num_small_subsets(TB, d);
    const uint32_t nlong = d >= 2 ? off13[min(d - 2, TB) + 1] : 0u;
    const uint32_t ncopy = off13[min(d, TB + 1)];
    const uint32_t ntiles = (uint32_t)nodes << h;
    const uint32_t wpb = blockDim.x >> 5;
    for (uint32_t tile = blockIdx.x * wpb + warp; tile < ntiles; tile += gridDim.x * wpb) {
        const int i = (int)(tile >> h);
        const uint32_t H = tile & ((1u << h) - 1u);
        const T* tb = tab + (size_t)i * K;
        T* out = A + BN_AT(((size_t)i << (n - 1)) + ((size_t)H << TB), TN, (size_t)nodes << (n - 1));
        const int hc = __popc(H);
        uint32_t total = 0;                      // rows of size <= d inside H
        for (int k = 0; k <= d && k <= hc; ++k) total += sb_binom(sb, hc, k);
        for (uint32_t p = lane; p < total; p += 32) {
            int k;
            const uint32_t loc = sb_unrank(sb, p, hc, &k);
            uint32_t rk = 0, hh = H;
            int q = 0, idx = 1;
            while (hh) {
                const int b = __ffs(hh) - 1;
                hh &= hh - 1;
                if (loc >> q & 1u) rk += sb_binom(sb, b, idx++);
                ++q;
            }
            rowbase[p] = rowoff_k[k] + rk * off13[min(d - k, TB) + 1];
        }
        __syncwarp();
        for (uint32_t c = lane; c < nlong; c += 32) {          // at most d - 2 low elements
            int j = 0;
            while (off13[j + 1] <= c) ++j;
            uint32_t rend = 0;
            for (int k = 0; k <= d - j && k <= hc; ++k) rend += sb_binom(sb, hc, k);
            LazySum<T> s;
#pragma unroll 4
            for (uint32_t rp = 0; rp < rend; ++rp) s.add(tb[BN_AT(rowbase[rp] + c, 1, K)]);
            out[c] = s.value();
        }
        const uint32_t rmid = 1u + (uint32_t)hc;               // d - 1 low elements
        for (uint32_t c = nlong + lane; c < ncopy; c += 32) {
            LazySum<T> s;
#pragma unroll 4
            for (uint32_t rp = 0; rp < rmid; ++rp) s.add(tb[BN_AT(rowbase[rp] + c, 1, K)]);
            out[c] = s.value();
        }
        for (uint32_t c = ncopy + lane; c < ncol; c += 32) out[c] = tb[c];   // d low elements
        __syncwarp();                                          // rowbase is reused
    }
}

// ===========================================================================
// Step 2 for n >= 14, part 2: one block per tile (i, H) of A_i.  The column
// sums of part 1 are placed at their low patterns (every other slot holds
// zero) and the truncated upward zeta over the 13 low bits follows.
// ===========================================================================
//
// TLO: the rows of A in tile-level order (see bn_device.cuh): output element
// e of the tile goes to row place(e >> lw) of the tile's block.
template <typename T, bool TLO>
__global__ void __launch_bounds__(TT, sizeof(T) == 4 ? 2 : 1)
k_upzeta13(int n, int d, const uint16_t* __restrict__ unrank13, T* __restrict__ A, size_t js)
{
    unrank13 = job_ptr(unrank13, js);
    A = job_ptr(A, js);
    using Lg = LogOps<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* A0 = reinterpret_cast<T*>(smem_raw);
    T* A1 = A0 + TN;
    T* wmax = A1 + TN;                           // each warp's largest column sum
    const uint32_t ncol = num_small_subsets(TB, d);
    const int h = n - 1 - TB;
    const int t = threadIdx.x, lane = t & 31;
    const int i = (int)(blockIdx.x >> h);
    const uint32_t H = blockIdx.x & ((1u << h) - 1u);
    T* out = A + BN_AT(((size_t)i << (n - 1)) + ((size_t)H << TB), TN, (size_t)gridDim.x << TB);
    // place of element e in the tile's block
    const int lw = i < 4 ? 3 : 4;                // row width of A_i in step 3
    const uint32_t lmask = (1u << lw) - 1u;
    auto opos = [&](uint32_t e) -> uint32_t {
        if (!TLO) return e;
        const uint32_t r = e >> lw;
        return ((lw == 4 ? g_place.p9[r] : g_place.p10[r]) << lw) | (e & lmask);
    };

    // |el1(r, t)| = |r| + |t| (disjoint bits): the slots with more than d
    // elements are no column (no input)
    const int pt = __popc(t);
    T tm = Lg::ninf();
    for (uint32_t c = t; c < ncol; c += TT) {
        const T v = out[c];
        const uint32_t sw = swz(BN_AT(unrank13[c], 1, TN));
        A0[sw] = A1[sw] = v;
        tm = v > tm ? v : tm;
    }
    for (int o = 16; o; o >>= 1) {
        const T o2 = __shfl_xor_sync(FULLMASK, tm, o);
        tm = o2 > tm ? o2 : tm;
    }
    if (lane == 0) wmax[t >> 5] = tm;
    __syncthreads();                             // columns placed, warp maxima written
    T tmx = wmax[0];
#pragma unroll
    for (int w = 1; w < TT / 32; ++w) tmx = wmax[w] > tmx ? wmax[w] : tmx;

    // --- single-scale passes (Window): pass p sums linear values 2^(x - s_p)
    //     (e^(x - s_p) in FP64) with s_p = M - top - p * win and writes the
    //     outputs it resolves; the last pass writes every output left.  Every
    //     output is at least C(empty) and at most M, so ceil((M - C(empty)) /
    //     win) passes resolve the tile.  Tiles that need more than
    //     Window::max_pass passes take the banded path below.
    {
        using Wn = Window<T>;
        const T M = tmx + T(TB);
        const T span = M - A1[0];
        // spans past max_pass windows (a zero weight held as -1e7 nats gives an
        // empty-set column far below the rest) and NaN go to the exact path
        // without converting the span to an integer
        const int npass = span < Wn::win ? 1
                          : span < T(Wn::max_pass) * Wn::win ? (int)ceil(span / Wn::win)
                                                             : Wn::max_pass + 1;
        if (npass == 1) {                        // one window holds the whole tile
            const T sp = M - Wn::top;
            T x[TR];
            ld1(A1, x, t);
#pragma unroll
            for (int r = 0; r < TR; ++r)
                x[r] = (__popc(r) + pt <= d) ? Lg::ex(x[r] - sp) : T(0);
            bfly_plain<true>(x, 0, 5);
            st1(A0, x, t);
            __syncthreads();
            ld2(A0, x, t);
            bfly_plain<true>(x, 0, 5);
            st2(A0, x, t);
            __syncthreads();
            ld3(A0, x, t);
            bfly_plain<true>(x, 0, 3);
#pragma unroll
            for (int r = 0; r < TR; ++r) x[r] = sp + Lg::lg(x[r]);
            if constexpr (TLO) {
                // a run of 8 consecutive elements stays inside one row (lw >= 3)
#pragma unroll
                for (int q = 0; q < TR / 8; ++q) {
                    float4* p = reinterpret_cast<float4*>(out + BN_AT(opos(el3(8 * q, t)), 8, TN));
                    p[0] = make_float4(x[8 * q], x[8 * q + 1], x[8 * q + 2], x[8 * q + 3]);
                    p[1] = make_float4(x[8 * q + 4], x[8 * q + 5], x[8 * q + 6], x[8 * q + 7]);
                }
            } else {
                st_out3(out, x, t);
            }
            return;
        }
        if (npass <= Wn::max_pass) {
            uint32_t done = 0u;                  // bit r: output el3(r, t) written
            // registers 8q..8q+7 (layout 3) are 8 consecutive elements of one
            // row: their places start at run3[q]
            uint32_t run3[TR / 8];
#pragma unroll
            for (int q = 0; q < TR / 8; ++q) run3[q] = BN_AT(opos(el3(8 * q, t)), 8, TN);
            T sp = M - Wn::top;
            for (int p = 0; p < npass; ++p, sp -= Wn::win) {
                const bool last = p + 1 == npass;
                T x[TR];
                ld1(A1, x, t);
#pragma unroll
                for (int r = 0; r < TR; ++r)
                    x[r] = (__popc(r) + pt <= d) ? Lg::ex(x[r] - sp) : T(0);
                bfly_plain<true>(x, 0, 5);
                st1(A0, x, t);
                __syncthreads();
                ld2(A0, x, t);
                bfly_plain<true>(x, 0, 5);
                st2(A0, x, t);
                __syncthreads();
                ld3(A0, x, t);
                bfly_plain<true>(x, 0, 3);
#pragma unroll
                for (int r = 0; r < TR; ++r) {
                    const T lx = Lg::lg(x[r]);
                    if (!(done >> r & 1u) && (last || lx >= Wn::lo)) {
                        out[run3[r >> 3] + (r & 7)] = sp + lx;
                        done |= 1u << r;
                    }
                }
                if (last) break;
                if (__syncthreads_and(done == 0xffffffffu)) break;   // also guards A0 reuse
            }
            return;
        }
    }

    // --- max-plus pass: layouts 1, 2, 3 ------------------------------------
#pragma unroll
    for (int r = 0; r < TR; ++r)                 // no term: zero (slots that are no column)
        if (__popc(r) + pt > d) A0[swz(el1(r, t))] = Lg::ninf();
    __syncthreads();
    T v[TR];
    ld1(A0, v, t);
    bfly_max<true>(v, 0, 5);
    st1(A0, v, t);
    __syncthreads();
    ld2(A0, v, t);
    bfly_max<true>(v, 0, 5);
    st2(A0, v, t);
    __syncthreads();
    ld3(A0, v, t);
    bfly_max<true>(v, 0, 3);

    // --- exact sum pass: layouts 3, 2, 1 ------------------------------------
    T sc[TR];
    sum_pass<true>(v, sc, A1, A0, t, d);
#pragma unroll
    for (int r = 0; r < TR; ++r) out[BN_AT(opos(el1(r, t)), 1, TN)] = scaled_log(v[r], sc[r]);
}

// The same tiles (FP32) in a persistent kernel: each block takes tiles
// blockIdx.x, blockIdx.x + gridDim.x, ...  Thread 0 keeps the next tile's
// column sums in flight while the block transforms the current one (one bulk
// copy into shared memory, counted by an mbarrier), and every finished tile
// leaves as one 32 KB bulk store from shared memory, so the block's threads
// issue neither the loads nor the stores.  The arithmetic and the outputs are
// those of k_upzeta13, bit for bit.  Shared memory: two blocks of 32 KB, the
// warps' maxima, the mbarrier and a flag, and the staged column sums (ncol
// floats rounded up to 16 bytes, and 48 bytes more).  The word after the flag
// keeps the tile's smallest output until the next tile's first barrier.
//
// What bounds it: 27 instructions an output at 16 warps per SM waited at the
// barriers (47 % issue with a block each for inputs, exchanges and outputs: two
// blocks per SM, one at d = 8).  A one-window tile now stays in one 32 KB
// block from its inputs to its outputs (a thread exchanges into the places it
// read) while the last tile's store leaves the other; of two windows the first
// exchanges in the other block, where the outputs then gather.  Three blocks
// per SM where kUp13ThreeM says so, two to d = 8.  Tiles, us, before -> now:
// n = 23, m = 500 146 -> 137, n = 29 11480 -> 10690, n = 25 d = 8 (one block
// per SM before) 1250 -> 865, n = 26, m = 2000 2264 -> 2222.
//
// With ncb < ncol the columns from ncb on (d low
// elements: the sum of one row, the empty high set) were not written by the
// column-sum kernel; they are the first ncol entries of node i's reordered
// score table `tab` (K entries per node, K a multiple of 4), and a second
// bulk copy stages them, from the 16-byte boundary at or below ncb.  A bulk
// copy that has not landed after `cap` polls of its mbarrier sets
// kErrDeviceTimeout in *err and the block returns after one more bounded
// wait for it.  `hold` (a test hook, 0 otherwise) withholds the block's
// first copies, so that its wait runs out.
template <bool TLO, int NB>
__global__ void __launch_bounds__(TT, NB)
k_upzeta13p(int n, int d, const uint16_t* __restrict__ unrank13, float* __restrict__ A, uint32_t ntiles,
            int* __restrict__ err, uint32_t cap, int hold, const float* __restrict__ tab, int64_t K,
            uint32_t ncb)
{
    using Lg = LogOps<float>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* const AA = reinterpret_cast<float*>(smem_raw);  // the two blocks
    float* wmax = AA + 2 * TN;                           // TT / 32 floats
    uint64_t* bar = reinterpret_cast<uint64_t*>(wmax + TT / 32);
    int* gave_up = reinterpret_cast<int*>(bar + 1);
    float* lowest = reinterpret_cast<float*>(gave_up + 1);   // the tile's smallest output
    float* S = reinterpret_cast<float*>(bar + 2);       // staged column sums
    const uint32_t ncol = num_small_subsets(TB, d);
    const int h = n - 1 - TB;
    const size_t asize = (size_t)ntiles << TB;
    // the tile's columns (before ncb) and, from the table, the rest
    const uint32_t ncb4 = ncb & ~3u;
    const uint32_t sbytes = (ncb * 4u + 15u) & ~15u;
    const uint32_t tbytes = ncb < ncol ? ((ncol - ncb4) * 4u + 15u) & ~15u : 0u;
    const int t = threadIdx.x, lane = t & 31;
    const int pt = __popc(t);
    // thread 0: the copies of tile `tl` on the barrier
    auto stage = [&](uint32_t tl) {
        mbar_expect(bar, sbytes + tbytes);
        bulk_copy_in(S, A + BN_AT((size_t)tl << TB, TN, asize), sbytes, bar);
        if (tbytes)
            bulk_copy_in(S + sbytes / 4, tab + BN_AT((size_t)(tl >> h) * K + ncb4, 4, (size_t)(ntiles >> h) * K), tbytes, bar);
    };
    if (t == 0) mbar_init(bar, 1);
    __syncthreads();
    uint32_t tile = blockIdx.x;
    if (t == 0 && tile < ntiles && !hold) stage(tile);
    uint32_t side = 0;                                   // the block the next tile's inputs go to
    for (uint32_t parity = 0; tile < ntiles; tile += gridDim.x, parity ^= 1u) {
        float* const A1 = AA + side * TN;                // inputs
        float* const A0 = AA + (side ^ 1u) * TN;         // the last tile's outputs, if one-window
        const int i = (int)(tile >> h);
        float* out = A + BN_AT((size_t)tile << TB, TN, asize);
        const int lw = i < 4 ? 3 : 4;
        const uint32_t lmask = (1u << lw) - 1u;
        auto opos = [&](uint32_t e) -> uint32_t {
            if (!TLO) return e;
            const uint32_t r = e >> lw;
            return ((lw == 4 ? g_place.p9[r] : g_place.p10[r]) << lw) | (e & lmask);
        };
        if (t == 0) {
            bulk_wait_read_but1();                       // the store before the last has read A1
            *gave_up = mbar_wait_bounded(bar, parity, cap) ? 0 : 1;
        }
        __syncthreads();
        if (*gave_up) {
            if (t == 0) {
                atomicOr(err, kErrDeviceTimeout);
                mbar_wait_bounded(bar, parity, cap);     // let a copy in flight land
                bulk_wait();
            }
            return;
        }
        // |el1(r, t)| = |r| + |t| (disjoint bits): the slots with more than d
        // elements are no column (no input)
        float tm = Lg::ninf();
        for (uint32_t c = t; c < ncol; c += TT) {
            const float v = c < ncb ? S[c] : S[sbytes / 4 + c - ncb4];
            A1[swz(BN_AT(unrank13[c], 1, TN))] = v;
            tm = v > tm ? v : tm;
        }
        for (int o = 16; o; o >>= 1) {
            const float o2 = __shfl_xor_sync(FULLMASK, tm, o);
            tm = o2 > tm ? o2 : tm;
        }
        if (lane == 0) wmax[t >> 5] = tm;
        // C(empty), in a word of its own: its place in A1 is thread 0's first
        // exchange below, before slower warps have read it
        if (t == 0) *lowest = S[0];
        fence_async_shared();                            // S is read: the next copy may land
        __syncthreads();
        if (t == 0 && tile + gridDim.x < ntiles) stage(tile + gridDim.x);
        float tmx = wmax[0];
#pragma unroll
        for (int w = 1; w < TT / 32; ++w) tmx = wmax[w] > tmx ? wmax[w] : tmx;

        // single-scale passes as in k_upzeta13
        using Wn = Window<float>;
        const float M = tmx + float(TB);
        const float span = M - *lowest;
        const int npass = span < Wn::win ? 1
                          : span < float(Wn::max_pass) * Wn::win ? (int)ceilf(span / Wn::win)
                                                                 : Wn::max_pass + 1;
        // outputs 8q .. 8q + 7 (a run stays inside one row: lw >= 3); half the
        // threads store the upper half first (bank conflicts)
        const int flip = (t >> 2) & 1;
        auto put8 = [&](float4* o, const float (&x)[TR], int q) {
            const float4 lo = make_float4(x[8 * q], x[8 * q + 1], x[8 * q + 2], x[8 * q + 3]);
            const float4 hi = make_float4(x[8 * q + 4], x[8 * q + 5], x[8 * q + 6], x[8 * q + 7]);
            o[flip] = flip ? hi : lo;
            o[!flip] = flip ? lo : hi;
        };
        float* out_s = A0;                               // where the finished tile lies
        if (npass == 1) {
            const float sp = M - Wn::top;
            float x[TR];
            ld1(A1, x, t);
#pragma unroll
            for (int r = 0; r < TR; ++r) x[r] = (__popc(r) + pt <= d) ? Lg::ex(x[r] - sp) : 0.0f;
            bfly_plain<true>(x, 0, 5);
            st1(A1, x, t);
            __syncthreads();
            ld2(A1, x, t);
            bfly_plain<true>(x, 0, 5);
            st2(A1, x, t);
            __syncthreads();
            ld3(A1, x, t);
            bfly_plain<true>(x, 0, 3);
#pragma unroll
            for (int r = 0; r < TR; ++r) x[r] = sp + Lg::lg(x[r]);
            out_s = A1;
            side ^= 1u;
            __syncthreads();                             // A1 is read: the outputs may land
#pragma unroll
            for (int q = 0; q < TR / 8; ++q)
                put8(reinterpret_cast<float4*>(A1 + BN_AT(opos(el3(8 * q, t)), 8, TN)), x, q);
        } else if (npass <= Wn::max_pass) {
            // the first window exchanges in A0 and keeps the inputs, the
            // second in A1; the outputs gather in A0
            static_assert(Wn::max_pass == 2, "two windows");
            uint32_t done = 0u;                          // bit r: output el3(r, t) written
            uint32_t run3[TR / 8];
#pragma unroll
            for (int q = 0; q < TR / 8; ++q) run3[q] = BN_AT(opos(el3(8 * q, t)), 8, TN);
            if (t == 0) bulk_wait_read();                // A0 is free
            __syncthreads();
            float sp = M - Wn::top;
            for (int p = 0; p < 2; ++p, sp -= Wn::win) {
                float* const E = p ? A1 : A0;
                float x[TR];
                ld1(A1, x, t);
#pragma unroll
                for (int r = 0; r < TR; ++r) x[r] = (__popc(r) + pt <= d) ? Lg::ex(x[r] - sp) : 0.0f;
                bfly_plain<true>(x, 0, 5);
                st1(E, x, t);
                __syncthreads();
                ld2(E, x, t);
                bfly_plain<true>(x, 0, 5);
                st2(E, x, t);
                __syncthreads();
                ld3(E, x, t);
                bfly_plain<true>(x, 0, 3);
                int all = 1;
                if (p == 0) {
#pragma unroll
                    for (int r = 0; r < TR; ++r) {
                        x[r] = Lg::lg(x[r]);
                        done |= (uint32_t)(x[r] >= Wn::lo) << r;
                    }
#pragma unroll
                    for (int r = 0; r < TR; ++r) x[r] += sp;
                    all = __syncthreads_and(done == 0xffffffffu);    // A0 is read
                } else {
#pragma unroll
                    for (int r = 0; r < TR; ++r) x[r] = sp + Lg::lg(x[r]);
                }
                // 8 consecutive outputs as two 16-byte stores, the upper first in
                // half the threads (bank conflicts); the second window keeps the
                // outputs of the first
#pragma unroll
                for (int q = 0; q < TR / 8; ++q) {
                    float4* o = reinterpret_cast<float4*>(A0 + run3[q]);
                    if (p) {
                        const float4 a = o[flip], b = o[!flip];
                        const float4 lo = flip ? b : a, hi = flip ? a : b;
                        const uint32_t dq = done >> (8 * q);
                        if (dq & 1u) x[8 * q] = lo.x;
                        if (dq & 2u) x[8 * q + 1] = lo.y;
                        if (dq & 4u) x[8 * q + 2] = lo.z;
                        if (dq & 8u) x[8 * q + 3] = lo.w;
                        if (dq & 16u) x[8 * q + 4] = hi.x;
                        if (dq & 32u) x[8 * q + 5] = hi.y;
                        if (dq & 64u) x[8 * q + 6] = hi.z;
                        if (dq & 128u) x[8 * q + 7] = hi.w;
                    }
                    put8(o, x, q);
                }
                if (all) break;
            }
        } else {
            if (t == 0) bulk_wait_read();                // A0 is free
            __syncthreads();
            // max-plus pass, then the exact sum pass (k_upzeta13)
#pragma unroll
            for (int r = 0; r < TR; ++r) {
                const uint32_t sw = swz(el1(r, t));
                A0[sw] = __popc(r) + pt > d ? Lg::ninf() : A1[sw];
            }
            __syncthreads();
            float v[TR];
            ld1(A0, v, t);
            bfly_max<true>(v, 0, 5);
            st1(A0, v, t);
            __syncthreads();
            ld2(A0, v, t);
            bfly_max<true>(v, 0, 5);
            st2(A0, v, t);
            __syncthreads();
            ld3(A0, v, t);
            bfly_max<true>(v, 0, 3);
            float sc[TR];
            sum_pass<true>(v, sc, A1, A0, t, d);
            __syncthreads();                             // A0 is read: the outputs may land
#pragma unroll
            for (int r = 0; r < TR; ++r) A0[BN_AT(opos(el1(r, t)), 1, TN)] = scaled_log(v[r], sc[r]);
        }
        fence_async_shared();                            // written: the store may read it
        __syncthreads();
        if (t == 0) bulk_store(out, out_s, TN * 4u);
    }
    if (t == 0) bulk_wait();
}

// ===========================================================================
// Step 4, phase 1 for n >= 14: one block per tile H of the n-1 bits of S
// (bit v removed); s_v(S) = F(S) + R'(S + {v}); keeps the outputs with at
// most d low elements in row H of W.
// ===========================================================================
//
// Relevance cut (when Aup is given).  Every output W[H][g] reaches a
// posterior only through B_v(G) Gamma_v(G) / F(V) with G inside the tile's
// full set S_H = H + all 13 low bits, and B_v(G) <= A_v(S_H).  An output
// below L = F(V) - margin - A_v(S_H) therefore moves no posterior by more than
// 2^-margin, and the K * 2^h outputs of v together by at most
// K 2^h 2^-margin; the launcher takes margin = 64 + log2(K 2^h) bits in FP64
// and 24 + log2(K 2^h) in FP32, so the total is below 2^-64 (resp. 2^-24,
// against the FP32 tolerance of 1e-4).  A tile whose upper bound M is below L writes every
// output as L - gap (no butterflies); a tile within one window of
// max(L, s(full)) takes the single-scale pass, its outputs held at >= L - gap.
// Outputs at or above L are exact as before.  The written value, like the
// true one, is below 2^L: the error of such an output is within the bound.
template <typename T, bool Q>
__global__ void __launch_bounds__(TT, sizeof(T) == 4 ? 3 : 1)
k_gamma13_p1(int n, int d, uint32_t nlow, const T* __restrict__ F,
             const T* __restrict__ Rc, const uint16_t* __restrict__ rank13, T* __restrict__ W,
             size_t js, const T* __restrict__ lq, const T* __restrict__ Aup, T margin,
             uint32_t vsel)
{
    // block x = tile H * n + endpoint v: the blocks running at once are
    // the n endpoints of a few neighbouring tiles, whose gathers of F and R'
    // fall on the same rows, so L2 serves most of them (against one endpoint's
    // tiles at a time: 1.99 -> 1.79 ms at n = 26)
    const int v = (int)(blockIdx.x % (unsigned)n);
    const uint32_t ntile = gridDim.x / (unsigned)n;
    if (!(vsel >> v & 1u)) return;                  // an endpoint another rank computes
    F = job_ptr(F, js);
    Rc = job_ptr(Rc, js);
    rank13 = job_ptr(rank13, js);
    const uint16_t* unrank13 = rank13 + TN;         // the inverse table follows
    W = job_ptr(W, js) + (size_t)endpoint_slot(vsel, v) * ntile * nlow;
    using Lg = LogOps<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* A0 = reinterpret_cast<T*>(smem_raw);
    T* A1 = A0 + TN;
    const int t = threadIdx.x;
    const uint32_t H = blockIdx.x / (unsigned)n;
    const uint32_t bv = 1u << v;

    using O = typename OrdInt<T>::type;
    constexpr bool kBases = sizeof(T) == 4;         // FP32: per-level bases of F and R'
    __shared__ O tmax_s;
    __shared__ T sfull_s;
    __shared__ T lq_s[Q ? 32 : 1];                  // q_v by |S| (Eq. 12), when given
    __shared__ float off_s[32];                     // F + R' - Z by level (bn_device.cuh)
    __shared__ int sh_s;
    __shared__ float fvrel_s;
    if (t == 0) tmax_s = ord_enc(Lg::ninf());
    if (Q && t < n) lq_s[t] = lq[v * n + t];
    T x[TR];
#pragma unroll
    for (int r = 0; r < TR; ++r) {                  // the tile's loads go out first
        const uint32_t S = expand((H << TB) | el1(r, t), v);
        x[r] = F[BN_AT(S, 1, (size_t)1 << n)] + Rc[BN_AT(S | bv, 1, (size_t)1 << n)];
    }
    if constexpr (kBases)                           // while they are in flight
        load_gamma_offsets(reinterpret_cast<const float*>(Rc), n, v, off_s, &sh_s, &fvrel_s);
    __syncthreads();
    T mx = Lg::ninf();
    // The level of element el1(r, t) is |S >> 4| = |H| + |t without its low
    // bits| + |r| (bit v, outside S, shifts the low bits of t by one when
    // v < 4), so a thread needs six offsets, indexed by |r| <= 5.
    float offr[6];
    if constexpr (kBases) {
        const int lowm = v >= kLevelShift ? 15 : 7;
        const int bt = sh_s == kLevelShift ? __popc(H) + __popc(t & ~lowm) : 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) offr[k] = off_s[BN_AT(sh_s == kLevelShift ? bt + k : 0, 1, 32)];
    }
#pragma unroll
    for (int r = 0; r < TR; ++r) {
        if constexpr (kBases) x[r] += offr[__popc(r)];
        if (Q) x[r] += lq_s[__popc(expand((H << TB) | el1(r, t), v))];
        mx = x[r] > mx ? x[r] : mx;
    }
    for (int o = 16; o; o >>= 1) {
        const T y = __shfl_xor_sync(FULLMASK, mx, o);
        mx = y > mx ? y : mx;
    }
    if ((t & 31) == 0) atomicMax(&tmax_s, ord_enc(mx));
    if (t == TT - 1) sfull_s = x[TR - 1];            // s of the full tile set (element 8191)
    __syncthreads();
    T* row = W + (size_t)H * nlow;
    {
        // every output T (|T| <= d) sums s over its supersets, the full set
        // included: it lies between s(full) and M, so a tile that spans
        // less than one window resolves in one single-scale pass (Window)
        const T M = ord_dec(tmax_s) + T(TB);
        T L = Lg::ninf();                           // relevance cut (see above)
        if (Aup) {
            T at = job_ptr(Aup, js)[BN_AT(((size_t)v << (n - 1)) + (((size_t)H << TB) | (TN - 1)), 1,
                                          (size_t)n << (n - 1))];
            // the bound is the sum of B_v: A_v without its factor q_v (a zero
            // factor is held as -1e7 nats, where FP32 counts in units of 1)
            if (Q) at += (sizeof(T) == 4 ? T(4) : T(1e-6)) - lq_s[__popc(H) + TB];
            // log P(D) in the units of s (FP32: relative to the integer Z)
            const T fv = kBases ? (T)fvrel_s : F[((size_t)1 << n) - 1];
            L = fv - margin - at;
        }
        const T floorv = L - Window<T>::gap;
        if (M < L) {                                // nothing in the tile matters
            for (uint32_t c = t; c < nlow; c += TT) row[BN_AT(c, 1, nlow)] = floorv;
            return;
        }
        if (M - (L > sfull_s ? L : sfull_s) < Window<T>::win) {
            const T sp = M - Window<T>::top;
#pragma unroll
            for (int r = 0; r < TR; ++r) x[r] = Lg::ex(x[r] - sp);
            bfly_plain<false>(x, 0, 5);
            st1(A0, x, t);
            __syncthreads();
            ld2(A0, x, t);
            bfly_plain<false>(x, 0, 5);
            st2(A0, x, t);
            __syncthreads();
            ld3(A0, x, t);
            bfly_plain<false>(x, 0, 3);
            if constexpr (sizeof(T) == 8) {
                // only the outputs with at most d elements are kept: back to
                // shared memory (each thread rewrites the slots it read), then
                // a logarithm (many FP64 instructions) per kept output, stored
                // in rank order
                st3(A0, x, t);
                __syncthreads();
                for (uint32_t c = t; c < nlow; c += TT) {
                    const T o = sp + Lg::lg(A0[swz(BN_AT(unrank13[c], 1, TN))]);
                    row[BN_AT(c, 1, nlow)] = o > floorv ? o : floorv;
                }
            } else {
                // FP32: a logarithm per register, kept outputs stored in place
#pragma unroll
                for (int r = 0; r < TR; ++r) {
                    const uint32_t el = el3(r, t);
                    const T o = sp + Lg::lg(x[r]);
                    if (__popc(el) <= d) row[BN_AT(rank13[el], 1, nlow)] = o > floorv ? o : floorv;
                }
            }
            return;
        }
    }
    st1(A1, x, t);                        // s_v kept for the band pass
    bfly_max<false>(x, 0, 5);
    st1(A0, x, t);
    __syncthreads();
    ld2(A0, x, t);
    bfly_max<false>(x, 0, 5);
    st2(A0, x, t);
    __syncthreads();
    ld3(A0, x, t);
    bfly_max<false>(x, 0, 3);

    T sc[TR];
    sum_pass<false>(x, sc, A1, A0, t, d);
    if constexpr (sizeof(T) == 8) {
        // the kept outputs in rank order, as in the single-scale pass; each
        // thread rewrites the layout-1 slots it has just read
        st1(A0, x, t);
        st1(A1, sc, t);
        __syncthreads();
        for (uint32_t c = t; c < nlow; c += TT) {
            const uint32_t e = swz(BN_AT(unrank13[c], 1, TN));
            row[BN_AT(c, 1, nlow)] = scaled_log(A0[e], A1[e]);
        }
    } else {
        const int pt = __popc((uint32_t)t);
#pragma unroll
        for (int r = 0; r < TR; ++r)
            if (pt + __popc((uint32_t)r) <= d) row[BN_AT(rank13[el1(r, t)], 1, nlow)] = scaled_log(x[r], sc[r]);
    }
}

// ===========================================================================
// The 13-dimension tiles of the linear FP64 form (X64, bn_device.cuh): the
// same transforms with the values themselves.  A pass takes the tile's values
// relative to one exponent `ref` as doubles (2^-1000 .. 2^1010: integer
// operations, no exponential), runs the butterflies as additions, and packs
// what it resolves (no logarithm): an output of at least 2^-900 there has lost
// at most 8192 terms below 2^-1000, under 2^-87 of it.  Later passes move ref
// down by 1900 bits until every output is resolved; values above 2^1010 are
// +inf there and belong to outputs already written.  Nearly every tile takes
// one pass.  What bounds it: the FP64 additions of the butterflies (6.5 per
// value, two lanes per clock and SM).
// ===========================================================================
constexpr int kXTop = 1010, kXKeep = -900, kXStep = 1900;

// Largest exponent of a block of TT threads (every thread gets it).
__device__ __forceinline__ int block_max(int e, int* red, int t)
{
    e = __reduce_max_sync(FULLMASK, e);
    if ((t & 31) == 0) red[t >> 5] = e;
    __syncthreads();
    int m = red[0];
#pragma unroll
    for (int w = 1; w < TT / 32; ++w) m = max(m, red[w]);
    return m;
}

// Column sums by butterflies over the high dimensions (k_upzeta13_colb).
template <int CPB>
__global__ void __launch_bounds__(kColbThreads)
k_colb_x(int n, int d, int64_t K, const X64* __restrict__ tab, X64* __restrict__ A, size_t js, int nodes,
         uint32_t ncb, int hc)
{
    tab = job_ptr(tab, js);
    A = job_ptr(A, js);
    __shared__ SBinom sb;
    __shared__ uint32_t off13[16];
    __shared__ uint32_t rowoff_k[32];
    __shared__ int wred[kColbThreads / 32][CPB];                     // the warps' column maxima (exponents)
    __shared__ int cmax_s[CPB], f0_s[CPB];
    __shared__ int ref_s[CPB];                       // a column's reference exponent
    __shared__ int lin_s[CPB], all_lin;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    X64* v = reinterpret_cast<X64*>(smem_raw);       // [column of the run][H]; doubles while linear
    const int h = n - 1 - TB;
    const int hl = h - hc;                           // hc: chunk bits (see k_upzeta13_colb)
    const uint32_t H2 = 1u << hl;
    const uint32_t ncol = num_small_subsets(TB, d);
    const uint32_t nrun = (ncb + CPB - 1) / CPB;
    const uint32_t nbb = ((uint32_t)nodes * nrun) << hc;
    const size_t asize = (size_t)nodes << (n - 1);
    if (blockIdx.x >= nbb) {                         // copies: a warp per tile
        const uint32_t tile = (blockIdx.x - nbb) * (blockDim.x >> 5) + (threadIdx.x >> 5);
        if (tile >= ((uint32_t)nodes << h)) return;
        const X64* tb = tab + (size_t)(tile >> h) * K;
        X64* out = A + BN_AT((size_t)tile << TB, TN, asize);
        for (uint32_t c = ncb + (threadIdx.x & 31); c < ncol; c += 32) out[c] = tb[BN_AT(c, 1, K)];
        return;
    }
    fill_sbinom(sb);
    if (threadIdx.x < 16) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= TB; ++k) o += binom(TB, k);
        off13[threadIdx.x] = o;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t o = 0;
        for (int k = 0; k < (int)threadIdx.x && k <= min(d, h); ++k)
            o += binom(h, k) * off13[min(d - k, TB) + 1];
        rowoff_k[threadIdx.x] = o;
    }
    __syncthreads();
    const uint32_t chunk = blockIdx.x & ((1u << hc) - 1u);
    const int i = (int)((blockIdx.x >> hc) / nrun);
    const uint32_t c0 = ((blockIdx.x >> hc) % nrun) * CPB;
    const uint32_t Hc = chunk << hl;
    const X64* tb = tab + (size_t)i * K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t cc = lane & (CPB - 1), c = c0 + cc;   // this lane's column
    int kl = 0;                                      // its low elements (-1: none)
    while (kl < TB && off13[kl + 1] <= c) ++kl;
    if (c >= ncb) kl = -1;
    const int kl0 = __shfl_sync(FULLMASK, kl, 0);
    int mx = -kXBias;
    for (uint32_t Hb = warp * 32; Hb < H2; Hb += blockDim.x) {
        const uint32_t Hf = Hc | Hb | lane;
        const int kh = __popc(Hf);
        uint32_t row = 0;                            // the row of G_H in the node's table
        if (kh <= d - kl0) {                         // some column reads it
            int t = 1;                               // colex rank of Hf among kh-subsets
            for (uint32_t x = Hf; x; x &= x - 1, ++t) row += sb_binom(sb, __ffs(x) - 1, t);
            row = rowoff_k[kh] + row * off13[min(d - kh, TB) + 1];
        }
#pragma unroll
        for (int j = 0; j < CPB; ++j) {
            const uint32_t src = j * (32 / CPB) + lane / CPB, H = Hb | src;
            const uint32_t rj = __shfl_sync(FULLMASK, row, src);
            const bool in = kl >= 0 && __popc(Hc | H) <= d - kl;
            const X64 val = in ? tb[BN_AT(rj + c, 1, K)] : X64{0ull};
            v[colb_pos<8, CPB>((cc << hl) | H, hl)] = val;
            mx = max(mx, x_exp(val));
        }
    }
    for (int o = 16; o >= CPB; o >>= 1) {
        mx = max(mx, __shfl_xor_sync(FULLMASK, mx, o));
    }
    if (lane < CPB) wred[warp][lane] = mx;
    __syncthreads();
    if (threadIdx.x < CPB) {
        int m = wred[0][threadIdx.x];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = max(m, wred[w][threadIdx.x]);
        cmax_s[threadIdx.x] = m;
        f0_s[threadIdx.x] = x_exp(v[colb_pos<8, CPB>(threadIdx.x << hl, hl)]);
    }
    if (hc) cluster_sync();
    else __syncthreads();
    if (threadIdx.x == 0) {
        // a column's outputs lie between its H = {} value and its largest
        // input times 2^h: one pass when both fit
        int all = 1;
        for (uint32_t q = 0; q < CPB; ++q) {
            int m = cmax_s[q];
            int f = f0_s[q];
            if (hc) {
                f = peer_ld(f0_s + q, 0);
                for (uint32_t p = 0; p < (1u << hc); ++p) m = max(m, peer_ld(cmax_s + q, p));
            }
            ref_s[q] = m + h + 1 - kXTop;
            lin_s[q] = c0 + q >= ncb || f - ref_s[q] >= kXKeep;
            all &= lin_s[q];
        }
        all_lin = all;
    }
    __syncthreads();
    const auto scaled = [&](X64 x, uint32_t cc) {
        return lin_s[cc] ? X64{(uint64_t)__double_as_longlong(x_scaled(x, ref_s[cc]))} : x;
    };
    const auto plus = [](X64 a, X64 b) {
        return X64{(uint64_t)__double_as_longlong(__longlong_as_double((long long)a.u) +
                                                  __longlong_as_double((long long)b.u))};
    };
    if (all_lin)
        colb_steps<CPB>(v, hl, scaled, [&](X64 a, X64 b, uint32_t) { return plus(a, b); });
    else
        colb_steps<CPB>(v, hl, scaled, [&](X64 a, X64 b, uint32_t cc) { return lin_s[cc] ? plus(a, b) : x_add(a, b); });
    if (hc) cluster_sync();                          // the peers' steps are done
    X64* Ai = A + ((size_t)i << (n - 1));
    if (c < ncb) {
        for (uint32_t H = warp * (32 / CPB) + lane / CPB; H < H2; H += (32 / CPB) * (blockDim.x >> 5)) {
            const X64* at = v + colb_pos<8, CPB>((cc << hl) | H, hl);
            const X64 x = hc ? chunk_sum(at, chunk, cc, [&](X64 a, X64 b, uint32_t q) {
                return lin_s[q] ? plus(a, b) : x_add(a, b);
            }) : *at;
            Ai[BN_AT(((size_t)(Hc | H) << TB) + c, 1, (size_t)1 << (n - 1))] =
                lin_s[cc] ? x_pack(__longlong_as_double((long long)x.u), ref_s[cc]) : x;
        }
    }
    if (hc) cluster_sync();                          // no peer reads this block's values any more
}

// Up-zeta tile (k_upzeta13): the tile's column sums are staged in shared
// memory (the outputs overwrite their slots), a thread reads its layout-1
// inputs by the rank of their patterns.  64 KB for the exchanges and 8 ncol
// bytes of columns: two blocks per SM.
__global__ void __launch_bounds__(TT, 2)
k_up13_x(int n, int d, const uint16_t* __restrict__ rank13, X64* __restrict__ A, size_t js)
{
    rank13 = job_ptr(rank13, js);
    A = job_ptr(A, js);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* A0 = reinterpret_cast<double*>(smem_raw);
    X64* col = reinterpret_cast<X64*>(A0 + TN);
    __shared__ int red[TT / 32];
    const uint32_t ncol = num_small_subsets(TB, d);
    const int h = n - 1 - TB;
    const int t = threadIdx.x;
    const int i = (int)(blockIdx.x >> h);
    const uint32_t H = blockIdx.x & ((1u << h) - 1u);
    X64* out = A + BN_AT(((size_t)i << (n - 1)) + ((size_t)H << TB), TN, (size_t)gridDim.x << TB);
    int e = -kXBias;
    for (uint32_t c = t; c < ncol; c += TT) {
        const X64 v = out[c];
        col[c] = v;
        e = max(e, x_exp(v));
    }
    const int M = block_max(e, red, t) + TB + 1;     // every output is below 2^M
    const int low = max(x_exp(col[0]), kXMin);       // and at least C(empty)
    const int pt = __popc(t);                        // |el1(r, t)| = |r| + |t|
    uint32_t done = 0u;                              // bit r: output el3(r, t) written
    for (int ref = M - kXTop;; ref -= kXStep) {
        const bool last = low - ref >= kXKeep;
        double x[TR];
#pragma unroll
        for (int r = 0; r < TR; ++r)
            x[r] = __popc(r) + pt <= d ? x_scaled(col[BN_AT(rank13[el1(r, t)], 1, ncol)], ref) : 0.0;
        bfly_plain<true>(x, 0, 5);
        st1(A0, x, t);
        __syncthreads();
        ld2(A0, x, t);
        bfly_plain<true>(x, 0, 5);
        st2(A0, x, t);
        __syncthreads();
        ld3(A0, x, t);
        bfly_plain<true>(x, 0, 3);
        if (last && done == 0u) {                    // one pass: whole runs of 8
#pragma unroll
            for (int q = 0; q < TR / 8; ++q) {
                ulonglong2* p = reinterpret_cast<ulonglong2*>(out + el3(8 * q, t));
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    p[k] = make_ulonglong2(x_pack(x[8 * q + 2 * k], ref).u, x_pack(x[8 * q + 2 * k + 1], ref).u);
            }
            return;
        }
#pragma unroll
        for (int r = 0; r < TR; ++r)
            if (!(done >> r & 1u) && (last || x[r] >= pow2d(kXKeep))) {
                out[el3(r, t)] = x_pack(x[r], ref);
                done |= 1u << r;
            }
        if (last) return;
        __syncthreads();                             // A0 is reused
    }
}

// Down-zeta tile (k_gamma13_p1).  The relevance cut works on exponents: an
// output below 2^L moves no posterior (L = log2 F(V) - margin - log2 A_v(S_H),
// rounded down), so a tile whose bound M is below L is all zeros and a pass is
// the last once it resolves max(L, s(full)).
template <bool Q>
__global__ void __launch_bounds__(TT, 2)
k_g13_x(int n, int d, uint32_t nlow, const X64* __restrict__ F, const X64* __restrict__ Rc,
        const uint16_t* __restrict__ rank13, X64* __restrict__ W, size_t js, const X64* __restrict__ lq,
        const X64* __restrict__ Aup, int margin, uint32_t vsel)
{
    const int v = (int)(blockIdx.x % (unsigned)n);   // the endpoint fastest (k_gamma13_p1)
    const uint32_t ntile = gridDim.x / (unsigned)n;
    if (!(vsel >> v & 1u)) return;
    F = job_ptr(F, js);
    Rc = job_ptr(Rc, js);
    const uint16_t* unrank13 = job_ptr(rank13, js) + TN;
    W = job_ptr(W, js) + (size_t)endpoint_slot(vsel, v) * ntile * nlow;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* A0 = reinterpret_cast<double*>(smem_raw);
    __shared__ int red[TT / 32];
    const int t = threadIdx.x;
    const uint32_t H = blockIdx.x / (unsigned)n;
    const uint32_t bv = 1u << v;
    X64* row = W + (size_t)H * nlow;
    int L = kXMin;
    if (Aup) {
        const X64 at = job_ptr(Aup, js)[BN_AT(((size_t)v << (n - 1)) + (((size_t)H << TB) | (TN - 1)), 1,
                                              (size_t)n << (n - 1))];
        // the bound is the sum of B_v: A_v without its factor q_v (unknown when
        // that is zero)
        const X64 q = Q ? lq[v * n + __popc(H) + TB] : x_one();
        if (at.u && q.u) L = max(L, x_exp(F[((size_t)1 << n) - 1]) - x_exp(at) + x_exp(q) - 2 - margin);
    }
    // s of the full tile set, the smallest output, is a load of its own: the
    // first reference puts the smallest output that matters at 2^kXKeep, and
    // the values are scaled as they arrive
    int efull;
    {
        const uint32_t S = expand((H << TB) | (TN - 1), v);
        efull = x_exp(F[BN_AT(S, 1, (size_t)1 << n)]) + x_exp(Rc[BN_AT(S | bv, 1, (size_t)1 << n)]);
        if (Q) efull += x_exp(lq[v * n + __popc(S)]);
    }
    const int low = max(L, efull);
    double x[TR];
    auto load = [&](int ref) {                       // s relative to ref; the largest exponent
        int mx = -2 * kXBias;
#pragma unroll
        for (int r = 0; r < TR; ++r) {
            const uint32_t S = expand((H << TB) | el1(r, t), v);
            const X64 f = F[BN_AT(S, 1, (size_t)1 << n)], g = Rc[BN_AT(S | bv, 1, (size_t)1 << n)];
            double p = x_mant(f) * x_mant(g);
            int e = x_exp(f) + x_exp(g);
            if (Q) {                                 // q_v(S) of Eq. 12
                const X64 q = lq[v * n + __popc(S)];
                p *= x_mant(q);
                e += x_exp(q);
            }
            mx = max(mx, e);
            x[r] = p * pow2d(min(e - ref, 1024));    // 0 or +inf outside a double's range
            // sixteen values' loads in flight: more would spill
            if ((r & 15) == 15) asm volatile("" ::: "memory");
        }
        return mx;
    };
    int ref = low - kXKeep;
    const int M = block_max(load(ref), red, t) + TB + 3;    // every output is below 2^M
    if (M < L) {                                     // nothing in the tile matters
        for (uint32_t c = t; c < nlow; c += TT) row[BN_AT(c, 1, nlow)] = X64{0ull};
        return;
    }
    if (M > ref + kXTop) {                           // wider than one pass: from the top
        ref = M - kXTop;
        load(ref);
    }
    uint32_t done = 0u;                              // bit k: output row[t + k TT] written
    for (;;) {
        const bool last = low - ref >= kXKeep;
        bfly_plain<false>(x, 0, 5);
        st1(A0, x, t);
        __syncthreads();
        ld2(A0, x, t);
        bfly_plain<false>(x, 0, 5);
        st2(A0, x, t);
        __syncthreads();
        ld3(A0, x, t);
        bfly_plain<false>(x, 0, 3);
        st3(A0, x, t);                               // each thread rewrites the slots it read
        __syncthreads();
        // the kept outputs (at most d elements) in rank order
        uint32_t k = 0;
        for (uint32_t c = t; c < nlow; c += TT, ++k) {
            const double o = A0[swz(BN_AT(unrank13[c], 1, TN))];
            if (!(done >> k & 1u) && (last || o >= pow2d(kXKeep))) {
                row[BN_AT(c, 1, nlow)] = x_pack(o, ref);
                done |= 1u << k;
            }
        }
        if (last) return;
        ref -= kXStep;
        load(ref);
        __syncthreads();                             // A0 is reused
    }
}

#ifndef BN_MEGA  // host launchers (bn_mega.cu includes only the device code)
#ifdef BN_CHECK_BOUNDS
BN_BOUNDS_READER(bounds_line_tile13)
#endif
// ===========================================================================
// Launchers.
// ===========================================================================
// Columns whose sums take more than one row: the low patterns with fewer
// than d elements.
static uint32_t colb_columns(const Plan& P)
{
    uint64_t c = 0;
    for (int k = 0; k < P.d && k <= TB; ++k) c += binom_host(TB, k);
    return (uint32_t)c;
}

// High bits whose chunks of a column lie in the blocks of a cluster: beyond
// h = 12, so that a block holds 4 columns (FP32; 2 in FP64) in 64 KB and three
// share an SM; at most 3 bits, the 8 blocks of a portable cluster.  Recorded
// launches have no clusters: a block holds whole columns of up to 128 KB
// there (4, more than is taken, past that).  n = 29 (h = 15), FP32: one
// column of 128 KB a block 13.4 ms, chunks in clusters of 8 blocks 4.9 ms.
static int colb_chunk_bits(const Plan& P)
{
    const int h = P.n - 1 - TB;
    const int hmax = P.prec == 0 ? 14 : 15;          // 2^h values of 8 or 4 bytes in 128 KB
    if (recording() || (P.spill && h > hmax)) return h <= hmax ? 0 : 4;
    const int hc = std::min(3, std::max(0, h - 12));
    return h - hc <= hmax ? hc : 4;
}

// Column sums by butterflies over the h high dimensions when they take at
// most four fifths (FP32; four times in FP64) of the steps of the direct sums
// (the columns with d low elements are copies either way) and a column run
// fits 128 KB of shared memory (5 <= h <= 15 in FP32, h <= 14 in FP64).
bool use_colb(const Plan& P)
{
    const int h = P.n - 1 - TB;
    // below h = 5 a column has at most 32 rows: the per-tile sums are cheap,
    // and the column kernel's many small blocks would cost a batch's
    // persistent kernel one work item each
    if (h < 5 || colb_chunk_bits(P) > 3) return false;
    double direct = 0.0, ncol = 0.0;
    for (int kl = 0; kl <= P.d && kl <= TB; ++kl) {
        ncol += (double)binom_host(TB, kl);
        double rows = 0.0;
        for (int kh = 0; kh <= P.d - kl && kh <= h; ++kh)
            rows += (double)binom_host(h, kh) * std::ldexp(1.0, h - kh);
        direct += (double)binom_host(TB, kl) * rows;
    }
    const double ncb = colb_columns(P);
    const double bfly = ncb * h * std::ldexp(1.0, h - 1) + (ncol - ncb) * std::ldexp(1.0, h);
    // FP64: a direct term costs an FP64 exponential, a linear-scale step one addition
    return direct >= (P.prec == 0 ? 0.25 : 1.25) * bfly;
}

size_t upzeta13_cols_smem_bytes(const Plan& P)
{
    const size_t es = P.prec == 0 ? 8 : 4;
    const int h = P.n - 1 - TB;
    uint64_t nrow = 0;
    for (int k = 0; k <= P.d && k <= h; ++k) nrow += binom_host(h, k);
    return 2 * 8 * 96 * es + sizeof(SBinom) + 64 * 4 + 16 * 4 + nrow * 4;
}

size_t upzeta13_smem_bytes(const Plan& P)
{
    const size_t es = P.prec == 0 ? 8 : 4;
    return (size_t)TN * (2 * es) + (TT / 32) * es;   // A0, A1, the warps' maxima
}

bool tile13_up_fits(const Plan& P)
{
    return P.n >= 14 && upzeta13_cols_smem_bytes(P) <= 227 * 1024 - 64;
}

size_t gamma13_smem_bytes(const Plan& P)
{
    const size_t es = P.prec == 0 ? 8 : 4;
    return (size_t)TN * (2 * es) + 16;
}

cudaError_t launch_reorder_up(const Plan& P, const void* lbs, void* tab, cudaStream_t s)
{
    const int64_t total = (int64_t)up_nodes(P) * P.K;
    const dim3 grid((unsigned)std::min<int64_t>((total + 255) / 256, 152 * 16), P.nj);
    if (P.lin)
        launch_or_record(KID_REORDER_X, k_reorder_up<X64>, grid, 256, 0, s, P.n, P.d, P.K, (const X64*)lbs, (X64*)tab,
                                                  P.js, up_nodes(P));
    else if (P.prec == 0)
        launch_or_record(KID_REORDER_D, k_reorder_up<double>, grid, 256, 0, s, P.n, P.d, P.K, (const double*)lbs, (double*)tab,
                                                  P.js, up_nodes(P));
    else
        launch_or_record(KID_REORDER_F, k_reorder_up<float>, grid, 256, 0, s, P.n, P.d, P.K, (const float*)lbs, (float*)tab,
                                                 P.js, up_nodes(P));
    return cudaGetLastError();
}

size_t upzeta13p_smem_bytes(const Plan& P)
{
    // two blocks of 32 KB, the warps' maxima, the mbarrier and a flag, the
    // staged column sums (16-byte multiple, and 48 bytes for the two copies'
    // rounding)
    return (size_t)TN * 4 * 2 + (TT / 32) * 4 + 16 + (((size_t)num_small_subsets_host(P.d) * 4 + 15) & ~(size_t)15) + 48;
}

// The persistent FP32 tile kernel runs single jobs whose A is in device
// memory (a spilled A may sit in host memory, where no bulk copy goes) and
// that are launched directly, not recorded for the persistent batch kernel.
static bool use_upzeta13p(const Plan& P, const int* err)
{
    return err && P.prec != 0 && P.nj == 1 && !P.spill && !recording();
}

// Three blocks per SM (80 registers; the exact path spills) for the sample
// counts whose tiles mostly take one window, two (128 registers) for the
// others and where the staged sums leave no room for three.  A tile's span
// grows with the evidence, so with m; the data decide the rest.  The tiles'
// time with three blocks over that with two, mean (and range) over eleven
// shapes, n = 21 to 28, d = 2 to 5, binary and arities 2 to 4: m = 150 0.91
// (0.90-0.95), 500 0.93 (0.90-0.97), 700 0.95 (0.92-1.02), 800 0.98 (0.92-1.02),
// 900 1.00 (0.92-1.04), 1000 1.02 (0.96-1.09), 1500 1.07 (0.97-1.15), 2000 1.14
// (1.05-1.28).  us, two / three: n = 26 d = 4, m = 800 1524 / 1478, m = 900
// 1759 / 1788; n = 21 d = 3 mixed, m = 700 44.0 / 43.0, m = 800 47.1 / 48.1.
constexpr int kUp13ThreeM = 800;

// The persistent tile kernel stages the columns with d low elements straight
// from the reordered score table when the column sums come from the column
// butterflies (which then leave them out), the table's node stride is a
// multiple of 16 bytes and every node's table holds at least 3 entries past
// its first ncol (h >= 1).
static bool upzeta_table_copies(const Plan& P, const void* tab, const int* err)
{
    const int h = P.n - 1 - TB;
    return use_upzeta13p(P, err) && use_colb(P) && colb_columns(P) < num_small_subsets_host(P.d) &&
           P.K % 4 == 0 && ((uintptr_t)tab & 15u) == 0 && h >= 1 && P.d >= 1;
}

// The per-tile column sums by a warp: its row list fits shared memory.
static bool colw_fits(const Plan& P)
{
    const int h = P.n - 1 - TB;
    uint64_t nrow = 0;
    for (int k = 0; k <= P.d && k <= h; ++k) nrow += binom_host(h, k);
    return nrow * 4 * 8 <= 160 * 1024;
}

// The linear FP64 form has the column butterflies and the warp's sums, and
// stages a tile's columns beside its 64 KB exchange array.
static size_t up13_x_smem(const Plan& P) { return (size_t)TN * 8 + (size_t)num_small_subsets_host(P.d) * 8; }
bool lin_tiles_fit(const Plan& P)
{
    if (P.n < 14) return true;
    return colw_fits(P) && up13_x_smem(P) <= 220 * 1024;
}

// A column-sum launch: plain (or recorded), or in clusters of 2^hc blocks.
struct ColbLaunch {
    dim3 grid;
    unsigned threads;
    size_t smem;
    int hc;
    cudaStream_t s;
    template <typename... P, typename... A> cudaError_t operator()(int kid, void (*k)(P...), A... a) const
    {
        if (!hc) return launch_or_record(kid, k, grid, threads, smem, s, a...);
        cudaLaunchAttribute attr = {};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = 1u << hc;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, k, static_cast<P>(a)...);
    }
};

cudaError_t launch_upzeta13(const Plan& P, const void* tab, const uint16_t* unrank13, void* A,
                            cudaStream_t s, cudaEvent_t sums_done, int* err)
{
    const int h = P.n - 1 - TB;
    const int nodes = up_nodes(P);
    const dim3 grid((unsigned)nodes << h, P.nj);
    const size_t sc = upzeta13_cols_smem_bytes(P), sm = upzeta13_smem_bytes(P);
    uint64_t nrow = 0;
    for (int k = 0; k <= P.d && k <= h; ++k) nrow += binom_host(h, k);
    if (use_colb(P)) {                                // butterflies over the high dims
        // columns per block: as many chunks as fit 64 KB, at most 8 (FP32) or
        // 4 (FP64), one where a chunk is 128 KB
        const size_t es = P.prec == 0 ? 8 : 4;
        const int hc = colb_chunk_bits(P);
        const int cpb = (int)std::max<size_t>(1, std::min<size_t>((size_t)(64 * 1024) / (es << (h - hc)), P.prec == 0 ? 4 : 8));
        uint64_t ncol = 0;
        for (int k = 0; k <= P.d && k <= TB; ++k) ncol += binom_host(TB, k);
        const uint32_t ncb = colb_columns(P);
        const uint64_t ntiles = (uint64_t)nodes << h;
        // the copy blocks follow the butterfly blocks (none when the tile
        // kernel stages those columns from the table itself), in whole clusters
        const bool copies = ncb < ncol && !upzeta_table_copies(P, tab, err);
        const unsigned threads = rec_block(kColbThreads), wpb = threads / 32;
        const unsigned ncopy = copies ? (unsigned)(((ntiles + wpb - 1) / wpb + ((1u << hc) - 1)) >> hc << hc) : 0;
        const unsigned nblk = (unsigned)((uint64_t)nodes * ((ncb + cpb - 1) / cpb) << hc) + ncopy;
        const size_t smb = ((size_t)cpb << (h - hc)) * es;
        const ColbLaunch L{dim3(nblk, P.nj), threads, smb, hc, s};
        if (P.lin) {
            const X64* tx = (const X64*)tab;
            X64* Ax = (X64*)A;
            if (cpb >= 4) L(KID_COLB4_X, k_colb_x<4>, P.n, P.d, P.K, tx, Ax, P.js, nodes, ncb, hc);
            else if (cpb == 2) L(KID_COLB2_X, k_colb_x<2>, P.n, P.d, P.K, tx, Ax, P.js, nodes, ncb, hc);
            else L(KID_COLB1_X, k_colb_x<1>, P.n, P.d, P.K, tx, Ax, P.js, nodes, ncb, hc);
        } else if (P.prec == 0) {
            const double* td = (const double*)tab;
            double* Ad = (double*)A;
            if (cpb >= 4) L(KID_COLB4_D, k_upzeta13_colb<double, 4>, P.n, P.d, P.K, td, Ad, P.js, nodes, ncb, hc);
            else if (cpb == 2) L(KID_COLB2_D, k_upzeta13_colb<double, 2>, P.n, P.d, P.K, td, Ad, P.js, nodes, ncb, hc);
            else L(KID_COLB1_D, k_upzeta13_colb<double, 1>, P.n, P.d, P.K, td, Ad, P.js, nodes, ncb, hc);
        } else {
            const float* tf = (const float*)tab;
            float* Af = (float*)A;
            if (cpb == 8) L(KID_COLB8, k_upzeta13_colb<float, 8>, P.n, P.d, P.K, tf, Af, P.js, nodes, ncb, hc);
            else if (cpb >= 4) L(KID_COLB4, k_upzeta13_colb<float, 4>, P.n, P.d, P.K, tf, Af, P.js, nodes, ncb, hc);
            else if (cpb == 2) L(KID_COLB2, k_upzeta13_colb<float, 2>, P.n, P.d, P.K, tf, Af, P.js, nodes, ncb, hc);
            else L(KID_COLB1, k_upzeta13_colb<float, 1>, P.n, P.d, P.K, tf, Af, P.js, nodes, ncb, hc);
        }
    } else if (colw_fits(P)) {                        // warp per tile, 8 tiles per block
        const uint64_t ntiles = (uint64_t)nodes << h;
        const dim3 gw((unsigned)std::min<uint64_t>((ntiles + 7) / 8, 152 * 16), P.nj);
        const size_t sw = (size_t)nrow * 4 * 8;
        if (P.lin)
            launch_or_record(KID_COLW_X, k_upzeta13_colw<X64>, gw, 256, sw, s, P.n, P.d, P.K, (const X64*)tab,
                                                        (X64*)A, P.js, nodes);
        else if (P.prec == 0)
            launch_or_record(KID_COLW_D, k_upzeta13_colw<double>, gw, 256, sw, s, P.n, P.d, P.K, (const double*)tab,
                                                        (double*)A, P.js, nodes);
        else
            launch_or_record(KID_COLW_F, k_upzeta13_colw<float>, gw, 256, sw, s, P.n, P.d, P.K, (const float*)tab,
                                                       (float*)A, P.js, nodes);
    } else if (P.prec == 0)
        launch_or_record(KID_COLS_D, k_upzeta13_cols<double>, grid, TT, sc, s, P.n, P.d, P.K, (const double*)tab, (double*)A,
                                                     P.js);
    else
        launch_or_record(KID_COLS_F, k_upzeta13_cols<float>, grid, TT, sc, s, P.n, P.d, P.K, (const float*)tab, (float*)A,
                                                    P.js);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (sums_done) {
        e = cudaEventRecord(sums_done, s);
        if (e != cudaSuccess) return e;
    }
    if (use_upzeta13p(P, err)) {
        const uint32_t ntiles = (uint32_t)nodes << h;
        const size_t smp = upzeta13p_smem_bytes(P);
        const auto launch = [&](auto kernel) {
            int dev = 0, nsm = 0, per_sm = 0;
            e = cudaGetDevice(&dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, TT, smp);
            if (e != cudaSuccess) return;
            const unsigned blocks = (unsigned)std::min<uint64_t>(ntiles, (uint64_t)std::max(per_sm, 1) * nsm);
            const uint32_t ncol = num_small_subsets_host(P.d);
            const uint32_t ncb = upzeta_table_copies(P, tab, err) ? colb_columns(P) : ncol;
            kernel<<<blocks, TT, smp, s>>>(P.n, P.d, unrank13, (float*)A, ntiles, err, kCopySpinCap, 0,
                                           (const float*)tab, P.K, ncb);
            e = cudaGetLastError();
        };
        const bool three = P.m <= kUp13ThreeM && P.d <= 5;
        if (use_tlo(P)) three ? launch(k_upzeta13p<true, 3>) : launch(k_upzeta13p<true, 2>);
        else three ? launch(k_upzeta13p<false, 3>) : launch(k_upzeta13p<false, 2>);
        return e;
    }
    if (P.lin)
        return launch_or_record(KID_UP13_X, k_up13_x, grid, TT, up13_x_smem(P), s, P.n, P.d, unrank13 - TN,
                                (X64*)A, P.js);
    if (P.prec == 0)
        launch_or_record(KID_UP13_D, k_upzeta13<double, false>, grid, TT, sm, s, P.n, P.d, unrank13, (double*)A, P.js);
    else if (use_tlo(P))
        launch_or_record(KID_UP13_F_TLO, k_upzeta13<float, true>, grid, TT, sm, s, P.n, P.d, unrank13, (float*)A, P.js);
    else
        launch_or_record(KID_UP13_F, k_upzeta13<float, false>, grid, TT, sm, s, P.n, P.d, unrank13, (float*)A, P.js);
    return cudaGetLastError();
}

// One block of the persistent tile kernel (n = 14, d = 4: one tile) with its
// first bulk copy withheld: its wait gives up after `polls` polls and sets
// kErrDeviceTimeout in *err.  A holds one tile (8192 floats).
cudaError_t launch_upzeta13p_withheld(float* A, const uint16_t* unrank13, int* err, uint32_t polls,
                                      cudaStream_t s)
{
    cudaError_t e = allow_max_dynamic_smem(k_upzeta13p<false, 3>);
    if (e != cudaSuccess) return e;
    Plan P{};
    P.n = 14;
    P.d = 4;
    P.prec = 1;
    k_upzeta13p<false, 3><<<1, TT, upzeta13p_smem_bytes(P), s>>>(14, 4, unrank13, A, 1u, err, polls, 1, nullptr,
                                                             int64_t(0), num_small_subsets_host(4));
    return cudaGetLastError();
}

cudaError_t launch_gamma13_p1(const Plan& P, const void* F, const void* Rc,
                              const uint16_t* rank13, void* W, cudaStream_t s, const void* lq,
                              const void* A)
{
    if (P.prec != 0) {
        const cudaError_t e = launch_gamma_table(P, F, Rc, s);
        if (e != cudaSuccess) return e;
    }
    const int h = P.n - 1 - TB;
    const size_t sm = gamma13_smem_bytes(P);
    const dim3 grid((1u << h) * (unsigned)P.n, P.nj, 1);
    // relevance margin: 64 (FP64) or 24 (FP32: its tolerance is 1e-4) bits +
    // log2(K 2^h), in bits (FP32) or nats (FP64)
    const double mbits = (P.prec == 0 ? 64.0 : 24.0) + std::ceil(std::log2((double)P.K)) + h;
    const double margin = P.prec == 0 ? mbits * 0.69314718055994531 : mbits;
    // the order prior is a separate instance: the plain kernel has no trace of it
    if (P.lin) {
        const size_t sx = (size_t)TN * 8;
        if (lq)
            launch_or_record(KID_G13_X_Q, k_g13_x<true>, grid, TT, sx, s, P.n, P.d, P.nlow_g, (const X64*)F,
                             (const X64*)Rc, rank13, (X64*)W, P.js, (const X64*)lq, (const X64*)A, (int)mbits, P.vsel);
        else
            launch_or_record(KID_G13_X, k_g13_x<false>, grid, TT, sx, s, P.n, P.d, P.nlow_g, (const X64*)F,
                             (const X64*)Rc, rank13, (X64*)W, P.js, nullptr, (const X64*)A, (int)mbits, P.vsel);
    } else if (P.prec == 0) {
        if (lq)
            launch_or_record(KID_G13_D_Q, k_gamma13_p1<double, true>, grid, TT, sm, s, 
                P.n, P.d, P.nlow_g, (const double*)F, (const double*)Rc, rank13, (double*)W, P.js,
                (const double*)lq, (const double*)A, margin, P.vsel);
        else
            launch_or_record(KID_G13_D, k_gamma13_p1<double, false>, grid, TT, sm, s, 
                P.n, P.d, P.nlow_g, (const double*)F, (const double*)Rc, rank13, (double*)W, P.js,
                nullptr, (const double*)A, margin, P.vsel);
    } else {
        if (lq)
            launch_or_record(KID_G13_F_Q, k_gamma13_p1<float, true>, grid, TT, sm, s, 
                P.n, P.d, P.nlow_g, (const float*)F, (const float*)Rc, rank13, (float*)W, P.js,
                (const float*)lq, (const float*)A, (float)margin, P.vsel);
        else
            launch_or_record(KID_G13_F, k_gamma13_p1<float, false>, grid, TT, sm, s, 
                P.n, P.d, P.nlow_g, (const float*)F, (const float*)Rc, rank13, (float*)W, P.js,
                nullptr, (const float*)A, (float)margin, P.vsel);
    }
    return cudaGetLastError();
}

cudaError_t set_tile13_attributes()
{
    cudaError_t e;
#define SETA(k)                      \
    e = allow_max_dynamic_smem(k); \
    if (e != cudaSuccess) return e;
    SETA(k_upzeta13_cols<double>)
    SETA(k_upzeta13_cols<float>)
    SETA(k_upzeta13_colw<double>)
    SETA(k_upzeta13_colw<float>)
    SETA((k_upzeta13_colb<float, 8>))
    SETA((k_upzeta13_colb<float, 4>))
    SETA((k_upzeta13_colb<float, 2>))
    SETA((k_upzeta13_colb<float, 1>))
    SETA((k_upzeta13_colb<double, 4>))
    SETA((k_upzeta13_colb<double, 2>))
    SETA((k_upzeta13_colb<double, 1>))
    SETA((k_upzeta13<double, false>))
    SETA((k_upzeta13<float, false>))
    SETA((k_upzeta13<float, true>))
    SETA((k_upzeta13p<false, 2>))
    SETA((k_upzeta13p<true, 2>))
    SETA((k_upzeta13p<false, 3>))
    SETA((k_upzeta13p<true, 3>))
    SETA((k_gamma13_p1<double, false>))
    SETA((k_gamma13_p1<float, false>))
    SETA((k_gamma13_p1<double, true>))
    SETA((k_gamma13_p1<float, true>))
    SETA(k_upzeta13_colw<X64>)
    SETA(k_colb_x<4>)
    SETA(k_colb_x<2>)
    SETA(k_colb_x<1>)
    SETA(k_up13_x)
    SETA(k_g13_x<false>)
    SETA(k_g13_x<true>)
#undef SETA
    return cudaSuccess;
}

#endif  // BN_MEGA

}  // namespace bn
