// bn_levels.cu -- F (Eq. 9) and R' (Eq. 10) over the subset lattice, one
// thread per tile of 2^B subsets: 16 in FP32 (base-2 logs), 8 in FP64 (X64
// values, or natural logs; a row of 8 is 64 bytes, like 16 floats).
//
// A tile is the 2^B subsets S = (Ht << B) | l that share their high bits Ht
// (l = the B low bits).  Tiles are launched one popcount level of Ht at a
// time (the sub-cube order of Section 3.2.2): every term that leaves the
// tile reads a tile of the previous level.  A thread
//   * adds the terms across tiles, one row of 2^B values of A_i and one row of
//     F (or R') per high bit, read as four 128-bit loads each;
//   * resolves the terms inside the tile in registers, in popcount order of l;
//   * writes its row of 2^B values.
// Every thread of a launch has the same number of terms (same |Ht|), so warps
// do not diverge, and the index arithmetic is shared by the 2^B subsets.
//
// Sums of logarithms are kept lazily: (m, s) stands for m + lg(s) with m the first
// term and s rescaled only when a term exceeds m by more than 2^64 (FP32) or
// e^40 (FP64), so a term costs one exponential.  s stays below that factor
// times 32, and every value entering is finite (A and F are logs of
// positive sums; a zero weight is a finite soft zero).
#include <algorithm>
#include <atomic>

#include "bn_device.cuh"
#include "bn_kernels.cuh"

namespace bn {
namespace {

constexpr int LB = 4;             // low bits of an FP32 tile
constexpr int LB64 = 3;           // low bits of an FP64 tile
constexpr int BT = 29;            // binomial table rows (n - B < 29: n <= 32 in FP32)
// k_sweeps: single jobs up to this n (FP32; linear FP64; a launch per level is
// faster from n = 22: FP32 330 us either way, FP64 640 against 748), vectors
// from kSweepVecN, up to kSweepBusyN while other served jobs run (the whole-GPU
// form of a wider job would hold every SM: 64 served jobs of n = 19 to 22 took
// 20.0 ms with it, 15.3 ms without); levels that fill more than kSweepGrid
// blocks run on the whole GPU; polls before a block gives up a wait (about 1 us each).
constexpr int kSweepMaxN = 21;
constexpr int kSweepMaxNX = 21;
// Largest n of any k_sweeps launch: the kernel's places among the n 2^(n-1)
// values of A are 32-bit numbers, and 28 2^27 is the last such size below 2^32
// (from n = 29 they wrap to other nodes' rows).  A batch group may come up to
// here; a level of a larger job fills the GPU by itself anyway.
constexpr int kSweepPlacesN = 28;
constexpr int kSweepVecN = 20;
constexpr int kSweepBusyN = 18;
constexpr uint64_t kSweepGrid = 12;
constexpr uint32_t kSweepSpinCap = 1u << 22;

__device__ const BinomTable g_binom_lanes = make_binom_table();

__device__ __forceinline__ void lazy_add(float& m, float& s, float x)
{
    const float dd = x - m;                       // +inf while the accumulator is empty
    const bool big = dd > 64.0f;
    const float e = ex2_approx(big ? -dd : dd);
    s = big ? __fmaf_rn(s, e, 1.0f) : s + e;
    m = big ? x : m;
}

__device__ __forceinline__ void lazy_add(double& m, double& s, double x)
{
    const double dd = x - m;                      // +inf while the accumulator is empty
    const bool big = dd > 40.0;
    const double e = exp_t(big ? -dd : dd);       // the library's table-driven exponential
    s = big ? fma(s, e, 1.0) : s + e;
    m = big ? x : m;
}

// The sum of one subset's terms A * F: (m, s) as above for logarithms (an
// empty sum has m far below any value, finite so that a left-out term of -inf
// changes nothing), LazySum for X64.  add() takes a term or leaves it out.
template <typename T> struct TileSum {
    T m = (T)-3.0e38f, s = T(0);
    __device__ __forceinline__ void add(T a, T f, bool take = true)
    {
        lazy_add(m, s, take ? a + f : LogOps<T>::ninf());
    }
    __device__ __forceinline__ void rebase(T r) { m -= r; }
    __device__ __forceinline__ T value() const { return m + LogOps<T>::lg(s); }
};
template <> struct TileSum<X64> {
    LazySum<X64> v;
    __device__ __forceinline__ void add(X64 a, X64 f, bool take = true)
    {
        const double p = x_mant(a) * x_mant(f);
        v.add(take ? p : 0.0, take ? x_exp(a) + x_exp(f) : -(1 << 28));
    }
    __device__ __forceinline__ void rebase(X64) {}
    __device__ __forceinline__ X64 value() const { return v.value(); }
};
template <typename T> __device__ __forceinline__ T unit() { return T(0); }         // log 1
template <> __device__ __forceinline__ X64 unit<X64>() { return x_one(); }

// x with bit i (i < B) removed: an index among the 2^(B-1) B-bit patterns
// without bit i.
__host__ __device__ constexpr int squeeze4(int x, int i)
{
    return (x & ((1 << i) - 1)) | ((x >> 1) & ~((1 << i) - 1));
}

// Load modes: LD_PLAIN, LD_STREAM (read once: evict first), LD_L2 (through
// L2 only: values another block of the same launch wrote).
enum { LD_PLAIN = 0, LD_STREAM = 1, LD_L2 = 2 };

// A row of N values, 128-bit loads (N * sizeof(T) is a multiple of 16).
template <int N>
__device__ __forceinline__ void load_row(const float* p, float (&v)[N], int mode)
{
    const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int k = 0; k < N / 4; ++k) {
        const float4 x = mode == LD_STREAM ? __ldcs(q + k) : mode == LD_L2 ? __ldcg(q + k) : q[k];
        v[4 * k] = x.x;
        v[4 * k + 1] = x.y;
        v[4 * k + 2] = x.z;
        v[4 * k + 3] = x.w;
    }
}

template <int N>
__device__ __forceinline__ void load_row(const double* p, double (&v)[N], int mode)
{
    const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
        const double2 x = mode == LD_STREAM ? __ldcs(q + k) : mode == LD_L2 ? __ldcg(q + k) : q[k];
        v[2 * k] = x.x;
        v[2 * k + 1] = x.y;
    }
}

template <int N>
__device__ __forceinline__ void load_row(const X64* p, X64 (&v)[N], int mode)
{
    const ulonglong2* q = reinterpret_cast<const ulonglong2*>(p);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
        const ulonglong2 x = mode == LD_STREAM ? __ldcs(q + k) : mode == LD_L2 ? __ldcg(q + k) : q[k];
        v[2 * k].u = x.x;
        v[2 * k + 1].u = x.y;
    }
}

// One value by load mode.
__device__ __forceinline__ float load_one(const float* p, int mode)
{
    return mode == LD_STREAM ? __ldcs(p) : mode == LD_L2 ? __ldcg(p) : *p;
}
__device__ __forceinline__ X64 load_one(const X64* p, int mode)
{
    const unsigned long long* q = &p->u;
    return X64{mode == LD_STREAM ? __ldcs(q) : mode == LD_L2 ? __ldcg(q) : *q};
}
__device__ __forceinline__ float shfl_one(unsigned mask, float v, int o) { return __shfl_xor_sync(mask, v, o); }
__device__ __forceinline__ X64 shfl_one(unsigned mask, X64 v, int o)
{
    return X64{__shfl_xor_sync(mask, v.u, o)};
}

template <int N>
__device__ __forceinline__ void store_row(float* p, const float (&v)[N])
{
    float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
    for (int k = 0; k < N / 4; ++k) q[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
}

template <int N>
__device__ __forceinline__ void store_row(double* p, const double (&v)[N])
{
    double2* q = reinterpret_cast<double2*>(p);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) q[k] = make_double2(v[2 * k], v[2 * k + 1]);
}

template <int N>
__device__ __forceinline__ void store_row(X64* p, const X64 (&v)[N])
{
    ulonglong2* q = reinterpret_cast<ulonglong2*>(p);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) q[k] = make_ulonglong2(v[2 * k].u, v[2 * k + 1].u);
}

// Tile g of the level: the g-th hl-element subset of nh bits in colex order.
__device__ __forceinline__ uint32_t tile_of(uint32_t g, int hl, int nh, const uint32_t (*bt)[BT])
{
    uint32_t H = 0, r = g;
    int c = nh - 1;
    for (int t = hl; t >= 1; --t) {
        while (bt[c][t] > r) --c;
        H |= 1u << c;
        r -= bt[c][t];
        --c;
    }
    return H;
}

// Tile g of level hl within the sub-lattice whose top kfix of the nh tile
// bits are rfix (a shard of a job split by its top variables; kfix = 0: the
// whole level).
__device__ __forceinline__ uint32_t level_tile(uint32_t g, int hl, int nh, uint32_t rfix, int kfix,
                                               const uint32_t (*bt)[BT])
{
    if (kfix == 0) return tile_of(g, hl, nh, bt);
    return tile_of(g, hl - __popc(rfix), nh - kfix, bt) | (rfix << (nh - kfix));
}

__device__ __forceinline__ void fill_table(uint32_t (*bt)[BT])
{
    for (int x = threadIdx.x; x < BT * BT; x += blockDim.x) bt[x / BT][x % BT] = g_binom_lanes.v[x / BT][x % BT];
}

// TLO (B = 4): the rows of A in tile-level order (see bn_device.cuh): a
// term across tiles reads row tlo_row(R, 9) of A_{B+j} (rows of 16 values,
// nine in-tile row bits); the in-tile rows of A_i (i < B: rows of 8 values,
// ten in-tile row bits) sit at tlo_row(Ht, 10).
//
// The 2^B values of F in tile Ht (its level's tiles of F already written):
//   F(S) = sum_{i in S} A_i(S - {i}) F(S - {i}),  F(empty) = 1
//
// rebase: the previous level's stored values are relative to a base larger by
// this much than this level's (the FP32 per-level bases, bn_device.cuh; 0
// otherwise).  Returns the largest value written.
//
// SLAB (a split job with divided A): A holds the rank's slabs of the nl = n -
// k low nodes, each over the nl - 1 low bits of its index (the top k bits are
// the rank's); Atop holds, for each top variable t = nl + q, its slab over
// the nl low variables.  A term of a low node reads its slab with the top
// bits of the row index dropped; a term of a top variable reads Atop.
template <typename T, int B, bool TLO = false, bool SLAB = false>
__device__ __forceinline__ T forward_tile(int n, uint32_t Ht, const T* __restrict__ A,
                                          T* __restrict__ F, T rebase = T{}, int nl = 0,
                                          const T* __restrict__ Atop = nullptr)
{
    constexpr int LN = 1 << B;
    [[maybe_unused]] const size_t full = (size_t)1 << n;
    const size_t half = (size_t)1 << ((SLAB ? nl : n) - 1);
    const uint32_t rmask = SLAB ? (1u << (nl - 1 - B)) - 1u : ~0u;   // slab row bits
    const uint32_t lmask = SLAB ? (1u << (nl - B)) - 1u : ~0u;       // low tile bits

    TileSum<T> s[LN];
    // terms across tiles: i = B + j for the set bits j of Ht
    for (uint32_t rest = Ht; rest; rest &= rest - 1) {
        const int j = __ffs(rest) - 1;
        const uint32_t Hm = Ht & ~(1u << j);
        T a[LN], f[LN];
        if (SLAB && B + j >= nl) {                  // a top variable: its slab
            load_row(Atop + BN_AT(((size_t)(B + j - nl) << nl) + ((size_t)(Ht & lmask) << B), LN,
                                  (size_t)(n - nl) << nl),
                     a, LD_STREAM);
        } else {
            const uint32_t row = TLO ? tlo_row(squeeze(Hm, j) & rmask, 9) : squeeze(Hm, j) & rmask;
            load_row(A + BN_AT((size_t)(B + j) * half + ((size_t)row << B), LN,
                               (SLAB ? nl : n) * half),
                     a, LD_STREAM);
        }
        load_row(F + BN_AT((size_t)Hm << B, LN, full), f, LD_PLAIN);
#pragma unroll
        for (int l = 0; l < LN; ++l) s[l].add(a[l], f[l]);
    }
    // the cross-tile sums moved to this level's base
#pragma unroll
    for (int l = 0; l < LN; ++l) s[l].rebase(rebase);
    // terms inside the tile: A_i(S - {i}) for i < B, 2^(B-1) values per i
    T ai[B][LN / 2];
#pragma unroll
    for (int i = 0; i < B; ++i)
        load_row(A + BN_AT((size_t)i * half + ((size_t)(TLO ? tlo_row(Ht & lmask, 10) : Ht & lmask) << (B - 1)),
                           LN / 2, (SLAB ? nl : n) * half),
                 ai[i], LD_STREAM);
    T Fv[LN];
    Fv[0] = Ht == 0u ? unit<T>() : s[0].value();
#pragma unroll
    for (int l = 1; l < LN; ++l) {
#pragma unroll
        for (int i = 0; i < B; ++i)
            if (l >> i & 1) s[l].add(ai[i][squeeze4(l ^ (1 << i), i)], Fv[l ^ (1 << i)]);
        Fv[l] = s[l].value();
    }
    store_row(F + BN_AT((size_t)Ht << B, LN, full), Fv);
    T mx = Fv[0];
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int l = 1; l < LN; ++l) mx = Fv[l] > mx ? Fv[l] : mx;
    }
    return mx;
}

// The 2^B values of R' in tile Ht (the tiles of the level above written):
//   R'(T) = sum_{i not in T} A_i(T) R'(T + {i}),  R'(V) = 1
template <typename T, int B, bool TLO = false, bool SLAB = false>
__device__ __forceinline__ T backward_tile(int n, uint32_t Ht, const T* __restrict__ A,
                                           T* __restrict__ Rc, T rebase = T{}, int nl = 0,
                                           const T* __restrict__ Atop = nullptr)
{
    constexpr int LN = 1 << B;
    const int nh = n - B;
    const uint32_t hmask = (1u << nh) - 1u;
    const size_t full = (size_t)1 << n;
    const size_t half = (size_t)1 << ((SLAB ? nl : n) - 1);
    const uint32_t rmask = SLAB ? (1u << (nl - 1 - B)) - 1u : ~0u;
    const uint32_t lmask = SLAB ? (1u << (nl - B)) - 1u : ~0u;

    TileSum<T> s[LN];
    for (uint32_t rest = ~Ht & hmask; rest; rest &= rest - 1) {
        const int j = __ffs(rest) - 1;
        T a[LN], r[LN];
        if (SLAB && B + j >= nl) {
            load_row(Atop + BN_AT(((size_t)(B + j - nl) << nl) + ((size_t)(Ht & lmask) << B), LN,
                                  (size_t)(n - nl) << nl),
                     a, LD_STREAM);
        } else {
            const uint32_t row = TLO ? tlo_row(squeeze(Ht, j) & rmask, 9) : squeeze(Ht, j) & rmask;
            load_row(A + BN_AT((size_t)(B + j) * half + ((size_t)row << B), LN,
                               (SLAB ? nl : n) * half),
                     a, LD_STREAM);
        }
        load_row(Rc + BN_AT((size_t)(Ht | (1u << j)) << B, LN, full), r, LD_PLAIN);
#pragma unroll
        for (int l = 0; l < LN; ++l) s[l].add(a[l], r[l]);
    }
#pragma unroll
    for (int l = 0; l < LN; ++l) s[l].rebase(rebase);
    // A_i(T) for i < B not in T, 2^(B-1) values per i
    T ai[B][LN / 2];
#pragma unroll
    for (int i = 0; i < B; ++i)
        load_row(A + BN_AT((size_t)i * half + ((size_t)(TLO ? tlo_row(Ht & lmask, 10) : Ht & lmask) << (B - 1)),
                           LN / 2, (SLAB ? nl : n) * half),
                 ai[i], LD_STREAM);
    T Rv[LN];
    Rv[LN - 1] = Ht == hmask ? unit<T>() : s[LN - 1].value();
#pragma unroll
    for (int l = LN - 2; l >= 0; --l) {
#pragma unroll
        for (int i = 0; i < B; ++i)
            if (!(l >> i & 1)) s[l].add(ai[i][squeeze4(l, i)], Rv[l | (1 << i)]);
        Rv[l] = s[l].value();
    }
    store_row(Rc + BN_AT((size_t)Ht << B, LN, full), Rv);
    T mx = Rv[0];
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int l = 1; l < LN; ++l) mx = Rv[l] > mx ? Rv[l] : mx;
    }
    return mx;
}

// The largest value a block wrote for its level, floored, into the level's
// word (one atomic per block; every thread of the block calls this).
__device__ __forceinline__ void block_level_max(int* word, float mx)
{
    __shared__ int wm[8];
    int v = __reduce_max_sync(0xffffffffu, level_floor(mx));
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = max(v, wm[w]);
        if (v != kLevelUnset) atomicMax(word, v);
    }
}
// The first level of a sweep (one tile, one thread) starts the level words.
__device__ __forceinline__ void level_words_start(int* lw, int level, float mx)
{
    for (int k = 0; k < kLevelMode; ++k) lw[k] = kLevelUnset;
    lw[kLevelMode] = kLevelShift;
    lw[level] = level_floor(mx);
}

}  // namespace

// FP32: 16-subset tiles at three blocks per SM (80 registers); FP64:
// 8-subset tiles at two.
//
// FP32 keeps the per-level bases (bn_device.cuh): level hl reads the
// previous level's word (its values' base minus this level's base), and
// every block adds its largest written value to the level's word.
template <typename T, bool TLO, bool SLAB = false>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 2)
k_forward_rows(int n, int hl, uint32_t ntiles, const T* __restrict__ A, T* __restrict__ F,
               size_t js, uint32_t rfix, int kfix, const T* __restrict__ Atop)
{
    constexpr int B = sizeof(T) == 4 ? LB : LB64;
    constexpr bool kBases = sizeof(T) == 4;
    A = job_ptr(A, js);
    F = job_ptr(F, js);
    __shared__ uint32_t bt[BT][BT];
    fill_table(bt);
    __syncthreads();
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (kBases) {
        int* lw = level_words(reinterpret_cast<float*>(F), n);
        const T rebase = hl > 0 ? (T)level_delta(lw, hl - 1) : T(0);
        T mx = LogOps<T>::ninf();
        if (g < ntiles)
            mx = forward_tile<T, B, TLO, SLAB>(n, level_tile(g, hl, n - B, rfix, kfix, bt), A, F, rebase,
                                               n - kfix, Atop);
        if (hl == 0) {
            if (g == 0) level_words_start(lw, 0, mx);
        } else {
            block_level_max(lw + hl, mx);
        }
    } else {
        if (g >= ntiles) return;
        forward_tile<T, B, TLO, SLAB>(n, level_tile(g, hl, n - B, rfix, kfix, bt), A, F, T{}, n - kfix, Atop);
    }
}

template <typename T, bool TLO, bool SLAB = false>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 2)
k_backward_rows(int n, int hl, uint32_t ntiles, const T* __restrict__ A, T* __restrict__ Rc,
                size_t js, uint32_t rfix, int kfix, const T* __restrict__ Atop)
{
    constexpr int B = sizeof(T) == 4 ? LB : LB64;
    constexpr bool kBases = sizeof(T) == 4;
    A = job_ptr(A, js);
    Rc = job_ptr(Rc, js);
    __shared__ uint32_t bt[BT][BT];
    fill_table(bt);
    __syncthreads();
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (kBases) {
        const int nh = n - B;
        int* lw = level_words(reinterpret_cast<float*>(Rc), n);
        const T rebase = hl < nh ? (T)level_delta(lw, hl + 1) : T(0);
        T mx = LogOps<T>::ninf();
        if (g < ntiles)
            mx = backward_tile<T, B, TLO, SLAB>(n, level_tile(g, hl, nh, rfix, kfix, bt), A, Rc, rebase,
                                                n - kfix, Atop);
        if (hl == nh) {
            if (g == 0) level_words_start(lw, nh, mx);
        } else {
            block_level_max(lw + hl, mx);
        }
    } else {
        if (g >= ntiles) return;
        backward_tile<T, B, TLO, SLAB>(n, level_tile(g, hl, n - B, rfix, kfix, bt), A, Rc, T{}, n - kfix, Atop);
    }
}

// F and R' of one or more jobs in one launch, every popcount level of a sweep
// separated by a barrier of the blocks that share it, instead of a launch per
// level.  A level launch of a job up to n of about 20 took 9 to 12 us, nearly
// all of it latency: the launch itself and one thread walking a tile's terms,
// each a dependent pair of row loads.  Here a tile's 16 (FP64: 8) subsets take several lanes
// (one value each, or a short vector), a lane issues the loads of up to eight (four) terms together,
// and the first tile's index and A values for the next level are fetched
// between arriving at the barrier and waiting on it.  The sums run in the
// order of forward_tile / backward_tile, so the results are the same bits.
//
// Item it (2 per job: F, then R') is shared by nb blocks.  R' is F's recursion
// read from the full set down: with bits = the elements of S (F) or the
// missing ones (R'), step st takes the tiles with st of them, a term per
// element j reads A_j at S without j and the neighbour tile S ^ {j}.
//
// SYNC 0: nb = 1, the block's own barrier.  SYNC 1: the item's blocks are one
// thread-block cluster (co-resident by construction; hardware barrier).
// SYNC 2: a cooperative launch (all blocks resident); a block arrives by an
// atomic on its sweep's counter and polls it, at most `cap` times: past that
// it sets kErrDeviceTimeout in *err and returns, and so does every other block
// of the sweep when its own wait runs out.  sync[0] / sync[16] count the
// arrivals of F / R', sync[8] / sync[24] the blocks done (the last resets
// both); they start at zero (k_step1_prep).
enum { SYNC_BLOCK = 0, SYNC_CLUSTER = 1, SYNC_GRID = 2 };

// N consecutive values (N * sizeof(T) bytes, aligned to them) by load mode;
// rev: in reverse order.
template <typename T, int N>
__device__ __forceinline__ void load_vals(const T* p, T (&v)[N], int mode, bool rev)
{
    if constexpr (N == 1) {
        v[0] = load_one(p, mode);
    } else if constexpr (sizeof(T) * N == 8) {      // two floats
        const float2* q = reinterpret_cast<const float2*>(p);
        const float2 x = mode == LD_STREAM ? __ldcs(q) : mode == LD_L2 ? __ldcg(q) : *q;
        v[0] = x.x;
        v[1] = x.y;
    } else {
        load_row(p, v, mode);
    }
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
        const T lo = v[k], hi = v[N - 1 - k];
        v[k] = rev ? hi : lo;
        v[N - 1 - k] = rev ? lo : hi;
    }
}
template <typename T, int N>
__device__ __forceinline__ void store_vals(T* p, const T (&v)[N], bool rev)
{
    T w[N];
#pragma unroll
    for (int k = 0; k < N; ++k) w[k] = rev ? v[N - 1 - k] : v[k];
    if constexpr (N == 1) *p = w[0];
    else store_row(p, w);
}

// VB: a lane holds the 2^VB values whose VB lowest bits vary (0: one value;
// 2, a 16-byte vector, in FP32).  One value per lane has the shortest chain,
// the faster form while latency bounds a level; vectors share the addresses,
// the index walk and half of the in-tile steps, the faster form once the
// levels are wide: n = 19 103 us (one value) and 117 (vectors), n = 20 145 and
// 135, n = 21 240 and 199.  (FP64 pairs were slower throughout: n = 20 232 us
// and 287.)
template <int VB> struct SweepShape {
    static constexpr int threads = VB ? 256 : 512;
    static constexpr int blocks = VB ? 3 : 2;       // resident per SM
};

template <typename T, bool TLO, int SYNC, int VB>
__global__ void __launch_bounds__(SweepShape<VB>::threads, SweepShape<VB>::blocks)
k_sweeps(int n, int nb, const T* __restrict__ A, T* __restrict__ F, T* __restrict__ Rc, size_t js,
         unsigned* __restrict__ sync, int* __restrict__ err, uint32_t cap)
{
    constexpr int B = sizeof(T) == 4 ? LB : LB64;
    constexpr int NV = 1 << VB, LNB = B - VB, LN = 1 << LNB;   // values per lane, lanes per tile
    constexpr int CH = sizeof(T) == 4 && VB == 0 ? 8 : 4;      // terms loaded together
    constexpr bool kBases = sizeof(T) == 4;
    constexpr int XMODE = SYNC == SYNC_BLOCK ? LD_PLAIN : LD_L2;
    __shared__ uint32_t bt[BT][BT];
    __shared__ int wm[SweepShape<VB>::threads / 32];
    __shared__ int ok_s;
    __shared__ uint16_t place[TLO ? 512 : 1];
    fill_table(bt);
    if (TLO)
        for (int x = threadIdx.x; x < 512; x += blockDim.x) place[x] = g_place.p9[x];
    __syncthreads();
    const int it = (int)(blockIdx.x / (unsigned)nb);
    const uint32_t rank = blockIdx.x % (unsigned)nb;
    const bool fwd = (it & 1) == 0;
    const size_t off = (size_t)(it >> 1) * js;
    A = reinterpret_cast<const T*>(reinterpret_cast<const char*>(A) + off);
    T* X = reinterpret_cast<T*>(reinterpret_cast<char*>(fwd ? F : Rc) + off);
    const int nh = n - B;
    const uint32_t hmask = (1u << nh) - 1u;
    const size_t half = (size_t)1 << (n - 1), full = (size_t)1 << n;
    // the lane's subsets: in-tile bits (l << VB) | r; value e has the in-lane
    // elements e (R': the missing ones, so the values sit in reverse order)
    const int l = threadIdx.x & (LN - 1);
    const uint32_t own = fwd ? (uint32_t)l : (uint32_t)l ^ (LN - 1);   // the lane's elements
    const int size = __popc(own);
    const unsigned tmask = (LN == 32 ? ~0u : (1u << LN) - 1u) << (threadIdx.x & 31 & ~(LN - 1));   // the tile's lanes
    // the groups of LN lanes number across the blocks: a narrow level spreads over them
    const uint32_t hw = (threadIdx.x >> LNB) * (uint32_t)nb + rank;
    const uint32_t nhw = (blockDim.x >> LNB) * (uint32_t)nb;
    int* lw = kBases ? level_words(reinterpret_cast<float*>(X), n) : nullptr;
    unsigned* arr = SYNC == SYNC_GRID ? sync + (fwd ? 0 : 16) : nullptr;

    // Places are 32-bit (n <= kSweepPlacesN).  That of the lane's values in the row
    // S-without-j of A_{B + j}, u = 1 << j: H with bit j squeezed out is
    // (H >> 1) with the bits below j taken from H.
    auto a_at = [&](uint32_t H, uint32_t u) {
        const uint32_t up = H >> 1, R = up ^ ((up ^ H) & (u - 1u));
        const uint32_t row = TLO ? (R & ~511u) | place[R & 511u] : R;
        return BN_AT(((uint32_t)(B + 31 - __clz(u)) << (n - 1)) + (row << B) + (l << VB), NV, n * half);
    };
    // the row of A_i (i < B) that the tile's in-tile terms read: for an in-lane
    // element i NV / 2 values, for a lane element NV
    auto in_at = [&](uint32_t H, int i) {
        const int at = i < VB ? l << (VB - 1) : squeeze4(l, i - VB) << VB;
        return BN_AT(((uint32_t)i << (n - 1)) + ((TLO ? tlo_row(H, 10) : H) << (B - 1)) + at,
                     i < VB ? (NV + 1) / 2 : NV, n * half);
    };
    // a group's run of tiles in step st: consecutive in colex order, so
    // only the first is unranked.  Its bits, the A values of its first terms
    // and of its in-tile terms are fetched ahead of the step.
    uint32_t bits = 0, g0 = 0, g1 = 0;
    constexpr bool kAhead = VB == 0;                // (vectors: more registers, one block fewer)
    T pa[kAhead ? CH : 1][NV], pin[VB ? VB : 1][NV > 1 ? NV / 2 : 1], plane[LNB][NV];
    auto load_a = [&](uint32_t H, uint32_t& rest, int st, T (&a)[CH][NV]) {
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            if (q < st) {
                load_vals(A + a_at(H, rest & (0u - rest)), a[q], LD_STREAM, !fwd);
                rest &= rest - 1;
            }
        }
    };
    auto load_in = [&](uint32_t H) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if (i < VB) load_vals(A + in_at(H, i), pin[i < VB ? i : 0], LD_STREAM, !fwd);
            else load_vals(A + in_at(H, i), plane[i < VB ? 0 : i - VB], LD_STREAM, !fwd);
        }
    };
    auto ahead = [&](int st) {
        const uint32_t nt = bt[nh][st], run = (nt + nhw - 1) / nhw;
        g0 = hw * run;
        g1 = min(nt, g0 + run);
        if (g0 >= g1) return;
        bits = tile_of(g0, st, nh, bt);
        if constexpr (kAhead) {
            const uint32_t H = fwd ? bits : hmask ^ bits;
            uint32_t rest = bits;
            load_a(H, rest, st, pa);
            load_in(H);
        }
    };
    ahead(0);
    for (int st = 0; st <= nh; ++st) {
        float mx = LogOps<float>::ninf();
        T rebase{};
        if constexpr (kBases)
            if (st > 0) {
                const int w = SYNC == SYNC_BLOCK ? *(volatile int*)(lw + (fwd ? st - 1 : nh - st + 1))
                                                 : __ldcg(lw + (fwd ? st - 1 : nh - st + 1));
                rebase = w == kLevelUnset ? T(0) : (T)w;
            }
        for (uint32_t g = g0; g < g1; ++g) {
            const uint32_t H = fwd ? bits : hmask ^ bits;
            uint32_t ra = bits, rf = bits;
            TileSum<T> s[NV];
            for (int c0 = 0; c0 < st; c0 += CH) {
                T a[CH][NV], f[CH][NV];
#pragma unroll
                for (int q = 0; q < CH; ++q) {
#pragma unroll
                    for (int e = 0; e < NV; ++e) f[q][e] = T{};
                    if (c0 + q < st) {
                        load_vals(X + BN_AT(((H ^ (rf & (0u - rf))) << B) + (l << VB), NV, full), f[q], XMODE,
                                  !fwd);
                        rf &= rf - 1;
                    }
                }
                if (kAhead && g == g0 && c0 == 0) {
#pragma unroll
                    for (int q = 0; q < CH; ++q) {
#pragma unroll
                        for (int e = 0; e < NV; ++e) a[q][e] = pa[kAhead ? q : 0][e];
                        ra &= ra - 1;
                    }
                } else {
                    load_a(H, ra, st - c0, a);
                }
#pragma unroll
                for (int q = 0; q < CH; ++q)
#pragma unroll
                    for (int e = 0; e < NV; ++e) s[e].add(a[q][e], f[q][e], c0 + q < st);
            }
            if (!kAhead || g != g0) load_in(H);
            // the in-tile terms, in popcount order of the lane's elements: in
            // round k the lanes with k elements add theirs.  One value per lane:
            // the others add a left-out term, so a warp's lanes stay together
            T v[NV];
#pragma unroll
            for (int e = 0; e < NV; ++e) {
                s[e].rebase(rebase);
                v[e] = unit<T>();
            }
#pragma unroll
            for (int k = 0; k <= LNB; ++k) {
                T y[LNB][NV];
                if (k > 0) {
#pragma unroll
                    for (int i = 0; i < LNB; ++i)
#pragma unroll
                        for (int e = 0; e < NV; ++e) {
                            y[i][e] = shfl_one(tmask, v[e], 1 << i);
                            if (VB == 0) s[e].add(plane[i][e], y[i][e], size == k && (own >> i & 1));
                        }
                }
                if (size == k) {
#pragma unroll
                    for (int e = 0; e < NV; ++e) {
#pragma unroll
                        for (int i = 0; i < VB; ++i)
                            if (e >> i & 1) s[e].add(pin[i][squeeze4(e, i)], v[e ^ (1 << i)]);
                        if (VB > 0 && k > 0) {
#pragma unroll
                            for (int i = 0; i < LNB; ++i) s[e].add(plane[i][e], y[i][e], own >> i & 1);
                        }
                        if (k > 0 || e > 0 || st > 0) v[e] = s[e].value();
                    }
                }
            }
            store_vals(X + BN_AT((H << B) + (l << VB), NV, full), v, !fwd);
            if constexpr (kBases) {
#pragma unroll
                for (int e = 0; e < NV; ++e) mx = v[e] > mx ? v[e] : mx;
            }
            if (g + 1 < g1) {                       // the next tile of the run
                const uint32_t u = bits & (0u - bits), w = bits + u;
                bits = w | (((w ^ bits) >> 2) >> (__ffs(u) - 1));
            }
        }
        // the level's largest value, for the next level's base
        if constexpr (kBases) {
            const int lv = fwd ? st : nh - st;
            if (st == 0) {
                // the one tile of the first level: its lanes' maximum
                if (hw == 0) {
                    for (int o = LN / 2; o; o >>= 1) {
                        const float y = __shfl_xor_sync(tmask, mx, o);
                        mx = y > mx ? y : mx;
                    }
                    if (l == 0) level_words_start(lw, lv, mx);
                }
            } else {
                int v = __reduce_max_sync(0xffffffffu, level_floor(mx));
                if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = v;
                __syncthreads();
                if (threadIdx.x < 32) {
                    v = threadIdx.x < (blockDim.x >> 5) ? wm[threadIdx.x] : kLevelUnset;
                    v = __reduce_max_sync(0xffffffffu, v);
                    if (threadIdx.x == 0 && v != kLevelUnset) atomicMax(lw + lv, v);
                }
            }
        }
        if (st == nh) break;
        if constexpr (SYNC == SYNC_CLUSTER) {
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
            ahead(st + 1);
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        } else {
            __syncthreads();
            if (SYNC == SYNC_GRID && threadIdx.x == 0) {
                __threadfence();
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arr) : "memory");
            }
            ahead(st + 1);
            if constexpr (SYNC == SYNC_GRID) {
                if (threadIdx.x == 0) {
                    const unsigned need = (unsigned)nb * (unsigned)(st + 1);
                    uint32_t k = 0;
                    unsigned v;
                    do {
                        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arr) : "memory");
                    } while (v < need && ++k < cap);
                    if (v < need) atomicOr(err, kErrDeviceTimeout);
                    ok_s = v >= need;
                }
                __syncthreads();
                if (!ok_s) return;
            }
        }
    }
    if (SYNC == SYNC_GRID && threadIdx.x == 0 && atomicAdd(arr + 8, 1u) == (unsigned)nb - 1u) {
        arr[0] = 0u;                                // every block has passed its last wait
        arr[8] = 0u;
    }
}

// The rows (2^B values each) of one level's tiles of the sub-lattice rsrc
// (top kfix tile bits), in tile order: dir 0 copies them from X into buf,
// dir 1 from buf into X.  The exchange of a job split over several ranks.
template <typename T>
__global__ void k_level_rows(int n, int hl, uint32_t ntiles, uint32_t rsrc, int kfix, T* __restrict__ X,
                             T* __restrict__ buf, int dir)
{
    constexpr int B = sizeof(T) == 4 ? LB : LB64;
    __shared__ uint32_t bt[BT][BT];
    fill_table(bt);
    __syncthreads();
    const uint64_t total = (uint64_t)ntiles << B;
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < total;
         x += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t g = (uint32_t)(x >> B);
        const size_t pos = BN_AT(((size_t)level_tile(g, hl, n - B, rsrc, kfix, bt) << B) |
                                     (x & ((1u << B) - 1u)),
                                 1, (size_t)1 << n);
        if (dir == 0) buf[x] = X[pos];
        else X[pos] = buf[x];
    }
}

// ---------------------------------------------------------------------------
// A split job's divided A (Eq. 7 restricted to a rank's sub-lattice).  With
// the top k variables V_t = {nl, .., n - 1} (nl = n - k) fixed to the rank's
// bits r, every entry a rank's tiles read is a truncated zeta transform over
// the nl low variables alone:
//   low node i < nl:  A_i(r + L) = sum over G <= L of B'_i(G),
//                     B'_i(G) = sum over G_t <= r, |G_t| + |G| <= d of B_i(G_t + G);
//   top variable t:   A_t(r' + L), r' = r - {t}, L over all nl low variables,
//                     = X1(L - {0}) when 0 is not in L, X1 + X2 when it is,
//                     X1, X2 the transforms over the low variables but 0 of
//                     the families G_t + G (0 not in G) and G_t + G + {0},
//                     G_t <= r'.
// So a rank forms the folded score tables of a virtual job of nl variables
// with nl + 2k tables over the same nl - 1-bit index space (table i < nl:
// node i, bit i squeezed out; tables nl + 2q and nl + 2q + 1: X1 and X2 of
// top variable nl + q, bit 0 squeezed out), runs the step-2 kernels on it,
// and combines X1 and X2 into each top variable's slab.  No exchange is
// needed: the score table is small and every rank holds it.
// ---------------------------------------------------------------------------

// The folded tables, in the virtual job's canonical family order (Kv per
// table), from the job's shifted scores lbs (K per node, the same shift).
template <typename T> struct FoldSum {
    using L = LogOps<T>;
    T m = L::ninf(), s = T(0);
    __device__ __forceinline__ void add(T v)
    {
        if (v == L::ninf()) return;
        if (v > m) {
            s = s * L::ex(m - v) + T(1);
            m = v;
        } else {
            s += L::ex(v - m);
        }
    }
    __device__ __forceinline__ T value() const { return m == L::ninf() ? m : m + L::lg(s); }
};
template <> struct FoldSum<X64> : LazySum<X64> {};

template <typename T>
__global__ void k_fold_scores(int n, int nl, int d, int64_t K, int64_t Kv, uint32_t r,
                              const T* __restrict__ lbs, T* __restrict__ out)
{
    const int k = n - nl;
    const int64_t total = (int64_t)(nl + 2 * k) * Kv;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int u = (int)(x / Kv);
        uint32_t f = (uint32_t)(x % Kv);
        int sz = 0;
        while (f >= binom(nl - 1, sz)) { f -= binom(nl - 1, sz); ++sz; }
        const uint32_t cm = colex_unrank(f, sz, nl - 1);
        int node;
        uint32_t G, tops;
        if (u < nl) {
            node = u;
            G = expand(cm, u);                          // over the nl low variables
            tops = r;
        } else {
            const int q = (u - nl) >> 1;
            node = nl + q;
            G = (cm << 1) | (uint32_t)((u - nl) & 1);   // X2: variable 0 in the family
            tops = r & ~(1u << q);
        }
        const int g = __popc(G);
        FoldSum<T> sum;
        if (g <= d) {
            for (uint32_t t = tops;; t = (t - 1) & tops) {
                if (g + __popc(t) <= d) {
                    const uint32_t c = squeeze(G | (t << nl), node);   // node's own index
                    sum.add(lbs[BN_AT((size_t)node * K + small_subset_rank(c, n - 1), 1, (size_t)n * K)]);
                }
                if (t == 0) break;
            }
        }
        out[x] = sum.value();
    }
}

__device__ __forceinline__ float add_logs(float a, float b) { return LogOps<float>::lse(a, b); }
__device__ __forceinline__ double add_logs(double a, double b) { return LogOps<double>::lse(a, b); }
__device__ __forceinline__ X64 add_logs(X64 a, X64 b) { return x_add(a, b); }

// The top variables' slabs (plain order over the nl low variables) from the
// X1 and X2 tables of the virtual job's A (its own layout: tile-level row
// order when TLO, rows of 16 for tables >= 4).
template <typename T, bool TLO>
__global__ void k_top_slabs(int nl, int k, const T* __restrict__ Av, T* __restrict__ Atop)
{
    const size_t per = (size_t)1 << nl;
    const size_t half = per >> 1;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < per * (size_t)k;
         x += (size_t)gridDim.x * blockDim.x) {
        const size_t q = x >> nl;
        const uint32_t Lw = (uint32_t)(x & (per - 1));
        const uint32_t c = Lw >> 1;
        const uint32_t pos = TLO ? (tlo_row(c >> 4, 9) << 4) | (c & 15u) : c;
        const T* X1 = Av + (size_t)(nl + 2 * q) * half;
        T v = X1[BN_AT(pos, 1, half)];
        if (Lw & 1u) v = add_logs(v, X1[half + BN_AT(pos, 1, half)]);
        Atop[x] = v;
    }
}

// *word = max(*word, *other): another rank's floored level maximum.
__global__ void k_word_max(int* __restrict__ word, const int* __restrict__ other)
{
    if (threadIdx.x == 0 && *other != kLevelUnset) atomicMax(word, *other);
}

#ifndef BN_MEGA  // host launchers (bn_mega.cu includes only the device code)
#ifdef BN_CHECK_BOUNDS
BN_BOUNDS_READER(bounds_line_levels)
#endif
namespace {

uint64_t choose(int n, int k)
{
    if (k < 0 || k > n) return 0;
    uint64_t r = 1;
    for (int t = 1; t <= k; ++t) r = r * (uint64_t)(n - k + t) / (uint64_t)t;
    return r;
}

}  // namespace

bool rows_levels_fit(const Plan& P)
{
    return P.prec != 0 && P.n >= LB + 1 && P.n - LB < BT;
}

bool rows64_fit(const Plan& P)
{
    return P.prec == 0 && P.n >= LB64 + 1 && P.n - LB64 < BT;
}

// Threads per block for a level of nt tiles: 256, or fewer for the small
// levels, so that a level's blocks spread over all SMs (two per SM at least).
static unsigned level_block(uint32_t nt)
{
    for (unsigned b = 256; b > 64; b >>= 1)
        if ((uint64_t)nt >= (uint64_t)b * 2 * 152) return b;
    return 64;
}

uint32_t shard_level_tiles(const Plan& P, int hl)
{
    const int nh = P.n - (P.prec == 0 ? LB64 : LB);
    const int k = P.shard_k, hr = __builtin_popcount(P.shard_r);
    if (hl - hr < 0 || hl - hr > nh - k) return 0;
    return (uint32_t)choose(nh - k, hl - hr);
}

// One level of a split job's sweep: the rank's tiles (P.shard_r, P.shard_k).
// With P.slab, A holds the rank's slabs of the low nodes and Atop the top
// variables' slabs (the kernels' SLAB form, launched directly: a split job
// is never recorded into a batch).
template <typename T, bool TLO>
static cudaError_t rows_level(const Plan& P, int sweep, int hl, uint32_t nt, unsigned tb, dim3 grid,
                              const void* A, void* X, const void* Atop, cudaStream_t s)
{
    const uint32_t rf = P.shard_r;
    const int kf = P.shard_k;
    const T* a = (const T*)A;
    const T* at = (const T*)Atop;
    if (P.slab) {
        if (sweep == 0)
            k_forward_rows<T, TLO, true><<<grid, tb, 0, s>>>(P.n, hl, nt, a, (T*)X, P.js, rf, kf, at);
        else
            k_backward_rows<T, TLO, true><<<grid, tb, 0, s>>>(P.n, hl, nt, a, (T*)X, P.js, rf, kf, at);
        return cudaGetLastError();
    }
    const int kid = std::is_same<T, X64>::value ? (sweep == 0 ? KID_FROWS_X : KID_BROWS_X)
                    : sizeof(T) == 8 ? (sweep == 0 ? KID_FROWS_D : KID_BROWS_D)
                    : TLO ? (sweep == 0 ? KID_FROWS_F_TLO : KID_BROWS_F_TLO)
                          : (sweep == 0 ? KID_FROWS_F : KID_BROWS_F);
    if (sweep == 0)
        return launch_or_record(kid, k_forward_rows<T, TLO>, grid, tb, 0, s, P.n, hl, nt, a, (T*)X, P.js,
                                rf, kf, at);
    return launch_or_record(kid, k_backward_rows<T, TLO>, grid, tb, 0, s, P.n, hl, nt, a, (T*)X, P.js, rf,
                            kf, at);
}

cudaError_t launch_rows_level(const Plan& P, int sweep, int hl, const void* A, void* X, cudaStream_t s,
                              const void* Atop)
{
    const uint32_t nt = shard_level_tiles(P, hl);
    if (nt == 0) return cudaSuccess;
    const unsigned tb = rec_block(level_block(nt));
    const dim3 grid((nt + tb - 1) / tb, P.nj);
    if (P.lin) return rows_level<X64, false>(P, sweep, hl, nt, tb, grid, A, X, Atop, s);
    if (P.prec == 0) return rows_level<double, false>(P, sweep, hl, nt, tb, grid, A, X, Atop, s);
    if (use_tlo(P)) return rows_level<float, true>(P, sweep, hl, nt, tb, grid, A, X, Atop, s);
    return rows_level<float, false>(P, sweep, hl, nt, tb, grid, A, X, Atop, s);
}

cudaError_t launch_fold_scores(const Plan& P, int nl, int64_t Kv, uint32_t r, const void* lbs, void* out,
                               cudaStream_t s)
{
    const int64_t total = (int64_t)(nl + 2 * (P.n - nl)) * Kv;
    const unsigned grid = (unsigned)std::min<int64_t>((total + 255) / 256, 152 * 16);
    if (P.lin)
        k_fold_scores<X64><<<grid, 256, 0, s>>>(P.n, nl, P.d, P.K, Kv, r, (const X64*)lbs, (X64*)out);
    else if (P.prec == 0)
        k_fold_scores<double><<<grid, 256, 0, s>>>(P.n, nl, P.d, P.K, Kv, r, (const double*)lbs, (double*)out);
    else
        k_fold_scores<float><<<grid, 256, 0, s>>>(P.n, nl, P.d, P.K, Kv, r, (const float*)lbs, (float*)out);
    return cudaGetLastError();
}

cudaError_t launch_top_slabs(const Plan& V, int k, const void* Av, void* Atop, cudaStream_t s)
{
    const int nl = V.n;
    const uint64_t total = (uint64_t)k << nl;
    if (total == 0) return cudaSuccess;                 // no top variables (one rank)
    const unsigned grid = (unsigned)std::min<uint64_t>((total + 255) / 256, 152 * 16);
    if (V.lin)
        k_top_slabs<X64, false><<<grid, 256, 0, s>>>(nl, k, (const X64*)Av, (X64*)Atop);
    else if (V.prec == 0)
        k_top_slabs<double, false><<<grid, 256, 0, s>>>(nl, k, (const double*)Av, (double*)Atop);
    else if (use_tlo(V))
        k_top_slabs<float, true><<<grid, 256, 0, s>>>(nl, k, (const float*)Av, (float*)Atop);
    else
        k_top_slabs<float, false><<<grid, 256, 0, s>>>(nl, k, (const float*)Av, (float*)Atop);
    return cudaGetLastError();
}

cudaError_t launch_word_max(int* word, const int* other, cudaStream_t s)
{
    k_word_max<<<1, 32, 0, s>>>(word, other);
    return cudaGetLastError();
}

uint32_t shard_rows_count(const Plan& P, uint32_t r, int hl)
{
    Plan Q = P;
    Q.shard_r = r;
    return shard_level_tiles(Q, hl);
}

cudaError_t launch_level_rows(const Plan& P, uint32_t r, int hl, void* X, void* buf, int dir,
                              cudaStream_t s)
{
    const uint32_t nt = shard_rows_count(P, r, hl);
    if (nt == 0) return cudaSuccess;
    const unsigned grid = std::min<uint64_t>(((uint64_t)nt * 16 + 255) / 256, 152 * 8);
    if (P.prec == 0)
        k_level_rows<double><<<grid, 256, 0, s>>>(P.n, hl, nt, r, P.shard_k, (double*)X, (double*)buf, dir);
    else
        k_level_rows<float><<<grid, 256, 0, s>>>(P.n, hl, nt, r, P.shard_k, (float*)X, (float*)buf, dir);
    return cudaGetLastError();
}

// Every level of one sweep (0 F, 1 R'), a launch each.
static cudaError_t rows_sweep(const Plan& P, int sweep, const void* A, void* X, cudaStream_t s, int* launches)
{
    const int nh = P.n - (P.prec == 0 ? LB64 : LB);
    for (int st = 0; st <= nh; ++st) {
        const cudaError_t e = launch_rows_level(P, sweep, sweep == 0 ? st : nh - st, A, X, s);
        if (e != cudaSuccess) return e;
        if (launches) ++*launches;
    }
    return cudaSuccess;
}

cudaError_t launch_forward_rows(const Plan& P, const void* A, void* F, cudaStream_t s, int* launches)
{
    return rows_sweep(P, 0, A, F, s, launches);
}

cudaError_t launch_backward_rows(const Plan& P, const void* A, void* Rc, cudaStream_t s, int* launches)
{
    return rows_sweep(P, 1, A, Rc, s, launches);
}

// The instance of k_sweeps that a plan takes.
template <typename V, bool L, int W> struct SweepForm {
    using T = V;
    static constexpr bool TLO = L;
    static constexpr int VB = W;
    static constexpr int threads = SweepShape<W>::threads;
    static constexpr int tiles = threads >> ((sizeof(V) == 4 ? LB : LB64) - W);    // of a block at a time
};
template <typename F> static auto with_sweep_form(const Plan& P, F f)
{
    const bool vec = P.n >= kSweepVecN;
    if (P.lin) return f(SweepForm<X64, false, 0>{});
    if (use_tlo(P)) return vec ? f(SweepForm<float, true, 2>{}) : f(SweepForm<float, true, 0>{});
    return vec ? f(SweepForm<float, false, 2>{}) : f(SweepForm<float, false, 0>{});
}

static uint64_t widest_level(const Plan& P)
{
    const int nh = P.n - (P.prec == 0 ? LB64 : LB);
    return choose(nh, nh / 2);
}

// Whether the whole GPU shares the two sweeps of a single job: levels that
// fill more than kSweepGrid blocks.
static bool whole_gpu(const Plan& P, int tiles) { return widest_level(P) > kSweepGrid * tiles; }

// Blocks that share one item of k_sweeps: enough that every tile of the
// widest level has its own lanes.  Clusters (at most 8 blocks, the portable
// size) serve the small jobs and every batch group.  The whole-GPU form takes
// at most `resident` blocks over both items, what the device holds at a time (its
// blocks wait on one another); 0: too few for it.
static int sweep_blocks(const Plan& P, int tiles, bool whole, int resident)
{
    const uint64_t need = (widest_level(P) + tiles - 1) / tiles;
    if (!whole) return (int)std::max<uint64_t>(1, std::min<uint64_t>(need, 8));
    return resident / 2 > 8 ? (int)std::min<uint64_t>(need, resident / 2) : 0;
}

// Blocks of the whole-GPU form that the current device holds at a time, asked
// once per device; 0 where it has no cooperative launches.
template <typename Form> static int resident_blocks()
{
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices];        // the answer + 1
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev < kDevices && known[dev].load() > 0) return known[dev].load() - 1;
    int coop = 0, nsm = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, k_sweeps<typename Form::T, Form::TLO, SYNC_GRID, Form::VB>, Form::threads, 0) != cudaSuccess)
        return 0;
    const int r = coop ? nsm * std::min(per_sm, SweepShape<Form::VB>::blocks) : 0;
    if (dev < kDevices) known[dev].store(r + 1);
    return r;
}

int debug_sweep_blocks(const Plan& P, int sms, int* per_sm)
{
    return with_sweep_form(P, [&](auto f) {
        *per_sm = SweepShape<f.VB>::blocks;
        return sweep_blocks(P, f.tiles, whole_gpu(P, f.tiles), sms * SweepShape<f.VB>::blocks);
    });
}

bool sweeps_fit(const Plan& P)
{
    return ((rows_levels_fit(P) && P.frows) || P.lin) && P.n <= kSweepPlacesN && P.shard_k == 0 && !P.slab &&
           !P.spill;
}

bool use_sweeps(const Plan& P, const int* err)
{
    const int most = P.busy ? kSweepBusyN : P.lin ? kSweepMaxNX : kSweepMaxN;
    if (!sweeps_fit(P) || P.n > most || !err || recording()) return false;
    return with_sweep_form(P, [&](auto f) {
        return !whole_gpu(P, f.tiles) || sweep_blocks(P, f.tiles, true, resident_blocks<decltype(f)>()) > 0;
    });
}

template <typename Form>
static cudaError_t sweeps(const Plan& P, const void* Av, void* Fv, void* Rv, int items, cudaStream_t s, int* err)
{
    using T = typename Form::T;
    constexpr bool TLO = Form::TLO;
    constexpr int VB = Form::VB, threads = Form::threads;
    const T* A = static_cast<const T*>(Av);
    T *F = static_cast<T*>(Fv), *Rc = static_cast<T*>(Rv);
    // the whole-GPU form needs the counters beside the job's error word
    const bool whole = err && whole_gpu(P, Form::tiles);
    const int nb = sweep_blocks(P, Form::tiles, whole, whole ? resident_blocks<Form>() : 0);
    if (nb == 0) return cudaErrorCooperativeLaunchTooLarge;     // (use_sweeps answers no)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(items * nb), 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    cfg.attrs = attr;
    cfg.numAttrs = nb > 1 ? 1 : 0;
    unsigned* sync = err ? reinterpret_cast<unsigned*>(err) + 16 : nullptr;
    if (nb == 1)
        return cudaLaunchKernelEx(&cfg, k_sweeps<T, TLO, SYNC_BLOCK, VB>, P.n, nb, A, F, Rc, P.js, sync, err, 0u);
    if (!whole) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = nb;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        return cudaLaunchKernelEx(&cfg, k_sweeps<T, TLO, SYNC_CLUSTER, VB>, P.n, nb, A, F, Rc, P.js, sync, err, 0u);
    }
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    return cudaLaunchKernelEx(&cfg, k_sweeps<T, TLO, SYNC_GRID, VB>, P.n, nb, A, F, Rc, P.js, sync, err,
                              kSweepSpinCap);
}

cudaError_t launch_sweeps(const Plan& P, const void* A, void* F, void* Rc, cudaStream_t s, int* err,
                          int* launches)
{
    if (P.n > kSweepPlacesN) return cudaErrorInvalidValue;
    const int items = Rc ? 2 * P.nj : 1;            // a feature's job: F alone
    const cudaError_t e =
        with_sweep_form(P, [&](auto f) { return sweeps<decltype(f)>(P, A, F, Rc, items, s, err); });
    if (e == cudaSuccess && launches) ++*launches;
    return e;
}

// Test hook: F of n = kWithheldN in the whole-GPU form with the last of its
// blocks missing, so that the others' first wait runs out after `polls` polls.
cudaError_t launch_sweeps_withheld(const float* A, float* F, int* err, uint32_t polls, cudaStream_t s)
{
    k_sweeps<float, false, SYNC_GRID, 0><<<kWithheldBlocks - 1, SweepShape<0>::threads, 0, s>>>(
        kWithheldN, kWithheldBlocks, A, F, nullptr, 0, reinterpret_cast<unsigned*>(err) + 16, err, polls);
    return cudaGetLastError();
}

#endif  // BN_MEGA

}  // namespace bn
