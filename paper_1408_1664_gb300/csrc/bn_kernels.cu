// bn_kernels.cu -- sm_103a kernels of steps 2 to 5 of Algorithm 1 (step 1 is in
// bn_scores.cu).
//
// Step 2  k_upzeta         truncated upward zeta (Eq. 7, Definition 1)
// Step 3  k_forward_level, k_backward_level   F (Eq. 9) and R (Eq. 10)
// Step 4  k_gamma_p1, k_gamma_p2, ..p2r, ..p2s, ..p2w   truncated downward zeta (Eq. 12)
// Step 5  k_edges          Eq. 11 and the division by P(D); k_tail: steps 4 and 5 for n < 14
//
// Values are base-2 logs in FP32 and the numbers themselves with a wide exponent
// in FP64 (X64), or natural logs where their range is not bounded (see
// bn_device.cuh, lin_range).  Every node's scores are shifted by their maximum c_i
// before step 2: replacing B_i by B_i / exp(c_i) scales every order's weight
// by the same factor prod_i exp(-c_i), which cancels in P(u->v | D), and
// keeps the log magnitudes of A, F, R and Gamma small.
#include "bn_device.cuh"
#include "bn_kernels.cuh"

#include <algorithm>
#include <cmath>

namespace bn {

static constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ unsigned long long to_fixed(double x) { return __double2ull_rn(x); }
__device__ __forceinline__ unsigned long long to_fixed(float x) { return __float2ull_rn(x); }
template <typename T> __device__ __forceinline__ T from_fixed(unsigned long long u);
template <> __device__ __forceinline__ double from_fixed<double>(unsigned long long u)
{
    return __ull2double_rn(u);
}
template <> __device__ __forceinline__ float from_fixed<float>(unsigned long long u)
{
    return __ull2float_rn(u);
}

// ===========================================================================
// Step 2: A_i(S) = sum_{G subset S, |G| <= d} B_i(G)  (Eq. 7, q_i = 1).
//
// Index space of node i: the n-1 bits of S with bit i removed.  One block per
// tile (i, H): H = the high n-1-b bits, the 2^b low-bit patterns L in shared
// memory.  The high dimensions of the transform are done by scattering every
// family G = (g_L, G_H) with G_H subset H into slot g_L (log-sum-exp via two
// shared-memory atomic passes: max, then sum of exp); the b low dimensions
// are then summed in shared memory one dimension at a time (the butterfly of
// Algorithm 2).  Every family has |G| <= d, so the truncation is exact; A is
// written to HBM exactly once, coalesced.
// ===========================================================================
template <typename T>
__global__ void __launch_bounds__(256)
k_upzeta(int n, int b, int64_t K, int qbits, const uint32_t* __restrict__ cmasks,
         const T* __restrict__ lbs, T* __restrict__ A, size_t js)
{
    cmasks = job_ptr(cmasks, js);
    lbs = job_ptr(lbs, js);
    A = job_ptr(A, js);
    using O = typename OrdInt<T>::type;
    using U = unsigned long long;
    using L = LogOps<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t tileN = 1u << b;
    U* sm = reinterpret_cast<U*>(smem_raw);
    T* vals = reinterpret_cast<T*>(sm + tileN);
    O* mx = reinterpret_cast<O*>(vals + tileN);
    const int h = n - 1 - b;
    const int i = (int)(blockIdx.x >> h);
    const uint32_t H = blockIdx.x & ((1u << h) - 1u);
    const uint32_t lowm = tileN - 1u;
    const O enc_ninf = ord_enc(L::ninf());
    const T qscale = (T)ldexp(1.0, qbits);

    for (uint32_t t = threadIdx.x; t < tileN; t += blockDim.x) {
        mx[t] = enc_ninf;
        sm[t] = 0ull;
    }
    __syncthreads();
    const uint32_t* cm_i = cmasks + (size_t)i * K;
    const T* lb_i = lbs + (size_t)i * K;
    for (int64_t f = threadIdx.x; f < K; f += blockDim.x) {
        const uint32_t c = cm_i[f];
        if (((c >> b) & ~H) == 0u) atomicMax(&mx[c & lowm], ord_enc(lb_i[f]));
    }
    __syncthreads();
    // Sum of exp(value - slot max) in fixed point: every term is in (0, 1] and
    // a slot holds at most K terms, so 2^qbits * K < 2^64; integer atomics
    // make the sum independent of the order of arrival.
    for (int64_t f = threadIdx.x; f < K; f += blockDim.x) {
        const uint32_t c = cm_i[f];
        if (((c >> b) & ~H) == 0u) {
            const uint32_t slot = c & lowm;
            const T e = L::ex(lb_i[f] - ord_dec(mx[slot]));
            atomicAdd(&sm[slot], to_fixed(e * qscale));
        }
    }
    __syncthreads();
    for (uint32_t t = threadIdx.x; t < tileN; t += blockDim.x) {
        const O e = mx[t];
        vals[t] = (e == enc_ninf) ? L::ninf()
                                  : ord_dec(e) + L::lg(from_fixed<T>(sm[t]) / qscale);
    }
    __syncthreads();
    for (int j = 0; j < b; ++j) {
        const uint32_t jm = (1u << j) - 1u;
        for (uint32_t p = threadIdx.x; p < (tileN >> 1); p += blockDim.x) {
            const uint32_t lo = ((p & ~jm) << 1) | (p & jm);
            const uint32_t hi = lo | (1u << j);
            vals[hi] = L::lse(vals[hi], vals[lo]);
        }
        __syncthreads();
    }
    T* out = A + ((size_t)i << (n - 1)) + ((size_t)H << b);
    for (uint32_t t = threadIdx.x; t < tileN; t += blockDim.x) out[t] = vals[t];
}

// ===========================================================================
// Step 3: F and R' = R(V - .) over the lattice, level by level.
//
// A warp owns a tile of 2^wb consecutive subsets (the low wb bits vary, one
// subset per lane).  Tiles are keyed by their high bits Ht and launched one
// popcount level of Ht at a time (the sub-cube order of Section 3.2.2).
// Terms across tiles read the previous level's tiles; the wb in-tile levels
// are resolved with warp shuffles.
//   F(S)  = sum_{i in S}     A_i(S - {i}) F(S - {i}),  F(empty) = 1  (Eq. 9)
//   R'(T) = sum_{i not in T} A_i(T) R'(T + {i}),       R'(V) = 1
// where R'(T) = R(V - T) turns Eq. 10 into a recursion over T.
// ===========================================================================
// Next subset with the same number of elements in increasing value order
// (the colexicographic successor); x != 0.
__device__ __forceinline__ uint32_t colex_next(uint32_t x)
{
    const uint32_t u = x & (0u - x);
    const uint32_t v = x + u;
    return v | (((v ^ x) >> 2) >> (__ffs(u) - 1));
}

// Branchless online log-sum-exp step: (m, s) represents m + lg(s).
template <typename T>
__device__ __forceinline__ void lse_step(T& m, T& s, T x)
{
    using L = LogOps<T>;
    const T mn = x > m ? x : m;
    if (mn == L::ninf()) return;
    s = s * L::ex(m - mn) + L::ex(x - mn);
    m = mn;
}

// A warp owns 2^wb consecutive subsets (one per lane); the tile's high bits
// Ht are the same for every lane, so the terms across tiles run over the set
// bits of Ht with warp-uniform addresses.  Each warp walks `tpw` tiles in
// colexicographic order of Ht.  A is read once, with a streaming hint so
// that F and R' stay in L2 for the next level.
template <typename T>
__global__ void __launch_bounds__(256)
k_forward_level(int n, int wb, int hl, uint32_t ntiles, int tpw, const T* __restrict__ A,
                T* __restrict__ F, size_t js)
{
    A = job_ptr(A, js);
    F = job_ptr(F, js);
    using L = LogOps<T>;
    // FP32: these tiles keep no per-level bases (bn_device.cuh)
    if (sizeof(T) == 4 && hl == 0 && blockIdx.x == 0 && threadIdx.x == 0)
        level_words(reinterpret_cast<float*>(F), n)[kLevelMode] = 0;
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t first = warp * (uint32_t)tpw;
    if (first >= ntiles) return;
    const int nh = n - wb;
    const uint32_t lb = (uint32_t)lane & ((1u << wb) - 1u);
    const bool active = lane < (1 << wb);
    const size_t half = (size_t)1 << (n - 1);
    uint32_t Ht = colex_unrank(first, hl, nh);
    for (uint32_t tile = first; tile < ntiles && tile < first + (uint32_t)tpw; ++tile) {
        const uint32_t S = (Ht << wb) | lb;
        // terms across tiles: i = wb + j for the set bits j of Ht (same for all lanes)
        T m = L::ninf(), sm = T(0);
        uint32_t rest = Ht;
        const int cnt = __popc(Ht);
#pragma unroll 4
        for (int q = 0; q < cnt; ++q) {
            const int j = __ffs(rest) - 1;
            rest &= rest - 1;
            const uint32_t Hm = Ht & ~(1u << j);
            const T* Ai = A + (size_t)(wb + j) * half + ((size_t)squeeze(Hm, j) << wb);
            const T* Fi = F + ((size_t)Hm << wb);
            if (active) lse_step(m, sm, __ldcs(Ai + lb) + Fi[lb]);
        }
        const T X = (m == L::ninf()) ? m : m + L::lg(sm);
        T a[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            a[i] = L::ninf();
            if (i < wb && active && (S >> i & 1u))
                a[i] = __ldcs(A + (size_t)i * half + squeeze(S & ~(1u << i), i));
        }
        T Fv = (S == 0u) ? T(0) : X;
        for (int l = 1; l <= wb; ++l) {
            T nb[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) nb[i] = __shfl_xor_sync(FULL, Fv, 1 << i);
            if (active && __popc(lb) == l) {
                T mm = X, ss = (X == L::ninf()) ? T(0) : T(1);
#pragma unroll
                for (int i = 0; i < 5; ++i)
                    if (lb >> i & 1u) lse_step(mm, ss, a[i] + nb[i]);
                Fv = mm + L::lg(ss);
            }
        }
        if (active) F[BN_AT(S, 1, (size_t)1 << n)] = Fv;
        if (Ht) Ht = colex_next(Ht);
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
k_backward_level(int n, int wb, int hl, uint32_t ntiles, int tpw, const T* __restrict__ A,
                 T* __restrict__ Rc, size_t js)
{
    A = job_ptr(A, js);
    Rc = job_ptr(Rc, js);
    using L = LogOps<T>;
    if (sizeof(T) == 4 && hl == n - wb && blockIdx.x == 0 && threadIdx.x == 0)
        level_words(reinterpret_cast<float*>(Rc), n)[kLevelMode] = 0;
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t first = warp * (uint32_t)tpw;
    if (first >= ntiles) return;
    const int nh = n - wb;
    const uint32_t wmask = (1u << wb) - 1u;
    const uint32_t lb = (uint32_t)lane & wmask;
    const bool active = lane < (1 << wb);
    const uint32_t full = (uint32_t)(((uint64_t)1 << n) - 1);   // n <= 32
    const uint32_t hmask = (1u << nh) - 1u;
    const size_t half = (size_t)1 << (n - 1);
    uint32_t Ht = colex_unrank(first, hl, nh);
    for (uint32_t tile = first; tile < ntiles && tile < first + (uint32_t)tpw; ++tile) {
        const uint32_t Tm = (Ht << wb) | lb;
        T m = L::ninf(), sm = T(0);
        uint32_t rest = ~Ht & hmask;
        const int cnt = __popc(rest);
#pragma unroll 4
        for (int q = 0; q < cnt; ++q) {
            const int j = __ffs(rest) - 1;
            rest &= rest - 1;
            const T* Ai = A + (size_t)(wb + j) * half + ((size_t)squeeze(Ht, j) << wb);
            const T* Ri = Rc + ((size_t)(Ht | (1u << j)) << wb);
            if (active) lse_step(m, sm, __ldcs(Ai + lb) + Ri[lb]);
        }
        const T X = (m == L::ninf()) ? m : m + L::lg(sm);
        T a[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            a[i] = L::ninf();
            if (i < wb && active && !(Tm >> i & 1u)) a[i] = __ldcs(A + (size_t)i * half + squeeze(Tm, i));
        }
        T Rv = (Tm == full) ? T(0) : X;
        for (int l = wb - 1; l >= 0; --l) {
            T nb[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) nb[i] = __shfl_xor_sync(FULL, Rv, 1 << i);
            if (active && __popc(lb) == l) {
                T mm = X, ss = (X == L::ninf()) ? T(0) : T(1);
#pragma unroll
                for (int i = 0; i < 5; ++i)
                    if (i < wb && !(lb >> i & 1u)) lse_step(mm, ss, a[i] + nb[i]);
                Rv = mm + L::lg(ss);
            }
        }
        if (active) Rc[BN_AT(Tm, 1, (size_t)1 << n)] = Rv;
        if (Ht) Ht = colex_next(Ht);
    }
}

// ===========================================================================
// Step 4: Gamma_v(G) = sum_{G subset S subset V-{v}} F(S) R'(S + {v}), |G|<=d
// (Eq. 12; F(S) R(V-{v}-S) = F(S) R'(S + {v}), the pairing of Section 3.1.2).
//
// Phase 1: one block per tile of the n-1 bits of S (bit v removed), 2^b low
// bits in shared memory: load s_v = F + R', run the downward butterflies over
// the b low dimensions with the guard of Algorithm 3 (only patterns with at
// most d elements among the dimensions done so far), and keep the outputs
// with at most d low elements: row H of W, nlow entries in canonical order.
// Phase 2: one block per column g of W (a low pattern, d' = d - |g|): the
// downward transform over the h high dimensions, truncated at d', chunk by
// chunk of 2^hc rows; each output is stored at its family index.
// ===========================================================================
template <typename T>
__global__ void __launch_bounds__(256)
k_gamma_p1(int n, int d, int b, uint32_t nlow, const T* __restrict__ F,
           const T* __restrict__ Rc, T* __restrict__ W, size_t js, const T* __restrict__ lq,
           uint32_t vsel)
{
    const int v = blockIdx.z;                       // endpoint: one slice of W each
    if (!(vsel >> v & 1u)) return;                  // an endpoint another rank computes
    F = job_ptr(F, js);
    Rc = job_ptr(Rc, js);
    W = job_ptr(W, js) + (size_t)endpoint_slot(vsel, v) * gridDim.x * nlow;
    using L = LogOps<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* vals = reinterpret_cast<T*>(smem_raw);
    const uint32_t tileN = 1u << b;
    const uint32_t H = blockIdx.x;
    const uint32_t bv = 1u << v;
    constexpr bool kBases = sizeof(T) == 4;         // FP32: per-level bases of F and R'
    __shared__ float off_s[32];
    __shared__ int sh_s;
    __shared__ float fvrel_s;
    if constexpr (kBases) {
        load_gamma_offsets(reinterpret_cast<const float*>(Rc), n, v, off_s, &sh_s, &fvrel_s);
        __syncthreads();
    }
    for (uint32_t t = threadIdx.x; t < tileN; t += blockDim.x) {
        const uint32_t S = expand((H << b) | t, v);
        vals[t] = F[BN_AT(S, 1, (size_t)1 << n)] + Rc[BN_AT(S | bv, 1, (size_t)1 << n)];
        if constexpr (kBases) vals[t] += off_s[BN_AT(__popc(S >> sh_s), 1, 32)];
        if (lq) vals[t] += lq[v * n + __popc(S)];   // q_v(S) of Eq. 12
    }
    __syncthreads();
    for (int j = 0; j < b; ++j) {
        const uint32_t jm = (1u << j) - 1u;
        for (uint32_t p = threadIdx.x; p < (tileN >> 1); p += blockDim.x) {
            const uint32_t lo = ((p & ~jm) << 1) | (p & jm);
            if (__popc(lo & jm) <= d) vals[lo] = L::lse(vals[lo], vals[lo | (1u << j)]);
        }
        __syncthreads();
    }
    T* row = W + (size_t)H * nlow;
    for (uint32_t t = threadIdx.x; t < tileN; t += blockDim.x)
        if (__popc(t) <= d) row[BN_AT(small_subset_rank(t, b), 1, nlow)] = vals[t];
}

// FP32: the down-zeta offsets of endpoint blockIdx.x (one warp; bn_device.cuh).
__global__ void k_gamma_table(int n, const float* __restrict__ F, float* __restrict__ Rc, size_t js,
                              uint32_t vsel)
{
    F = job_ptr(F, js);
    Rc = job_ptr(Rc, js);
    const int v = blockIdx.x;
    if (!(vsel >> v & 1u)) return;
    __shared__ float off[32];
    __shared__ int sh;
    __shared__ float fvrel;
    if (threadIdx.x < 32) off[threadIdx.x] = 0.f;
    __syncwarp();
    gamma_offsets(n, v, F, Rc, off, &sh, &fvrel);
    __syncwarp();
    float* tab = gamma_table(Rc, n) + v * 32;
    const int l = threadIdx.x;
    tab[l] = l < 30 ? off[l] : l == 30 ? __int_as_float(sh) : fvrel;
}

__device__ __forceinline__ float p2_add(float a, float b) { return LogOps<float>::lse(a, b); }
__device__ __forceinline__ double p2_add(double a, double b) { return LogOps<double>::lse(a, b); }
__device__ __forceinline__ X64 p2_add(X64 a, X64 b) { return x_add(a, b); }
__device__ __forceinline__ void p2_zero(float& a) { a = LogOps<float>::ninf(); }
__device__ __forceinline__ void p2_zero(double& a) { a = LogOps<double>::ninf(); }
__device__ __forceinline__ void p2_zero(X64& a) { a.u = 0ull; }

template <typename T>
__global__ void __launch_bounds__(256)
k_gamma_p2(int n, int d, int b, int hc, uint32_t nlow, int64_t K, const T* __restrict__ W,
           T* __restrict__ Gam, size_t js, uint32_t vsel)
{
    const int v = blockIdx.z;                       // endpoint: its slice of W, its K outputs
    if (!(vsel >> v & 1u)) return;
    W = job_ptr(W, js) + ((size_t)endpoint_slot(vsel, v) << (n - 1 - b)) * nlow;
    Gam = job_ptr(Gam, js) + (size_t)v * K;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int h = n - 1 - b;
    const int hh = h - hc;
    const uint32_t col = blockIdx.x;
    // low pattern g of this column
    int kg = 0;
    uint32_t r = col;
    while (r >= binom(b, kg)) { r -= binom(b, kg); ++kg; }
    const uint32_t g = colex_unrank(r, kg, b);
    const int dp = d - kg;
    const uint32_t nout = num_small_subsets(h, dp);
    const uint32_t chunkN = 1u << hc;
    T* vals = reinterpret_cast<T*>(smem_raw);
    T* acc = vals + chunkN;
    uint32_t* gh = reinterpret_cast<uint32_t*>(acc + nout);
    for (uint32_t o = threadIdx.x; o < nout; o += blockDim.x) {
        uint32_t ro = o;
        int k = 0;
        while (ro >= binom(h, k)) { ro -= binom(h, k); ++k; }
        gh[o] = colex_unrank(ro, k, h);
        p2_zero(acc[o]);
    }
    const uint32_t lowc = chunkN - 1u;
    for (uint32_t Hhi = 0; Hhi < (1u << hh); ++Hhi) {
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < chunkN; t += blockDim.x)
            vals[t] = W[BN_AT((size_t)((Hhi << hc) | t) * nlow + col, 1, ((size_t)nlow << h))];
        __syncthreads();
        for (int j = 0; j < hc; ++j) {
            const uint32_t jm = (1u << j) - 1u;
            for (uint32_t p = threadIdx.x; p < (chunkN >> 1); p += blockDim.x) {
                const uint32_t lo = ((p & ~jm) << 1) | (p & jm);
                if (__popc(lo & jm) <= dp) vals[lo] = p2_add(vals[lo], vals[lo | (1u << j)]);
            }
            __syncthreads();
        }
        for (uint32_t o = threadIdx.x; o < nout; o += blockDim.x) {
            const uint32_t G = gh[o];
            if (((G >> hc) & ~Hhi) == 0u) acc[o] = p2_add(acc[o], vals[G & lowc]);
        }
    }
    __syncthreads();
    for (uint32_t o = threadIdx.x; o < nout; o += blockDim.x) {
        const uint32_t cm = g | (gh[o] << b);      // mask over the n-1 bits of V-{v}
        const int k = __popc(cm);
        uint32_t f = 0;
        for (int s = 0; s < k; ++s) f += binom(n - 1, s);
        int t = 1;
        for (uint32_t x = cm; x; x &= x - 1, ++t) f += binom(__ffs(x) - 1, t);
        Gam[BN_AT(f, 1, K)] = acc[o];
    }
}

// Phase 2 for the columns with at least two high elements left, a block per
// endpoint and run of CPB consecutive columns: the 2^h values of each column
// sit in shared memory (one column after another, the columns' starts four
// banks apart), the downward steps run three dimensions at a time in registers
// (eight values per thread) and the outputs with at most d - |g| high elements
// go to their families.  A run of columns reads whole sectors of W's rows and
// a step touches shared memory once per three dimensions (n = 22, d = 8: phase 2
// 612 us with a block per column and a step per dimension, k_gamma_p2, and 277
// here; p2r_columns has the other sizes).
//
// The steps are additions relative to one scale (an exponential per input, a
// logarithm per output resolved), in one or a few passes like the tiles': a
// pass resolves the outputs of at least 2^low in its scale, the next moves
// down by the range.  A column's outputs lie between W at the full high set
// and the largest input times 2^h, and those below L = log2 F(V) - margin -
// log2 (sum of B_v) move no posterior (the cut of phase 1 with the largest
// set): the passes end at max(W(full), L).  Columns that would take more than
// kP2Passes passes sum logarithms instead.
template <bool LIN>
__device__ __forceinline__ void p2_steps(float* v, uint32_t H2, uint32_t HS, int h, int cpb)
{
    for (int j0 = 0; j0 < h; j0 += 3) {
        const int nb = min(3, h - j0);
        const uint32_t lowm = (1u << j0) - 1u;
        const uint32_t np = H2 >> nb;
        for (uint32_t g = threadIdx.x; g < np * cpb; g += blockDim.x) {
            const uint32_t cc = g >> (h - nb), p = g & (np - 1u);
            const uint32_t base = cc * HS + (((p & ~lowm) << nb) | (p & lowm));
            float x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < (1 << nb)) x[q] = v[base + ((uint32_t)q << j0)];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                if (k >= nb) continue;
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < (1 << nb) && !(q >> k & 1)) {
                        if constexpr (LIN) x[q] = x[q] + x[q | (1 << k)];
                        else x[q] = p2_add(x[q], x[q | (1 << k)]);
                    }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < (1 << nb)) v[base + ((uint32_t)q << j0)] = x[q];
        }
        __syncthreads();
    }
}

// Logarithms and sums in the scale of an integer (2^ref, as the sums of a
// pass).  The integer part of a logarithm goes straight into the exponent and
// back: w - ref itself is rounded to the bits of a number of up to 126 (2^-18)
// where w may have more, and so is the logarithm of a sum of up to 2^126.
__device__ __forceinline__ int p2_mag(float w) { return w > -2.0e9f ? (int)floorf(w) : -2000000000; }
__device__ __forceinline__ float p2_pow2(int k)    // 2^k; 0 below 2^-126, +inf above 2^127
{
    return __uint_as_float((unsigned)(min(max(k, -127), 128) + 127) << 23);
}
struct P2Scale {
    // w - ref is exact from |ref| = 2^21 on; below, the integer part of w comes
    // from an addition that rounds to it (1.5 2^23: the low bits hold it)
    float base, low;
    int bias;
    __device__ __forceinline__ explicit P2Scale(int ref)
    {
        const bool wide = abs(ref) > (1 << 21);
        base = wide ? (float)ref : 0.0f;
        const int i = wide ? 0 : ref;
        low = (float)(i - 127);
        bias = 127 - i;
    }
    // 2^(w - ref): 0 below 2^-126, +inf above 2^127 (TOP: w may lie there)
    template <bool TOP> __device__ __forceinline__ float value(float w) const
    {
        w = fmaxf(w - base, low);
        if (TOP) w = fminf(w, low + 255.0f);
        const float t = w + 12582912.0f;
        return ex2_approx(w - (t - 12582912.0f)) * __uint_as_float((unsigned)(__float_as_int(t) + bias) << 23);
    }
};
__device__ __forceinline__ float p2_log(float s, int ref)      // s at least 2^-126
{
    const int b = __float_as_int(s);
    return (float)(ref + (b >> 23) - 127) + lg2_approx(__int_as_float((b & 0x7fffff) | 0x3f800000));
}
// Largest sum and smallest exact output of a pass, in bits above its
// reference (Window<float> of bn_tile13.cu).
constexpr int kP2Top = 126, kP2Low = -80;
constexpr float kP2Keep = 8.271806125530277e-25f;  // 2^-80
constexpr int kP2Passes = 4;

template <int CPB>
__global__ void __launch_bounds__(256)
k_gamma_p2r(int n, int d, int b, uint32_t nlow, uint32_t c0, int64_t K, const float* __restrict__ W,
            float* __restrict__ Gam, const float* __restrict__ Aup, const float* __restrict__ lq, int margin, size_t js, uint32_t vsel)
{
    const int v = blockIdx.z;
    if (!(vsel >> v & 1u)) return;
    const int h = n - 1 - b;
    const uint32_t H2 = 1u << h, HS = H2 + 4;
    W = job_ptr(W, js) + ((size_t)endpoint_slot(vsel, v) << h) * nlow;
    Gam = job_ptr(Gam, js) + (size_t)v * K;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* vals = reinterpret_cast<float*>(smem_raw);
    __shared__ uint32_t hb[18][20];                 // C(b + bit, t)
    __shared__ int mag_s[CPB], ref_s[CPB], span_s;
    __shared__ uint32_t base_s[CPB], soff[20];
    __shared__ int kg_s[CPB];
    const int tid = threadIdx.x;
    const uint32_t cb = blockIdx.x * CPB;
    const int cols = min((uint32_t)CPB, c0 - cb);
    for (int x = tid; x < 18 * 20; x += blockDim.x) hb[x / 20][x % 20] = binom(b + x / 20, x % 20);
    if (tid < CPB) {
        mag_s[tid] = -2000000000;
        int kg = 0;
        uint32_t r = cb + min(tid, cols - 1);
        while (r >= binom(b, kg)) { r -= binom(b, kg); ++kg; }
        kg_s[tid] = kg;
        base_s[tid] = r;                            // its rank among the kg-subsets
    }
    if (tid < 20) {
        uint32_t o = 0;
        for (int s = 0; s < tid; ++s) o += binom(n - 1, s);
        soff[tid] = o;
    }
    if (tid == 0) span_s = 0;
    __syncthreads();
    // blockDim.x is a multiple of CPB: a thread's column is fixed in these loops
    const int mycol = tid % CPB;
    const float* Wc = W + cb + min(mycol, cols - 1);
    int mag = -2000000000;
    for (uint32_t H = tid / CPB; H < H2; H += blockDim.x / CPB)
        mag = max(mag, p2_mag(Wc[BN_AT((size_t)H * nlow, 1, (size_t)nlow << h)]));
    atomicMax(&mag_s[mycol], mag);
    __syncthreads();
    if (tid < CPB) {
        int L = -2000000000;
        if (Aup) {
            // log2 F(V), in [0, 1) relative to the integer Z, and the sum of B_v
            // over all parent sets: A_v(V - {v}) without its factor q_v (a zero
            // factor is held as -1.4e7, in units of 1)
            const float at = job_ptr(Aup, js)[BN_AT(((size_t)(v + 1) << (n - 1)) - 1, 1, (size_t)n << (n - 1))];
            const int av = p2_mag(at) - (lq ? p2_mag(lq[v * n + n - 1]) - 4 : 0);
            L = -av - 2 - margin;
        }
        const int top = mag_s[tid] + h + 2;         // every output is below 2^top
        const int low = max(L, p2_mag(Wc[BN_AT((size_t)(H2 - 1) * nlow, 1, (size_t)nlow << h)]));
        ref_s[tid] = top - kP2Top;
        atomicMax(&span_s, top - low);
    }
    __syncthreads();
    constexpr int range = kP2Top - kP2Low;
    const int span = span_s;
    const int passes = span <= range ? 1 : span <= kP2Passes * range ? (span + range - 1) / range : 0;
    unsigned long long done = 0ull;                 // bit i: the thread's i-th output is written
    for (int pass = 0; pass < max(passes, 1); ++pass) {
        const int down = pass * range;
        const bool last = pass + 1 >= passes;
        const P2Scale sc(ref_s[mycol] - down);
        for (uint32_t H = tid / CPB; H < H2; H += blockDim.x / CPB) {
            const float w = Wc[BN_AT((size_t)H * nlow, 1, (size_t)nlow << h)];
            vals[mycol * HS + H] = passes ? sc.value<true>(w) : w;
        }
        __syncthreads();
        if (passes) p2_steps<true>(vals, H2, HS, h, cols);
        else p2_steps<false>(vals, H2, HS, h, cols);
        int i = 0;
        for (uint32_t e = tid; e < H2 * cols; e += blockDim.x, ++i) {
            const uint32_t cc = e >> h, t = e & (H2 - 1u);
            const int kg = kg_s[cc], k = kg + __popc(t);
            if (k > d || (done >> (i & 63) & 1ull)) continue;
            float o = vals[cc * HS + t];
            if (passes) {
                if (!last && o < kP2Keep) continue;
                // a sum flushed in the last pass is irrelevant: kept finite
                const int ref = ref_s[cc] - down;
                o = o < 1.1754943508222875e-38f ? (float)(ref - 126) : p2_log(o, ref);
                done |= 1ull << (i & 63);
            }
            // family index of g with the high part t: sizes below k, then the
            // colex rank (the low part's, then one entry per high bit)
            uint32_t f = base_s[cc] + soff[k];
            int pos = kg + 1;
            for (uint32_t x = t; x; x &= x - 1, ++pos) f += hb[__ffs(x) - 1][pos];
            Gam[BN_AT(f, 1, K)] = o;
        }
        __syncthreads();                            // the values are reused
    }
}

// Family index of the mask cm over the n-1 bits of V - {v}: by size, then
// colexicographic rank (the canonical order of the scores).
__device__ __forceinline__ uint32_t family_index(uint32_t cm, int n)
{
    const int k = __popc(cm);
    uint32_t f = 0;
    for (int s = 0; s < k; ++s) f += binom(n - 1, s);
    int t = 1;
    for (uint32_t x = cm; x; x &= x - 1, ++t) f += binom(__ffs(x) - 1, t);
    return f;
}

// Lazy log-sum-exp step (one exponential per term): (m, s) is m + log(s).
template <typename T>
__device__ __forceinline__ void lse_lazy_k(T& m, T& s, T x)
{
    using L = LogOps<T>;
    const T dd = x - m;                             // +inf while empty
    const bool big = dd > T(64);
    const T e = L::ex(big ? -dd : dd);
    s = big ? s * e + T(1) : s + e;
    m = big ? x : m;
}

// Warp-wide log-sum of the lanes' (m, s), in a fixed tree order.
template <typename T>
__device__ __forceinline__ T warp_lse(T m, T s)
{
    using L = LogOps<T>;
    for (int o = 16; o; o >>= 1) {
        const T m2 = __shfl_xor_sync(FULL, m, o);
        const T s2 = __shfl_xor_sync(FULL, s, o);
        const T mn = m2 > m ? m2 : m;
        if (mn != L::ninf()) {
            s = s * L::ex(m - mn) + s2 * L::ex(m2 - mn);
            m = mn;
        }
    }
    return m + L::lg(s);
}

// Phase 2 for the columns whose low pattern g has at least d - 1 elements
// (d' = d - |g| <= 1, at most one high element left): the outputs are
// Gamma(g) = log-sum of W[H][g] over every H and, for d' = 1, Gamma(g + {b})
// = log-sum over the H that contain b, for every high bit b -- the truncated
// transform over the high dimensions, written out.  One warp per column,
// eight consecutive columns per block (they share the sectors of W's rows).
// Lane l takes the rows H = l + 32k: high bits 0-4 are its lane bits, the
// bits from 5 up are summed per lane.
template <typename T>
__global__ void __launch_bounds__(256)
k_gamma_p2s(int n, int d, int b, uint32_t nlow, uint32_t c0, int64_t K, const T* __restrict__ W,
            T* __restrict__ Gam, size_t js, uint32_t vsel)
{
    constexpr int MB = 14;                          // high bits from 5 up (h <= 18, n <= 32)
    const int v = blockIdx.z;
    if (!(vsel >> v & 1u)) return;
    W = job_ptr(W, js) + ((size_t)endpoint_slot(vsel, v) << (n - 1 - b)) * nlow;
    Gam = job_ptr(Gam, js) + (size_t)v * K;
    using L = LogOps<T>;
    const int h = n - 1 - b;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t col = c0 + blockIdx.x * 8 + warp;
    if (col >= nlow) return;                        // whole warps leave
    int kg = 0;
    uint32_t r = col;
    while (r >= binom(b, kg)) { r -= binom(b, kg); ++kg; }
    const uint32_t g = colex_unrank(r, kg, b);
    const bool one = d - kg == 1;
    T m0 = L::ninf(), s0 = T(0);
    T mb[MB], sb[MB];
#pragma unroll
    for (int q = 0; q < MB; ++q) { mb[q] = L::ninf(); sb[q] = T(0); }
    const uint32_t nH = 1u << h;
    const size_t wsize = (size_t)nlow << h;
    // the rows two and three steps ahead are in flight while a row is added
    // (the loop waits on load latency, each lane reading its own row; four
    // rows ahead cost registers: 61 against 48, one block per SM fewer)
    T wa = lane < nH ? W[BN_AT((size_t)lane * nlow + col, 1, wsize)] : T(0);
    T wb = lane + 32 < nH ? W[BN_AT((size_t)(lane + 32) * nlow + col, 1, wsize)] : T(0);
    for (uint32_t H = lane; H < nH; H += 32) {
        const T w = wa;
        wa = wb;
        if (H + 64 < nH) wb = W[BN_AT((size_t)(H + 64) * nlow + col, 1, wsize)];
        lse_lazy_k(m0, s0, w);
        if (one) {
#pragma unroll
            for (int q = 0; q < MB; ++q)
                if (5 + q < h && (H >> (5 + q) & 1u)) lse_lazy_k(mb[q], sb[q], w);
        }
    }
    const T all = warp_lse(m0, s0);
    if (lane == 0) Gam[BN_AT(family_index(g, n), 1, K)] = all;
    if (!one) return;
    for (int bb = 0; bb < h && bb < 5; ++bb) {
        const bool in = lane >> bb & 1;
        const T x = warp_lse(in ? m0 : L::ninf(), in ? s0 : T(0));
        if (lane == 0) Gam[BN_AT(family_index(g | (1u << (b + bb)), n), 1, K)] = x;
    }
#pragma unroll
    for (int q = 0; q < MB; ++q) {
        if (5 + q >= h) break;
        const T x = warp_lse(mb[q], sb[q]);
        if (lane == 0) Gam[BN_AT(family_index(g | (1u << (b + 5 + q)), n), 1, K)] = x;
    }
}

// The same columns in FP32 for h >= 8, a block per eight consecutive columns.
// A warp's load takes eight columns of four rows: four whole sectors, where a
// lane per row touched 32 (the L1 was 96 % busy with them).  Lane 8 r + c takes
// column c and the rows whose two lowest bits are r, warp w those whose three
// highest bits are w; the bits between are the loop's, the same for the whole
// warp, so eight rows at a time are summed over their three lowest loop bits
// and enter the other sums as one term.  A lane's sums share one scale: one
// exponential per row (one per sum before).  The scale lies 90 to 102 bits
// below the lane's largest value, which uses the upper part of the exponent
// range too: a sum 178 bits below the largest (2^-88 in its scale, where the
// terms flushed are below 2^-108 together) is still exact, as strongly
// dependent data need; one below that is formed again in logarithms by a warp.
__global__ void __launch_bounds__(256)
k_gamma_p2w(int n, int d, int b, uint32_t nlow, uint32_t c0, int64_t K, const float* __restrict__ W,
            float* __restrict__ Gam, size_t js, uint32_t vsel)
{
    constexpr int MB = 13;                          // loop bits (h <= 18)
    using L = LogOps<float>;
    const int v = blockIdx.z;
    if (!(vsel >> v & 1u)) return;
    W = job_ptr(W, js) + ((size_t)endpoint_slot(vsel, v) << (n - 1 - b)) * nlow;
    Gam = job_ptr(Gam, js) + (size_t)v * K;
    __shared__ float part[8][8][20];                // [warp][column][sum]
    __shared__ int scale_s[8][8];                   // [warp][column]
    __shared__ uint32_t g_s[8];
    __shared__ int redo_s[8];                       // per column: sums to form again
    const int h = n - 1 - b, hi = h - 5;            // hi: loop bits, 2 .. h - 4
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = lane & 7, r = lane >> 3;
    const uint32_t cb = c0 + blockIdx.x * 8;
    const int cols = min(8u, nlow - cb);
    const size_t wsize = (size_t)nlow << h;
    if (threadIdx.x < 8) {
        int kg = 0;
        uint32_t x = cb + min((int)threadIdx.x, cols - 1);
        while (x >= binom(b, kg)) { x -= binom(b, kg); ++kg; }
        g_s[threadIdx.x] = colex_unrank(x, kg, b);
        redo_s[threadIdx.x] = 0;
    }
    __syncthreads();
    // the last column's values stand in for those past the end
    const float* Wc = W + cb + min(c, cols - 1);
    const uint32_t base = ((uint32_t)warp << (h - 3)) | (uint32_t)r;
    int m = -(1 << 30);                             // the scale
    P2Scale sc(m);
    float s = 0.0f, sb[MB];
#pragma unroll
    for (int q = 0; q < MB; ++q) sb[q] = 0.0f;
    for (uint32_t k = 0; k < (1u << hi); k += 8) {
        float w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = Wc[BN_AT((size_t)(base + ((k + q) << 2)) * nlow, 1, wsize)];
        float top = w[0];
#pragma unroll
        for (int q = 1; q < 8; ++q) top = fmaxf(top, w[q]);
        const int mt = p2_mag(top);
        if (mt - m > 102) {
            const float r0 = p2_pow2((m - (mt - 90)) >> 1), r1 = p2_pow2((m - (mt - 90) + 1) >> 1);
            s = s * r0 * r1;
#pragma unroll
            for (int q = 0; q < MB; ++q) sb[q] = sb[q] * r0 * r1;
            m = mt - 90;
            sc = P2Scale(m);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = sc.value<false>(w[q]);
        const float p1 = w[2] + w[3], p2 = w[4] + w[5], p3 = w[6] + w[7];
        const float t = (w[0] + w[1]) + p1 + (p2 + p3);
        s += t;
        sb[0] += (w[1] + w[3]) + (w[5] + w[7]);
        sb[1] += p1 + p3;
        sb[2] += p2 + p3;
#pragma unroll
        for (int q = 3; q < MB; ++q)
            if (k >> q & 1u) sb[q] += t;
    }
    // over the four row phases: the largest scale, every sum relative to it
    int top = max(m, __shfl_xor_sync(FULL, m, 8));
    top = max(top, __shfl_xor_sync(FULL, top, 16));
    // in halves: the sums are up to 2^102
    const float r0 = p2_pow2((m - top) >> 1), r1 = p2_pow2((m - top + 1) >> 1);
    s = s * r0 * r1;
    const float s1 = s + __shfl_xor_sync(FULL, s, 16);      // phases r and r ^ 2
    const float s2 = s + __shfl_xor_sync(FULL, s, 8);       // phases r and r ^ 1
    const float all = s1 + __shfl_xor_sync(FULL, s1, 8);
    if (r == 3) {                                   // phases 1, 3 and 2, 3: bits 0 and 1
        scale_s[warp][c] = top;
        part[warp][c][0] = all;
        part[warp][c][1] = s1;
        part[warp][c][2] = s2;
    }
#pragma unroll
    for (int q = 0; q < MB; ++q) {
        if (q >= hi) break;
        float x = sb[q] * r0 * r1;
        x += __shfl_xor_sync(FULL, x, 16);
        x += __shfl_xor_sync(FULL, x, 8);
        if (r == 0) part[warp][c][3 + q] = x;
    }
    __syncthreads();
    // output o of column c: 0 every row, 1 + j the rows with high bit j
    auto store = [&](int col, int o, float x) {
        const uint32_t cm = g_s[col] | (o ? 1u << (b + o - 1) : 0u);
        Gam[BN_AT(family_index(cm, n), 1, K)] = x;
    };
    for (int x = threadIdx.x; x < 8 * (h + 1); x += blockDim.x) {
        const int col = x & 7, o = x >> 3;
        if (col >= cols || (o && d - __popc(g_s[col]) != 1)) continue;
        const int j = o - 1;                        // the high bit
        const int at = j < h - 3 ? o : 0;           // warp bits: sums of the warps with the bit
        int t = scale_s[0][col];
#pragma unroll
        for (int w = 1; w < 8; ++w) t = max(t, scale_s[w][col]);
        float sum = 0.0f;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const int k = scale_s[w][col] - t;
            if (j < h - 3 || (w >> (j - (h - 3)) & 1)) sum += part[w][col][at] * p2_pow2(k >> 1) * p2_pow2((k + 1) >> 1);
        }
        if (sum > 3.2311742677852644e-27f) store(col, o, p2_log(sum, t));     // 2^-88
        else atomicOr(&redo_s[col], 1 << o);
    }
    __syncthreads();
    for (int x = warp; x < 8 * (h + 1); x += 8) {
        const int col = x & 7, o = x >> 3;
        if (!(redo_s[col] >> o & 1)) continue;
        float mm = L::ninf(), ss = 0.0f;
        for (uint32_t H = lane; H < (1u << h); H += 32)
            if (H >> (o - 1) & 1u) lse_lazy_k(mm, ss, W[BN_AT((size_t)H * nlow + cb + col, 1, wsize)]);
        const float y = warp_lse(mm, ss);
        if (lane == 0) store(col, o, y);
    }
}

// ===========================================================================
// Step 5: P(u->v, D) = sum_{G: u in G} B_v(G) Gamma_v(G)  (Eq. 11) and
// P(u->v | D) = P(u->v, D) / P(D), in FP64, in one launch.
// Every term B_v(G) Gamma_v(G) is at most their sum over G, which is F(V)
// (Eq. 11 summed over all G), so e(G) = B_v(G) Gamma_v(G) / F(V) <= 1 (up to
// rounding) needs no maximum pass.  Blocks over (families of v, v) add e(G)
// in fixed point (2^qbits, integer atomics: the sums do not depend on the
// order of arrival) into acc[v*n + u] for every u in G and into acc[n*n + v]
// for all G; the last block to finish divides.  The FP64 path divides by F(V)
// (Algorithm 1), i.e. takes acc[v*n + u] / 2^qbits; the FP32 path divides by
// Z_v = acc[n*n + v] (the same quantity from the same Gamma_v, so rounding
// common to numerator and denominator cancels).  log P(D) = F~(V) + sum_i c_i.
// Most families weigh less than half a unit of the fixed point: they are
// left out by a comparison in the working precision, before the FP64
// exponential and the atomics (n = 25, d = 8: 31.8 M families, 2.06 -> 0.28 ms).
// ===========================================================================
// The weight e(G) 2^qbits of family x, rounded: 0 without an exponential when
// it is certainly below one half.
struct EdgeScale {
    double cv, lnfv, qscale, inv;                   // logs: c_v, ln F(V), 2^qbits; X64: 1 / F(V)'s fraction
    float cut;                                      // FP32: log2 of a weight that rounds to 0
    int eq;                                         // X64: qbits - F(V)'s exponent
};
__device__ __forceinline__ EdgeScale edge_scale(const float* F, int n, int qbits, double cv)
{
    // Gamma is relative to the integer Z = floor of log P(D) in the
    // level-based units (see gamma_offsets), so P(D) enters as F(V) - Z
    const double fv = (double)F[(uint32_t)(((uint64_t)1 << n) - 1)];   // n <= 32
    const double rel = fv - floor(fv);
    return {cv, LogOps<float>::to_ln(rel), ldexp(1.0, qbits), 0.0, (float)rel - (float)(qbits + 3), 0};
}
__device__ __forceinline__ EdgeScale edge_scale(const double* F, int n, int qbits, double cv)
{
    const double fv = F[(uint32_t)(((uint64_t)1 << n) - 1)];
    return {cv, fv, ldexp(1.0, qbits), 0.0, -0.69314718f * (float)(qbits + 3), 0};
}
__device__ __forceinline__ EdgeScale edge_scale(const X64* F, int n, int qbits, double)
{
    const X64 fv = F[(uint32_t)(((uint64_t)1 << n) - 1)];
    return {0.0, 0.0, 0.0, 1.0 / x_mant(fv), 0.f, qbits - x_exp(fv)};
}
__device__ __forceinline__ unsigned long long edge_weight(const EdgeScale& s, double logB, float lb, float g)
{
    // lb is log B - c_v in log2 units to a few 1e-4: three bits of margin
    if (lb + g < s.cut) return 0ull;
    return __double2ull_rn(exp(logB - s.cv + LogOps<float>::to_ln((double)g) - s.lnfv) * s.qscale);
}
__device__ __forceinline__ unsigned long long edge_weight(const EdgeScale& s, double logB, double, double g)
{
    const double x = logB - s.cv + g - s.lnfv;
    if (x < (double)s.cut) return 0ull;
    return __double2ull_rn(exp(x) * s.qscale);
}
__device__ __forceinline__ unsigned long long edge_weight(const EdgeScale& s, double, X64 b, X64 g)
{
    const int e = x_exp(b) + x_exp(g) + s.eq;       // the weight is at most 2^qbits
    return e < -8 ? 0ull : __double2ull_rn(x_mant(b) * x_mant(g) * s.inv * pow2d(min(e, 64)));
}

// ln F(V) of the shifted scores.
__device__ __forceinline__ double ln_full(const float* F, int n)
{
    // FP32: add the level base of F(V)
    return LogOps<float>::to_ln((double)F[((size_t)1 << n) - 1] +
                                level_base_fwd(level_words(F, n), n - kLevelShift));
}
__device__ __forceinline__ double ln_full(const double* F, int n) { return F[((size_t)1 << n) - 1]; }
__device__ __forceinline__ double ln_full(const X64* F, int n)
{
    const X64 f = F[((size_t)1 << n) - 1];
    return f.u ? (double)x_exp(f) * 0.69314718055994530942 + log(x_mant(f)) : -INFINITY;
}
template <typename T>
__device__ __forceinline__ double log_evidence(int n, const double* cmax, const T* F)
{
    double c = 0.0;
    for (int i = 0; i < n; ++i) c += cmax[i];
    return ln_full(F, n) + c;
}

// acc: n * (n + 1) sums, zero before the launch and left zero by it; acc[0]
// (no edge 0 -> 0) counts the finished blocks.
template <typename T>
__global__ void __launch_bounds__(256)
k_edges(int n, int64_t K, int qbits, const double* __restrict__ logB, const T* __restrict__ lbs,
        const double* __restrict__ cmax, const uint32_t* __restrict__ masks, const T* __restrict__ Gam,
        const T* __restrict__ F, const int* __restrict__ err, unsigned long long* __restrict__ acc,
        double* __restrict__ post, double* __restrict__ log_PD, size_t js, uint32_t vsel)
{
    // an endpoint another rank computes (a rank without any: its first block
    // still writes the zeros and log P(D))
    const int mine = __popc(vsel & (uint32_t)(((uint64_t)1 << n) - 1));
    if (!(vsel >> blockIdx.z & 1u) && (mine || blockIdx.x || blockIdx.z)) return;
    logB = job_ptr(logB, js);
    lbs = job_ptr(lbs, js);
    cmax = job_ptr(cmax, js);
    masks = job_ptr(masks, js);
    Gam = job_ptr(Gam, js);
    F = job_ptr(F, js);
    acc = job_ptr(acc, js);
    __shared__ unsigned long long Nu[32], Nz;
    __shared__ int last_s;
    const int v = blockIdx.z;
    const int tid = threadIdx.x;
    if (tid < 32) Nu[tid] = 0ull;
    if (tid == 0) Nz = 0ull;
    __syncthreads();
    const EdgeScale sc = edge_scale(F, n, qbits, cmax[v]);
    unsigned long long z = 0ull;
    for (int64_t f = mine ? blockIdx.x * (int64_t)blockDim.x + tid : K; f < K;
         f += (int64_t)gridDim.x * blockDim.x) {
        const size_t x = (size_t)v * K + f;
        const unsigned long long q = edge_weight(sc, logB[x], lbs[x], Gam[x]);
        if (q) {
            z += q;
            for (uint32_t g = masks[x]; g; g &= g - 1) atomicAdd(&Nu[BN_AT(__ffs(g) - 1, 1, 32)], q);
        }
    }
    for (int o = 16; o; o >>= 1) z += __shfl_xor_sync(FULL, z, o);
    if ((tid & 31) == 0) atomicAdd(&Nz, z);
    __syncthreads();
    if (tid < n && Nu[tid]) atomicAdd(&acc[(size_t)v * n + tid], Nu[tid]);
    if (tid == 0) atomicAdd(&acc[(size_t)n * n + v], Nz);
    __threadfence();                                // this block's sums before its count
    __syncthreads();
    if (tid == 0) {
        last_s = !mine || atomicAdd(&acc[0], 1ull) + 1ull == (unsigned long long)mine * gridDim.x;
        __threadfence();
    }
    __syncthreads();
    if (!last_s) return;
    err = job_ptr(err, js);
    post = job_ptr(post, js);
    log_PD = job_ptr(log_PD, js);
    const bool bad = err && *err;
    for (int t = tid; t < n * n; t += blockDim.x) {
        const int u = t / n, w = t % n;
        const unsigned long long num = __ldcg(acc + (size_t)w * n + u);
        double p = 0.0;
        if (u != w && num > 0ull)
            p = sizeof(T) == 4 ? __ull2double_rn(num) / __ull2double_rn(__ldcg(acc + (size_t)n * n + w))
                               : __ull2double_rn(num) / ldexp(1.0, qbits);
        post[t] = bad ? NAN : (vsel >> w & 1u) ? p : 0.0;   // other ranks' endpoints: 0
    }
    if (tid == 0 && log_PD) *log_PD = bad ? NAN : log_evidence(n, cmax, F);
    __syncthreads();
    for (int t = tid; t < n * (n + 1); t += blockDim.x) acc[t] = 0ull;
}

// Steps 4 and 5 for n < 14 in one launch, a block per endpoint v: the whole
// down-zeta of v fits one tile in shared memory (no phase 2), its families'
// Gamma come straight out of it, and the block divides its own column.  It
// replaces six launches (the FP32 offsets, two phases, three of step 5), about
// 45 of the 150 us of an n = 12 job.
__device__ __forceinline__ void tail_input(float& y, const float* F, const float* Rc, uint32_t S, uint32_t bv,
                                           size_t full, const float* off, int sh)
{
    y = F[BN_AT(S, 1, full)] + Rc[BN_AT(S | bv, 1, full)];
    y += off[BN_AT(__popc(S >> sh), 1, 32)];
}
__device__ __forceinline__ void tail_input(double& y, const double* F, const double* Rc, uint32_t S, uint32_t bv,
                                           size_t full, const float*, int)
{
    y = F[BN_AT(S, 1, full)] + Rc[BN_AT(S | bv, 1, full)];
}
__device__ __forceinline__ void tail_input(X64& y, const X64* F, const X64* Rc, uint32_t S,
                                           uint32_t bv, size_t full, const float*, int)
{
    y = x_mul(F[BN_AT(S, 1, full)], Rc[BN_AT(S | bv, 1, full)]);
}
__device__ __forceinline__ void apply_weight(float& a, float w) { a += w; }
__device__ __forceinline__ void apply_weight(double& a, double w) { a += w; }
__device__ __forceinline__ void apply_weight(X64& a, X64 w) { a = x_mul(a, w); }

template <typename T>
__global__ void __launch_bounds__(1024)
k_tail(int n, int d, int64_t K, int qbits, const T* __restrict__ F, const T* __restrict__ Rc,
       const T* __restrict__ lq, const double* __restrict__ logB, const T* __restrict__ lbs,
       const double* __restrict__ cmax, const uint32_t* __restrict__ masks,
       const uint32_t* __restrict__ cmasks, T* __restrict__ Gam, const int* __restrict__ err,
       double* __restrict__ post, double* __restrict__ log_PD, size_t js, uint32_t vsel)
{
    const int v = blockIdx.x;
    F = job_ptr(F, js);
    Rc = job_ptr(Rc, js);
    logB = job_ptr(logB, js);
    lbs = job_ptr(lbs, js);
    cmax = job_ptr(cmax, js);
    masks = job_ptr(masks, js);
    cmasks = job_ptr(cmasks, js);
    Gam = job_ptr(Gam, js);
    err = job_ptr(err, js);
    post = job_ptr(post, js);
    const int tid = threadIdx.x;
    const bool bad = err && *err;
    if (!(vsel >> v & 1u)) {                        // an endpoint another rank computes
        if (tid < n) post[(size_t)tid * n + v] = bad ? NAN : 0.0;
        if (tid == 0 && v == 0 && log_PD && !(vsel & (uint32_t)(((uint64_t)1 << n) - 1)))
            *job_ptr(log_PD, js) = bad ? NAN : log_evidence(n, cmax, F);
        return;
    }
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* vals = reinterpret_cast<T*>(smem_raw);
    __shared__ unsigned long long Nu[32], Nz;
    __shared__ float off_s[32];
    __shared__ int sh_s;
    __shared__ float fvrel_s;
    if (tid < 32) {
        Nu[tid] = 0ull;
        if (tid == 0) Nz = 0ull;
        if constexpr (sizeof(T) == 4) {             // FP32: the level bases of F and R'
            off_s[tid] = 0.f;
            __syncwarp();
            gamma_offsets(n, v, reinterpret_cast<const float*>(F), reinterpret_cast<const float*>(Rc), off_s, &sh_s,
                          &fvrel_s);
        }
    }
    __syncthreads();
    const uint32_t N = 1u << (n - 1);
    const size_t full = (size_t)1 << n;
    const int sh = sizeof(T) == 4 ? sh_s : 0;
    for (uint32_t t = tid; t < N; t += blockDim.x) {
        const uint32_t S = expand(t, v);
        T y;
        tail_input(y, F, Rc, S, 1u << v, full, off_s, sh);
        if (lq) apply_weight(y, lq[v * n + __popc(S)]);     // q_v(S) of Eq. 12
        vals[t] = y;
    }
    __syncthreads();
    for (int j = 0; j < n - 1; ++j) {
        const uint32_t jm = (1u << j) - 1u;
        for (uint32_t p = tid; p < (N >> 1); p += blockDim.x) {
            const uint32_t lo = ((p & ~jm) << 1) | (p & jm);
            if (__popc(lo & jm) <= d) vals[lo] = p2_add(vals[lo], vals[lo | (1u << j)]);
        }
        __syncthreads();
    }
    const EdgeScale sc = edge_scale(F, n, qbits, cmax[v]);
    unsigned long long z = 0ull;
    const int64_t rounds = (K + blockDim.x - 1) / blockDim.x;
    for (int64_t r = 0; r < rounds; ++r) {
        const int64_t f = r * blockDim.x + tid;
        if (f >= K) continue;
        const size_t x = (size_t)v * K + f;
        const T g = vals[BN_AT(cmasks[x], 1, N)];
        Gam[x] = g;
        const unsigned long long q = edge_weight(sc, logB[x], lbs[x], g);
        if (q) {
            z += q;
            for (uint32_t y = masks[x]; y; y &= y - 1) atomicAdd(&Nu[BN_AT(__ffs(y) - 1, 1, 32)], q);
        }
    }
    for (int o = 16; o; o >>= 1) z += __shfl_xor_sync(FULL, z, o);
    if ((tid & 31) == 0) atomicAdd(&Nz, z);
    __syncthreads();
    if (tid < n) {
        double p = 0.0;
        if (tid != v && Nu[tid] > 0ull)
            p = sizeof(T) == 4 ? __ull2double_rn(Nu[tid]) / __ull2double_rn(Nz)
                               : __ull2double_rn(Nu[tid]) / ldexp(1.0, qbits);
        post[(size_t)tid * n + v] = bad ? NAN : p;
    }
    // one block writes log P(D): that of the first endpoint computed
    if (tid == 0 && log_PD && (vsel & ((1u << v) - 1u)) == 0u)
        *job_ptr(log_PD, js) = bad ? NAN : log_evidence(n, cmax, F);
}

// ===========================================================================
// Priors beyond the defaults and single features (Eqs. 4-9).
// ===========================================================================

// A_i(S) += log q_i(S), q_i a function of |S| (Eq. 7): lq[i * n + |S|] in
// the working precision and log base; A is [i * 2^(n-1) + c], c = S with
// bit i removed, so |S| = popc(c).
template <typename T>
__global__ void k_apply_q(int n, const T* __restrict__ lq, T* __restrict__ A, int tlo)
{
    const int64_t total = (int64_t)n << (n - 1);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t >> (n - 1));
        const uint32_t c = (uint32_t)(t & (((int64_t)1 << (n - 1)) - 1));
        int size = __popc(c);
        if (tlo) {
            // in tile-level order the in-tile row part of c is a place p:
            // its size is the number of row sizes whose places end at or
            // before p (places of size k start at sum_{q<k} C(rb, q))
            const int lw = i < 4 ? 3 : 4, rb = 13 - lw;
            const uint32_t p = (c >> lw) & ((1u << rb) - 1u);
            int k = 0;
            for (uint32_t end = 1; end <= p; end += binom(rb, k)) ++k;
            size = __popc(c >> 13) + k + __popc(c & ((1u << lw) - 1u));
        }
        apply_weight(A[t], lq[i * n + size]);
    }
}

// ===========================================================================
// The linear FP64 form (X64, bn_device.cuh) of steps 2 (n < 14) and 4.
// ===========================================================================

// Step 2 for n < 14: one block per node, every family in its slot of the
// 2^(n-1) values in shared memory, then the butterflies of Algorithm 2.
__global__ void __launch_bounds__(256)
k_upzeta_x(int n, int64_t K, const uint32_t* __restrict__ cmasks, const X64* __restrict__ lbs,
           X64* __restrict__ A, size_t js)
{
    cmasks = job_ptr(cmasks, js);
    lbs = job_ptr(lbs, js);
    A = job_ptr(A, js);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    X64* v = reinterpret_cast<X64*>(smem_raw);
    const uint32_t N = 1u << (n - 1);
    const int i = (int)blockIdx.x;
    for (uint32_t t = threadIdx.x; t < N; t += blockDim.x) v[t] = X64{0ull};
    __syncthreads();
    for (int64_t f = threadIdx.x; f < K; f += blockDim.x)
        v[BN_AT(cmasks[(size_t)i * K + f], 1, N)] = lbs[(size_t)i * K + f];
    __syncthreads();
    for (int j = 0; j < n - 1; ++j) {
        const uint32_t jm = (1u << j) - 1u;
        for (uint32_t p = threadIdx.x; p < (N >> 1); p += blockDim.x) {
            const uint32_t lo = ((p & ~jm) << 1) | (p & jm), hi = lo | (1u << j);
            v[hi] = x_add(v[hi], v[lo]);
        }
        __syncthreads();
    }
    for (uint32_t t = threadIdx.x; t < N; t += blockDim.x) A[BN_AT((size_t)i * N + t, 1, (size_t)n * N)] = v[t];
}

// Warp-wide sum of the lanes' LazySums, in a fixed tree order.
__device__ __forceinline__ X64 warp_sum_x(LazySum<X64> a)
{
    for (int o = 16; o; o >>= 1) {
        const int e2 = __shfl_xor_sync(FULL, a.e, o);
        const double s2 = __shfl_xor_sync(FULL, a.s, o);
        const int m = max(a.e, e2);
        // both lanes of a pair form the same sum (the operands swap)
        a.s = a.s * pow2d(a.e - m) + s2 * pow2d(e2 - m);
        a.e = m;
    }
    return a.value();
}

// Phase 2 for the columns with at most one high element left (k_gamma_p2s).
// One unpacking per value of W; each sum it enters costs an aligned addition.
__global__ void __launch_bounds__(256)
k_gamma_p2s_x(int n, int d, int b, uint32_t nlow, uint32_t c0, int64_t K, const X64* __restrict__ W,
              X64* __restrict__ Gam, size_t js, uint32_t vsel)
{
    constexpr int MB = 14;                          // high bits from 5 up (h <= 18)
    const int v = blockIdx.z;
    if (!(vsel >> v & 1u)) return;
    W = job_ptr(W, js) + ((size_t)endpoint_slot(vsel, v) << (n - 1 - b)) * nlow;
    Gam = job_ptr(Gam, js) + (size_t)v * K;
    const int h = n - 1 - b;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t col = c0 + blockIdx.x * 8 + warp;
    if (col >= nlow) return;                        // whole warps leave
    int kg = 0;
    uint32_t r = col;
    while (r >= binom(b, kg)) { r -= binom(b, kg); ++kg; }
    const uint32_t g = colex_unrank(r, kg, b);
    const bool one = d - kg == 1;
    LazySum<X64> s0, sb[MB];
    const uint32_t nH = 1u << h;
    const size_t wsize = (size_t)nlow << h;
    X64 wa = lane < nH ? W[BN_AT((size_t)lane * nlow + col, 1, wsize)] : X64{0ull};
    X64 wb = lane + 32 < nH ? W[BN_AT((size_t)(lane + 32) * nlow + col, 1, wsize)] : X64{0ull};
    for (uint32_t H = lane; H < nH; H += 32) {
        const double p = x_mant(wa);
        const int e = x_exp(wa);
        wa = wb;
        if (H + 64 < nH) wb = W[BN_AT((size_t)(H + 64) * nlow + col, 1, wsize)];
        s0.add(p, e);
        if (one) {
#pragma unroll
            for (int q = 0; q < MB; ++q)
                if (5 + q < h && (H >> (5 + q) & 1u)) sb[q].add(p, e);
        }
    }
    const X64 all = warp_sum_x(s0);
    if (lane == 0) Gam[BN_AT(family_index(g, n), 1, K)] = all;
    if (!one) return;
    for (int bb = 0; bb < h && bb < 5; ++bb) {
        LazySum<X64> s = s0;
        if (!(lane >> bb & 1)) s = LazySum<X64>();
        const X64 x = warp_sum_x(s);
        if (lane == 0) Gam[BN_AT(family_index(g | (1u << (b + bb)), n), 1, K)] = x;
    }
#pragma unroll
    for (int q = 0; q < MB; ++q) {
        if (5 + q >= h) break;
        const X64 x = warp_sum_x(sb[q]);
        if (lane == 0) Gam[BN_AT(family_index(g | (1u << (b + 5 + q)), n), 1, K)] = x;
    }
}

// out = lbs + lf: the shifted scores of B_i(G) f_i(G) (Eq. 6 with a feature).
template <typename T>
__global__ void k_add_feature(const T* __restrict__ lbs, const T* __restrict__ lf,
                              T* __restrict__ out, int64_t nK)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < nK;
         x += (int64_t)gridDim.x * blockDim.x)
    {
        T y = lbs[x];
        apply_weight(y, lf[x]);
        out[x] = y;
    }
}

// Byte copies between scattered device regions, one block per segment: the
// batch upload (a staging buffer to every job's data) and download (every
// job's results to a staging buffer).
__global__ void k_copy_segments(const CopySeg* __restrict__ segs, int nseg)
{
    for (int q = blockIdx.x; q < nseg; q += gridDim.x) {
        const CopySeg sg = segs[q];
        for (uint64_t i = threadIdx.x; i < sg.bytes; i += blockDim.x) sg.dst[i] = sg.src[i];
    }
}

// ===========================================================================
// Launchers.
// ===========================================================================
// exp_t / log_t (bn_device.cuh) beside CUDA's exp / log, for the test of
// the table-driven functions: out[4i..4i+3] = exp_t, exp, log_t, log of x[i].
__global__ void k_explog_check(const double* __restrict__ x, int64_t count, double* __restrict__ out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double v = x[i];
        out[4 * i] = exp_t(v);
        out[4 * i + 1] = exp(v);
        out[4 * i + 2] = log_t(v);
        out[4 * i + 3] = log(v);
    }
}

#ifndef BN_MEGA  // host launchers (bn_mega.cu includes only the device code)
#ifdef BN_CHECK_BOUNDS
BN_BOUNDS_READER(bounds_line_kernels)
#endif
static int grid_for(int64_t work, int threads, int cap = 152 * 32)
{
    int64_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

static uint32_t host_binom(int n, int k);

cudaError_t launch_apply_q(const Plan& P, const void* lq, void* A, cudaStream_t s)
{
    const int64_t total = (int64_t)P.n << (P.n - 1);
    const int grid = grid_for(total, 256, 152 * 16);
    if (P.lin)
        launch_or_record(KID_APPLY_Q_X, k_apply_q<X64>, grid, 256, 0, s, P.n, (const X64*)lq, (X64*)A, 0);
    else if (P.prec == 0)
        launch_or_record(KID_APPLY_Q_D, k_apply_q<double>, grid, 256, 0, s, P.n, (const double*)lq, (double*)A, 0);
    else
        launch_or_record(KID_APPLY_Q_F, k_apply_q<float>, grid, 256, 0, s, P.n, (const float*)lq, (float*)A,
                                              use_tlo(P) ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_add_feature(const Plan& P, const void* lbs, const void* lf, void* out,
                               cudaStream_t s)
{
    const int64_t nK = (int64_t)P.n * P.K;
    if (P.lin)
        launch_or_record(KID_ADD_FEATURE_X, k_add_feature<X64>, grid_for(nK, 256), 256, 0, s,
            (const X64*)lbs, (const X64*)lf, (X64*)out, nK);
    else if (P.prec == 0)
        launch_or_record(KID_ADD_FEATURE_D, k_add_feature<double>, grid_for(nK, 256), 256, 0, s, 
            (const double*)lbs, (const double*)lf, (double*)out, nK);
    else
        launch_or_record(KID_ADD_FEATURE_F, k_add_feature<float>, grid_for(nK, 256), 256, 0, s, 
            (const float*)lbs, (const float*)lf, (float*)out, nK);
    return cudaGetLastError();
}

size_t upzeta_smem_bytes(const Plan& P)
{
    const size_t es = P.prec == 0 ? 8 : 4;
    return ((size_t)1 << P.b_up) * (8 + 2 * es);
}

// Fractional bits of a fixed-point sum of at most `terms` values in (0, 1].
static int fixed_bits(int64_t terms)
{
    int b = 0;
    while (((int64_t)1 << b) <= terms) ++b;
    return 63 - b;
}

cudaError_t launch_upzeta(const Plan& P, const uint32_t* cmasks, const void* lbs, void* tab,
                          const uint16_t* rk13, void* A, cudaStream_t s, cudaEvent_t sums_done, int* err,
                          bool reordered)
{
    if (use_tile13_up(P)) {
        if (!reordered) {
            const cudaError_t e = launch_reorder_up(P, lbs, tab, s);
            if (e != cudaSuccess) return e;
        }
        return launch_upzeta13(P, tab, rk13 + 8192, A, s, sums_done, err);
    }
    if (P.lin)                                      // n < 14: a node per block
        return launch_or_record(KID_UPZETA_X, k_upzeta_x, dim3(P.n, P.nj), 256, (size_t)8 << (P.n - 1), s, P.n,
                                P.K, cmasks, (const X64*)lbs, (X64*)A, P.js);
    const int h = P.n - 1 - P.b_up;
    const dim3 grid((unsigned)P.n << h, P.nj);
    const size_t sm = upzeta_smem_bytes(P);
    if (P.prec == 0)
        launch_or_record(KID_UPZETA_D, k_upzeta<double>, grid, 256, sm, s, P.n, P.b_up, P.K, fixed_bits(P.K), cmasks,
                                               (const double*)lbs, (double*)A, P.js);
    else
        launch_or_record(KID_UPZETA_F, k_upzeta<float>, grid, 256, sm, s, P.n, P.b_up, P.K, fixed_bits(P.K), cmasks,
                                              (const float*)lbs, (float*)A, P.js);
    return cudaGetLastError();
}

static uint32_t host_binom(int n, int k)
{
    if (k < 0 || k > n) return 0;
    uint64_t r = 1;
    for (int t = 1; t <= k; ++t) r = r * (uint64_t)(n - k + t) / (uint64_t)t;
    return (uint32_t)r;
}

// Tiles per warp: enough warps to fill the GPU a few times over, at most 8.
static int tiles_per_warp(uint32_t ntiles)
{
    int tpw = 1;
    while (tpw < 8 && (uint64_t)ntiles >= (uint64_t)tpw * 2 * 152 * 64 * 4) tpw *= 2;
    return tpw;
}

cudaError_t launch_forward(const Plan& P, const void* A, void* F, cudaStream_t s, int* launches)
{
    if (use_rows_levels(P) || rows64_fit(P)) return launch_forward_rows(P, A, F, s, launches);
    const int nh = P.n - P.wb;
    for (int hl = 0; hl <= nh; ++hl) {
        const uint32_t nt = host_binom(nh, hl);
        const int tpw = tiles_per_warp(nt);
        const uint32_t warps = (nt + tpw - 1) / tpw;
        const dim3 grid((unsigned)(((uint64_t)warps * 32 + 255) / 256), P.nj);
        if (P.prec == 0)
            launch_or_record(KID_FWD_LEVEL_D, k_forward_level<double>, grid, 256, 0, s, P.n, P.wb, hl, nt, tpw, (const double*)A,
                                                         (double*)F, P.js);
        else
            launch_or_record(KID_FWD_LEVEL_F, k_forward_level<float>, grid, 256, 0, s, P.n, P.wb, hl, nt, tpw, (const float*)A,
                                                        (float*)F, P.js);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (launches) ++*launches;
    }
    return cudaSuccess;
}

cudaError_t launch_backward(const Plan& P, const void* A, void* Rc, cudaStream_t s, int* launches)
{
    if (use_rows_levels(P) || rows64_fit(P)) return launch_backward_rows(P, A, Rc, s, launches);
    const int nh = P.n - P.wb;
    for (int hl = nh; hl >= 0; --hl) {
        const uint32_t nt = host_binom(nh, hl);
        const int tpw = tiles_per_warp(nt);
        const uint32_t warps = (nt + tpw - 1) / tpw;
        const dim3 grid((unsigned)(((uint64_t)warps * 32 + 255) / 256), P.nj);
        if (P.prec == 0)
            launch_or_record(KID_BWD_LEVEL_D, k_backward_level<double>, grid, 256, 0, s, P.n, P.wb, hl, nt, tpw,
                                                          (const double*)A, (double*)Rc, P.js);
        else
            launch_or_record(KID_BWD_LEVEL_F, k_backward_level<float>, grid, 256, 0, s, P.n, P.wb, hl, nt, tpw, (const float*)A,
                                                         (float*)Rc, P.js);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (launches) ++*launches;
    }
    return cudaSuccess;
}

size_t gamma_p1_smem_bytes(const Plan& P)
{
    return ((size_t)1 << P.b_g) * (P.prec == 0 ? 8 : 4);
}

size_t gamma_p2_smem_bytes(const Plan& P)
{
    const int h = P.n - 1 - P.b_g;
    uint64_t nout = 0;
    for (int k = 0; k <= P.d && k <= h; ++k) nout += host_binom(h, k);
    const size_t es = P.prec == 0 ? 8 : 4;
    return ((size_t)1 << P.hc_g) * es + nout * es + nout * 4 + 16;
}

cudaError_t launch_gamma_table(const Plan& P, const void* F, const void* Rc, cudaStream_t s)
{
    launch_or_record(KID_GAMMA_TABLE, k_gamma_table, dim3(P.n, P.nj), 32, 0, s, P.n, (const float*)F, (float*)const_cast<void*>(Rc),
                                                 P.js, P.vsel);
    return cudaGetLastError();
}

cudaError_t launch_gamma_p1(const Plan& P, const void* F, const void* Rc, const uint16_t* rk13,
                            void* W, cudaStream_t s, const void* lq, const void* A)
{
    if (use_tail(P)) return cudaSuccess;            // launch_edges does steps 4 and 5
    if (use_tile13_gamma(P)) return launch_gamma13_p1(P, F, Rc, rk13, W, s, lq, A);
    if (P.prec != 0) {
        const cudaError_t e = launch_gamma_table(P, F, Rc, s);
        if (e != cudaSuccess) return e;
    }
    const int h = P.n - 1 - P.b_g;
    const size_t sm1 = gamma_p1_smem_bytes(P);
    const dim3 grid(1u << h, P.nj, P.n);
    if (P.prec == 0)
        launch_or_record(KID_GAMMA_P1_D, k_gamma_p1<double>, grid, 256, sm1, s, P.n, P.d, P.b_g, P.nlow_g,
                                                  (const double*)F, (const double*)Rc,
                                                  (double*)W, P.js, (const double*)lq, P.vsel);
    else
        launch_or_record(KID_GAMMA_P1_F, k_gamma_p1<float>, grid, 256, sm1, s, P.n, P.d, P.b_g, P.nlow_g,
                                                 (const float*)F, (const float*)Rc,
                                                 (float*)W, P.js, (const float*)lq, P.vsel);
    return cudaGetLastError();
}

// Phase 2's columns: those before c0 (at least two high elements left) go to
// the block butterfly kernel, the others (at least d - 1 low elements) to
// the warp kernel.
uint32_t gamma_p2_split(const Plan& P)
{
    const int h = P.n - 1 - P.b_g;
    uint32_t c0 = 0;
    for (int k = 0; k <= P.d - 2 && k <= P.b_g; ++k) c0 += host_binom(P.b_g, k);
    if (h > 18) c0 = P.nlow_g;                      // beyond the warp kernel's bit count
    return c0;
}

int gamma_launches(const Plan& P)
{
    if (use_tail(P)) return 0;
    const uint32_t c0 = gamma_p2_split(P);
    return 1 + (P.prec != 0 ? 1 : 0) + (c0 > 0 ? 1 : 0) + (c0 < P.nlow_g ? 1 : 0);
}

// Columns per block of k_gamma_p2r: 64 KB of values (at most 64 outputs per
// thread), 8 or 4 columns; 0: k_gamma_p2.  The full transform of eight columns
// at a time beats the guarded one of a column per block where columns are short
// or enough of their high parts are outputs, and there are columns enough for the
// GPU.  Phase 2, us, k_gamma_p2 against k_gamma_p2r (m = 500): h = 7, d = 3 29 and
// 30, d = 4 51 and 48; h = 8, d = 3 25 and 29, d = 4 43 and 40, d = 8 612 and 277;
// h = 9, d = 4 53 and 58, d = 5 119 and 104; h = 10, d = 5 171 and 174, d = 6 390
// and 338, d = 8 1240 and 917; h = 11, d = 7 1348 and 1448, d = 8 2334 and 2373;
// h = 12, d = 7 4135 and 3072, d = 8 5897 and 5210; h = 13, d = 7 7507 and 8588.
// FP32: the linear FP64 form gained nothing (n = 23).
static int p2r_columns(const Plan& P)
{
    const int h = P.n - 1 - P.b_g;
    if (P.prec == 0 || P.d > 18) return 0;
    if (h <= 7 || (h <= 10 && P.d >= h - 4)) return 8;
    return h == 12 && P.d >= 7 ? 4 : 0;
}

template <int CPB>
static cudaError_t gamma_p2r(const Plan& P, int kid, uint32_t c0, const void* W, void* Gam, const void* A,
                             const void* lq, cudaStream_t s)
{
    const int h = P.n - 1 - P.b_g;
    // the K outputs of an endpoint move no posterior by more than 2^-24 together
    const int margin = 24 + (int)std::ceil(std::log2((double)P.K));
    return launch_or_record(kid, k_gamma_p2r<CPB>, dim3((c0 + CPB - 1) / CPB, P.nj, P.n), 256,
                            (((size_t)1 << h) + 4) * CPB * sizeof(float), s, P.n, P.d, P.b_g, P.nlow_g, c0, P.K,
                            (const float*)W, (float*)Gam, (const float*)A, (const float*)lq, margin, P.js, P.vsel);
}

cudaError_t launch_gamma_p2(const Plan& P, const void* W, void* Gam, const void* A, const void* lq,
                            cudaStream_t s)
{
    if (use_tail(P)) return cudaSuccess;
    const uint32_t c0 = gamma_p2_split(P);
    if (c0 > 0) {
        const int cpb = p2r_columns(P);
        cudaError_t e = cudaSuccess;
        const size_t sm2 = gamma_p2_smem_bytes(P);
        const dim3 grid(c0, P.nj, P.n);
        if (cpb == 8) e = gamma_p2r<8>(P, KID_P2R8, c0, W, Gam, A, lq, s);
        else if (cpb == 4) e = gamma_p2r<4>(P, KID_P2R4, c0, W, Gam, A, lq, s);
        else if (P.lin)
            launch_or_record(KID_GAMMA_P2_X, k_gamma_p2<X64>, grid, 256, sm2, s, P.n, P.d, P.b_g, P.hc_g, P.nlow_g,
                             P.K, (const X64*)W, (X64*)Gam, P.js, P.vsel);
        else if (P.prec == 0)
            launch_or_record(KID_GAMMA_P2_D, k_gamma_p2<double>, grid, 256, sm2, s, P.n, P.d, P.b_g, P.hc_g, P.nlow_g, P.K,
                                                      (const double*)W, (double*)Gam, P.js, P.vsel);
        else
            launch_or_record(KID_GAMMA_P2_F, k_gamma_p2<float>, grid, 256, sm2, s, P.n, P.d, P.b_g, P.hc_g, P.nlow_g, P.K,
                                                     (const float*)W, (float*)Gam, P.js, P.vsel);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (c0 < P.nlow_g) {
        const int h2 = P.n - 1 - P.b_g;             // high bits
        const dim3 grid((P.nlow_g - c0 + 7) / 8, P.nj, P.n);
        if (P.lin)
            launch_or_record(KID_GAMMA_P2S_X, k_gamma_p2s_x, grid, 256, 0, s, P.n, P.d, P.b_g, P.nlow_g, c0, P.K,
                             (const X64*)W, (X64*)Gam, P.js, P.vsel);
        else if (P.prec != 0 && h2 >= 8)
            launch_or_record(KID_GAMMA_P2W, k_gamma_p2w, grid, 256, 0, s, P.n, P.d, P.b_g, P.nlow_g, c0, P.K,
                             (const float*)W, (float*)Gam, P.js, P.vsel);
        else if (P.prec == 0)
            launch_or_record(KID_GAMMA_P2S_D, k_gamma_p2s<double>, grid, 256, 0, s, P.n, P.d, P.b_g, P.nlow_g, c0, P.K,
                                                     (const double*)W, (double*)Gam, P.js, P.vsel);
        else
            launch_or_record(KID_GAMMA_P2S_F, k_gamma_p2s<float>, grid, 256, 0, s, P.n, P.d, P.b_g, P.nlow_g, c0, P.K,
                                                    (const float*)W, (float*)Gam, P.js, P.vsel);
    }
    return cudaGetLastError();
}

// The one-launch form of steps 4 and 5 (k_tail).
bool use_tail(const Plan& P) { return P.n < 14; }

template <typename T>
static cudaError_t edges(const Plan& P, int kid, int kid_tail, const double* logB, const void* lbs,
                         const double* cmax, const uint32_t* masks, const uint32_t* cmasks, void* Gam,
                         const void* F, const void* Rc, const void* lq, const int* err, unsigned long long* acc,
                         double* post, double* log_PD, cudaStream_t s)
{
    if (use_tail(P)) {
        // a thread per pair of values, at most 1024
        const unsigned tb = rec_block((unsigned)std::min(1024, std::max(128, (1 << (P.n - 1)) >> 1)));
        return launch_or_record(kid_tail, k_tail<T>, dim3(P.n, P.nj), tb, sizeof(T) << (P.n - 1), s, P.n, P.d, P.K,
                                fixed_bits(P.K), (const T*)F, (const T*)Rc, (const T*)lq, logB, (const T*)lbs, cmax,
                                masks, cmasks, (T*)Gam, err, post, log_PD, P.js, P.vsel);
    }
    const unsigned chunks = (unsigned)std::min<int64_t>((P.K + 1023) / 1024, 64);
    return launch_or_record(kid, k_edges<T>, dim3(chunks, P.nj, P.n), 256, 0, s, P.n, P.K, fixed_bits(P.K), logB,
                            (const T*)lbs, cmax, masks, (const T*)Gam, (const T*)F, err, acc, post, log_PD, P.js,
                            P.vsel);
}

cudaError_t launch_edges(const Plan& P, const double* logB, const void* lbs, const double* cmax,
                         const uint32_t* masks, const uint32_t* cmasks, void* Gam, const void* F, const void* Rc,
                         const void* lq, const int* err, unsigned long long* acc, double* post, double* log_PD,
                         cudaStream_t s)
{
    if (P.lin)
        return edges<X64>(P, KID_EDGES_X, KID_TAIL_X, logB, lbs, cmax, masks, cmasks, Gam, F, Rc, lq, err, acc, post,
                          log_PD, s);
    if (P.prec == 0)
        return edges<double>(P, KID_EDGES_D, KID_TAIL_D, logB, lbs, cmax, masks, cmasks, Gam, F, Rc, lq, err, acc,
                             post, log_PD, s);
    return edges<float>(P, KID_EDGES_F, KID_TAIL_F, logB, lbs, cmax, masks, cmasks, Gam, F, Rc, lq, err, acc, post,
                        log_PD, s);
}

cudaError_t launch_explog_check(const double* x, int64_t count, double* out, cudaStream_t s)
{
    if (count < 1) return cudaSuccess;
    k_explog_check<<<(unsigned)std::min<int64_t>((count + 255) / 256, 152 * 8), 256, 0, s>>>(x, count, out);
    return cudaGetLastError();
}

cudaError_t launch_copy_segments(const CopySeg* segs, int nseg, cudaStream_t s)
{
    if (nseg < 1) return cudaSuccess;
    return launch_or_record(KID_NONE, k_copy_segments, dim3((unsigned)std::min(nseg, 152 * 8)), 256,
                            0, s, segs, nseg);
}

cudaError_t set_kernel_attributes()
{
    cudaError_t e;
#define SETA(k)                      \
    e = allow_max_dynamic_smem(k); \
    if (e != cudaSuccess) return e;
    SETA(k_upzeta<double>)
    SETA(k_upzeta<float>)
    SETA(k_gamma_p1<double>)
    SETA(k_gamma_p1<float>)
    SETA(k_gamma_p2<double>)
    SETA(k_gamma_p2<float>)
    SETA(k_upzeta_x)
    SETA(k_gamma_p2<X64>)
    SETA(k_gamma_p2r<8>)
    SETA(k_gamma_p2r<4>)
    SETA(k_tail<float>)
    SETA(k_tail<double>)
    SETA(k_tail<X64>)
#undef SETA
    e = set_scores_attributes();
    if (e != cudaSuccess) return e;
    return set_tile13_attributes();
}

#endif  // BN_MEGA

}  // namespace bn
