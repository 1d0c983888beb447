// admm.cu -- G4: batched LASSO-ADMM (Sec. II-E, Eq. 5) over bootstraps x equations x lambdas.
//
// Scaled-form ADMM for (1/(2 n_k)) ||y - X b||^2_{W_k} + lambda ||b||_1 with the
// factor cached as M_k = (G_k/n_k + rho I)^{-1} and c_k = M_k b_k / n_k:
//   x = c_k + rho M_k (z - u)            x-minimisation (a multi-RHS product)
//   v = x + u,  z = S_{lambda/rho}(v)    z-minimisation (soft threshold)
//   u = v - z                            dual update
//   stop when ||x - z|| <= sqrt(p) abs + rel max(||x||, ||z||)
//        and rho ||z - z_prev|| <= sqrt(p) abs + rel rho ||u||, or at max_iter.
// A "chain" is one (bootstrap g, equation e) path over lambda_0 > lambda_1 > ...
// (warm = path: column j starts from column j-1's (z, u)) or one single
// (g, e, j) column (warm = none: z = u = 0).
//
// Schedules:
//  * chain (FP64, and FP32 with few chains): one cluster of CTAs iterates one chain
//    (or four) at a time from start to end in a single launch, see k_admm_chain.
//  * wide (FP32, many chains, 64 < p <= 512): admm_wide.cu.
//  * resident (FP32, many chains, p <= 64; with a given start p <= 192): one CTA keeps M_g in shared
//    memory; each warp runs its own chains to completion with no block-wide
//    barrier (the warp only reads its own columns of V = z - u), pulling new
//    chains from a per-group counter.  One launch solves everything.
//  * streaming (FP64 past the chain schedule's shared memory): one launch per
//    iteration computes x for every active
//    chain (row tiles x chain tiles x groups) with the soft-threshold / dual
//    update / partial norms fused into the epilogue; a second launch reduces the
//    norms in a fixed order, finishes converged columns and compacts the active
//    list.  The host checks the active count every few iterations.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "fixed_dot.cuh"
#include "kernels.h"

namespace uoi {

namespace {

template <typename T>
struct AdmmDev {
    int32_t G, q, max_iter, warm;
    int32_t p, r, W;
    const T* M;
    const T* c;
    const double* lambdas;
    T rho, abs_tol, rel_tol, sqrtp;
    double* beta;
    int32_t* iters;
    uint8_t* conv;
    uint64_t* family;
    double* u_out;       // final scaled dual per column (nullable)
    const float* z0;     // initial state per column, cold schedule only (nullable)
    const float* u0;
    unsigned long long* near_count;   // near-threshold features (nullable)
};

template <typename T>
__device__ __forceinline__ void and_family_bits(const AdmmDev<T>& P, int64_t col_je, int a,
                                                unsigned ballot)
{
    // rows 32a .. 32a+31 form half of 64-bit word a/2
    const int shift = (a & 1) * 32;
    const uint64_t mask = ((uint64_t)ballot << shift) | ~(0xFFFFFFFFull << shift);
    atomicAnd((unsigned long long*)&P.family[col_je * P.W + (a >> 1)], (unsigned long long)mask);
}

// ----------------------------------------------------------------------------
// Resident schedule
// ----------------------------------------------------------------------------
template <typename T, int A, int SW>
__global__ void __launch_bounds__(256, 1) k_admm_resident(AdmmDev<T> P, int32_t* chain_next)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int LD = A * 32;
    const int p = P.p;
    const int p4 = (p + 3) & ~3;
    T* Ms = reinterpret_cast<T*>(smem_raw);                  // p4 x LD, zero padded
    T* Vs = Ms + (size_t)p4 * LD;                             // 8 warps x SW x LD
    const int g = blockIdx.y;
    const T* Mg = P.M + (size_t)g * p * p;
    for (int idx = threadIdx.x; idx < p4 * LD; idx += blockDim.x) {
        const int row = idx / LD, col = idx % LD;
        Ms[idx] = (row < p && col < p) ? Mg[(size_t)row * p + col] : T(0);
    }
    __syncthreads();

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T* Vw = Vs + (size_t)warp * SW * LD;
    const int nchains = P.warm ? P.r : P.r * P.q;

    int e_[SW], j_[SW], jend_[SW], it_[SW];
    bool act[SW];
    T kappa[SW];
    T z[A][SW], u[A][SW];

    auto fetch = [&](int b) {
        int cid = 0;
        if (lane == 0) cid = atomicAdd(&chain_next[g], 1);
        cid = __shfl_sync(0xffffffffu, cid, 0);
        act[b] = cid < nchains;
        if (!act[b]) return;
        if (P.warm) { e_[b] = cid; j_[b] = 0; jend_[b] = P.q; }
        else        { e_[b] = cid % P.r; j_[b] = cid / P.r; jend_[b] = j_[b] + 1; }
        it_[b] = 0;
        kappa[b] = (T)P.lambdas[j_[b]] / P.rho;
        const int64_t col0 = ((int64_t)g * P.q + j_[b]) * P.r + e_[b];
#pragma unroll
        for (int a = 0; a < A; ++a) {
            const int i = lane + 32 * a;
            const bool init = P.z0 && !P.warm && i < p;
            z[a][b] = init ? (T)P.z0[col0 * p + i] : T(0);
            u[a][b] = init ? (T)P.u0[col0 * p + i] : T(0);
        }
    };
#pragma unroll
    for (int b = 0; b < SW; ++b) fetch(b);

    for (;;) {
        bool any = false;
#pragma unroll
        for (int b = 0; b < SW; ++b) any |= act[b];
        if (!any) break;
#pragma unroll
        for (int b = 0; b < SW; ++b)
#pragma unroll
            for (int a = 0; a < A; ++a) {
                const int i = lane + 32 * a;
                Vw[b * LD + i] = (act[b] && i < p) ? z[a][b] - u[a][b] : T(0);
            }
        __syncwarp();
        T acc[A][SW];
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
            for (int b = 0; b < SW; ++b) acc[a][b] = T(0);
        for (int k = 0; k < p4; k += 4) {
            T v[SW][4];
#pragma unroll
            for (int b = 0; b < SW; ++b)
#pragma unroll
                for (int t = 0; t < 4; ++t) v[b][t] = Vw[b * LD + k + t];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                T mrow[A];
#pragma unroll
                for (int a = 0; a < A; ++a) mrow[a] = Ms[(size_t)(k + t) * LD + lane + 32 * a];
#pragma unroll
                for (int a = 0; a < A; ++a)
#pragma unroll
                    for (int b = 0; b < SW; ++b) acc[a][b] = fma(mrow[a], v[b][t], acc[a][b]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < SW; ++b) {
            if (!act[b]) continue;
            const T* cg = P.c + ((size_t)g * P.r + e_[b]) * p;
            T r2 = 0, s2 = 0, x2 = 0, z2 = 0, u2 = 0;
#pragma unroll
            for (int a = 0; a < A; ++a) {
                const int i = lane + 32 * a;
                if (i < p) {
                    const T x = cg[i] + P.rho * acc[a][b];
                    const T zp = z[a][b];
                    const T v = x + u[a][b];
                    const T zn = soft_threshold(v, kappa[b]);
                    const T un = v - zn;
                    z[a][b] = zn;
                    u[a][b] = un;
                    const T d = x - zn, dz = zn - zp;
                    r2 += d * d; s2 += dz * dz; x2 += x * x; z2 += zn * zn; u2 += un * un;
                }
            }
            r2 = warp_sum(r2); s2 = warp_sum(s2); x2 = warp_sum(x2);
            z2 = warp_sum(z2); u2 = warp_sum(u2);
            it_[b] += 1;
            const T xn = sqrt(x2), zn = sqrt(z2);
            const T eps_pri = P.sqrtp * P.abs_tol + P.rel_tol * (xn > zn ? xn : zn);
            const T eps_dual = P.sqrtp * P.abs_tol + P.rel_tol * P.rho * sqrt(u2);
            const bool converged = sqrt(r2) <= eps_pri && P.rho * sqrt(s2) <= eps_dual;
            if (converged || it_[b] >= P.max_iter) {
                const int64_t col_je = (int64_t)j_[b] * P.r + e_[b];
                const int64_t col = (int64_t)g * P.q * P.r + col_je;
                if (P.beta) {
#pragma unroll
                    for (int a = 0; a < A; ++a) {
                        const int i = lane + 32 * a;
                        if (i < p && UOI_IN_BOUNDS(col * p + i, (int64_t)P.G * P.q * P.r * p, 201))
                            P.beta[col * p + i] = (double)z[a][b];
                    }
                }
                if (P.u_out) {
#pragma unroll
                    for (int a = 0; a < A; ++a) {
                        const int i = lane + 32 * a;
                        if (i < p) P.u_out[col * p + i] = (double)u[a][b];
                    }
                }
                if (P.family) {
#pragma unroll
                    for (int a = 0; a < A; ++a) {
                        const int i = lane + 32 * a;
                        const unsigned bal = __ballot_sync(0xffffffffu, i < p && z[a][b] != T(0));
                        if (lane == 0 && 32 * a < p) and_family_bits(P, col_je, a, bal);
                    }
                }
                if (P.near_count) {
#pragma unroll
                    for (int a = 0; a < A; ++a)
                        count_near_threshold<T>(lane + 32 * a < p, z[a][b], u[a][b], kappa[b],
                                                (T)kNearThreshold, P.near_count);
                }
                if (lane == 0) {
                    if (P.iters) P.iters[col] = it_[b];
                    if (P.conv) P.conv[col] = converged ? 1 : 0;
                }
                j_[b] += 1;
                if (j_[b] < jend_[b]) {
                    it_[b] = 0;
                    kappa[b] = (T)P.lambdas[j_[b]] / P.rho;
                } else {
                    fetch(b);
                }
            }
        }
    }
}

// ----------------------------------------------------------------------------
// Chain schedule
// ----------------------------------------------------------------------------
// A cluster of `cs` CTAs owns one group's chains, NC at a time.  CTA `rank` holds a
// run of 16-row blocks of x, z, u and c in shared memory (and its rows of M_g too when
// they fit; else M_g streams from L2).  One iteration:
//   product   lane = (row of a block, one of two k), each warp its own k: the warp
//             reads 16 consecutive entries of two rows of the symmetric M and adds
//             into up to 8 independent accumulators; partial sums over the warps
//             go through shared memory;
//   update    one thread per row: x, soft threshold, dual, and V = z - u of the
//             next iteration written into every CTA of the cluster;
//   stop      the CTAs exchange five partial norms; one cluster barrier ends the
//             iteration, after which every thread takes the same decision.
// FP64 products run on the integer pipe (fixed_dot.cuh).  M and V are equilibrated first, by
// powers of two and so exactly: with 2^(2 f_i) above M_ii, M^ = M_ij 2^(-f_i - f_j) has entries
// below 1, and V^ = V_j 2^(f_j) is scaled by its largest value of this step.  (One scale for
// all of M cost features whose columns are larger than others' their bits: 2^-57 of the
// largest M_ii.)  Both become integers of h + l bits, and
//   x_i - c_i = rho 2^(f_i + ..) sum_k hi hi' 2^(2 l) + (hi lo' + lo hi') 2^l   (+ lo lo', below the last bit)
// is summed exactly in 64 bits by three 32 x 32 + 64 -> 64 multiply-adds per entry.  h comes
// from the largest row sum R of |M^|, which bounds every sum by R 2^(2 h) (R is 1 to 4 where
// the number of terms is 50 to 1000: 30 bits instead of 26 to 28), l from what is then left
// for the terms of one thread: 57 to 60 bits in all.  This part's FP64 pipe charges 19 clocks
// and SM per warp instruction, the integer pipe 1 per multiply-add.  The error is that of
// rounding M^ and V^, 2^-58 to 2^-61 of 1 and of V^'s largest value, where an FP64 dot product
// rounds every partial sum at 2^-53.  Against 80-bit iterates after 60 steps (a model of this
// arithmetic on the CPU, p = 24..1000, columns of equal scale and up to 1e3 apart) the 2-norm
// error of z is 0.2 to 0.7 times that of FP64 sums (1.3 times in one of eight), that of u 0.4 to
// 1.0 times; where columns are 1e5 apart, entries of u far below its largest are off by 4e-13 of
// themselves (2e-15 with FP64 sums).  The rest of an iteration is FP64:
// no instruction of it may run on few lanes, and the norms are first taken in FP32 (from the
// FP64 differences): only when those say that the stop test may pass are they formed in
// FP64, so that decisions are those of the FP64 norms.
// What bounds it: for small p the length of one iteration (about 10 dependent FP64 operations
// at 64 clocks, two block barriers, the exchange); past L2 the stream of M.
// Measured (one call; one warp per chain or two launches per iteration, then this schedule
// with FP64 products, then as it is): 200 x 50, 20 chains, 598 iterations each: 12.7, 2.3,
// 1.6 ms; p = 400, 20 chains: 38, 6.9, 3.8 ms; p = 1000 (M 160 MB): 124, 52, 13.5 ms
// (26 ms with 8 and 3 blocks per pass instead of 6 and 5: a pass of few blocks has few
// loads in flight);
// p = 150, 128 chains: 110, 5.1, 3.0 ms.
constexpr int CH_RB = 16;            // rows per block
constexpr int CH_NB = 8;             // blocks accumulated together
constexpr int CH_CLUSTER_MAX = 8;
constexpr int CH_KAPPA = 256;        // thresholds kept in shared memory
constexpr float CH_SCREEN = 1.0001f; // FP32 norms decide alone outside this margin

struct ChainGeom {
    int32_t cs;                      // CTAs per cluster
    int32_t nrp;                     // rows of the largest CTA, a multiple of CH_RB
    int32_t kp;                      // k extent padded to a multiple of 2 * warps
    int32_t ldm;                     // row length of the shared copy of M, 0: M stays in global memory
    int32_t lg_terms;                // FP64: log2 of the products one thread sums, rounded up
    size_t smem;
};

__device__ __forceinline__ uint32_t ch_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Store to the variable at `p` in CTA `rank` of the cluster.
template <typename V>
__device__ __forceinline__ void ch_store_rank(V* p, int rank, V v)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(ch_smem(p)), "r"(rank));
    if constexpr (sizeof(V) == 8)
        asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(a), "l"(*reinterpret_cast<long long*>(&v)) : "memory");
    else
        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(*reinterpret_cast<int*>(&v)) : "memory");
}

__device__ __forceinline__ void ch_barrier(int cs)
{
    if (cs == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                     "barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// |x| truncated to FP32 by integer operations (0 below 2^-126, Inf past FP32).
__device__ __forceinline__ float ch_abs32(double x)
{
    const uint32_t h = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
    const uint32_t f = __funnelshift_l((uint32_t)__double2loint(x), h, 3) + 0x40000000u;   // exponent bias 1023 -> 127
    return __uint_as_float(h < 0x38100000u ? 0u : h >= 0x47F00000u ? (h > 0x7FF00000u ? 0x7FC00000u : 0x7F800000u) : f);
}
__device__ __forceinline__ float ch_abs32(float x) { return x; }

__device__ __forceinline__ float ch_sqrt(float x)            // to 2^-22
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// soft_threshold with the comparisons on the integer pipe (FP64, k >= 0): one FP64
// subtraction.
__device__ __forceinline__ double ch_threshold(double v, double k)
{
    const long long kb = __double_as_longlong(k);
    if (kb < 0) return soft_threshold(v, k);
    const long long a = __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFll;
    if (!(a > kb && a <= 0x7FF0000000000000ll)) return 0.0;             // |v| <= k, or v is NaN
    const long long sign = __double_as_longlong(v) & (1ll << 63);
    return v - __longlong_as_double(kb | sign);
}
__device__ __forceinline__ float ch_threshold(float v, float k) { return soft_threshold(v, k); }

// An entry of M or V as the kernel multiplies it: FP32 itself, or (FP64) an integer of up to
// 57 bits as two balanced 28-bit digits, hi 2^28 + lo.
template <typename T> struct ChNumOf;
template <> struct ChNumOf<float> { using type = float; };
template <> struct ChNumOf<double> { using type = int2; };

// Digits of the FP64 products: sums of |M^ V^| are below 2^(lg_sum), one thread's have 2^lg_terms
// terms; all sums of upper digits' products then stay within 2^62, and those of the mixed ones.
struct ChDigits { int bits, lo; };
__device__ __forceinline__ ChDigits ch_digits_for(int lg_sum, int lg_terms)
{
    const int h = min(30, (62 - lg_sum) / 2);
    const int lo = min(30, 62 - h - max(lg_sum, lg_terms));
    return { h + lo, lo };
}

// f with x 2^(-2 f) in [1/4, 1) for x > 0.
__device__ __forceinline__ int ch_scale(double x) { return (fx_exponent(fx_high(x)) + 1) >> 1; }

// |x| 2^-e in FP32, cut off to 23 bits (0 below 2^-126).
__device__ __forceinline__ float ch_scaled32(double x, int e)
{
    const uint32_t h = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu, m = __funnelshift_l((uint32_t)__double2loint(x), h, 3) & 0x7FFFFFu;
    const int ex = (int)(h >> 20) - e - 896;                 // exponent bias 1023 -> 127
    return ex <= 0 ? 0.f : ex >= 255 ? __uint_as_float(0x7F800000u) : __uint_as_float((uint32_t)ex << 23 | m);
}

// log2, rounded up, of a bound on what sums of ch_scaled32 stand for.
__device__ __forceinline__ int ch_log2_bound(float sum)
{
    const int e = (int)(__float_as_uint(sum * 1.001f + 1e-30f) >> 23) - 126;
    return max(0, min(e, 40));
}

// Exponent of x 2^f as a number that grows with it: 0 for x = 0, past any other for Inf or NaN.
constexpr uint32_t CH_KEY_BIAS = 16384, CH_KEY_NONFINITE = 0x7FFFFFFF;
__device__ __forceinline__ uint32_t ch_key(double x, int f)
{
    const uint32_t h = fx_high(x);
    return h >= 0x7FF00000u ? CH_KEY_NONFINITE : h == 0 ? 0u : (uint32_t)(fx_exponent(h) + f + (int)CH_KEY_BIAS);
}

// acc += m v.  FP64: exact 64-bit sums of the digits' products; value() is the sum in units
// of 2^(2 lo), rounded.  FP32: the rounding errors of the product and of the sum go to a second
// word.
struct ChSumF {
    using Out = float;
    float a = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float m, float v)
    {
        const float p = __fmul_rn(m, v), e = fmaf(m, v, -p);
        const float s = __fadd_rn(a, p), b = __fsub_rn(s, a);
        c += (__fsub_rn(a, __fsub_rn(s, b)) + __fsub_rn(p, b)) + e;
        a = s;
    }
    __device__ __forceinline__ float value(int) const { return a + c; }
};
template <typename T> struct ChSumOf;
template <> struct ChSumOf<double> { using type = FxSum; };
template <> struct ChSumOf<float> { using type = ChSumF; };

// NB blocks of one warp: out[(block * 16 + row)] of each slot (row stride `ostr` per
// slot) = sum over this warp's k of M[k][row] V_slot[k].  m points at (k = 0, the
// lane's row of the first block); rows of a block past the CTA's last repeat it.
template <typename T, int NB, int NC, bool SHARED>
__device__ __forceinline__ void ch_product(const typename ChNumOf<T>::type* m, size_t ld, int p,
                                           const typename ChNumOf<T>::type* V, int kp, int k0, int kstep, int row,
                                           int nrows, typename ChSumOf<T>::type::Out* out, int ostr, int lob)
{
    using Num = typename ChNumOf<T>::type;
    typename ChSumOf<T>::type acc[NB][NC];
    int off[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) off[b] = min(row + b * CH_RB, nrows - 1) - min(row, nrows - 1);
    // rows of the shared copy reach to kp (its padding meets zeros of V); streamed rows past
    // p - 1 repeat the last
    const size_t step = (size_t)kstep * ld;
    const Num* mk = m + (size_t)min(k0, p - 1) * ld;
#pragma unroll(NB > (SHARED ? 4 : 6) ? 2 : 4)
    for (int k = k0; k < kp; k += kstep, mk += step) {
        const Num* mr = SHARED ? mk : m + (size_t)min(k, p - 1) * ld;
        Num v[NC], x[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) x[b] = mr[off[b]];
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c] = V[c * kp + k];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[b][c].add(x[b], v[c]);
    }
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            typename ChSumOf<T>::type::Out s = acc[b][c].value(lob);
            s += __shfl_xor_sync(0xffffffffu, s, CH_RB);
            if ((threadIdx.x & 31) < CH_RB) out[c * ostr + b * CH_RB] = s;
        }
}

template <typename T, int NC>
__global__ void __launch_bounds__(NC == 1 ? 512 : 256) k_admm_chain(AdmmDev<T> P, int32_t* chain_next, ChainGeom geo,
                                                   const int32_t* m_scale)
{
    using Num = typename ChNumOf<T>::type;
    using Sum = typename ChSumOf<T>::type::Out;
    constexpr bool F64 = sizeof(T) == 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ T s_kappa[CH_KAPPA];
    __shared__ __align__(16) float s_red[5][16];
    __shared__ float s_norm[2][CH_CLUSTER_MAX][NC][5];
    __shared__ T s_redx[16][5], s_exact[CH_CLUSTER_MAX][NC][5];
    __shared__ int s_cid[NC];
    __shared__ uint32_t s_max[2][CH_CLUSTER_MAX][NC], s_redm[16];   // largest exponent key of V^'
    const int p = P.p, cs = geo.cs, nrp = geo.nrp, kp = geo.kp;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, NW = blockDim.x >> 5;
    int rank = 0;
    if (cs > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int g = blockIdx.y;
    const int nbt = (p + CH_RB - 1) / CH_RB;
    const int b0 = rank * nbt / cs, nblk = (rank + 1) * nbt / cs - b0;
    const int row0 = b0 * CH_RB, nrows = min(p - row0, nblk * CH_RB);
    const T* Mg = P.M + (size_t)g * p * p;
    // shared memory: [M] | V, two buffers of NC | [FP64: V's digits] | partial products | z u c x z_prev |
    // [FP64 with M: the rows' f]
    Num* Ms = reinterpret_cast<Num*>(smem_raw);
    T* V = reinterpret_cast<T*>(Ms + (size_t)geo.ldm * kp);
    Num* Vi = reinterpret_cast<Num*>(V + (size_t)2 * NC * kp);
    Sum* part = reinterpret_cast<Sum*>(Vi + (F64 ? (size_t)NC * kp : 0));
    T* zs = reinterpret_cast<T*>(part + (size_t)NW * NC * nrp);
    T* us = zs + NC * nrp;
    T* cv = us + NC * nrp;
    T* xs = cv + NC * nrp;
    T* zq = xs + NC * nrp;
    const Num* Mi = reinterpret_cast<const Num*>(Mg);        // streamed M: digits already
    // FP64: f of the features k = threadIdx.x and + blockDim.x in registers (with M in shared
    // memory there are no more), of this CTA's rows in rowf, of all in feat (streamed M)
    int f0 = 0, f1 = 0, bits = 0, lob = 0;
    int* rowf_s = reinterpret_cast<int*>(zq + NC * nrp);
    const int* rowf = rowf_s;
    const int* feat = nullptr;
    if constexpr (F64) {
        const int ka = threadIdx.x, kb = threadIdx.x + blockDim.x;
        if (geo.ldm) {
            if (ka < p) f0 = ch_scale(Mg[(size_t)ka * p + ka]);
            if (kb < p) f1 = ch_scale(Mg[(size_t)kb * p + kb]);
            for (int i = threadIdx.x; i < nrows; i += blockDim.x) rowf_s[i] = ch_scale(Mg[(size_t)(row0 + i) * p + row0 + i]);
            __syncthreads();
            // the largest row sum of |M^|: over the columns k of a warp, the warps, the rows, the cluster
            float* ps = reinterpret_cast<float*>(part) + (size_t)warp * nrp;
            for (int i = lane; i < nrows; i += 32) {
                float sum = 0.f;
#pragma unroll 4
                for (int k = warp; k < p; k += NW)
                    sum += ch_scaled32(Mg[(size_t)k * p + row0 + i], rowf_s[i] + ch_scale(Mg[(size_t)k * p + k]));
                ps[i] = sum;
            }
            __syncthreads();
            float top = 0.f;
            for (int i = threadIdx.x; i < nrows; i += blockDim.x) {
                float sum = 0.f;
                for (int w = 0; w < NW; ++w) sum += reinterpret_cast<float*>(part)[(size_t)w * nrp + i];
                top = fmaxf(top, sum);
            }
            uint32_t h = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
            if (lane == 0) s_redm[warp] = h;
            ch_barrier(cs);                                  // and every CTA of the cluster has started
            for (int w = 0; w < NW; ++w) h = max(h, s_redm[w]);
            if (cs > 1) {
                if (threadIdx.x < cs) ch_store_rank(&s_max[1][rank][0], (int)threadIdx.x, h);
                ch_barrier(cs);
                for (int k = 0; k < cs; ++k) h = max(h, s_max[1][k][0]);
            }
            const ChDigits d = ch_digits_for(ch_log2_bound(__uint_as_float(h)), geo.lg_terms);
            bits = d.bits;
            lob = d.lo;
            for (int k = warp; k < p; k += NW) {
                const int fk = ch_scale(Mg[(size_t)k * p + k]);
                for (int i = lane; i < nrows; i += 32)
                    Ms[(size_t)k * geo.ldm + i] = fx_digits(Mg[(size_t)k * p + row0 + i], fk + rowf_s[i], bits, lob);
            }
        } else {
            feat = m_scale + P.G + (size_t)g * p;
            rowf = feat + row0;
            if (ka < p) f0 = feat[ka];
            if (kb < p) f1 = feat[kb];
            const ChDigits d = ch_digits_for(ch_log2_bound(__int_as_float(m_scale[g])), geo.lg_terms);
            bits = d.bits;
            lob = d.lo;
        }
    } else if (geo.ldm) {
        for (int k = warp; k < kp; k += NW)
            for (int i = lane; i < nrows; i += 32)
                Ms[(size_t)k * geo.ldm + i] = k < p ? Mg[(size_t)k * p + row0 + i] : T(0);
    }
    auto feature_scale = [&](int k) {                        // f_k of a feature k this thread owns in V
        return k >= p ? 0 : k == (int)threadIdx.x ? f0 : k == (int)(threadIdx.x + blockDim.x) ? f1 : feat[k];
    };
    // digits of V^_slot from buffer `buf`, their scale's exponent in re[slot]:
    // x = c + rho 2^(re + f) (sum of digits)
    constexpr int RE_NAN = 1 << 30;
    int re[NC];
    int rho_e = 0;                                           // exponent field of rho (0: subnormal, scaled by scalbn)
    if constexpr (F64) {
        rho_e = (__double2hiint(P.rho) >> 20) & 0x7FF;
        if (rho_e == 0) rho_e = -100000;
    }
    auto digits = [&](int buf, int s, uint32_t key) {
        if constexpr (F64) {
            const int ev = key == 0 ? 0 : (int)key - (int)CH_KEY_BIAS;
            const T* src = V + ((size_t)buf * NC + s) * kp;
            for (int k = threadIdx.x; k < kp; k += blockDim.x)
                Vi[s * kp + k] = fx_digits(src[k], ev - feature_scale(k), bits, lob);
            // M^ = Q 2^-bits, V^ = P 2^(ev - bits), sums in units of 2^(2 lob); NaN if V holds Inf or NaN
            re[s] = key == CH_KEY_NONFINITE ? RE_NAN : ev - 2 * (bits - lob);
        }
    };
    for (int i = threadIdx.x; i < 2 * NC * kp; i += blockDim.x) V[i] = T(0);
    for (int i = threadIdx.x; i < min(P.q, CH_KAPPA); i += blockDim.x) s_kappa[i] = (T)P.lambdas[i] / P.rho;

    const int nchains = P.warm ? P.r : P.r * P.q;
    int e_[NC], j_[NC], jend_[NC], it_[NC];
    bool act[NC];
    T kappa[NC];
    auto kappa_of = [&](int j) { return j < CH_KAPPA ? s_kappa[j] : (T)P.lambdas[j] / P.rho; };
    // takes the next chain of the group for each slot of `need`, its V in buffer `buf`
    auto fetch = [&](unsigned need, int buf) {
        if (rank == 0 && threadIdx.x == 0)
            for (int s = 0; s < NC; ++s)
                if ((need >> s) & 1u) {
                    const int cid = atomicAdd(&chain_next[g], 1);
                    for (int t = 0; t < cs; ++t) {
                        if (cs == 1) s_cid[s] = cid;
                        else ch_store_rank(&s_cid[s], t, cid);
                    }
                }
        ch_barrier(cs);
#pragma unroll
        for (int s = 0; s < NC; ++s) {
            if (!((need >> s) & 1u)) continue;
            const int cid = s_cid[s];
            act[s] = cid < nchains;
            if (!act[s]) continue;
            if (P.warm) { e_[s] = cid; j_[s] = 0; jend_[s] = P.q; }
            else        { e_[s] = cid % P.r; j_[s] = cid / P.r; jend_[s] = j_[s] + 1; }
            it_[s] = 0;
            kappa[s] = kappa_of(j_[s]);
            const int64_t col0 = ((int64_t)g * P.q + j_[s]) * P.r + e_[s];
            const bool init = P.z0 && !P.warm;
            for (int i = threadIdx.x; i < nrows; i += blockDim.x) {
                zs[s * nrp + i] = init ? (T)P.z0[col0 * p + row0 + i] : T(0);
                us[s * nrp + i] = init ? (T)P.u0[col0 * p + row0 + i] : T(0);
                cv[s * nrp + i] = P.c[((size_t)g * P.r + e_[s]) * p + row0 + i];
            }
            T* Vn = V + ((size_t)buf * NC + s) * kp;
            uint32_t h = 0;
            for (int k = threadIdx.x; k < p; k += blockDim.x) {
                const T v0 = init ? (T)P.z0[col0 * p + k] - (T)P.u0[col0 * p + k] : T(0);
                Vn[k] = v0;
                if constexpr (F64) h = max(h, ch_key(v0, feature_scale(k)));
            }
            if constexpr (F64) {
                if (init) {                              // the largest value of the start, over the block
                    h = __reduce_max_sync(0xffffffffu, h);
                    __syncthreads();
                    if (lane == 0) s_redm[warp] = h;
                    __syncthreads();
                    for (int w = 0; w < NW; ++w) h = max(h, s_redm[w]);
                }
                digits(buf, s, h);                       // a zero start needs no barrier: every digit is zero
            }
        }
        __syncthreads();
    };
    // s_kappa and V, and every CTA of the cluster has started: only then may rank 0 store into the
    // others' shared memory
    ch_barrier(cs);
    fetch((1u << NC) - 1u, 0);

    const int slot = warp % NC, wi = warp / NC, nwi = NW / NC;   // this warp's slot in the row-wise steps
    for (int cur = 0;; cur ^= 1) {
        bool any = false;
#pragma unroll
        for (int s = 0; s < NC; ++s) any |= act[s];
        if (!any) break;
        // product
        {
            const int kk = lane / CH_RB, ri = lane % CH_RB;
            const Num* Vc;
            if constexpr (F64) Vc = Vi;
            else Vc = V + (size_t)cur * NC * kp;
            Sum* pw = part + (size_t)warp * NC * nrp;
            const size_t ld = geo.ldm ? (size_t)geo.ldm : (size_t)p;
            const Num* base = geo.ldm ? Ms : Mi + row0;
            // blocks per pass over k, as equal as they come: loads in flight hide a streamed M's latency
            constexpr int CB_MAX = NC == 1 ? CH_NB : CH_NB / 2;
            const int CB = geo.ldm ? CB_MAX : (nblk + (nblk + CB_MAX - 1) / CB_MAX - 1) / ((nblk + CB_MAX - 1) / CB_MAX);
            for (int c0 = 0; c0 < nblk; c0 += CB) {
                const int row = c0 * CH_RB + ri;
                const Num* m = base + min(row, nrows - 1);
                Sum* o = pw + row;
                const int k0 = 2 * warp + kk, ks = 2 * NW;
                auto run = [&](auto nb) {
                    constexpr int NB = decltype(nb)::value;
                    if (geo.ldm) ch_product<T, NB, NC, true>(m, ld, p, Vc, kp, k0, ks, row, nrows, o, nrp, lob);
                    else if constexpr (F64) ch_product<T, NB, NC, false>(m, ld, p, Vc, kp, k0, ks, row, nrows, o, nrp, lob);
                };
                switch (min(CB, nblk - c0)) {
                case 1: run(std::integral_constant<int, 1>{}); break;
                case 2: run(std::integral_constant<int, 2>{}); break;
                case 3: run(std::integral_constant<int, 3>{}); break;
                case 4: run(std::integral_constant<int, 4>{}); break;
                default:
                    if constexpr (NC == 1) {
                        switch (min(CB, nblk - c0)) {
                        case 5: run(std::integral_constant<int, 5>{}); break;
                        case 6: run(std::integral_constant<int, 6>{}); break;
                        case 7: run(std::integral_constant<int, 7>{}); break;
                        default: run(std::integral_constant<int, 8>{}); break;
                        }
                    }
                }
            }
        }
        __syncthreads();
        // update
        {
            T kap = T(0);
            bool on = false;
            int rexp = 0;
            uint32_t big = 0;                                // largest exponent key of V^'
#pragma unroll
            for (int s = 0; s < NC; ++s)
                if (slot == s) { kap = kappa[s]; on = act[s]; rexp = re[s]; }
            float n5[5] = { 0.f, 0.f, 0.f, 0.f, 0.f };
            if (on)
                for (int i = wi * 32 + lane; i < nrows; i += nwi * 32) {
                    const int o = slot * nrp + i;
                    T x;
                    int fi = 0;
                    if constexpr (F64) {
                        fi = rowf[i];
                        long long sum = 0;                   // within 2^62, however it is split (ch_digits_for)
                        for (int w = 0; w < NW; ++w) sum += part[(size_t)w * NC * nrp + o];
                        const int xe = rexp + fi;
                        T scale;
                        if (rexp == RE_NAN) scale = __longlong_as_double(0x7FF8000000000000ll);
                        else if (xe + rho_e > 0 && xe + rho_e < 2046)
                            scale = __longlong_as_double(__double_as_longlong(P.rho) + ((long long)xe << 52));
                        else scale = scalbn(P.rho, xe);
                        x = cv[o] + scale * (double)sum;
                    } else {
                        T sum = part[o];
                        for (int w = 1; w < NW; ++w) sum += part[(size_t)w * NC * nrp + o];
                        x = cv[o] + P.rho * sum;
                    }
                    const T zp = zs[o];
                    const T v = x + us[o];
                    const T zn = ch_threshold(v, kap);
                    const T un = v - zn;
                    const T vn = zn - un;
                    if constexpr (F64) big = max(big, ch_key(vn, fi));
                    const T d = x - zn, dz = zn - zp;
                    zs[o] = zn;
                    us[o] = un;
                    xs[o] = x;
                    zq[o] = zp;
                    T* dst = V + ((size_t)(cur ^ 1) * NC + slot) * kp + row0 + i;
                    if (cs == 1) *dst = vn;
                    else
                        for (int t = 0; t < cs; ++t) ch_store_rank(dst, t, vn);
                    const float fd = ch_abs32(d), fz = ch_abs32(dz), fx = ch_abs32(x), fn = ch_abs32(zn), fu = ch_abs32(un);
                    n5[0] += fd * fd; n5[1] += fz * fz; n5[2] += fx * fx; n5[3] += fn * fn; n5[4] += fu * fu;
                }
#pragma unroll
            for (int t = 0; t < 5; ++t) {
                const float w = warp_sum(n5[t]);
                if (lane == 0) s_red[t][warp] = w;
            }
            if constexpr (F64) {
                big = __reduce_max_sync(0xffffffffu, big);
                if (lane == 0) s_redm[warp] = big;
            }
        }
        __syncthreads();
        // the CTA's norms and largest V' to every CTA of the cluster, one thread per value and CTA;
        // a CTA alone reads its warps' values as they are
        if (cs > 1) {
            constexpr int per = NC * 6;
            for (int i = threadIdx.x; i < per * cs; i += blockDim.x) {
                const int k = i / per, s = (i % per) / 6, t = i % 6;
                if (t < 5) {
                    float w = 0.f;
                    for (int q = 0; q < nwi; ++q) w += s_red[t][q * NC + s];
                    ch_store_rank(&s_norm[cur][rank][s][t], k, w);
                } else if (F64) {
                    uint32_t h = 0;
                    for (int q = 0; q < nwi; ++q) h = max(h, s_redm[q * NC + s]);
                    ch_store_rank(&s_max[cur][rank][s], k, h);
                }
            }
            ch_barrier(cs);
        }
        if constexpr (F64) {
#pragma unroll
            for (int s = 0; s < NC; ++s) {
                if (!act[s]) continue;
                uint32_t h = 0;
                if (cs == 1)
                    for (int q = 0; q < nwi; ++q) h = max(h, s_redm[q * NC + s]);
                else
                    for (int k = 0; k < cs; ++k) h = max(h, s_max[cur][k][s]);
                digits(cur ^ 1, s, h);                       // of the next product
            }
        }
        // stop test
        bool conv[NC];
        unsigned maybe = 0;
#pragma unroll
        for (int s = 0; s < NC; ++s) {
            conv[s] = false;
            if (!act[s]) continue;
            float n[5] = { 0.f, 0.f, 0.f, 0.f, 0.f };
            if (cs > 1) {
                for (int k = 0; k < cs; ++k)
#pragma unroll
                    for (int t = 0; t < 5; ++t) n[t] += s_norm[cur][k][s][t];
            } else {
                for (int q = 0; q < nwi; ++q)
#pragma unroll
                    for (int t = 0; t < 5; ++t) n[t] += s_red[t][q * NC + s];
            }
            const float base = (float)P.sqrtp * (float)P.abs_tol, rel = (float)P.rel_tol, rho = (float)P.rho;
            if constexpr (!F64) {
                const float ep = base + rel * fmaxf(sqrtf(n[2]), sqrtf(n[3])), ed = base + rel * rho * sqrtf(n[4]);
                conv[s] = sqrtf(n[0]) <= ep && rho * sqrtf(n[1]) <= ed;
            } else {
                const float ep = CH_SCREEN * (base + rel * ch_sqrt(fmaxf(n[2], n[3])));
                const float ed = CH_SCREEN * (base + rel * rho * ch_sqrt(n[4]));
                if (!(ch_sqrt(n[0]) > ep) && !(rho * ch_sqrt(n[1]) > ed)) maybe |= 1u << s;
            }
        }
        if constexpr (sizeof(T) == 8) {
            if (maybe) {                                     // the same in every thread of the cluster
                T n5[5] = {};
                if ((maybe >> slot) & 1u)
                    for (int i = wi * 32 + lane; i < nrows; i += nwi * 32) {
                        const int o = slot * nrp + i;
                        const T x = xs[o], zn = zs[o], un = us[o], d = x - zn, dz = zn - zq[o];
                        n5[0] += d * d; n5[1] += dz * dz; n5[2] += x * x; n5[3] += zn * zn; n5[4] += un * un;
                    }
#pragma unroll
                for (int t = 0; t < 5; ++t) {
                    const T w = warp_sum(n5[t]);
                    if (lane == 0) s_redx[warp][t] = w;
                }
                __syncthreads();
                if (threadIdx.x < NC * 5) {
                    const int s = threadIdx.x / 5, t = threadIdx.x % 5;
                    T w = T(0);
                    for (int k = 0; k < nwi; ++k) w += s_redx[k * NC + s][t];
                    if (cs == 1) s_exact[0][s][t] = w;
                    else
                        for (int k = 0; k < cs; ++k) ch_store_rank(&s_exact[rank][s][t], k, w);
                }
                ch_barrier(cs);
#pragma unroll
                for (int s = 0; s < NC; ++s) {
                    if (!((maybe >> s) & 1u)) continue;
                    T n[5] = {};
                    for (int k = 0; k < cs; ++k)
#pragma unroll
                        for (int t = 0; t < 5; ++t) n[t] += s_exact[k][s][t];
                    const T xn = sqrt(n[2]), zn = sqrt(n[3]);
                    const T eps_pri = P.sqrtp * P.abs_tol + P.rel_tol * (xn > zn ? xn : zn);
                    const T eps_dual = P.sqrtp * P.abs_tol + P.rel_tol * P.rho * sqrt(n[4]);
                    conv[s] = sqrt(n[0]) <= eps_pri && P.rho * sqrt(n[1]) <= eps_dual;
                }
            }
        }
        unsigned need = 0;
#pragma unroll
        for (int s = 0; s < NC; ++s) {
            if (!act[s]) continue;
            it_[s] += 1;
            if (!conv[s] && it_[s] < P.max_iter) continue;
            const int64_t col_je = (int64_t)j_[s] * P.r + e_[s];
            const int64_t col = (int64_t)g * P.q * P.r + col_je;
            for (int i0 = warp * 32; i0 < nrows; i0 += NW * 32) {
                const int i = i0 + lane;
                const bool in = i < nrows;
                const T zi = in ? zs[s * nrp + i] : T(0), ui = in ? us[s * nrp + i] : T(0);
                const int64_t o = col * p + row0 + i;
                if (P.beta && in && UOI_IN_BOUNDS(o, (int64_t)P.G * P.q * P.r * p, 203)) P.beta[o] = (double)zi;
                if (P.u_out && in) P.u_out[o] = (double)ui;
                if (P.family) {
                    // 32 rows from row0 + i0, a multiple of 16: within one word or across two
                    const uint64_t out = (uint64_t)__ballot_sync(0xffffffffu, in && zi == T(0));
                    const int bit = (row0 + i0) & 63;
                    unsigned long long* w = (unsigned long long*)&P.family[col_je * P.W + ((row0 + i0) >> 6)];
                    if (lane == 0 && (out << bit)) atomicAnd(w, ~(unsigned long long)(out << bit));
                    if (lane == 0 && bit > 32 && (out >> (64 - bit)))
                        atomicAnd(w + 1, ~(unsigned long long)(out >> (64 - bit)));
                }
                if (P.near_count)
                    count_near_threshold<T>(in, zi, ui, kappa[s], (T)kNearThreshold, P.near_count);
            }
            if (rank == 0 && threadIdx.x == 0) {
                if (P.iters) P.iters[col] = it_[s];
                if (P.conv) P.conv[col] = conv[s] ? 1 : 0;
            }
            j_[s] += 1;
            if (j_[s] < jend_[s]) {
                it_[s] = 0;
                kappa[s] = kappa_of(j_[s]);
            } else {
                need |= 1u << s;
            }
        }
        if (need) {
            __syncthreads();                                 // every thread has read the finished chain's z, u
            fetch(need, cur ^ 1);
        } else if (F64) {
            __syncthreads();                                 // V's digits
        }
    }
    if (cs > 1) ch_barrier(cs);                              // no CTA leaves while another may store into it
}

// Streamed M of the FP64 chain schedule.  ms: G row-sum bounds (FP32 bits, zero before), then
// G x p exponents f; then M turns into its digits in place.
__global__ void __launch_bounds__(256) k_chain_scales(const double* M, int p, int G, int32_t* ms)
{
    const int g = blockIdx.y, i = blockIdx.x * 256 + threadIdx.x;
    if (i < p) ms[G + (size_t)g * p + i] = ch_scale(M[((size_t)g * p + i) * p + i]);
}

__global__ void __launch_bounds__(256) k_chain_row_sums(const double* __restrict__ M, int p, int G, int32_t* ms)
{
    const int g = blockIdx.y, i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= p) return;
    const double* m = M + ((size_t)g * p + i) * p;
    const int32_t* f = ms + G + (size_t)g * p;
    const int fi = f[i];
    float sum = 0.f;
#pragma unroll 4
    for (int k = lane; k < p; k += 32) sum += ch_scaled32(m[k], fi + f[k]);
    sum = warp_sum(sum);
    if (lane == 0) atomicMax(&ms[g], __float_as_int(sum));
}

__global__ void __launch_bounds__(256) k_chain_digits(double* M, int p, int G, const int32_t* ms, int lg_terms)
{
    const int g = blockIdx.y;
    const ChDigits d = ch_digits_for(ch_log2_bound(__int_as_float(ms[g])), lg_terms);
    const int32_t* f = ms + G + (size_t)g * p;
    for (int i = blockIdx.x; i < p; i += gridDim.x) {
        double* m = M + ((size_t)g * p + i) * p;
        const int fi = f[i];
        for (int k = threadIdx.x; k < p; k += 256) {
            const int2 v = fx_digits(m[k], fi + f[k], d.bits, d.lo);
            m[k] = __hiloint2double(v.y, v.x);               // the pair's first member in the low word
        }
    }
}

// ----------------------------------------------------------------------------
// Streaming schedule
// ----------------------------------------------------------------------------
struct StreamState {
    int32_t* slot_j;      // current lambda index per slot
    int32_t* slot_jend;
    int32_t* slot_it;
    int32_t* act[2];      // G x nchains active lists (double-buffered)
    int32_t* cnt[2];      // G counts
    int32_t* total[2];    // total active count
    int32_t nchains;
};

constexpr int GV_ROWS = 8;  // rows per GEMV block (one warp per row)

template <typename T>
__device__ __forceinline__ void slot_coords(const AdmmDev<T>& P, int32_t nchains, int32_t s,
                                            int& g, int& e)
{
    g = s / nchains;
    const int cid = s % nchains;
    e = P.warm ? cid : cid % P.r;
}

// Epilogue for one (row i, slot s) element; returns the five partial sums.
template <typename T>
__device__ __forceinline__ void admm_elem(const AdmmDev<T>& P, T acc, int g, int e, int64_t s,
                                          int i, T kappa, T* z, T* u, T* Vn, T (&part)[5])
{
    const int p = P.p;
    const T x = P.c[((size_t)g * P.r + e) * p + i] + P.rho * acc;
    const size_t o = (size_t)s * p + i;
    const T zp = z[o];
    const T v = x + u[o];
    const T zn = soft_threshold(v, kappa);
    const T un = v - zn;
    z[o] = zn;
    u[o] = un;
    Vn[o] = zn - un;
    const T d = x - zn, dz = zn - zp;
    part[0] += d * d; part[1] += dz * dz; part[2] += x * x; part[3] += zn * zn; part[4] += un * un;
}

// x-update tile: 128 rows x 64 chains, 256 threads with an 8 x 4 register block
// each (rows 8*ty .. +7, chains 4*tx .. +3).  M is symmetric, so the tile's
// column k (rows i0 .. i0+127) is the contiguous segment M[k][i0 .. i0+127]:
// it is copied row by row with coalesced loads and conflict-free stores.  The
// next K step is prefetched into registers while the current one is consumed
// (two shared-memory buffers).  The soft threshold, dual update and partial
// norms run in the epilogue; V = z - u of the next iteration goes to the other
// V buffer.
constexpr int SG_TM = 128;
constexpr int SG_TN = 64;

template <typename T>
__global__ void __launch_bounds__(256)
k_stream_gemm(AdmmDev<T> P, StreamState S, int cur, const T* __restrict__ Vc, T* Vn, T* z, T* u,
              T* norms, int RT)
{
    constexpr int TK = sizeof(T) == 8 ? 8 : 16;              // K per stage
    constexpr int LDB = SG_TN + 4;
    constexpr int A_PER = SG_TM * TK / 256;                  // M elements per thread per stage
    constexpr int B_PER = SG_TN * TK / 256;                  // V elements per thread per stage
    const int g = blockIdx.z;
    const int rt = blockIdx.x;
    const int i0 = rt * SG_TM;
    const int s0 = blockIdx.y * SG_TN;
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x < 32) {
        for (int t = threadIdx.x; t < P.G; t += 32) S.cnt[cur ^ 1][t] = 0;
        if (threadIdx.x == 0) *S.total[cur ^ 1] = 0;
    }
    const int count = S.cnt[cur][g];
    if (s0 >= count) return;
    const int ncols = min(SG_TN, count - s0);
    const int32_t* act = S.act[cur] + (size_t)g * S.nchains + s0;
    const int p = P.p;
    const T* __restrict__ Mg = P.M + (size_t)g * p * p;

    __shared__ __align__(16) T As[2][TK][SG_TM];
    __shared__ __align__(16) T Bs[2][TK][LDB];
    __shared__ int32_t slots[SG_TN];
    __shared__ T red[8][SG_TN][5];
    if (threadIdx.x < SG_TN) slots[threadIdx.x] = threadIdx.x < ncols ? act[threadIdx.x] : -1;
    __syncthreads();

    T ra[A_PER], rb[B_PER];
    auto fetch = [&](int kb) {
#pragma unroll
        for (int h = 0; h < A_PER; ++h) {                    // A: row kb+kk of M, cols i0..
            const int e = threadIdx.x + 256 * h;
            const int kk = e / SG_TM, il = e % SG_TM;
            const int k = kb + kk, i = i0 + il;
            ra[h] = (k < p && i < p) ? Mg[(size_t)k * p + i] : T(0);
        }
#pragma unroll
        for (int h = 0; h < B_PER; ++h) {                    // B: V[slot][kb .. kb+TK)
            const int e = threadIdx.x + 256 * h;
            const int cl = e / TK, kk = e % TK;
            const int sl = slots[cl], k = kb + kk;
            rb[h] = (sl >= 0 && k < p) ? Vc[(size_t)sl * p + k] : T(0);
        }
    };
    auto stash = [&](int buf) {
#pragma unroll
        for (int h = 0; h < A_PER; ++h) {
            const int e = threadIdx.x + 256 * h;
            As[buf][e / SG_TM][e % SG_TM] = ra[h];
        }
#pragma unroll
        for (int h = 0; h < B_PER; ++h) {
            const int e = threadIdx.x + 256 * h;
            Bs[buf][e % TK][e / TK] = rb[h];
        }
    };

    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    fetch(0);
    stash(0);
    __syncthreads();
    int buf = 0;
    for (int kb = 0; kb < p; kb += TK) {
        const bool more = kb + TK < p;
        if (more) fetch(kb + TK);                            // in flight during the FMAs
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            T a[8], b[4];
#pragma unroll
            for (int w = 0; w < 8; ++w) a[w] = As[buf][kk][ty * 8 + w];
#pragma unroll
            for (int w = 0; w < 4; ++w) b[w] = Bs[buf][kk][tx * 4 + w];
#pragma unroll
            for (int w = 0; w < 8; ++w)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[w][v] = fma(a[w], b[v], acc[w][v]);
        }
        if (more) stash(buf ^ 1);
        __syncthreads();
        buf ^= 1;
    }
    // epilogue: thread owns chains 4*tx + v and rows 8*ty + w
    T part[4][5];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
#pragma unroll
        for (int t = 0; t < 5; ++t) part[v][t] = T(0);
        const int sl = slots[tx * 4 + v];
        if (sl < 0) continue;
        int gg, e;
        slot_coords(P, S.nchains, sl, gg, e);
        const T kappa = (T)P.lambdas[S.slot_j[sl]] / P.rho;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const int i = i0 + ty * 8 + w;
            if (i < p) admm_elem(P, acc[w][v], g, e, sl, i, kappa, z, u, Vn, part[v]);
        }
    }
    // lanes l and l^16 hold rows of the same chains (ty differs by one)
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int t = 0; t < 5; ++t) part[v][t] += __shfl_xor_sync(0xffffffffu, part[v][t], 16);
    if ((threadIdx.x & 31) < 16)
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int t = 0; t < 5; ++t) red[threadIdx.x >> 5][tx * 4 + v][t] = part[v][t];
    __syncthreads();
    if (threadIdx.x < ncols) {
        const int sl = slots[threadIdx.x];
        T tot[5] = {};
        for (int w = 0; w < 8; ++w)                        // fixed order over row groups
#pragma unroll
            for (int t = 0; t < 5; ++t) tot[t] += red[w][threadIdx.x][t];
#pragma unroll
        for (int t = 0; t < 5; ++t) norms[((size_t)sl * RT + rt) * 5 + t] = tot[t];
    }
}

// Few chains per group (path-warm LASSO: one): one warp per row computes the
// dot products of M_g[i, :] with every active chain of the group.
template <typename T, int NC>
__global__ void __launch_bounds__(256)
k_stream_gemv(AdmmDev<T> P, StreamState S, int cur, const T* __restrict__ Vc, T* Vn, T* z, T* u,
              T* norms, int RT)
{
    const int g = blockIdx.y;
    const int rt = blockIdx.x;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 32) {
        for (int t = threadIdx.x; t < P.G; t += 32) S.cnt[cur ^ 1][t] = 0;
        if (threadIdx.x == 0) *S.total[cur ^ 1] = 0;
    }
    const int count = min(S.cnt[cur][g], NC);
    if (count == 0) return;
    const int p = P.p;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = rt * GV_ROWS + warp;
    const int32_t* act = S.act[cur] + (size_t)g * S.nchains;
    __shared__ T red[GV_ROWS][NC][5];
    int sl[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) sl[c] = c < count ? act[c] : -1;
    T part[NC][5];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int t = 0; t < 5; ++t) part[c][t] = T(0);
    if (i < p) {
        const T* Mi = P.M + (size_t)g * p * p + (size_t)i * p;
        T acc[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = T(0);
        for (int k = lane; k < p; k += 32) {
            const T mv = Mi[k];
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (sl[c] >= 0) acc[c] = fma(mv, Vc[(size_t)sl[c] * p + k], acc[c]);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = warp_sum(acc[c]);
        if (lane == 0) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (sl[c] < 0) continue;
                int gg, e;
                slot_coords(P, S.nchains, sl[c], gg, e);
                const T kappa = (T)P.lambdas[S.slot_j[sl[c]]] / P.rho;
                admm_elem(P, acc[c], g, e, sl[c], i, kappa, z, u, Vn, part[c]);
            }
        }
    }
    if (lane == 0)
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int t = 0; t < 5; ++t) red[warp][c][t] = part[c][t];
    __syncthreads();
    if (threadIdx.x < count) {
        const int c = threadIdx.x;
        T tot[5] = {};
        for (int w = 0; w < GV_ROWS; ++w)
#pragma unroll
            for (int t = 0; t < 5; ++t) tot[t] += red[w][c][t];
#pragma unroll
        for (int t = 0; t < 5; ++t) norms[((size_t)act[c] * RT + rt) * 5 + t] = tot[t];
    }
}

// One warp per active slot: reduce the row-tile partial norms in order, test
// convergence, finish the column and advance the chain, compact the list.
template <typename T>
__global__ void k_stream_check(AdmmDev<T> P, StreamState S, int cur, T* z, T* u, T* Vn,
                               const T* norms, int RT)
{
    const int warp_global = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int g = blockIdx.y;
    const int count = S.cnt[cur][g];
    if (warp_global >= count) return;
    const int sl = S.act[cur][(size_t)g * S.nchains + warp_global];
    const int p = P.p;
    T tot[5] = {};
    for (int t0 = 0; t0 < RT; t0 += 32) {
        T loc[5] = {};
        const int t = t0 + lane;
        if (t < RT)
#pragma unroll
            for (int c = 0; c < 5; ++c) loc[c] = norms[((size_t)sl * RT + t) * 5 + c];
        // fixed-order tree over 32 lanes, then sequential over 32-chunks
#pragma unroll
        for (int c = 0; c < 5; ++c) tot[c] += warp_sum(loc[c]);
    }
    int it = S.slot_it[sl] + 1;
    const T xn = sqrt(tot[2]), zn = sqrt(tot[3]);
    const T eps_pri = P.sqrtp * P.abs_tol + P.rel_tol * (xn > zn ? xn : zn);
    const T eps_dual = P.sqrtp * P.abs_tol + P.rel_tol * P.rho * sqrt(tot[4]);
    const bool converged = sqrt(tot[0]) <= eps_pri && P.rho * sqrt(tot[1]) <= eps_dual;
    bool still = true;
    if (converged || it >= P.max_iter) {
        int gg, e;
        slot_coords(P, S.nchains, sl, gg, e);
        const int j = S.slot_j[sl];
        const int64_t col_je = (int64_t)j * P.r + e;
        const int64_t col = (int64_t)g * P.q * P.r + col_je;
        const T* zs = z + (size_t)sl * p;
        const T* us = u + (size_t)sl * p;
        // threshold lambda_j / rho, once per column (FP64 division off the loop)
        const T kappa_j = P.near_count ? (T)(P.lambdas[j] / (double)P.rho) : T(0);
        for (int a = 0; 32 * a < p; ++a) {
            const int i = lane + 32 * a;
            const T zi = i < p ? zs[i] : T(0);
            if (P.beta && i < p && UOI_IN_BOUNDS(col * p + i, (int64_t)P.G * P.q * P.r * p, 202))
                P.beta[col * p + i] = (double)zi;
            if (P.u_out && i < p) P.u_out[col * p + i] = (double)us[i];
            if (P.family) {
                const unsigned bal = __ballot_sync(0xffffffffu, zi != T(0));
                if (lane == 0) and_family_bits(P, col_je, a, bal);
            }
            if (P.near_count)
                count_near_threshold<T>(i < p, zi, i < p ? us[i] : T(0), kappa_j, (T)kNearThreshold,
                                        P.near_count);
        }
        if (lane == 0) {
            if (P.iters) P.iters[col] = it;
            if (P.conv) P.conv[col] = converged ? 1 : 0;
        }
        const int jn = j + 1;
        if (jn < S.slot_jend[sl]) {
            if (lane == 0) S.slot_j[sl] = jn;
            it = 0;
        } else {
            still = false;
        }
    }
    if (lane == 0) {
        S.slot_it[sl] = it;
        if (still) {
            const int pos = atomicAdd(&S.cnt[cur ^ 1][g], 1);
            S.act[cur ^ 1][(size_t)g * S.nchains + pos] = sl;
            atomicAdd(S.total[cur ^ 1], 1);
        }
    }
}

// Cold schedule with a learned start: slot s is column s, so z, u and
// V = z - u start from the given state.
template <typename T>
__global__ void k_stream_init_state(AdmmDev<T> P, int64_t count, T* z, T* u, T* V)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * blockDim.x) {
        const T zz = (T)P.z0[t], uu = (T)P.u0[t];
        z[t] = zz;
        u[t] = uu;
        V[t] = zz - uu;
    }
}

template <typename T>
__global__ void k_stream_init(AdmmDev<T> P, StreamState S)
{
    const int64_t total = (int64_t)P.G * S.nchains;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < total;
         s += (int64_t)gridDim.x * blockDim.x) {
        const int cid = (int)(s % S.nchains);
        const int g = (int)(s / S.nchains);
        if (P.warm) { S.slot_j[s] = 0; S.slot_jend[s] = P.q; }
        else        { S.slot_j[s] = cid / P.r; S.slot_jend[s] = cid / P.r + 1; }
        S.slot_it[s] = 0;
        S.act[0][s] = (int32_t)s;
        if (cid == 0) S.cnt[0][g] = S.nchains;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *S.total[0] = (int32_t)total;
}

template <typename T>
AdmmDev<T> to_dev(const AdmmProblem<T>& P)
{
    AdmmDev<T> d;
    d.G = P.G; d.q = P.q; d.max_iter = P.max_iter; d.warm = P.warm;
    d.p = (int32_t)P.p; d.r = (int32_t)P.r; d.W = (int32_t)((P.p + 63) / 64);
    d.M = P.M; d.c = P.c; d.lambdas = P.lambdas;
    d.rho = (T)P.rho; d.abs_tol = (T)P.abs_tol; d.rel_tol = (T)P.rel_tol;
    d.sqrtp = (T)sqrt((double)P.p);
    d.beta = P.beta; d.iters = P.iters; d.conv = P.conv; d.family = P.family;
    d.u_out = P.u_out; d.z0 = P.z0; d.u0 = P.u0; d.near_count = P.near_count;
    return d;
}

template <typename T, int A, int SW>
void launch_resident(const AdmmDev<T>& d, int32_t* chain_next, cudaStream_t s)
{
    const int p4 = (d.p + 3) & ~3;
    const size_t smem = sizeof(T) * ((size_t)p4 * A * 32 + (size_t)8 * SW * A * 32);
    auto kern = k_admm_resident<T, A, SW>;
    allow_max_dynamic_smem((const void*)kern);
    const int nchains = d.warm ? d.r : d.r * d.q;
    const int per_cta = 8 * SW;
    int ctas = (int)ceil_div(nchains, per_cta);
    const int fill = std::max(1, 152 / std::max(1, d.G));
    ctas = std::max(1, std::min(ctas, fill));
    k_admm_resident<T, A, SW><<<dim3((unsigned)ctas, (unsigned)d.G), 256, smem, s>>>(d, chain_next);
    UOI_CHECK_LAUNCH();
    count_launch();
}

// Launches the chain schedule if its rows fit in shared memory; false (nothing
// launched) when p is too large for it.
//
// Cluster size: with at least one chain per SM, one CTA per chain (the FP64 pipes are
// all busy and a cluster barrier would only add to each step); with fewer, as many
// CTAs per chain as keep every chain on the device at once, but at least 32 rows
// each (below that the barrier costs more than the rows).  M goes to shared memory
// where it fits; where it does not and a group has four chains or more, four share
// each read of M.
template <typename T, int NC>
bool launch_chain_nc(const AdmmDev<T>& d, int32_t* chain_next, int nw, int cs, bool m_smem, int nchains,
                     cudaStream_t s)
{
    const int nbt = (int)ceil_div(d.p, CH_RB);
    ChainGeom geo{};
    geo.cs = cs;
    geo.nrp = (int)ceil_div(nbt, cs) * CH_RB;
    geo.kp = (int)ceil_div(d.p, 2 * nw) * 2 * nw;
    // FP32 rows of M 64 bytes apart modulo 128, so that a warp's two rows use all banks
    geo.ldm = m_smem ? (sizeof(T) == 4 && geo.nrp % 32 == 0 ? geo.nrp + CH_RB : geo.nrp) : 0;
    geo.smem = sizeof(T) * ((size_t)geo.ldm * geo.kp + (size_t)(sizeof(T) == 8 ? 3 : 2) * NC * geo.kp +
                            (size_t)(nw + 5) * NC * geo.nrp);
    if (sizeof(T) == 8) {
        if (m_smem && geo.kp > 2 * 32 * nw) return false;   // two features a thread (their f in registers)
        if (m_smem) geo.smem += sizeof(int32_t) * (size_t)geo.nrp;
        while ((1 << geo.lg_terms) < geo.kp / (2 * nw)) ++geo.lg_terms;
    }
    auto kern = k_admm_chain<T, NC>;
    int dev = 0, optin = 0, nsm = 0;
    UOI_CUDA(cudaGetDevice(&dev));
    UOI_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    UOI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    cudaFuncAttributes fa;
    UOI_CUDA(cudaFuncGetAttributes(&fa, (const void*)kern));
    if (geo.smem + fa.sharedSizeBytes > (size_t)optin) return false;
    allow_max_dynamic_smem((const void*)kern);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3((unsigned)(32 * nw));
    cfg.dynamicSmemBytes = geo.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)cs, (unsigned)d.G);
    int resident = 0;
    if (cs > 1) {
        UOI_CUDA(cudaOccupancyMaxActiveClusters(&resident, kern, &cfg));
        if (resident < 1) return false;
    } else {
        UOI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, kern, 32 * nw, geo.smem));
        resident *= nsm;
    }
    const int per = std::max(1, std::min((int)ceil_div(nchains, NC), resident / std::max(1, d.G)));
    cfg.gridDim = dim3((unsigned)(cs * per), (unsigned)d.G);
    int32_t* ms = chain_next + d.G;                  // scales of the streamed M
    if constexpr (sizeof(T) == 8) {
        if (!geo.ldm) {
            // the solve is M's last reader: its entries turn into their digits in place
            double* M = const_cast<double*>(d.M);
            k_chain_scales<<<dim3((unsigned)ceil_div(d.p, 256), (unsigned)d.G), 256, 0, s>>>(M, d.p, d.G, ms);
            UOI_CHECK_LAUNCH();
            k_chain_row_sums<<<dim3((unsigned)ceil_div(d.p, 8), (unsigned)d.G), 256, 0, s>>>(M, d.p, d.G, ms);
            UOI_CHECK_LAUNCH();
            k_chain_digits<<<dim3((unsigned)std::min(d.p, 1024), (unsigned)d.G), 256, 0, s>>>(M, d.p, d.G, ms, geo.lg_terms);
            UOI_CHECK_LAUNCH();
            count_launch(3);
        }
    }
    UOI_CUDA(cudaLaunchKernelEx(&cfg, kern, d, chain_next, geo, (const int32_t*)ms));
    UOI_CHECK_LAUNCH();
    count_launch();
    return true;
}

template <typename T>
bool try_chain(const AdmmDev<T>& d, int32_t* chain_next, cudaStream_t s)
{
    const int nchains = d.warm ? d.r : d.r * d.q;
    const int64_t total = (int64_t)d.G * nchains;
    constexpr int NSM = 152, GPC_FIT = 128;       // SMs, and those that clusters of up to 8 can fill
    int cs = 1;
    if (total < NSM)
        cs = (int)std::max<int64_t>(1, std::min<int64_t>({ CH_CLUSTER_MAX, GPC_FIT / total, d.p / 32 }));
    const int NW_S = sizeof(T) == 8 && d.p <= 96 ? 4 : 8;   // warps with M in shared memory
    for (; cs <= CH_CLUSTER_MAX; ++cs) {
        if (launch_chain_nc<T, 1>(d, chain_next, NW_S, cs, true, nchains, s)) return true;
        if constexpr (sizeof(T) == 8) {
            if (nchains >= 4 && launch_chain_nc<T, 4>(d, chain_next, 8, cs, false, nchains, s)) return true;
            if (launch_chain_nc<T, 1>(d, chain_next, nchains >= 4 ? 8 : 16, cs, false, nchains, s)) return true;
        }
    }
    return false;
}

template <typename T>
bool try_resident(const AdmmDev<T>& d, int32_t* chain_next, cudaStream_t s);

template <>
bool try_resident<double>(const AdmmDev<double>& d, int32_t* chain_next, cudaStream_t s)
{
    return try_chain<double>(d, chain_next, s);
}

template <>
bool try_resident<float>(const AdmmDev<float>& d, int32_t* chain_next, cudaStream_t s)
{
    // few chains per group (a path start with few responses): the chain schedule while
    // the cluster's shared memory holds M
    if ((d.warm ? d.r : d.r * d.q) <= 4 && try_chain<float>(d, chain_next, s)) return true;
    if (d.p <= 64) { launch_resident<float, 2, 4>(d, chain_next, s); return true; }
    if (d.p <= 128) { launch_resident<float, 4, 4>(d, chain_next, s); return true; }
    if (d.p <= 192) { launch_resident<float, 6, 4>(d, chain_next, s); return true; }
    return false;
}

}  // namespace

thread_local bool g_admm_streaming = false;

namespace {

// One launch per iteration and one to check it (FP64 past the chain schedule's shared memory, p of
// about 5000 and more).
void solve_streaming(const AdmmProblem<double>& P, const AdmmDev<double>& d, int32_t nchains, cudaStream_t s)
{
    const int64_t slots = (int64_t)P.G * nchains;
    const int p = (int)P.p;
    const bool gemv = nchains <= 4;
    const int RT = gemv ? (int)ceil_div(p, GV_ROWS) : (int)ceil_div(p, SG_TM);
    DevBuf zb(sizeof(double) * slots * p, s), ub(sizeof(double) * slots * p, s);
    DevBuf v0(sizeof(double) * slots * p, s), v1(sizeof(double) * slots * p, s);
    DevBuf nb(sizeof(double) * slots * RT * 5, s);
    DevBuf sj(sizeof(int32_t) * slots, s), sje(sizeof(int32_t) * slots, s), sit(sizeof(int32_t) * slots, s);
    DevBuf a0(sizeof(int32_t) * slots, s), a1(sizeof(int32_t) * slots, s);
    DevBuf c0(sizeof(int32_t) * P.G, s), c1(sizeof(int32_t) * P.G, s);
    DevBuf tot(sizeof(int32_t) * 2, s);
    UOI_CUDA(cudaMemsetAsync(zb.ptr, 0, zb.bytes, s));
    UOI_CUDA(cudaMemsetAsync(ub.ptr, 0, ub.bytes, s));
    UOI_CUDA(cudaMemsetAsync(v0.ptr, 0, v0.bytes, s));
    UOI_CUDA(cudaMemsetAsync(c0.ptr, 0, c0.bytes, s));
    StreamState S;
    S.slot_j = sj.as<int32_t>(); S.slot_jend = sje.as<int32_t>(); S.slot_it = sit.as<int32_t>();
    S.act[0] = a0.as<int32_t>(); S.act[1] = a1.as<int32_t>();
    S.cnt[0] = c0.as<int32_t>(); S.cnt[1] = c1.as<int32_t>();
    S.total[0] = tot.as<int32_t>(); S.total[1] = tot.as<int32_t>() + 1;
    S.nchains = nchains;
    k_stream_init<double><<<(unsigned)std::min<int64_t>(ceil_div(slots, 256), 4096), 256, 0, s>>>(d, S);
    UOI_CHECK_LAUNCH();
    count_launch();
    if (P.z0 && !P.warm) {
        k_stream_init_state<double><<<(unsigned)std::min<int64_t>(ceil_div(slots * p, 256), 8192), 256, 0, s>>>(
            d, slots * p, zb.as<double>(), ub.as<double>(), v0.as<double>());
        UOI_CHECK_LAUNCH();
        count_launch();
    }

    int32_t* host_total = pinned_scratch_i32();
    const int64_t bound = (int64_t)(P.warm ? P.q : 1) * P.max_iter + 2;
    const int check_every = 8;
    double* V[2] = { v0.as<double>(), v1.as<double>() };
    int cur = 0;
    bool done = false;
    for (int64_t it = 0; it < bound && !done; ++it) {
        if (gemv) {
            dim3 grid((unsigned)RT, (unsigned)P.G);
            k_stream_gemv<double, 4><<<grid, 256, 0, s>>>(d, S, cur, V[cur], V[cur ^ 1], zb.as<double>(),
                                                      ub.as<double>(), nb.as<double>(), RT);
        } else {
            dim3 grid((unsigned)RT, (unsigned)ceil_div(nchains, SG_TN), (unsigned)P.G);
            ktimer_begin(TK_XUPDATE, s);
            k_stream_gemm<double><<<grid, 256, 0, s>>>(d, S, cur, V[cur], V[cur ^ 1], zb.as<double>(),
                                                  ub.as<double>(), nb.as<double>(), RT);
            ktimer_end(TK_XUPDATE, s, 0.0, 0.0);
        }
        UOI_CHECK_LAUNCH();
        dim3 gc((unsigned)ceil_div(nchains, 8), (unsigned)P.G);
        k_stream_check<double><<<gc, 256, 0, s>>>(d, S, cur, zb.as<double>(), ub.as<double>(), V[cur ^ 1],
                                              nb.as<double>(), RT);
        UOI_CHECK_LAUNCH();
        count_launch(2);
        cur ^= 1;
        if ((it + 1) % check_every == 0 || it + 1 == bound) {
            UOI_CUDA(cudaMemcpyAsync(host_total, S.total[cur], sizeof(int32_t),
                                     cudaMemcpyDeviceToHost, s));
            UOI_CUDA(cudaStreamSynchronize(s));
            done = *host_total == 0;
        }
    }
    if (!done) throw Error(UOI_ERR_TIMEOUT, "ADMM streaming loop exceeded its iteration bound");
}

}  // namespace

template <typename T>
void admm_solve(const AdmmProblem<T>& P, cudaStream_t s)
{
    if (P.G <= 0 || P.p <= 0 || P.r <= 0 || P.q <= 0) return;
    AdmmDev<T> d = to_dev(P);
    const int32_t nchains = P.warm ? (int32_t)P.r : (int32_t)(P.r * P.q);
    if constexpr (sizeof(T) == 4)
        if (nchains > 4 && admm_solve_wide(P, s)) return;
    if (sizeof(T) == 4 || !g_admm_streaming) {
        // chain counters and (FP64) row-sum bounds, zero, then the exponents of a streamed M
        DevBuf next(sizeof(int32_t) * (size_t)P.G * (2 + (sizeof(T) == 8 ? (size_t)P.p : 0)), s);
        UOI_CUDA(cudaMemsetAsync(next.ptr, 0, sizeof(int32_t) * 2 * (size_t)P.G, s));
        if (try_resident<T>(d, next.as<int32_t>(), s)) return;
    }
    if constexpr (sizeof(T) == 4) {
        // FP32 state: x-update on the tensor cores
        if (!admm_tc_available()) throw Error(UOI_ERR_UNSUPPORTED, "the mixed form's ADMM needs sm_103a tensor cores");
        if (admm_batch_try_join(P, s)) return;   // solved with the rest of a batch
        admm_solve_tc(P, s);
    } else {
        solve_streaming(P, d, nchains, s);
    }
}

template void admm_solve<double>(const AdmmProblem<double>&, cudaStream_t);
template void admm_solve<float>(const AdmmProblem<float>&, cudaStream_t);

template <typename T>
bool admm_solve_resident_with(const AdmmProblem<T>& P, int32_t* chain_next, cudaStream_t s)
{
    if (P.G <= 0 || P.p <= 0 || P.r <= 0 || P.q <= 0) return true;
    if (P.p > 128) return false;                     // up to here M fits in shared memory: no scales
    const AdmmDev<T> d = to_dev(P);
    return try_resident<T>(d, chain_next, s);
}

template bool admm_solve_resident_with<double>(const AdmmProblem<double>&, int32_t*, cudaStream_t);

}  // namespace uoi
