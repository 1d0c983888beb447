// estimate.cu -- G5-G7: support family, support-restricted OLS, held-out loss,
// argmin over the family and bagging (Alg. 1/2 model estimation, Eq. 3-4).
//
// For estimation bootstrap k and family member S_j (per response e):
//   beta = argmin || W^{1/2} (y_e - X_S b) ||   from G'_k[S,S] (FP64 moments):
//   FP32 inverse or Cholesky + FP64-accurate iterative refinement, FP64 Cholesky
//   where FP32 is not safe (see k_ols_warp, k_ols_block, k_ols_mixed)
//   L_kje = sum_{t in E^k} (y_te - x_t beta)^2
//         = y_E'y_E - 2 beta' (X_E'y_E)_S + beta' G^E_k[S,S] beta
// j*_k = argmin_j sum_e L_kje (ties -> smallest j); beta*_e = median (or mean)
// over k of the chosen estimates (zero outside the support).
// Singular supports (a Cholesky pivot <= 1e-12 max diag) are solved as the
// paper states OLS, the LASSO ADMM at lambda = 0: with no threshold z = x and
// u stays 0, so the iteration is x_{t+1} = (G + rho I)^{-1} (b + rho x_t) from
// x_0 = 0, whose iterates stay in the range of G and converge to the
// minimum-norm least-squares solution; they are flagged.
#include <algorithm>
#include <mutex>
#include <vector>

#include "fixed_dot.cuh"
#include "kernels.h"

namespace uoi {

namespace {

constexpr int OLS_SMEM_MAX = 160;   // supports up to this size factor in shared memory (FP64 path)
// mixed path: a warp, a CTA with 4 x 4 or 8 x 8 register tiles, a CTA with a blocked factor
constexpr int OLS_CLASSES = 4;
constexpr int OLS_CLASS_MAX[OLS_CLASSES] = { 32, 64, 128, 0x7fffffff };
// ADMM at lambda = 0 for singular supports: rho relative to the largest diagonal
// (directions with eigenvalue >> rho converge in a few steps), the stopping
// test on the relative change, and the iteration cap.
constexpr double OLS_PROX_RHO = 1e-6;
constexpr double OLS_PROX_TOL = 1e-14;
constexpr int OLS_PROX_MAX = 500;

struct OlsArgs {
    const double* Gt; const double* Bt;      // B2 x p x p, B2 x p x r
    const double* Ge; const double* Be;      // B2 x p x p, B2 x p x r
    const double* yye;                       // B2 x r
    const uint64_t* family;                  // q x r x W
    int64_t p, r; int32_t q, B2, W;
    const int32_t* jstar;                    // chosen pass: B2 (else null)
    const int32_t* dup;                      // q x r: first j with the same support (or null)
    double* losses;                          // B2 x q x r
    int32_t* singular;                       // B2 x q x r (nullable)
    double* chosen;                          // chosen pass: B2 x r x p
    double* scratch;                         // global factor scratch (per CTA), or null
    int64_t solves;
    int smax;                                // max support size
    int s_lo;                                // mixed pass: solves with fewer or more than smax are another kernel's
    bool use_smem;
    const int32_t* list;                     // solve indices to run (null: 0 .. solves-1)
    // Moments restricted to the union U of the family supports: Gt, Ge are
    // B2 x pu x pu and Bt, Be B2 x pu x r over U's columns; upos[i] = position of
    // feature i in U, ucols[t] = feature at position t.
    const int32_t* upos;
    const int32_t* ucols;
    int64_t pu;
    int32_t* fb_list;                        // mixed pass: solves left to the FP64 kernel
    int32_t* fb_count;
    float* fscratch;                         // mixed pass: global packed factor (per CTA), or null
    // mixed loss pass: the (j*r + e) it covers, taken in order from the counter `next`
    // (preset to 0), support-major (t = rank of je in je_list * B2 + k), so a list sorted
    // by decreasing support size runs the largest factors first
    const int32_t* je_list;
    unsigned long long* next;
};

// The t-th solve of a mixed pass: bootstrap k, lambda j, response e, and its index in the
// numbering of k_ols (for the FP64 hand-over).
struct OlsSolve { int k, j, e; int64_t tg; };
__device__ __forceinline__ OlsSolve ols_solve(const OlsArgs& a, int64_t t)
{
    OlsSolve o;
    if (a.jstar) {
        o.k = (int)(t / a.r); o.e = (int)(t % a.r); o.j = a.jstar[o.k];
        o.tg = t;
    } else {
        const int32_t je = a.je_list[t / a.B2];
        o.k = (int)(t % a.B2); o.j = (int)(je / a.r); o.e = (int)(je % a.r);
        o.tg = ((int64_t)o.k * a.q + o.j) * a.r + o.e;
    }
    return o;
}

// Set bits of W words (bits below p) in increasing order, plus `base`, the first `cap` to idx,
// and their number, by one warp: a word per lane, offsets by a prefix sum of their counts.
__device__ __forceinline__ int warp_support(const uint64_t* bits, int W, int64_t p, int lane, int* idx, int cap,
                                            int base = 0)
{
    int cnt = 0;
    for (int w0 = 0; w0 < W; w0 += 32) {
        const int wi = w0 + lane;
        uint64_t word = wi < W ? bits[wi] : 0;
        if (p < (int64_t)(wi + 1) * 64) word &= (1ull << (p & 63)) - 1ull;
        const int c = __popcll(word);
        int pos = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, pos, o);
            if (lane >= o) pos += v;
        }
        const int total = __shfl_sync(0xffffffffu, pos, 31);
        for (pos += cnt - c; word; word &= word - 1, ++pos)
            if (pos < cap) idx[pos] = base + wi * 64 + __ffsll((long long)word) - 1;
        cnt += total;
    }
    __syncwarp();
    return cnt;
}

__global__ void __launch_bounds__(256) k_ols(OlsArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int* idx = reinterpret_cast<int*>(smem_raw);                         // p ints
    double* bs = reinterpret_cast<double*>(smem_raw + sizeof(int) * ((a.smax + 1) & ~1));
    double* xs = bs + a.smax + 1;                                        // solution
    double* ws = xs + a.smax + 1;                                        // work vector
    double* red = ws + a.smax + 1;                                       // 32 doubles
    double* Gs = a.use_smem ? red + 32 : a.scratch + (size_t)blockIdx.x * a.smax * a.smax;
    __shared__ int s_count;
    __shared__ int s_bad;
    __shared__ int s_done;
    __shared__ double s_dmax;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    for (int64_t it = blockIdx.x; it < a.solves; it += gridDim.x) {
        const int64_t t = a.list ? a.list[it] : it;
        int k, j, e;
        if (a.jstar) { k = (int)(t / a.r); e = (int)(t % a.r); j = a.jstar[k]; }
        else { k = (int)(t / ((int64_t)a.q * a.r)); const int64_t rem = t % ((int64_t)a.q * a.r);
               j = (int)(rem / a.r); e = (int)(rem % a.r);
               if (a.dup && a.dup[rem] != j) continue; }       // duplicate support: filled later
        const uint64_t* bits = a.family + ((int64_t)j * a.r + e) * a.W;
        // support indices (warp 0, ballot compaction in increasing i)
        if (warp == 0) {
            int cnt = 0;
            for (int64_t i0 = 0; i0 < a.p; i0 += 32) {
                const int64_t i = i0 + lane;
                const bool in = i < a.p && ((bits[i >> 6] >> (i & 63)) & 1ull);
                const unsigned bal = __ballot_sync(0xffffffffu, in);
                if (in) idx[cnt + __popc(bal & ((1u << lane) - 1u))] = a.upos[i];
                cnt += __popc(bal);
            }
            if (lane == 0) { s_count = cnt; s_bad = 0; }
        }
        __syncthreads();
        const int s = s_count;
        const double* Gk = a.Gt + (size_t)k * a.pu * a.pu;
        const double* Bk = a.Bt + (size_t)k * a.pu * a.r;
        double ridge = 0.0;                   // rho of the lambda = 0 ADMM (0: plain solve)
        for (int attempt = 0; attempt < 2 && s > 0; ++attempt) {
            double dm = 0.0;
            for (int x = threadIdx.x; x < s * s; x += blockDim.x) {
                const int r0 = x / s, c0 = x % s;
                const double v = Gk[(size_t)idx[r0] * a.pu + idx[c0]];
                Gs[x] = v + (r0 == c0 ? ridge : 0.0);
                if (r0 == c0) dm = fmax(dm, v);
            }
            for (int x = threadIdx.x; x < s; x += blockDim.x) bs[x] = Bk[(size_t)idx[x] * a.r + e];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dm = fmax(dm, __shfl_xor_sync(0xffffffffu, dm, o));
            if (lane == 0) red[warp] = dm;
            __syncthreads();
            if (threadIdx.x == 0) {
                double m = 0.0;
                for (int w = 0; w < 8; ++w) m = fmax(m, red[w]);
                s_dmax = m;
                s_bad = 0;
            }
            __syncthreads();
            const double thr = 1e-12 * s_dmax;
            // unblocked right-looking Cholesky of Gs (lower)
            for (int c = 0; c < s; ++c) {
                if (threadIdx.x == 0) {
                    const double d = Gs[c * s + c];
                    if (!(d > thr)) { s_bad = 1; Gs[c * s + c] = 1.0; } else Gs[c * s + c] = sqrt(d);
                }
                __syncthreads();
                const double lcc = Gs[c * s + c];
                for (int i = c + 1 + threadIdx.x; i < s; i += blockDim.x) Gs[i * s + c] /= lcc;
                __syncthreads();
                const int rem = s - c - 1;
                for (int x = threadIdx.x; x < rem * rem; x += blockDim.x) {
                    const int i = c + 1 + x / rem, jj = c + 1 + x % rem;
                    if (jj <= i) Gs[i * s + jj] -= Gs[i * s + c] * Gs[jj * s + c];
                }
                __syncthreads();
            }
            if (!s_bad) break;
            ridge = OLS_PROX_RHO * s_dmax;    // factor G + rho I for the lambda = 0 ADMM
            __syncthreads();
        }
        const bool singular = s > 0 && ridge > 0.0;
        // x = (G + rho I)^{-1} (b + rho x): once with rho = 0 (plain Cholesky solve),
        // else the lambda = 0 ADMM iterations from x = 0
        for (int x = threadIdx.x; x < s; x += blockDim.x) xs[x] = 0.0;
        for (int itp = 0; s > 0; ++itp) {
            for (int x = threadIdx.x; x < s; x += blockDim.x) ws[x] = bs[x] + ridge * xs[x];
            __syncthreads();
            // forward / back substitution by warp 0
            if (warp == 0) {
                for (int i = 0; i < s; ++i) {
                    double acc = 0.0;
                    for (int c = lane; c < i; c += 32) acc += Gs[i * s + c] * ws[c];
                    acc = warp_sum(acc);
                    if (lane == 0) ws[i] = (ws[i] - acc) / Gs[i * s + i];
                    __syncwarp();
                }
                for (int i = s - 1; i >= 0; --i) {
                    double acc = 0.0;
                    for (int c = i + 1 + lane; c < s; c += 32) acc += Gs[c * s + i] * ws[c];
                    acc = warp_sum(acc);
                    if (lane == 0) ws[i] = (ws[i] - acc) / Gs[i * s + i];
                    __syncwarp();
                }
            }
            __syncthreads();
            double dmx = 0.0, xmx = 0.0;
            for (int x = threadIdx.x; x < s; x += blockDim.x) {
                dmx = fmax(dmx, fabs(ws[x] - xs[x]));
                xmx = fmax(xmx, fabs(ws[x]));
                xs[x] = ws[x];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                dmx = fmax(dmx, __shfl_xor_sync(0xffffffffu, dmx, o));
                xmx = fmax(xmx, __shfl_xor_sync(0xffffffffu, xmx, o));
            }
            if (lane == 0) { red[warp] = dmx; red[8 + warp] = xmx; }
            __syncthreads();
            if (threadIdx.x == 0) {
                double d = 0.0, xm = 0.0;
                for (int w = 0; w < 8; ++w) { d = fmax(d, red[w]); xm = fmax(xm, red[8 + w]); }
                s_done = (!singular || d <= OLS_PROX_TOL * xm || itp + 1 >= OLS_PROX_MAX) ? 1 : 0;
            }
            __syncthreads();
            if (s_done) break;
        }
        __syncthreads();
        if (a.jstar) {
            double* out = a.chosen + ((size_t)k * a.r + e) * a.p;
            for (int x = threadIdx.x; x < s; x += blockDim.x) out[a.ucols[idx[x]]] = xs[x];
        } else {
            // held-out loss via the evaluation moments
            const double* Gek = a.Ge + (size_t)k * a.pu * a.pu;
            const double* Bek = a.Be + (size_t)k * a.pu * a.r;
            double part = 0.0;
            for (int x = threadIdx.x; x < s * s; x += blockDim.x) {
                const int r0 = x / s, c0 = x % s;
                part += xs[r0] * Gek[(size_t)idx[r0] * a.pu + idx[c0]] * xs[c0];
            }
            for (int x = threadIdx.x; x < s; x += blockDim.x)
                part -= 2.0 * xs[x] * Bek[(size_t)idx[x] * a.r + e];
            part = warp_sum(part);
            __syncthreads();
            if (lane == 0) red[warp] = part;
            __syncthreads();
            if (threadIdx.x == 0) {
                double tot = 0.0;
                for (int w = 0; w < 8; ++w) tot += red[w];
                const int64_t o = ((int64_t)k * a.q + j) * a.r + e;
                a.losses[o] = a.yye[(size_t)k * a.r + e] + tot;
                if (a.singular) a.singular[o] = singular ? 1 : 0;
            }
        }
        __syncthreads();
    }
}

// Mixed-precision form of the same solve: an FP32 inverse or factor of G'_k[S,S], then iterative
// refinement with FP64 residuals r = b - G x until the correction is at FP64 rounding level, so
// the result agrees with an FP64 factorisation to ~kappa * 1e-16.  A solve whose FP32 pivots
// fall below 1e-3 of the largest diagonal (where FP32 cannot certify the 1e-12 singularity
// test) or whose refinement stalls is queued for k_ols.
//
// Up to 128 columns (k_ols_warp, k_ols_block) the solve is a symmetric Gauss-Jordan sweep in
// registers, which leaves -G^{-1}: a refinement step is then a matrix-vector product instead of
// two substitutions, whose s dependent steps were most of a small solve's time.  The pivots are
// those of the Cholesky factor.  Rows and columns of G are scaled by powers of two 2^-e_i that
// bring its diagonal to [1/4, 1) (exact; one scale for all of G lost the bits of its small
// columns), and the result is kept as integers (fixed_dot.cuh) for the residuals: the FP64
// pipe would take 19 clocks per 32 entries and the gather of G from L2 would be repeated at
// each step.
// Measured (all solves of a fit, against one CTA with a packed factor for every size): VAR
// p = 192, 30 bootstraps x 32 lambdas (supports of a few to 30 columns): 4.1 -> 0.25 ms;
// 4999 x 301, 24 x 32 (15 to 111 columns): 0.43 -> 0.13 ms.
constexpr float OLS_F32_PIVOT = 1e-3f;
constexpr int OLS_REFINE_MAX = 8;

__device__ __forceinline__ int packed_row(int i) { return (i * (i + 1)) >> 1; }

// w <- L^{-T} L^{-1} w with L packed lower, by the whole block: 32-row diagonal
// blocks are solved by warp 0 in registers (one shuffle per column), the rows
// beyond them are updated by all threads.
__device__ __forceinline__ void chol_solve_f32(const float* L, const float* dinv, float* w, int s, int warp,
                                               int lane)
{
    for (int c0 = 0; c0 < s; c0 += 32) {
        const int nb = min(32, s - c0);
        if (warp == 0) {
            float wi = lane < nb ? w[c0 + lane] : 0.f;
            for (int c = 0; c < nb; ++c) {
                if (lane == c) wi *= dinv[c0 + c];
                const float wc = __shfl_sync(0xffffffffu, wi, c);
                if (lane > c && lane < nb) wi -= L[packed_row(c0 + lane) + c0 + c] * wc;
            }
            if (lane < nb) w[c0 + lane] = wi;
        }
        __syncthreads();
        for (int i = c0 + nb + threadIdx.x; i < s; i += blockDim.x) {
            const float* row = L + packed_row(i) + c0;
            float acc = 0.f;
            for (int c = 0; c < nb; ++c) acc += row[c] * w[c0 + c];
            w[i] -= acc;
        }
        __syncthreads();
    }
    for (int c0 = ((s - 1) / 32) * 32; c0 >= 0; c0 -= 32) {
        const int nb = min(32, s - c0);
        if (warp == 0) {
            float xi = lane < nb ? w[c0 + lane] : 0.f;
            for (int c = nb - 1; c >= 0; --c) {
                if (lane == c) xi *= dinv[c0 + c];
                const float xc = __shfl_sync(0xffffffffu, xi, c);
                if (lane < c) xi -= L[packed_row(c0 + c) + c0 + lane] * xc;
            }
            if (lane < nb) w[c0 + lane] = xi;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < c0; i += blockDim.x) {
            float acc = 0.f;
            for (int c = 0; c < nb; ++c) acc += L[packed_row(c0 + c) + i] * w[c0 + c];
            w[i] -= acc;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ double block_max(double v, double* red, int lane, int warp)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double m = red[0];
    for (int w = 1; w < 8; ++w) m = fmax(m, red[w]);
    return m;
}

__device__ __forceinline__ double block_sum(double v, double* red, int lane, int warp)
{
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    return t;
}

// Tests of one refinement step on dmx = max |correction|, xmx = max |x| (FP32 is enough for
// them).  Converged: the correction is at the level of FP64 rounding of the residual, or it no
// longer shrinks (the residual is rounding noise).  1: done, -1: not to be had, 0: go on.
__device__ __forceinline__ int ols_converged(int itr, float dmx, float xmx, float prev)
{
    if (itr > 0 && (dmx <= 1e-14f * xmx || (dmx > 0.5f * prev && dmx <= 1e-12f * xmx))) return 1;
    if (itr == OLS_REFINE_MAX) return dmx <= 1e-12f * xmx ? 1 : -1;
    return 0;
}

// e with d 2^(-2 e) in [1/4, 1) for d > 0 with high word h.
__device__ __forceinline__ int ols_scale(uint32_t h) { return (fx_exponent(h) + 1) >> 1; }

// Whether |v| 2^-e is 1 or more, or v is Inf or NaN.
__device__ __forceinline__ bool ols_exceeds(double v, int e)
{
    const uint32_t h = fx_high(v);
    return h >= 0x7FF00000u || (h != 0 && fx_exponent(h) > e);
}

// Least pivot of a scaled column: OLS_F32_PIVOT of the largest diagonal (high word hg) before
// scaling, in the scale of a column with exponent e.
__device__ __forceinline__ float ols_pivot(uint32_t hg, int e)
{
    const float top = __uint_as_float(0x3F000000u | (hg & 0xFFFFFu) << 3);       // hg's value over 2^fx_exponent
    return hg == 0 ? 1.f : ldexpf(OLS_F32_PIVOT * top, min(fx_exponent(hg) - 2 * e, 100));
}

// Exponent of v 2^-e as a number that grows with it (0 for v = 0, past any other for Inf or NaN).
constexpr uint32_t OLS_EXP_BIAS = 16384, OLS_EXP_NONFINITE = 0x7FFFFFFF;
__device__ __forceinline__ uint32_t ols_exponent_key(double v, int e)
{
    const uint32_t h = fx_high(v);
    return h >= 0x7FF00000u ? OLS_EXP_NONFINITE : h == 0 ? 0u : (uint32_t)(fx_exponent(h) - e + (int)OLS_EXP_BIAS);
}
__device__ __forceinline__ int ols_key_exponent(uint32_t k) { return k == 0 ? 0 : (int)k - (int)OLS_EXP_BIAS; }

// Solves of at most 32 columns, one per warp: lane i holds row i of the swept matrix.
// Bound by issue slots and the latency of a few hundred dependent steps; a warp per solve keeps
// 16 or more in flight on an SM, and needs no block barrier.  The line at 32 is the warp's width.
constexpr int OLS_WARPS = 4;
struct OlsWarpSmem {
    int2 xd[32];
    double xb[32];
    float buf[2][32];
    int idx[32], ex[32];
};
__global__ void __launch_bounds__(32 * OLS_WARPS) k_ols_warp(OlsArgs a)
{
    constexpr int BITS = 57, LOB = 29;                      // sums of 32 products fit 62 bits
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    OlsWarpSmem& m = reinterpret_cast<OlsWarpSmem*>(smem_raw)[warp];
    int2* Gd = reinterpret_cast<int2*>(smem_raw + sizeof(OlsWarpSmem) * OLS_WARPS) + (size_t)warp * a.smax * a.smax;
    const int64_t wid = (int64_t)blockIdx.x * OLS_WARPS + warp, nwarps = (int64_t)gridDim.x * OLS_WARPS;
    auto fetch = [&](int64_t t) -> int64_t {
        if (!a.next) return t < 0 ? wid : t + nwarps;
        unsigned long long v = 0;
        if (lane == 0) v = atomicAdd(a.next, 1ull);
        return (int64_t)__shfl_sync(0xffffffffu, v, 0);
    };
    for (int64_t t = fetch(-1); t < a.solves; t = fetch(t)) {
        const OlsSolve o = ols_solve(a, t);
        __syncwarp();
        const int s = warp_support(a.family + ((int64_t)o.j * a.r + o.e) * a.W, a.W, a.p, lane, m.idx, a.smax);
        if (s < a.s_lo || s > a.smax) continue;
        const bool in = lane < s;
        const int my = in ? a.upos[m.idx[lane]] : 0;
        __syncwarp();
        m.idx[lane] = my;
        __syncwarp();
        const double* Gk = a.Gt + (size_t)o.k * a.pu * a.pu;
        const double dg = in ? __ldg(Gk + (size_t)my * a.pu + my) : 0.0;
        const double b = in ? __ldg(a.Bt + ((size_t)o.k * a.pu + my) * a.r + o.e) : 0.0;
        const uint32_t hg = __reduce_max_sync(0xffffffffu, fx_high(dg));
        const int e = ols_scale(fx_high(dg));
        const uint32_t hb = __reduce_max_sync(0xffffffffu, ols_exponent_key(b, e));
        const int eb = ols_key_exponent(hb);
        m.ex[lane] = e;
        __syncwarp();
        bool bad = hb == OLS_EXP_NONFINITE;                  // scaled entries of G at 1 or above: below
        float g[32];
        constexpr float unit = 1.f / (float)(1 << (BITS - LOB));
#pragma unroll
        for (int c0 = 0; c0 < 32; c0 += 8) {
            if (c0 < s) {
                double v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    v[i] = in && c0 + i < s ? __ldg(Gk + (size_t)m.idx[c0 + i] * a.pu + my) : 0.0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int ev = e + m.ex[c0 + i];
                    const int2 d = fx_digits(v[i], ev, BITS, LOB);
                    bad |= ols_exceeds(v[i], ev);
                    if (in && c0 + i < s) Gd[(c0 + i) * s + lane] = d;
                    g[c0 + i] = (float)d.x * unit;
                }
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) g[c0 + i] = 0.f;
            }
        }
        bool ok = !__any_sync(0xffffffffu, bad);
        const float thr = ols_pivot(hg, e);                  // of this lane's column
        // sweep of column c: g_ij -= g_ic g_cj / d, row and column c times 1 / d, g_cc = -1 / d.
        // Row c is column c (symmetry), and in lane c the same update with 1 - 1/d for g_ic / d
        // leaves g_cj / d.
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            if (c < s && ok) {                               // the same in every lane
                const float d = __shfl_sync(0xffffffffu, g[c], c);
                if (__any_sync(0xffffffffu, lane == c && !(d > thr))) ok = false;
                else {
                    float* row = m.buf[c & 1];
                    row[lane] = g[c];
                    __syncwarp();
                    const float inv = __frcp_rn(d), q = g[c] * inv;
                    const float f = lane == c ? 1.f - inv : q;
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        if (j < s) {
                            const float4 r = *reinterpret_cast<const float4*>(row + j);
                            g[j] -= f * r.x; g[j + 1] -= f * r.y; g[j + 2] -= f * r.z; g[j + 3] -= f * r.w;
                        }
                    g[c] = lane == c ? -inv : q;
                }
            }
        }
        const double bs = scalbn(b, -e - eb);                // x comes out times 2^(e - eb)
        double x = 0.0;
        bool done = false;
        if (ok) {
            float w = f64_to_f32_int(bs), prev = 0.f;
            for (int itr = 0; itr <= OLS_REFINE_MAX; ++itr) {
                __syncwarp();
                m.buf[0][lane] = w;
                __syncwarp();
                float y0 = 0.f, y1 = 0.f;
#pragma unroll
                for (int c = 0; c < 32; c += 4)
                    if (c < s) {
                        const float4 r = *reinterpret_cast<const float4*>(m.buf[0] + c);
                        y0 += g[c] * r.x; y1 += g[c + 1] * r.y; y0 += g[c + 2] * r.z; y1 += g[c + 3] * r.w;
                    }
                const float y = -(y0 + y1);
                x += (double)y;
                const uint32_t hx = __reduce_max_sync(0xffffffffu, fx_high(x));
                const float dmx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(y))));
                const float xmx = __uint_as_float(
                    __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(f64_to_f32_int(x)))));
                const int st = ols_converged(itr, dmx, xmx, prev);
                if (st) { done = st > 0; break; }
                prev = dmx;
                const int ev = hx ? fx_exponent(hx) : 0;
                m.xd[lane] = fx_digits(x, ev, BITS, LOB);
                __syncwarp();
                FxFull sum;
                if (in)
#pragma unroll 4
                    for (int c = 0; c < s; ++c) sum.add(Gd[c * s + lane], m.xd[c]);
                w = f64_to_f32_int(fx_residual(bs, sum.hh, sum.low(LOB), ev - 2 * BITS, LOB));
            }
        }
        if (s > 0 && !done) {
            if (lane == 0) a.fb_list[atomicAdd(a.fb_count, 1)] = (int32_t)o.tg;
            continue;
        }
        x = scalbn(x, eb - e);
        if (a.jstar) {
            if (in) a.chosen[((size_t)o.k * a.r + o.e) * a.p + a.ucols[my]] = x;
            continue;
        }
        m.xb[lane] = x;
        __syncwarp();
        const double* Ge = a.Ge + (size_t)o.k * a.pu * a.pu;
        double acc = 0.0, part = 0.0;
        if (in) {
#pragma unroll 8
            for (int c = 0; c < s; ++c) acc += __ldg(Ge + (size_t)m.idx[c] * a.pu + my) * m.xb[c];
            part = x * (acc - 2.0 * a.Be[((size_t)o.k * a.pu + my) * a.r + o.e]);
        }
        const double tot = warp_sum(part);
        if (lane == 0) {
            a.losses[o.tg] = a.yye[(size_t)o.k * a.r + o.e] + tot;
            if (a.singular) a.singular[o.tg] = 0;
        }
    }
}

// Solves of at most 16 T columns, one CTA each: thread (ty, tx) holds entries (ty + 16 u,
// tx + 16 v) of the swept matrix.  One barrier per swept column (column c through two
// alternating buffers); residuals by threads = (row, part of the columns).  Bound by the s
// barriers of the sweep (about 200 clocks each at T = 4, 350 at T = 8).  T = 8 ends where the
// integers of G[S,S] fill an SM's shared memory (128 columns) and the tile its registers.
template <int T>
struct OlsBlockSmem {
    double bs[16 * T], x[16 * T];
    long long part[256];
    double part_low[256];
    int2 xd[16 * T];
    float buf[2][16 * T], w[16 * T], y[16 * T], thr[16 * T];
    int idx[16 * T], ex[16 * T];
    uint32_t red[3][8];
    double redd[8];
    int64_t next;
    int count;
};
template <int T>
__global__ void __launch_bounds__(256, T == 4 ? 4 : 2) k_ols_block(OlsArgs a)
{
    constexpr int R = 16 * T, PARTS = 256 / R;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    OlsBlockSmem<T>& m = *reinterpret_cast<OlsBlockSmem<T>*>(smem_raw);
    int2* Gd = reinterpret_cast<int2*>(smem_raw + sizeof(OlsBlockSmem<T>));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, tx = tid & 15, ty = tid >> 4;
    // upper digits: sums of all 16 T products fit 62 bits; the others: sums of one part's
    constexpr int BITS = T == 4 ? 58 : 56, LOB = T == 4 ? 30 : 29;
    constexpr float unit = 1.f / (float)(1 << (BITS - LOB));
    auto fetch = [&](int64_t t) -> int64_t {
        if (!a.next) return t < 0 ? (int64_t)blockIdx.x : t + gridDim.x;
        __syncthreads();
        if (tid == 0) m.next = (int64_t)atomicAdd(a.next, 1ull);
        __syncthreads();
        return m.next;
    };
    // maxima of up to three words over the block
    auto block_max3 = [&](uint32_t& p0, uint32_t& p1, uint32_t& p2) {
        p0 = __reduce_max_sync(0xffffffffu, p0);
        p1 = __reduce_max_sync(0xffffffffu, p1);
        p2 = __reduce_max_sync(0xffffffffu, p2);
        if (lane == 0) { m.red[0][warp] = p0; m.red[1][warp] = p1; m.red[2][warp] = p2; }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            p0 = max(p0, m.red[0][i]);
            p1 = max(p1, m.red[1][i]);
            p2 = max(p2, m.red[2][i]);
        }
    };
    for (int64_t t = fetch(-1); t < a.solves; t = fetch(t)) {
        const OlsSolve o = ols_solve(a, t);
        __syncthreads();                                     // the last solve's shared memory is free
        if (warp == 0) {
            const int c = warp_support(a.family + ((int64_t)o.j * a.r + o.e) * a.W, a.W, a.p, lane, m.idx,
                                       a.smax);
            if (lane == 0) m.count = c;
        }
        __syncthreads();
        const int s = m.count;
        if (s < a.s_lo || s > a.smax) continue;
        int my = 0;
        if (tid < s) my = a.upos[m.idx[tid]];
        __syncthreads();
        if (tid < s) m.idx[tid] = my;
        const double* Gk = a.Gt + (size_t)o.k * a.pu * a.pu;
        const double dg = tid < s ? __ldg(Gk + (size_t)my * a.pu + my) : 0.0;
        const double b = tid < s ? __ldg(a.Bt + ((size_t)o.k * a.pu + my) * a.r + o.e) : 0.0;
        const int e = ols_scale(fx_high(dg));
        if (tid < R) m.ex[tid] = e;
        uint32_t hg = fx_high(dg), hb = tid < s ? ols_exponent_key(b, e) : 0u, zero = 0;
        block_max3(hg, hb, zero);                            // its barrier: idx and ex are complete
        const int eb = ols_key_exponent(hb);
        bool bad = hb == OLS_EXP_NONFINITE;
        for (int c = warp; c < s; c += 8) {
            const double* row = Gk + (size_t)m.idx[c] * a.pu;
            double v[R / 32];
#pragma unroll
            for (int i = 0; i < R / 32; ++i) v[i] = lane + 32 * i < s ? __ldg(row + m.idx[lane + 32 * i]) : 0.0;
#pragma unroll
            for (int i = 0; i < R / 32; ++i) {
                const int ev = m.ex[c] + m.ex[lane + 32 * i];
                bad |= ols_exceeds(v[i], ev);
                if (lane + 32 * i < s) Gd[c * s + lane + 32 * i] = fx_digits(v[i], ev, BITS, LOB);
            }
        }
        const double bs = scalbn(b, -e - eb);
        if (tid < R) {
            m.bs[tid] = bs;
            m.thr[tid] = ols_pivot(hg, e);
            m.x[tid] = 0.0;
            m.w[tid] = f64_to_f32_int(bs);                   // zero past s
            m.xd[tid] = make_int2(0, 0);
        }
        bool ok = __syncthreads_or(bad) == 0;
        float g[T][T];
#pragma unroll
        for (int u = 0; u < T; ++u)
#pragma unroll
            for (int v = 0; v < T; ++v) {
                const int i = ty + 16 * u, j = tx + 16 * v;
                g[u][v] = i < s && j < s ? (float)Gd[j * s + i].x * unit : 0.f;
            }
#pragma unroll
        for (int v0 = 0; v0 < T; ++v0) {
            for (int l = 0; l < 16 && ok; ++l) {
                const int c = 16 * v0 + l;
                if (c >= s) break;
                float* col = m.buf[c & 1];
                if (tx == l) {
#pragma unroll
                    for (int u = 0; u < T; ++u) col[ty + 16 * u] = g[u][v0];
                }
                __syncthreads();
                const float d = col[c];
                if (!(d > m.thr[c])) { ok = false; break; }
                const float inv = __frcp_rn(d);
                float r[T], f[T];
#pragma unroll
                for (int v = 0; v < T; ++v) r[v] = col[tx + 16 * v];
#pragma unroll
                for (int u = 0; u < T; ++u) {
                    const float q = col[ty + 16 * u] * inv;
                    f[u] = ty + 16 * u == c ? 1.f - inv : q;
#pragma unroll
                    for (int v = 0; v < T; ++v) g[u][v] -= f[u] * r[v];
                    if (tx == l) g[u][v0] = ty + 16 * u == c ? -inv : q;
                }
            }
        }
        bool done = false;
        double x = 0.0;                                      // threads below s
        if (ok) {
            float prev = 0.f;
            for (int itr = 0; itr <= OLS_REFINE_MAX; ++itr) {
                __syncthreads();                             // w
                float r[T];
#pragma unroll
                for (int v = 0; v < T; ++v) r[v] = m.w[tx + 16 * v];
#pragma unroll
                for (int u = 0; u < T; ++u) {
                    float y = 0.f;
#pragma unroll
                    for (int v = 0; v < T; ++v) y -= g[u][v] * r[v];
#pragma unroll
                    for (int k = 8; k > 0; k >>= 1) y += __shfl_xor_sync(0xffffffffu, y, k);
                    if (tx == 0) m.y[ty + 16 * u] = y;
                }
                __syncthreads();
                uint32_t hx = 0, hd = 0, hm = 0;
                if (tid < s) {
                    const float y = m.y[tid];
                    x += (double)y;
                    hx = fx_high(x);
                    hd = __float_as_uint(fabsf(y));
                    hm = __float_as_uint(fabsf(f64_to_f32_int(x)));
                }
                block_max3(hx, hd, hm);
                const float dmx = __uint_as_float(hd);
                const int st = ols_converged(itr, dmx, __uint_as_float(hm), prev);
                if (st) { done = st > 0; break; }
                prev = dmx;
                const int ev = hx ? fx_exponent(hx) : 0;
                if (tid < s) m.xd[tid] = fx_digits(x, ev, BITS, LOB);
                __syncthreads();
                const int row = tid % R, part = tid / R;
                if (row < s) {
                    FxFull sum;
#pragma unroll 4
                    for (int c = part; c < s; c += PARTS) sum.add(Gd[c * s + row], m.xd[c]);
                    m.part[tid] = sum.hh;
                    m.part_low[tid] = sum.low(LOB);
                }
                __syncthreads();
                if (tid < s) {
                    long long q = 0;
                    double low = 0.0;
#pragma unroll
                    for (int k = 0; k < PARTS; ++k) {
                        q += m.part[k * R + tid];
                        low += m.part_low[k * R + tid];
                    }
                    m.w[tid] = f64_to_f32_int(fx_residual(m.bs[tid], q, low, ev - 2 * BITS, LOB));
                }
            }
        }
        if (!done) {                                         // s >= s_lo > 0
            if (tid == 0) a.fb_list[atomicAdd(a.fb_count, 1)] = (int32_t)o.tg;
            continue;
        }
        x = scalbn(x, eb - e);
        if (a.jstar) {
            if (tid < s) a.chosen[((size_t)o.k * a.r + o.e) * a.p + a.ucols[my]] = x;
            continue;
        }
        if (tid < s) m.x[tid] = x;
        __syncthreads();
        // x' Ge x - 2 x' be
        const double* Ge = a.Ge + (size_t)o.k * a.pu * a.pu;
        double part = tid < s ? -2.0 * x * a.Be[((size_t)o.k * a.pu + my) * a.r + o.e] : 0.0;
        const int row = tid % R;
        if (row < s) {
            const int col = m.idx[row];
            double acc = 0.0;
#pragma unroll 8
            for (int c = tid / R; c < s; c += PARTS) acc += __ldg(Ge + (size_t)m.idx[c] * a.pu + col) * m.x[c];
            part += m.x[row] * acc;
        }
        part = warp_sum(part);
        if (lane == 0) m.redd[warp] = part;
        __syncthreads();
        if (tid == 0) {
            double tot = 0.0;
            for (int w = 0; w < 8; ++w) tot += m.redd[w];
            a.losses[o.tg] = a.yye[(size_t)o.k * a.r + o.e] + tot;
            if (a.singular) a.singular[o.tg] = 0;
        }
    }
}

// Supports of more than 128 columns: packed FP32 Cholesky factor.
__global__ void __launch_bounds__(256) k_ols_mixed(OlsArgs a)
{
    constexpr int PB = 8;                               // k chunk of the trailing update's register tiles
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int sm2 = (a.smax + 1) & ~1;
    int* idx = reinterpret_cast<int*>(smem_raw);                        // smax ints
    double* b64 = reinterpret_cast<double*>(smem_raw + sizeof(int) * sm2);
    double* x64 = b64 + sm2;
    double* red = x64 + sm2;                                            // 32 doubles
    float* w = reinterpret_cast<float*>(red + 32);                      // smax floats
    float* dinv = w + sm2;                                              // 1 / diagonal of the factor
    float* L = a.fscratch ? a.fscratch + (size_t)blockIdx.x * ((size_t)a.smax * (a.smax + 1) / 2) : dinv + sm2;
    __shared__ int s_count;
    __shared__ int64_t s_next;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    // the next solve of this CTA: a fixed stride, or the shared counter (block-uniform)
    auto fetch = [&](int64_t cur) -> int64_t {
        if (!a.next) return cur < 0 ? (int64_t)blockIdx.x : cur + gridDim.x;
        __syncthreads();                               // every thread is done with s_next
        if (threadIdx.x == 0) s_next = (int64_t)atomicAdd(a.next, 1ull);
        __syncthreads();
        return s_next;
    };

    for (int64_t t = fetch(-1); t < a.solves; t = fetch(t)) {
        const OlsSolve o = ols_solve(a, t);
        const int k = o.k, j = o.j, e = o.e;
        const int64_t tg = o.tg;
        if (warp == 0) {
            const int c = warp_support(a.family + ((int64_t)j * a.r + e) * a.W, a.W, a.p, lane, idx, a.smax);
            if (lane == 0) s_count = c;
        }
        __syncthreads();
        const int s = s_count;
        if (s < a.s_lo || s > a.smax) { __syncthreads(); continue; }
        for (int x = threadIdx.x; x < s; x += blockDim.x) idx[x] = a.upos[idx[x]];
        __syncthreads();
        const double* Gk = a.Gt + (size_t)k * a.pu * a.pu;
        const double* Bk = a.Bt + (size_t)k * a.pu * a.r;
        // gather the packed lower triangle in FP32, b in FP64
        double dm = 0.0;
        for (int i = warp; i < s; i += 8) {
            const double* grow = Gk + (size_t)idx[i] * a.pu;
            float* lrow = L + packed_row(i);
#pragma unroll 4
            for (int c = lane; c <= i; c += 32) {
                const double v = grow[idx[c]];
                lrow[c] = f64_to_f32_int(v);
                if (c == i) dm = fmax(dm, v);
            }
        }
        for (int x = threadIdx.x; x < s; x += blockDim.x) b64[x] = Bk[(size_t)idx[x] * a.r + e];
        const double dmax = block_max(dm, red, lane, warp);
        const float thr = OLS_F32_PIVOT * (float)dmax;
        // blocked right-looking Cholesky with 32-column panels: warp 0 factors the
        // diagonal block in registers (no block barrier per column), every
        // thread solves one row of the panel below it against that block, then the
        // trailing triangle takes the rank-32 update in 4 x 4 register tiles
        // (k chunks of PB) over 64 x 64 blocks of 16 x 16 threads: three barriers
        // per 32 columns
        __shared__ int s_ok;
        bool ok = true;
        for (int c0 = 0; c0 < s; c0 += 32) {
            const int c1 = min(s, c0 + 32);
            if (warp == 0) {
                // lane i holds row c0 + i of the diagonal block in registers;
                // column c of the factor travels between lanes by shuffles
                const int nb = c1 - c0;
                const bool has = lane < nb;
                float* lrow = L + packed_row(c0 + (has ? lane : 0)) + c0;
                float a[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) a[j] = (has && j <= lane) ? lrow[j] : 0.f;
                bool wok = true;
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    if (c >= nb || !wok) continue;                   // same in every lane
                    const float d = __shfl_sync(0xffffffffu, a[c], c);
                    if (!(d > thr)) { wok = false; continue; }
                    const float lcc = sqrtf(d);
                    const float inv = 1.f / lcc;
                    const float lic = lane > c ? a[c] * inv : 0.f;
                    if (lane == c) a[c] = lcc;
                    else if (lane > c) a[c] = lic;
                    if (lane == 0) dinv[c0 + c] = inv;
#pragma unroll
                    for (int j = c + 1; j < 32; ++j) {
                        const float ljc = __shfl_sync(0xffffffffu, lic, j);
                        if (lane >= j) a[j] -= lic * ljc;
                    }
                }
                if (wok && has) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j <= lane) lrow[j] = a[j];
                }
                if (lane == 0) s_ok = wok ? 1 : 0;
            }
            __syncthreads();
            if (!s_ok) { ok = false; break; }
            // panel rows below the block: L21 = A21 L11^{-T}, one row per thread
            for (int r = c1 + threadIdx.x; r < s; r += blockDim.x) {
                float* lr = L + packed_row(r);
                for (int c = c0; c < c1; ++c) {
                    const float* lc = L + packed_row(c);
                    float acc = lr[c];
                    for (int t = c0; t < c; ++t) acc -= lr[t] * lc[t];
                    lr[c] = acc * dinv[c];
                }
            }
            __syncthreads();
            const int T = s - c1;
            const int nbk = (T + 63) / 64;
            for (int pr = 0; pr < nbk * (nbk + 1) / 2; ++pr) {
                int bi = (int)((sqrtf(8.f * pr + 1.f) - 1.f) * 0.5f);
                while ((bi + 1) * (bi + 2) / 2 <= pr) ++bi;
                while (bi * (bi + 1) / 2 > pr) --bi;
                const int bj = pr - bi * (bi + 1) / 2;
                const int i0 = c1 + bi * 64, j0 = c1 + bj * 64;
                float acc[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
                for (int k0 = c0; k0 < c1; k0 += PB) {
                    float li[4][PB], lj[4][PB];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = i0 + ty + 16 * u, j = j0 + tx + 16 * u;
#pragma unroll
                        for (int t = 0; t < PB; ++t) {
                            const bool kin = k0 + t < c1;
                            li[u][t] = (i < s && kin) ? L[packed_row(i) + k0 + t] : 0.f;
                            lj[u][t] = (j < s && kin) ? L[packed_row(j) + k0 + t] : 0.f;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int v = 0; v < 4; ++v)
#pragma unroll
                            for (int t = 0; t < PB; ++t) acc[u][v] += li[u][t] * lj[v][t];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + ty + 16 * u;
                    if (i >= s) break;
                    float* lrow = L + packed_row(i);
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int j = j0 + tx + 16 * v;
                        if (j > i) break;
                        lrow[j] -= acc[u][v];
                    }
                }
            }
            __syncthreads();
        }
        bool done = false;
        if (ok) {
            // x = solve(b) in FP32, then x += solve(b - G x) with FP64 residuals
            for (int x = threadIdx.x; x < s; x += blockDim.x) { w[x] = (float)b64[x]; x64[x] = 0.0; }
            __syncthreads();
            double prev = 0.0;
            for (int itr = 0; itr <= OLS_REFINE_MAX; ++itr) {
                chol_solve_f32(L, dinv, w, s, warp, lane);
                double dd = 0.0, xx = 0.0;
                for (int x = threadIdx.x; x < s; x += blockDim.x) {
                    const double nx = x64[x] + (double)w[x];
                    dd = fmax(dd, fabs((double)w[x]));
                    xx = fmax(xx, fabs(nx));
                    x64[x] = nx;
                }
                const double dmx = block_max(dd, red, lane, warp);
                const double xmx = block_max(xx, red, lane, warp);
                // converged: the correction is at the level of FP64 rounding of the
                // residual, or it no longer shrinks (the residual is rounding noise)
                if (itr > 0 && (dmx <= 1e-14 * xmx || (dmx > 0.5 * prev && dmx <= 1e-12 * xmx))) {
                    done = true;
                    break;
                }
                if (itr == OLS_REFINE_MAX) { done = dmx <= 1e-12 * xmx; break; }
                prev = dmx;
                // residual r_i = b_i - sum_c G[S_i, S_c] x_c (one warp per row)
                for (int i = warp; i < s; i += 8) {
                    const double* grow = Gk + (size_t)idx[i] * a.pu;
                    double acc = 0.0;
#pragma unroll 4
                    for (int c = lane; c < s; c += 32) acc += grow[idx[c]] * x64[c];
                    acc = warp_sum(acc);
                    if (lane == 0) w[i] = (float)(b64[i] - acc);
                }
                __syncthreads();
            }
        }
        if (s > 0 && !done) {
            if (threadIdx.x == 0) a.fb_list[atomicAdd(a.fb_count, 1)] = (int32_t)tg;
            __syncthreads();
            continue;
        }
        if (a.jstar) {
            double* out = a.chosen + ((size_t)k * a.r + e) * a.p;
            for (int x = threadIdx.x; x < s; x += blockDim.x) out[a.ucols[idx[x]]] = x64[x];
        } else {
            const double* Gek = a.Ge + (size_t)k * a.pu * a.pu;
            const double* Bek = a.Be + (size_t)k * a.pu * a.r;
            double part = 0.0;
            for (int i = warp; i < s; i += 8) {
                const double* grow = Gek + (size_t)idx[i] * a.pu;
                double acc = 0.0;
#pragma unroll 4
                for (int c = lane; c < s; c += 32) acc += grow[idx[c]] * x64[c];
                acc = warp_sum(acc);
                if (lane == 0) part += x64[i] * acc;
            }
            for (int x = threadIdx.x; x < s; x += blockDim.x)
                part -= 2.0 * x64[x] * Bek[(size_t)idx[x] * a.r + e];
            const double tot = block_sum(part, red, lane, warp);
            if (threadIdx.x == 0) {
                const int64_t o = ((int64_t)k * a.q + j) * a.r + e;
                a.losses[o] = a.yye[(size_t)k * a.r + e] + tot;
                if (a.singular) a.singular[o] = 0;
            }
        }
        __syncthreads();
    }
}

// out[k][a][b] = G[k][cols[a]][cols[b]] (restriction to the union U).
__global__ void k_gather_gram(const double* G, int64_t p, const int32_t* cols, int64_t u, int32_t B,
                              double* out)
{
    const int64_t per = u * u, total = (int64_t)B * per;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / per, rem = t % per;
        out[t] = G[(k * p + cols[rem / u]) * p + cols[rem % u]];
    }
}

// out[k][a][e] = Bm[k][cols[a]][e].
__global__ void k_gather_rhs(const double* Bm, int64_t p, int64_t r, const int32_t* cols, int64_t u,
                             int32_t B, double* out)
{
    const int64_t per = u * r, total = (int64_t)B * per;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / per, rem = t % per;
        out[t] = Bm[(k * p + cols[rem / r]) * r + rem % r];
    }
}

__global__ void k_union_pos(const int32_t* cols, int64_t u, int32_t* pos)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < u;
         t += (int64_t)gridDim.x * blockDim.x)
        pos[cols[t]] = (int32_t)t;
}

// dup[j*r + e] = smallest j' <= j whose support for response e equals S_{j,e}.
__global__ void k_family_dedup(const uint64_t* fam, int32_t q, int64_t r, int W, int32_t* dup)
{
    const int64_t total = (int64_t)q * r;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(t / r);
        const int64_t e = t % r;
        const uint64_t* a = fam + t * W;
        int first = j;
        for (int jj = 0; jj < j; ++jj) {
            const uint64_t* b = fam + ((int64_t)jj * r + e) * W;
            bool same = true;
            for (int w = 0; w < W && same; ++w) same = a[w] == b[w];
            if (same) { first = jj; break; }
        }
        dup[t] = first;
    }
}

// Copy the loss (and flag) of the representative to every duplicate (k, j, e).
__global__ void k_fill_duplicates(const int32_t* dup, int32_t B2, int32_t q, int64_t r,
                                  double* losses, int32_t* singular)
{
    const int64_t total = (int64_t)B2 * q * r;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / ((int64_t)q * r), rem = t % ((int64_t)q * r);
        const int64_t e = rem % r;
        const int32_t j0 = dup[rem];
        if (j0 == (int32_t)(rem / r)) continue;
        const int64_t src = (k * q + j0) * r + e;
        losses[t] = losses[src];
        if (singular) singular[t] = singular[src];
    }
}

__global__ void k_support_sizes(const uint64_t* fam, int64_t count, int W, int32_t* out)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * blockDim.x) {
        int c = 0;
        for (int w = 0; w < W; ++w) c += __popcll(fam[t * W + w]);
        out[t] = c;
    }
}

__global__ void k_support_max(const uint64_t* fam, int64_t count, int W, int32_t* out)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * blockDim.x) {
        int c = 0;
        for (int w = 0; w < W; ++w) c += __popcll(fam[t * W + w]);
        atomicMax(out, c);
    }
}

// Lane = lambda, each adding its responses in order; ties go to the smallest j.
__global__ void k_argmin(const double* losses, int32_t q, int64_t r, int32_t* jstar)
{
    const int k = blockIdx.x, lane = threadIdx.x;
    int best = 0x7fffffff;
    double bv = 0.0;
    bool nan0 = false;
    for (int j = lane; j < q; j += 32) {
        double s = 0.0;
#pragma unroll 8
        for (int64_t e = 0; e < r; ++e) s += losses[((int64_t)k * q + j) * r + e];
        if (j == 0) nan0 = s != s;
        if (s == s && (best == 0x7fffffff || s < bv)) { bv = s; best = j; }
    }
    // a NaN at j = 0 is never improved on, one at a later j never chosen
    nan0 = __shfl_sync(0xffffffffu, nan0 ? 1 : 0, 0) != 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int ob = __shfl_xor_sync(0xffffffffu, best, o);
        const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
        if (ob != 0x7fffffff && (best == 0x7fffffff || ov < bv || (ov == bv && ob < best))) { bv = ov; best = ob; }
    }
    if (nan0) best = 0;
    if (lane == 0) jstar[k] = best;
}

__device__ void bag_sorted(double* v, int n, double* out)    // by insertion, in place
{
    for (int k = 1; k < n; ++k) {
        const double x = v[k * 33];
        int t = k;
        while (t > 0 && v[(t - 1) * 33] > x) { v[t * 33] = v[(t - 1) * 33]; --t; }
        v[t * 33] = x;
    }
    *out = (n & 1) ? v[n / 2 * 33] : 0.5 * (v[(n / 2 - 1) * 33] + v[n / 2 * 33]);
}

// Mean: one thread per coefficient.  Median: 32 coefficients per CTA through shared memory,
// a warp per coefficient; each lane holds up to four of the B2 <= 128 values and counts those
// before them (by value, then by bootstrap) on integer keys that order as the values do.
__global__ void __launch_bounds__(256) k_bagging(const double* chosen, int32_t B2, int64_t count, int32_t mode,
                                                 double* out)
{
    if (mode == UOI_BAG_MEAN) {
        for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < count;
             c += (int64_t)gridDim.x * blockDim.x) {
            double s = 0.0;
            for (int k = 0; k < B2; ++k) s += chosen[(int64_t)k * count + c];
            out[c] = s / (double)B2;
        }
        return;
    }
    __shared__ double v[128 * 33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = B2 < 128 ? B2 : 128;
    for (int64_t c0 = blockIdx.x * (int64_t)32; c0 < count; c0 += (int64_t)gridDim.x * 32) {
        __syncthreads();
        for (int k = warp; k < n; k += 8)
            if (c0 + lane < count) v[k * 33 + lane] = chosen[(int64_t)k * count + c0 + lane];
        __syncthreads();
        for (int i = warp; i < 32 && c0 + i < count; i += 8) {
            double x[4];
            long long key[4];
            bool zero = true, nan = false;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = lane + 32 * u;
                x[u] = k < n ? v[k * 33 + i] : 0.0;
                const long long b = __double_as_longlong(x[u]), mag = b & 0x7FFFFFFFFFFFFFFFll;
                zero &= b == 0;
                nan |= mag > 0x7FF0000000000000ll;
                key[u] = b < 0 ? -mag : mag;
            }
            if (__all_sync(0xffffffffu, zero)) {             // outside every chosen support
                if (lane == 0) out[c0 + i] = 0.0;
                continue;
            }
            if (__any_sync(0xffffffffu, nan)) {
                if (lane == 0) bag_sorted(v + i, n, out + c0 + i);
                continue;
            }
            int before[4] = { 0, 0, 0, 0 };
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const int m = min(32, n - 32 * w);
                for (int l = 0; l < m; ++l) {
                    const long long o = __shfl_sync(0xffffffffu, key[w], l);
                    const int k = 32 * w + l;
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (32 * u < n) before[u] += o < key[u] || (o == key[u] && k < lane + 32 * u) ? 1 : 0;
                }
            }
            // the values of rank n / 2 and n / 2 - 1, each held by one lane
            double hi = 0.0, lo = 0.0;
            bool has_hi = false, has_lo = false;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (lane + 32 * u >= n) continue;
                if (before[u] == n / 2) { hi = x[u]; has_hi = true; }
                if (before[u] == n / 2 - 1) { lo = x[u]; has_lo = true; }
            }
            const unsigned bh = __ballot_sync(0xffffffffu, has_hi), bl = __ballot_sync(0xffffffffu, has_lo);
            hi = __shfl_sync(0xffffffffu, hi, __ffs(bh) - 1);
            if (!(n & 1)) hi = 0.5 * (__shfl_sync(0xffffffffu, lo, __ffs(bl) - 1) + hi);
            if (lane == 0) out[c0 + i] = hi;
        }
    }
}

__global__ void k_mask_tail(uint64_t* fam, int64_t count, int W, uint64_t mask)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * blockDim.x)
        fam[t * W + (W - 1)] &= mask;
}

int32_t family_support_max(const OlsArgs& a, cudaStream_t s)
{
    DevBuf mx(sizeof(int32_t), s);
    UOI_CUDA(cudaMemsetAsync(mx.ptr, 0, sizeof(int32_t), s));
    const int64_t fam_count = (int64_t)a.q * a.r;
    k_support_max<<<(unsigned)std::min<int64_t>(ceil_div(fam_count, 256), 1024), 256, 0, s>>>(
        a.family, fam_count, a.W, mx.as<int32_t>());
    UOI_CHECK_LAUNCH();
    count_launch();
    int32_t smax = 0;
    UOI_CUDA(cudaMemcpyAsync(&smax, mx.ptr, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    UOI_CUDA(cudaStreamSynchronize(s));
    return smax;
}

// FP64 solves (all of a.solves, or those listed in a.list); a.smax set.
void launch_ols_fp64(OlsArgs a, cudaStream_t s)
{
    a.use_smem = a.smax <= OLS_SMEM_MAX;
    size_t smem = sizeof(int) * ((a.smax + 1) & ~1) + sizeof(double) * (3 * (a.smax + 1) + 32);
    DevBuf scratch;
    int grid = (int)std::min<int64_t>(a.solves, 152 * 8);
    if (a.use_smem) {
        smem += sizeof(double) * (size_t)a.smax * a.smax;
    } else {
        grid = (int)std::min<int64_t>(a.solves, 152 * 2);
        scratch.alloc(sizeof(double) * (size_t)grid * a.smax * a.smax, s);
        a.scratch = scratch.as<double>();
    }
    allow_max_dynamic_smem((const void*)k_ols);
    if (a.solves > 0) {
        k_ols<<<grid, 256, smem, s>>>(a);
        UOI_CHECK_LAUNCH();
        count_launch();
    }
}

// Mixed pass: launches the kernel of class `cls` (OLS_CLASS_MAX) over a.solves; those it hands
// back go to a.fb_list.
void launch_ols_class(OlsArgs a, int cls, DevBuf& fscratch, cudaStream_t s)
{
    if (a.solves == 0) return;
    a.s_lo = cls == 0 ? 0 : OLS_CLASS_MAX[cls - 1] + 1;
    a.smax = std::max(1, std::min(a.smax, OLS_CLASS_MAX[cls]));
    int dev = 0, nsm = 0, per = 0, threads = 256;
    UOI_CUDA(cudaGetDevice(&dev));
    UOI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const void* kern;
    size_t smem;
    int64_t work = a.solves;
    const size_t digits = sizeof(int2) * (size_t)a.smax * a.smax;
    if (cls == 0) {
        kern = (const void*)k_ols_warp;
        threads = 32 * OLS_WARPS;
        smem = OLS_WARPS * (sizeof(OlsWarpSmem) + digits);
        work = ceil_div(a.solves, OLS_WARPS);
    } else if (cls == 1) {
        kern = (const void*)k_ols_block<4>;
        smem = sizeof(OlsBlockSmem<4>) + digits;
    } else if (cls == 2) {
        kern = (const void*)k_ols_block<8>;
        smem = sizeof(OlsBlockSmem<8>) + digits;
    } else {
        kern = (const void*)k_ols_mixed;
        const int sm2 = (a.smax + 1) & ~1;
        const size_t base = sizeof(int) * sm2 + 2 * sizeof(double) * sm2 + 32 * sizeof(double) +
                            2 * sizeof(float) * sm2;
        const size_t lbytes = sizeof(float) * (size_t)a.smax * (a.smax + 1) / 2;
        const bool in_smem = base + lbytes <= 227 * 1024 - 64;
        smem = base + (in_smem ? lbytes : 0);
        if (!in_smem) {
            allow_max_dynamic_smem(kern);
            UOI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem));
            fscratch.alloc(lbytes * (size_t)std::min<int64_t>(work, (int64_t)nsm * std::max(1, per)), s);
            a.fscratch = fscratch.as<float>();
        }
    }
    allow_max_dynamic_smem(kern);
    UOI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem));
    const int grid = (int)std::min<int64_t>(work, (int64_t)nsm * std::max(1, per));
    if (cls == 0) k_ols_warp<<<grid, threads, smem, s>>>(a);
    else if (cls == 1) k_ols_block<4><<<grid, threads, smem, s>>>(a);
    else if (cls == 2) k_ols_block<8><<<grid, threads, smem, s>>>(a);
    else k_ols_mixed<<<grid, threads, smem, s>>>(a);
    UOI_CHECK_LAUNCH();
    count_launch();
}

// Work on `side` between the constructor and done() follows what s has queued and precedes
// what s queues afterwards (also when an exception leaves the scope: the buffers go back to
// their pool in the order of s).
struct SideJoin {
    cudaStream_t side, s;
    cudaEvent_t ev = nullptr;
    SideJoin(cudaStream_t side_, cudaStream_t s_) : side(side_), s(s_)
    {
        if (side == s) return;
        UOI_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        UOI_CUDA(cudaEventRecord(ev, s));
        UOI_CUDA(cudaStreamWaitEvent(side, ev, 0));
    }
    SideJoin(const SideJoin&) = delete;
    SideJoin& operator=(const SideJoin&) = delete;
    void done()
    {
        if (!ev) return;
        UOI_CUDA(cudaEventRecord(ev, side));
        UOI_CUDA(cudaStreamWaitEvent(s, ev, 0));
        cudaEventDestroy(ev);
        ev = nullptr;
    }
    ~SideJoin()
    {
        if (!ev) return;
        if (cudaEventRecord(ev, side) == cudaSuccess) cudaStreamWaitEvent(s, ev, 0);
        cudaEventDestroy(ev);
    }
};

// The FP64 kernel for the solves that the mixed pass handed back (waits for their count).
int64_t finish_ols(OlsArgs a, int smax, cudaStream_t s)
{
    int32_t nfb = 0;
    UOI_CUDA(cudaMemcpyAsync(&nfb, a.fb_count, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    UOI_CUDA(cudaStreamSynchronize(s));
    if (nfb > 0) {
        a.smax = smax;
        a.list = a.fb_list;
        a.solves = nfb;
        launch_ols_fp64(a, s);
    }
    return nfb;
}

// U = union over (j, e) of the family supports, compacted in increasing order.  One block:
// every thread ORs one word over its share of the members, then warp 0 lists the set bits.
constexpr int UNION_WORDS = 1024;
__global__ void __launch_bounds__(UNION_WORDS) k_union_cols(const uint64_t* fam, int64_t count, int W, int64_t p,
                                                            int32_t* cols, int32_t* n_out)
{
    __shared__ unsigned long long word[UNION_WORDS];
    const int lane = threadIdx.x & 31;
    int n = 0;                                               // columns listed so far (warp 0)
    for (int w0 = 0; w0 < W; w0 += UNION_WORDS) {
        const int wc = min(W - w0, UNION_WORDS), shares = UNION_WORDS / wc;
        const int w = threadIdx.x % wc, share = threadIdx.x / wc;
        word[threadIdx.x] = 0;
        __syncthreads();
        unsigned long long acc = 0;
        if (share < shares)
#pragma unroll 4
            for (int64_t t = share; t < count; t += shares) acc |= fam[t * W + w0 + w];
        if (acc) atomicOr(&word[w], acc);
        __syncthreads();
        if (threadIdx.x < 32)
            n += warp_support((const uint64_t*)word, wc, p - (int64_t)w0 * 64, lane, cols + n, 0x7fffffff, w0 * 64);
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_out = n;
}

}  // namespace

// A second stream per host thread and device, for work that runs beside the thread's main
// stream (the smaller classes of the loss pass, half of the batch of the tensor-core
// inverse, sums of the warm-start gradient).  A thread takes one on first use and hands it on
// when it ends (idle: every user waits for it), so there are as many as threads were at work at
// once; uoi_shutdown destroys those no thread holds.  Destroying them with each batch's workers
// cost 2 to 4 % of a batch of 24.
namespace {
struct SidePool {
    std::mutex mu;
    std::vector<std::vector<cudaStream_t>> idle;             // by device
};
SidePool& side_pool()
{
    static SidePool* pool = new SidePool;                    // outlives the threads that hand streams back
    return *pool;
}
struct SideStreams {
    std::vector<cudaStream_t> of;                            // by device
    ~SideStreams()
    {
        SidePool& p = side_pool();
        std::lock_guard<std::mutex> lock(p.mu);
        if (p.idle.size() < of.size()) p.idle.resize(of.size());
        for (size_t d = 0; d < of.size(); ++d)
            if (of[d]) p.idle[d].push_back(of[d]);
    }
};
}  // namespace

cudaStream_t side_stream()
{
    thread_local SideStreams mine;
    int dev = 0;
    UOI_CUDA(cudaGetDevice(&dev));
    if ((size_t)dev >= mine.of.size()) mine.of.resize((size_t)dev + 1, nullptr);
    cudaStream_t& q = mine.of[(size_t)dev];
    if (!q) {
        SidePool& p = side_pool();
        std::lock_guard<std::mutex> lock(p.mu);
        if ((size_t)dev < p.idle.size() && !p.idle[(size_t)dev].empty()) {
            q = p.idle[(size_t)dev].back();
            p.idle[(size_t)dev].pop_back();
        }
    }
    if (!q) UOI_CUDA(cudaStreamCreateWithFlags(&q, cudaStreamNonBlocking));
    return q;
}

void release_side_streams(int dev)
{
    SidePool& p = side_pool();
    std::lock_guard<std::mutex> lock(p.mu);
    if ((size_t)dev >= p.idle.size()) return;
    for (cudaStream_t q : p.idle[(size_t)dev]) cudaStreamDestroy(q);
    p.idle[(size_t)dev].clear();
}

int32_t union_columns(const uint64_t* family, int64_t count, int64_t p, int32_t* cols,
                      cudaStream_t s)
{
    DevBuf n(sizeof(int32_t), s);
    k_union_cols<<<1, UNION_WORDS, 0, s>>>(family, count, (int)((p + 63) / 64), p, cols, n.as<int32_t>());
    UOI_CHECK_LAUNCH();
    count_launch();
    int32_t h = 0;
    UOI_CUDA(cudaMemcpyAsync(&h, n.ptr, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    UOI_CUDA(cudaStreamSynchronize(s));
    return h;
}

void family_init(uint64_t* fam, int64_t words, cudaStream_t s)
{
    UOI_CUDA(cudaMemsetAsync(fam, 0xFF, sizeof(uint64_t) * (size_t)words, s));
}

void family_mask_tail(uint64_t* fam, int64_t count, int64_t p, cudaStream_t s)
{
    if ((p & 63) == 0) return;
    const int W = (int)((p + 63) / 64);
    k_mask_tail<<<(unsigned)std::min<int64_t>(ceil_div(count, 256), 1024), 256, 0, s>>>(
        fam, count, W, (1ull << (p & 63)) - 1ull);
    UOI_CHECK_LAUNCH();
    count_launch();
}

namespace {

// The OLS solves only touch rows and columns in the union U of the family
// supports: restricting the moments to U once per call makes every later
// access a read of a small, L2-resident matrix.
struct UnionMoments {
    DevBuf cols, pos, Gt, Bt, Ge, Be;
    int64_t pu = 0;
};

void restrict_to_union(const uint64_t* family, int64_t p, int64_t r, int32_t q, int32_t B2,
                       const double* Gt, const double* Bt, const double* Ge, const double* Be,
                       UnionMoments& U, cudaStream_t s)
{
    U.cols.alloc(sizeof(int32_t) * (size_t)std::max<int64_t>(p, 1), s);
    U.pu = union_columns(family, (int64_t)q * r, p, U.cols.as<int32_t>(), s);
    const int64_t u1 = std::max<int64_t>(U.pu, 1);
    U.pos.alloc(sizeof(int32_t) * (size_t)std::max<int64_t>(p, 1), s);
    UOI_CUDA(cudaMemsetAsync(U.pos.ptr, 0xFF, sizeof(int32_t) * (size_t)p, s));
    k_union_pos<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(U.pu, 256), 64)), 256, 0, s>>>(
        U.cols.as<int32_t>(), U.pu, U.pos.as<int32_t>());
    UOI_CHECK_LAUNCH();
    count_launch();
    auto gram = [&](const double* G, DevBuf& out) {
        out.alloc(sizeof(double) * (size_t)(B2 * u1 * u1), s);
        const int64_t total = (int64_t)B2 * U.pu * U.pu;
        if (total == 0) return;
        k_gather_gram<<<(unsigned)std::min<int64_t>(ceil_div(total, 256), 152 * 32), 256, 0, s>>>(
            G, p, U.cols.as<int32_t>(), U.pu, B2, out.as<double>());
        UOI_CHECK_LAUNCH();
        count_launch();
    };
    auto rhs = [&](const double* Bm, DevBuf& out) {
        out.alloc(sizeof(double) * (size_t)(B2 * u1 * r), s);
        const int64_t total = (int64_t)B2 * U.pu * r;
        if (total == 0) return;
        k_gather_rhs<<<(unsigned)std::min<int64_t>(ceil_div(total, 256), 152 * 32), 256, 0, s>>>(
            Bm, p, r, U.cols.as<int32_t>(), U.pu, B2, out.as<double>());
        UOI_CHECK_LAUNCH();
        count_launch();
    };
    gram(Gt, U.Gt);
    rhs(Bt, U.Bt);
    if (Ge) { gram(Ge, U.Ge); rhs(Be, U.Be); }
}

void use_union(OlsArgs& a, const UnionMoments& U)
{
    a.Gt = U.Gt.as<double>(); a.Bt = U.Bt.as<double>();
    a.Ge = U.Ge.ptr ? U.Ge.as<double>() : nullptr;
    a.Be = U.Be.ptr ? U.Be.as<double>() : nullptr;
    a.upos = U.pos.as<int32_t>(); a.ucols = U.cols.as<int32_t>(); a.pu = U.pu;
}

}  // namespace

int64_t ols_losses(const double* Gt, const double* Bt, const double* Ge, const double* Be,
                const double* yye, const uint64_t* family, int64_t p, int64_t r, int32_t q,
                int32_t B2, double* losses, int32_t* singular, cudaStream_t s)
{
    UnionMoments U;
    restrict_to_union(family, p, r, q, B2, Gt, Bt, Ge, Be, U, s);
    OlsArgs a{};
    use_union(a, U);
    a.yye = yye; a.family = family;
    a.p = p; a.r = r; a.q = q; a.B2 = B2; a.W = (int32_t)((p + 63) / 64);
    a.losses = losses; a.singular = singular;
    a.solves = (int64_t)B2 * q * r;
    DevBuf dup(sizeof(int32_t) * (size_t)(q * r), s);
    const unsigned gd = (unsigned)std::min<int64_t>(ceil_div((int64_t)q * r, 256), 1024);
    k_family_dedup<<<gd, 256, 0, s>>>(family, q, r, a.W, dup.as<int32_t>());
    UOI_CHECK_LAUNCH();
    a.dup = dup.as<int32_t>();
    // Size classes: small supports run with little shared memory per CTA (many
    // CTAs per SM hide the latency of their short dependent steps); large ones
    // with room for their factor.  Only first occurrences of a support are listed.
    const int64_t qr = (int64_t)q * r;
    DevBuf sizes(sizeof(int32_t) * (size_t)qr, s);
    k_support_sizes<<<(unsigned)std::min<int64_t>(ceil_div(qr, 256), 1024), 256, 0, s>>>(
        family, qr, a.W, sizes.as<int32_t>());
    UOI_CHECK_LAUNCH();
    count_launch();
    std::vector<int32_t> hsz((size_t)qr), hdup((size_t)qr);
    UOI_CUDA(cudaMemcpyAsync(hsz.data(), sizes.ptr, sizeof(int32_t) * qr, cudaMemcpyDeviceToHost, s));
    UOI_CUDA(cudaMemcpyAsync(hdup.data(), dup.ptr, sizeof(int32_t) * qr, cudaMemcpyDeviceToHost, s));
    UOI_CUDA(cudaStreamSynchronize(s));
    std::vector<int32_t> lists[OLS_CLASSES];
    int32_t smax = 1;
    for (int64_t t = 0; t < qr; ++t) {
        if (hdup[t] != (int32_t)(t / r)) continue;
        int cls = 0;
        while (hsz[t] > OLS_CLASS_MAX[cls]) ++cls;
        lists[cls].push_back((int32_t)t);
        smax = std::max(smax, hsz[t]);
    }
    if (smax > 46000) throw Error(UOI_ERR_UNSUPPORTED, "OLS support larger than 46000 columns");
    DevBuf ctr(sizeof(unsigned long long) * OLS_CLASSES, s), fbc(sizeof(int32_t), s);
    DevBuf fbl(sizeof(int32_t) * (size_t)std::max<int64_t>(a.solves, 1), s);
    UOI_CUDA(cudaMemsetAsync(ctr.ptr, 0, ctr.bytes, s));
    UOI_CUDA(cudaMemsetAsync(fbc.ptr, 0, fbc.bytes, s));
    a.fb_list = fbl.as<int32_t>();
    a.fb_count = fbc.as<int32_t>();
    // largest supports first within each class, taken from a counter as CTAs or warps
    // free up (the factor costs grow as the cube of the support size)
    std::vector<int32_t> order;
    int64_t start[OLS_CLASSES + 1] = {};
    int classes = 0, top = 0;
    for (int cls = 0; cls < OLS_CLASSES; ++cls) {
        std::stable_sort(lists[cls].begin(), lists[cls].end(),
                         [&](int32_t x, int32_t y) { return hsz[(size_t)x] > hsz[(size_t)y]; });
        order.insert(order.end(), lists[cls].begin(), lists[cls].end());
        start[cls + 1] = (int64_t)order.size();
        if (!lists[cls].empty()) { ++classes; top = cls; }
    }
    DevBuf jl(sizeof(int32_t) * std::max<size_t>(order.size(), 1), s);
    UOI_CUDA(cudaMemcpyAsync(jl.ptr, order.data(), sizeof(int32_t) * order.size(), cudaMemcpyHostToDevice, s));
    // the classes run side by side: the one of the largest supports on s, the others on a
    // second stream that starts after everything s has queued so far
    DevBuf fscratch;
    cudaStream_t side = classes < 2 ? s : side_stream();
    SideJoin join(side, s);
    for (int cls = OLS_CLASSES - 1; cls >= 0; --cls) {
        if (lists[cls].empty()) continue;
        OlsArgs b = a;
        b.je_list = jl.as<int32_t>() + start[cls];
        b.next = ctr.as<unsigned long long>() + cls;
        b.solves = (int64_t)B2 * (int64_t)lists[cls].size();
        b.smax = hsz[(size_t)lists[cls][0]];
        launch_ols_class(b, cls, fscratch, cls == top ? s : side);
    }
    join.done();
    const int64_t nfb = finish_ols(a, smax, s);
    const unsigned gf = (unsigned)std::min<int64_t>(ceil_div(a.solves, 256), 4096);
    k_fill_duplicates<<<gf, 256, 0, s>>>(dup.as<int32_t>(), B2, q, r, losses, singular);
    UOI_CHECK_LAUNCH();
    count_launch(2);
    return nfb;
}

void loss_argmin(const double* losses, int32_t B2, int32_t q, int64_t r, int32_t* jstar,
                 cudaStream_t s)
{
    k_argmin<<<B2, 32, 0, s>>>(losses, q, r, jstar);
    UOI_CHECK_LAUNCH();
    count_launch();
}

int64_t ols_chosen(const double* Gt, const double* Bt, const uint64_t* family, const int32_t* jstar,
                int64_t p, int64_t r, int32_t q, int32_t B2, double* chosen, cudaStream_t s)
{
    UOI_CUDA(cudaMemsetAsync(chosen, 0, sizeof(double) * (size_t)(B2 * r * p), s));
    UnionMoments U;
    restrict_to_union(family, p, r, q, B2, Gt, Bt, nullptr, nullptr, U, s);
    OlsArgs a{};
    use_union(a, U);
    a.family = family;
    a.p = p; a.r = r; a.q = q; a.B2 = B2; a.W = (int32_t)((p + 63) / 64);
    a.jstar = jstar; a.chosen = chosen;
    a.solves = (int64_t)B2 * r;
    const int smax = std::max(1, (int)family_support_max(a, s));
    if (smax > 46000) throw Error(UOI_ERR_UNSUPPORTED, "OLS support larger than 46000 columns");
    DevBuf fbl(sizeof(int32_t) * (size_t)a.solves, s), fbc(sizeof(int32_t), s), fscratch;
    UOI_CUDA(cudaMemsetAsync(fbc.ptr, 0, fbc.bytes, s));
    a.fb_list = fbl.as<int32_t>();
    a.fb_count = fbc.as<int32_t>();
    a.smax = smax;
    // the sizes of the chosen supports are on the device: each class runs its own and skips the rest
    for (int cls = 0; cls < OLS_CLASSES && (cls == 0 || smax > OLS_CLASS_MAX[cls - 1]); ++cls)
        launch_ols_class(a, cls, fscratch, s);
    return finish_ols(a, smax, s);
}

void bagging(const double* chosen, int32_t B2, int64_t count, int32_t mode, double* out,
             cudaStream_t s)
{
    k_bagging<<<(unsigned)std::min<int64_t>(ceil_div(count, 32), 4096), 256, 0, s>>>(
        chosen, B2, count, mode, out);
    UOI_CHECK_LAUNCH();
    count_launch();
}

}  // namespace uoi
