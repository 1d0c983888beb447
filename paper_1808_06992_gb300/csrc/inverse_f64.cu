// inverse_f64.cu -- G3 in FP64 accuracy without an FP64 factorisation: M_k = (G_k/n_k + rho I)^{-1}
// by Newton's iteration from an FP32 inverse.
//
// The system is equilibrated by powers of two, A^ = D A D with diagonal in [1/8, 1), which is
// exact and makes the iteration (as a Cholesky factor is) indifferent to the scale of the
// columns.  M_0 is the FP32 inverse of A^.  Each step forms R = I - A^ M with FP64-accurate
// products (exact integer slices on the tensor cores, gram_f64tc.cu) and adds M R: as R is
// small, an FP32 product is enough, and the error of M falls from e to e (e + c 2^-24).  A step
// whose residual is at most 2^-30 (largest row sum) is the last: what it leaves is below
// 2^-52 of M.  Each system stops on its own residual, summed in a fixed order: its bits are those
// it has alone.  Two steps do for condition numbers of a few hundred, three or four for 10^5.
// A system whose residual starts at 1 or more, or stops shrinking, is left to the FP64 Cholesky
// factor.
//
// Why: this part's FP64 pipe takes 19 clocks per warp multiply-add, and factor, triangular
// inverse and product need p^3 / 2 of them per system; here FP64 work is p^2 per step.
// Measured, 20 systems, factor stage against Cholesky, triangular inverse and product in FP64:
// p = 1000 33.3 -> 9.0 ms (residuals 4, FP32 products 2.8, FP32 inverse 1.5), 600 10.9 -> 3.15,
// 400 4.9 -> 1.6, 150 1.26 -> 0.43, 65 0.40 -> 0.30; below 64 columns the
// factor's 0.35 ms are not beaten.  |M b| against 80-bit arithmetic: the factor's error or
// less (tests/test_gpu_inverse_newton.py).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "kernels.h"
#include "tile.cuh"

namespace uoi {

namespace {

// e_i with (G_ii / n + rho) 2^(-2 e_i) in [1/8, 1).
__global__ void k_equil_exponents(const double* G, const double* nk, double rho, int64_t p, int32_t B, int32_t* ex)
{
    const int64_t total = (int64_t)B * p;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / p, i = t % p;
        const double a = G[(k * p + i) * p + i] * (1.0 / nk[k]) + rho;
        int e = 0;
        if (a > 0.0 && a < INFINITY) frexp(a, &e);
        ex[t] = (e + 1) >> 1;
    }
}

// A^ in FP64 and in FP32 (block.y: system; rows over blocks).
__global__ void __launch_bounds__(256) k_build_equil(const double* __restrict__ G, const double* nk, double rho, int64_t p,
                                                     const int32_t* ex, double* __restrict__ A, float* __restrict__ A32)
{
    const int64_t k = blockIdx.y;
    const double inv_n = 1.0 / nk[k];
    const int32_t* e = ex + k * p;
    for (int64_t i = blockIdx.x; i < p; i += gridDim.x) {
        const int64_t o = (k * p + i) * p;
        const double si = scalbn(1.0, -e[i]);
#pragma unroll 4
        for (int64_t j = threadIdx.x; j < p; j += blockDim.x) {
            const double v = (__ldg(G + o + j) * inv_n + (i == j ? rho : 0.0)) * si * scalbn(1.0, -e[j]);
            A[o + j] = v;
            A32[o + j] = f64_to_f32_int(v);
        }
    }
}

__global__ void k_widen(const float* __restrict__ src, double* __restrict__ dst, int64_t count)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x)
        dst[t] = (double)src[t];
}

// What a system does with its residual.
enum NewtonAction : int32_t { NEWTON_NONE = 0, NEWTON_STEP = 1, NEWTON_FINISH = -1 };

// M += M32 R (FP32 product), M32out = M rounded.
__global__ void __launch_bounds__(256) k_newton_step(const int32_t* action, double* M, const float* M32, const float* R,
                                                     float* M32out, int64_t p)
{
    if (action[blockIdx.y] != NEWTON_STEP) return;
    const int64_t base = blockIdx.y * p * p, tt = (p + 63) / 64;
    const int64_t i0 = (blockIdx.x / tt) * 64, j0 = (blockIdx.x % tt) * 64;
    float acc[4][4] = {};
    tile64_acc<float, true, false>(
        acc, [&](int il, int64_t s) { return i0 + il < p ? __ldg(M32 + base + (i0 + il) * p + s) : 0.f; },
        [&](int64_t s, int jl) { return j0 + jl < p ? __ldg(R + base + s * p + j0 + jl) : 0.f; }, 0, p);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
            if (i >= p || j >= p) continue;
            const double m = M[base + i * p + j] + (double)acc[u][v];
            M[base + i * p + j] = m;
            M32out[base + i * p + j] = f64_to_f32_int(m);
        }
}

// The last step: lower tiles, back to the scale of A, and their mirror.
__global__ void __launch_bounds__(256) k_newton_last(const int32_t* action, double* M, const float* M32, const float* R,
                                                     const int32_t* ex, int64_t p)
{
    if (action[blockIdx.y] != NEWTON_FINISH) return;
    const int64_t base = blockIdx.y * p * p;
    const int32_t* e = ex + blockIdx.y * p;
    int64_t ti, tj;
    tri_index(blockIdx.x, ti, tj);
    const int64_t i0 = ti * 64, j0 = tj * 64;
    float acc[4][4] = {};
    tile64_acc<float, true, false>(
        acc, [&](int il, int64_t s) { return i0 + il < p ? __ldg(M32 + base + (i0 + il) * p + s) : 0.f; },
        [&](int64_t s, int jl) { return j0 + jl < p ? __ldg(R + base + s * p + j0 + jl) : 0.f; }, 0, p);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
            if (i >= p || j > i) continue;
            const double m = scalbn(M[base + i * p + j] + (double)acc[u][v], -e[i] - e[j]);
            M[base + i * p + j] = m;
            M[base + j * p + i] = m;
        }
}

constexpr int NEWTON_MAX = 8;
constexpr float NEWTON_LAST = 0x1p-30f;
constexpr size_t NEWTON_SCRATCH = 2ull << 30;   // FP32 copies of the systems in flight

void newton(const double* G, const double* nk, double rho, int64_t p, int32_t B, double* A, double* M, uint8_t* settled,
            cudaStream_t s)
{
    const size_t per = 3 * sizeof(float) * (size_t)(p * p);
    const int32_t group = (int32_t)std::max<size_t>(1, std::min<size_t>((size_t)B, scratch_share(NEWTON_SCRATCH) / per));
    const size_t words = (size_t)group * p * p;
    DevBuf ex(sizeof(int32_t) * (size_t)(group * p), s);
    DevBuf a32(sizeof(float) * words, s), m32(sizeof(float) * words, s), r32(sizeof(float) * words, s);
    // status of the FP32 inverse and, read together: pipeline error, then per system the norm, whether
    // its FP32 inverse failed, and its action (the residual is taken where it is to step)
    DevBuf st(sizeof(DevStatus), s), info(sizeof(int32_t) * (size_t)(1 + 3 * group), s);
    int32_t* err = info.as<int32_t>();
    float* norm = reinterpret_cast<float*>(err + 1);
    int32_t* bad = err + 1 + group;
    int32_t* action = bad + group;
    std::vector<int32_t> h((size_t)(1 + 2 * group)), act((size_t)group);
    std::vector<float> prev((size_t)group);
    for (int32_t b0 = 0; b0 < B; b0 += group) {
        const int32_t nb = std::min(group, B - b0);
        const int64_t o = (int64_t)b0 * p * p, count = (int64_t)nb * p * p;
        const dim3 rows((unsigned)std::min<int64_t>(p, 1024), (unsigned)nb);
        UOI_CUDA(cudaMemsetAsync(st.ptr, 0, st.bytes, s));
        UOI_CUDA(cudaMemsetAsync(info.ptr, 0, sizeof(int32_t) * (size_t)(1 + 2 * group), s));
        k_equil_exponents<<<(unsigned)std::min<int64_t>(ceil_div(nb * p, 256), 1024), 256, 0, s>>>(
            G + o, nk + b0, rho, p, nb, ex.as<int32_t>());
        UOI_CHECK_LAUNCH();
        k_build_equil<<<rows, 256, 0, s>>>(G + o, nk + b0, rho, p, ex.as<int32_t>(), A + o, a32.as<float>());
        UOI_CHECK_LAUNCH();
        spd_inverse_tc(a32.as<float>(), p, nb, m32.as<float>(), st.as<DevStatus>(), s, bad);
        k_widen<<<(unsigned)std::min<int64_t>(ceil_div(count, 1024), 152 * 16), 256, 0, s>>>(m32.as<float>(), M + o, count);
        UOI_CHECK_LAUNCH();
        count_launch(3);
        float* cur = m32.as<float>();
        float* other = a32.as<float>();                  // A32 is read by the FP32 inverse alone
        std::fill(prev.begin(), prev.end(), 1.f);
        int32_t at_work = nb;
        std::fill(act.begin(), act.begin() + nb, (int32_t)NEWTON_STEP);
        UOI_CUDA(cudaMemcpyAsync(action, act.data(), sizeof(int32_t) * (size_t)nb, cudaMemcpyHostToDevice, s));
        for (int it = 0; it < NEWTON_MAX && at_work > 0; ++it) {
            residual_f64(A + o, M + o, p, nb, action, r32.as<float>(), norm, err, s);
            UOI_CUDA(cudaMemcpyAsync(h.data(), err, sizeof(int32_t) * (size_t)(1 + 2 * group), cudaMemcpyDeviceToHost, s));
            UOI_CUDA(cudaStreamSynchronize(s));
            if (h[0]) throw Error(h[0], "tensor-core FP64 residual: a bounded pipeline wait expired");
            int32_t steps = 0, last = 0;
            for (int32_t k = 0; k < nb; ++k) {
                int32_t& a = act[(size_t)k];
                if (a != NEWTON_STEP) { a = NEWTON_NONE; continue; }
                float n;
                std::memcpy(&n, &h[(size_t)(1 + k)], sizeof(n));
                if (h[(size_t)(1 + group + k)] || !(n < prev[(size_t)k])) a = NEWTON_NONE;     // left to the factor
                else if (n <= NEWTON_LAST) { a = NEWTON_FINISH; settled[b0 + k] = 1; ++last; }
                else ++steps;
                prev[(size_t)k] = 0.5f * n;
            }
            UOI_CUDA(cudaMemcpyAsync(action, act.data(), sizeof(int32_t) * (size_t)nb, cudaMemcpyHostToDevice, s));
            const unsigned tt = (unsigned)ceil_div(p, 64);
            if (last) {
                k_newton_last<<<dim3(tt * (tt + 1) / 2, (unsigned)nb), 256, 0, s>>>(action, M + o, cur, r32.as<float>(),
                                                                                   ex.as<int32_t>(), p);
                UOI_CHECK_LAUNCH();
                count_launch();
            }
            if (steps) {
                k_newton_step<<<dim3(tt * tt, (unsigned)nb), 256, 0, s>>>(action, M + o, cur, r32.as<float>(), other, p);
                UOI_CHECK_LAUNCH();
                count_launch();
                std::swap(cur, other);
            }
            at_work = steps;
        }
    }
}

}  // namespace

std::vector<uint8_t> inverse_newton(const double* G, const double* nk, double rho, int64_t p, int32_t B, double* A,
                                    double* M, cudaStream_t s)
{
    std::vector<uint8_t> settled((size_t)B, 0);
    if (p < INVERSE_NEWTON_MIN || 3 * sizeof(float) * (size_t)(p * p) > NEWTON_SCRATCH || !inverse_tc_available())
        return settled;
    try {
        newton(G, nk, rho, p, B, A, M, settled.data(), s);
    } catch (const Error& e) {
        if (e.status != UOI_ERR_OOM) throw;                  // the factor needs none of the scratch
        cudaGetLastError();
    }
    return settled;
}

}  // namespace uoi
