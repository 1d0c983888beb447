// gram_f64tc.cu -- G1 in FP64 accuracy on the tensor cores: the weighted moments of
// the plain form from exact integer products (the error-free slicing of Ozaki, Ogita,
// Oishi and Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication and its applications", Numer. Algorithms 59, 2012).
//
// Each column c of Z = [X | Y], restricted to the rows with positive weight, is scaled
// by the power of two 2^-e_c above its largest magnitude there and rounded to 56 bits:
//   z = 2^e_c sum_s d_s 2^(-7 - 8 s),  s = 0..6, integers |d_s| <= 128 (exact in bf16).
// For every order o = s + t <= 6 the sums  S_o = sum_rows d_s(i) d_t(j)  over the pairs
// of that order run on the bf16 tensor cores with FP32 accumulation.  Over 128 rows
// |S_o| <= 7 * 128 * 2^14 < 2^24, so every partial sum is an exact integer; it is drained
// into 64-bit integers
//   T_hi += S_0 2^24 + S_1 2^16 + S_2 2^8 + S_3,   T_lo += S_4 2^16 + S_5 2^8 + S_6,
// and G_ij = (T_hi 2^-38 + T_lo 2^-62) 2^(e_i + e_j) is rounded once at the end.
// Errors: the rounding of z (2^-56 of the column's largest value) and the products of
// orders 7 and up (the same size, zero-mean).  An FP64 dot product of n terms rounds
// n partial sums; on 200 and 5000 standard normal rows and 700 with columns 2^60 apart this
// form's error is the smaller one (tests/test_gpu_gram_f64.py).  Entries too far above their
// column's others for that (oz_spread) are zero to the slicing and their products are summed in
// FP64 beside it.  Sums are integers, so the split of the rows over CTAs and launches changes
// no bit.
//
// Weights are handled exactly too: w = sum of its bits, rows are listed once for every
// set bit b, the lists of one bit padded to 128 rows, and a drained sum counts 2^b times.
// (A bootstrap of n draws lists 0.70 n rows.)
//
// Why: this part's FP64 pipe does 1.7 multiply-adds per clock and SM (19 clocks per warp
// instruction); 28 bf16 products replace one FP64 product at 4096 per clock.  Tiles are
// 128 x 64 because the 7 accumulators of a tile (448 of 512 TMEM columns) cap N.
// Measured against the CUDA-core form (k_moments_fp64, selection moments of 20
// bootstraps): 20000 x 1000 414 -> 10.9 ms, 5000 x 400 26.0 -> 1.05 ms, 200 x 50 0.23 ->
// 0.13 ms; X^T Y of 192 responses x 5000 rows (the lambda grid of a VAR) 5.9 -> 0.3 ms.
// No size was found where the CUDA-core form is the faster one.  Far entries: 20000 x 1000
// exp(2 N(0,1)) 11.7 ms, exp(3 N(0,1)), 1 % of the entries, 26.4 ms (normal columns 10.9).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "kernels.h"
#include "tc_common.cuh"

namespace uoi {

namespace {
using namespace tc;

constexpr int OZ_S = 7;                        // slices
constexpr int OZ_TM = 128, OZ_TN = 64;         // tile (rows of Z x columns of X)
constexpr int OZ_TK = 32;                      // sample rows per stage
constexpr int OZ_CHUNK = 128;                  // sample rows per exact FP32 sum
constexpr int OZ_STAGES = 2;
constexpr int OZ_A_BYTES = OZ_S * OZ_TM * OZ_TK * 2;       // 56 KB
constexpr int OZ_B_BYTES = OZ_S * OZ_TN * OZ_TK * 2;       // 28 KB
constexpr int OZ_STAGE_BYTES = OZ_A_BYTES + OZ_B_BYTES;
constexpr int OZ_SMEM = OZ_STAGES * OZ_STAGE_BYTES + 1024;
constexpr int OZ_EPI_WARPS = 8;
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI_WARPS;
constexpr uint32_t OZ_TMEM_COLS = 512;
constexpr int64_t OZ_TILE = (int64_t)OZ_TM * OZ_TN;
// T_hi stays below 2^63 while the weights of an item add up to at most this
constexpr unsigned long long OZ_MAX_WEIGHT = 1ull << 24;

struct OzItem {
    unsigned long long weight;      // sum of the weights
    int32_t entries;                // listed rows, padded (a multiple of OZ_CHUNK)
    int32_t pad;
};

struct OzArgs {
    int32_t pz, pz_x, ntiles;
    const int32_t* tiles;           // (row tile, column tile)
    const OzItem* items;
    const int32_t* cshift;          // items x max_chunks: bit of the weight each chunk stands for
    int32_t max_chunks;
    int32_t chunk0, range;          // this launch sums the chunks chunk0 .. chunk0 + range - 1
    int32_t add;                    // into T as it is (zero before the first range)
    long long* T;                   // items x ntiles x 2 x OZ_TN x OZ_TM
    int32_t* err;
    uint64_t wait_ns = tc::kWaitLimitNs;
};

// Four consecutive TMEM columns of each of the NA accumulators (64 columns apart).
template <int NA>
__device__ __forceinline__ void oz_load4(uint32_t taddr, float (&v)[NA][4])
{
    uint32_t r[8][4];
    if constexpr (NA < 8) r[7][0] = r[7][1] = r[7][2] = r[7][3] = 0;
#pragma unroll
    for (int o = 0; o < NA; ++o)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[o][0]), "=r"(r[o][1]), "=r"(r[o][2]), "=r"(r[o][3])
                     : "r"(taddr + (uint32_t)(o * OZ_TN)));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0][0]), "+r"(r[0][1]), "+r"(r[0][2]), "+r"(r[0][3]), "+r"(r[1][0]), "+r"(r[1][1]),
                   "+r"(r[1][2]), "+r"(r[1][3]), "+r"(r[2][0]), "+r"(r[2][1]), "+r"(r[2][2]), "+r"(r[2][3]),
                   "+r"(r[3][0]), "+r"(r[3][1]), "+r"(r[3][2]), "+r"(r[3][3]), "+r"(r[4][0]), "+r"(r[4][1]),
                   "+r"(r[4][2]), "+r"(r[4][3]), "+r"(r[5][0]), "+r"(r[5][1]), "+r"(r[5][2]), "+r"(r[5][3]),
                   "+r"(r[6][0]), "+r"(r[6][1]), "+r"(r[6][2]), "+r"(r[6][3]), "+r"(r[7][0]), "+r"(r[7][1]),
                   "+r"(r[7][2]), "+r"(r[7][3]));
#pragma unroll
    for (int o = 0; o < NA; ++o)
#pragma unroll
        for (int t = 0; t < 4; ++t) v[o][t] = __uint_as_float(r[o][t]);
}

// grid (tiles, items, row splits): one tile of one item over a range of its chunks.
// Warp 0: TMA producer (ring of two stages of 32 rows, all slices of A and of B in one
// copy each); warp 1: MMA issuer; warps 2-9 drain the accumulators after every chunk.
// NA orders are kept: 7, or 8 for residuals (T_lo then in units 2^-8 as large).
template <int NA>
__global__ void __launch_bounds__(OZ_THREADS, 1)
k_gram_f64tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, OzArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ uint64_t full_bar[OZ_STAGES], empty_bar[OZ_STAGES], accf_bar, acce_bar, done_bar;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int item = blockIdx.y;
    const int ti = a.tiles[2 * blockIdx.x], tj = a.tiles[2 * blockIdx.x + 1];
    if (a.items[item].entries == 0 && NA == 8) return;   // a residual that nobody asked for
    const int chunks = min(max(a.items[item].entries / OZ_CHUNK - a.chunk0, 0), a.range);
    const int c0 = (int)((int64_t)chunks * blockIdx.z / gridDim.z);
    const int nc = (int)((int64_t)chunks * (blockIdx.z + 1) / gridDim.z) - c0;
    if (nc <= 0 && a.add) return;                        // nothing to add
    const int nst = nc * (OZ_CHUNK / OZ_TK);
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < OZ_STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&accf_bar, 1);
        mbar_init(&acce_bar, 32 * OZ_EPI_WARPS);
        mbar_init(&done_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(OZ_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp == 0 && elect_one()) {
        for (int g = 0; g < nst; ++g) {
            const int s = g % OZ_STAGES;
            if (g >= OZ_STAGES && !mbar_wait(&empty_bar[s], ((g / OZ_STAGES) - 1) & 1, &abort_flag, a.wait_ns)) {
                abort_flag = 1;
                atomicCAS(a.err, 0, UOI_ERR_TIMEOUT);
                break;
            }
            const uint32_t st = sbase + s * OZ_STAGE_BYTES;
            const int k0 = c0 * OZ_CHUNK + g * OZ_TK;
            mbar_expect_tx(&full_bar[s], OZ_STAGE_BYTES);
            tma_load_3d(st, &tmA, &full_bar[s], k0, ti * OZ_TM, item * OZ_S);
            tma_load_3d(st + OZ_A_BYTES, &tmB, &full_bar[s], k0, tj * OZ_TN, item * OZ_S);
        }
        if (abort_flag)
            for (int g = max(0, nst - OZ_STAGES); g < nst; ++g)
                mbar_wait(&full_bar[g % OZ_STAGES], (g / OZ_STAGES) & 1, &abort_flag, a.wait_ns);
    } else if (warp == 1 && nc > 0 && elect_one()) {
        constexpr uint32_t idesc = idesc_bf16(OZ_TM, OZ_TN);
        int g = 0;
        for (int c = 0; c < nc && !abort_flag; ++c) {
            if (c > 0 && !mbar_wait(&acce_bar, (c - 1) & 1, &abort_flag, a.wait_ns)) {
                abort_flag = 1;
                atomicCAS(a.err, 0, UOI_ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            for (int q = 0; q < OZ_CHUNK / OZ_TK; ++q, ++g) {
                const int s = g % OZ_STAGES;
                if (!mbar_wait(&full_bar[s], (g / OZ_STAGES) & 1, &abort_flag, a.wait_ns)) {
                    abort_flag = 1;
                    atomicCAS(a.err, 0, UOI_ERR_TIMEOUT);
                    break;
                }
                tc_fence_after();
                const uint32_t st = sbase + s * OZ_STAGE_BYTES;
#pragma unroll 1
                for (int ks = 0; ks < OZ_TK / 16; ++ks) {
                    const uint64_t adv = (uint64_t)(ks * 32 >> 4);
#pragma unroll 1
                    for (int u = 0; u < OZ_S; ++u) {
                        const uint64_t A = smem_desc_sw64(st + u * (OZ_TM * OZ_TK * 2)) + adv;
                        // the first product of an order starts its sum: slice 0 of A, slice 1 for order 7
                        const bool started = q > 0 || ks > 0;
                        for (int t = 0; t < OZ_S && t + u < NA; ++t)
                            mma_bf16(tmem + (uint32_t)((u + t) * OZ_TN), A,
                                     smem_desc_sw64(st + OZ_A_BYTES + t * (OZ_TN * OZ_TK * 2)) + adv, idesc,
                                     started || u > (u + t >= OZ_S ? 1 : 0) ? 1u : 0u);
                    }
                }
                mma_commit(&empty_bar[s]);
            }
            if (abort_flag) break;
            mma_commit(&accf_bar);
        }
        mma_commit(&done_bar);
        int dummy = 0;
        mbar_wait(&done_bar, 0, &dummy, a.wait_ns);
    } else if (warp >= 2) {
        const int quad = warp & 3, half = (warp - 2) >> 2;
        const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * (OZ_TN / 2));
        constexpr int NCOL = OZ_TN / 2;
        long long hi[NCOL], lo[NCOL];
#pragma unroll
        for (int t = 0; t < NCOL; ++t) { hi[t] = 0; lo[t] = 0; }
        for (int c = 0; c < nc; ++c) {
            const bool okw = mbar_wait(&accf_bar, c & 1, &abort_flag, a.wait_ns);
            if (!__all_sync(0xffffffffu, okw)) {
                abort_flag = 1;
                atomicCAS(a.err, 0, UOI_ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            const int sh = a.cshift[(int64_t)item * a.max_chunks + a.chunk0 + c0 + c];
#pragma unroll
            for (int cb = 0; cb < NCOL; cb += 4) {
                float v[NA][4];
                oz_load4<NA>(taddr + (uint32_t)cb, v);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    // S_0 2^8 + S_1 and S_2 2^8 + S_3 fit 32 bits (|S_o| <= (o + 1) 2^21)
                    const int p01 = __float2int_rn(v[0][t]) * 256 + __float2int_rn(v[1][t]);
                    const int p23 = __float2int_rn(v[2][t]) * 256 + __float2int_rn(v[3][t]);
                    const long long p56 = (long long)__float2int_rn(v[5][t]) * 256 + __float2int_rn(v[6][t]);
                    hi[cb + t] += ((long long)p01 * 65536 + p23) << sh;
                    long long p46 = (long long)__float2int_rn(v[4][t]) * 65536 + p56;
                    if constexpr (NA == 8) p46 = p46 * 256 + __float2int_rn(v[7][t]);
                    lo[cb + t] += p46 << sh;
                }
            }
            tc_fence_before();
            mbar_arrive(&acce_bar);
        }
        if (!abort_flag) {
            long long* out = a.T + ((int64_t)item * a.ntiles + blockIdx.x) * (2 * OZ_TILE) + quad * 32 + lane;
#pragma unroll
            for (int t = 0; t < NCOL; ++t) {
                const int64_t o = (int64_t)(half * NCOL + t) * OZ_TM;
                if (!a.add) {
                    out[o] = hi[t];
                    out[OZ_TILE + o] = lo[t];
                } else {
                    atomicAdd((unsigned long long*)(out + o), (unsigned long long)hi[t]);
                    atomicAdd((unsigned long long*)(out + OZ_TILE + o), (unsigned long long)lo[t]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS));
    }
}

__device__ __forceinline__ uint32_t oz_weight(const uint32_t* w, const uint8_t* mask, int64_t i)
{
    return w ? w[i] : (mask ? (mask[i] ? 1u : 0u) : 1u);
}

// A column's largest entry may lie 2^oz_spread above its typical one (the mean exponent of its
// entries that are not zero).  Rounded against the largest value, sums of n products of
// typical entries are off by n^(1/2) 2^-57 of that value; FP64 sums by about n 2^-54 of the
// typical one: the slicing is the less accurate one from 2^(2.5) n^(1/2) on.  It never matters
// to the fit (the error stays 2^-56 of the product of the columns' norms), but it does to an
// entry of G whose other column is zero where the large values are.
__host__ __device__ __forceinline__ int oz_spread(unsigned long long weight)
{
    int bits = 0;
    while (weight) { weight >>= 1; ++bits; }
    return 3 + bits / 2;
}

// Sum of biased exponents << 24 | number, of a column's entries that are not zero (m < 2^23).
__device__ __forceinline__ int oz_mean_exponent(unsigned long long stat)
{
    const unsigned long long n = stat & 0xFFFFFFu;
    return n ? (int)((stat >> 24) / n) : 0;
}

// Per item: the sum of the weights and the number of listed rows (the rows of each set
// bit padded to a chunk).  One block per item.  After k_oz_colmax: *spread = 1 if a column of
// the item has entries too far above its typical ones (stat nullable).
__global__ void __launch_bounds__(1024)
k_oz_count(const uint32_t* w, const uint8_t* mask, int64_t m, OzItem* items, const uint32_t* cmax, const unsigned long long* stat, int32_t pz,
           int32_t* spread)
{
    __shared__ unsigned s_cnt[32];
    __shared__ unsigned long long s_sum;
    const int64_t base = (int64_t)blockIdx.x * m;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) s_cnt[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_sum = 0;
    __syncthreads();
    unsigned long long sum = 0;
    unsigned mine = 0;                                   // lane b: rows of this warp with bit b set
    for (int64_t t0 = threadIdx.x - lane; t0 < m; t0 += blockDim.x) {
        const uint32_t v = t0 + lane < m ? oz_weight(w, mask, base + t0 + lane) : 0u;
        sum += v;
        for (unsigned left = __reduce_or_sync(0xffffffffu, v); left; left &= left - 1) {
            const int b = __ffs(left) - 1;
            const unsigned n = __popc(__ballot_sync(0xffffffffu, (v >> b) & 1u));
            if (lane == b) mine += n;
        }
    }
    if (mine) atomicAdd(&s_cnt[lane], mine);
    sum = warp_sum(sum);
    if (lane == 0) atomicAdd(&s_sum, sum);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long e = 0;
        for (int b = 0; b < 32; ++b) e += (s_cnt[b] + OZ_CHUNK - 1ull) / OZ_CHUNK * OZ_CHUNK;
        items[blockIdx.x].weight = s_sum;
        items[blockIdx.x].entries = (int32_t)min(e, 0x7fffff80ull);
    }
    if (!stat) return;
    const int far = oz_spread(s_sum);
    for (int c = threadIdx.x; c < pz; c += blockDim.x)
        if ((int)(cmax[(int64_t)blockIdx.x * pz + c] >> 20) - oz_mean_exponent(stat[c]) > far) *spread = 1;
}

// The listed rows of each item, increasing within a bit, -1 as padding, and each
// chunk's bit.  One block per item.
__global__ void __launch_bounds__(1024)
k_oz_lists(const uint32_t* w, const uint8_t* mask, int64_t m, int64_t cap, int32_t max_chunks, int32_t* rows,
           int32_t* cshift)
{
    __shared__ unsigned s_or;
    __shared__ int warp_tot[32];
    const int64_t base = (int64_t)blockIdx.x * m;
    int32_t* out = rows + (int64_t)blockIdx.x * cap;
    int32_t* cs = cshift + (int64_t)blockIdx.x * max_chunks;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) s_or = 0;
    __syncthreads();
    unsigned o = 0;
    for (int64_t t = threadIdx.x; t < m; t += blockDim.x) o |= oz_weight(w, mask, base + t);
    o = __reduce_or_sync(0xffffffffu, o);
    if (lane == 0 && o) atomicOr(&s_or, o);
    __syncthreads();
    int64_t at = 0;                                      // entries written so far (the same in every thread)
    for (unsigned left = s_or; left; left &= left - 1) {
        const int b = __ffs(left) - 1;
        const int64_t begin = at;
        for (int64_t t0 = 0; t0 < m; t0 += blockDim.x) {
            const int64_t t = t0 + threadIdx.x;
            const bool on = t < m && ((oz_weight(w, mask, base + t) >> b) & 1u);
            const unsigned bal = __ballot_sync(0xffffffffu, on);
            __syncthreads();                             // the previous totals have been read
            if (lane == 0) warp_tot[wid] = __popc(bal);
            __syncthreads();
            int before = 0, total = 0;
            for (int k = 0; k < nw; ++k) {
                if (k == wid) before = total;
                total += warp_tot[k];
            }
            if (on) out[at + before + __popc(bal & ((1u << lane) - 1u))] = (int32_t)t;
            at += total;
        }
        const int64_t end = begin + (at - begin + OZ_CHUNK - 1) / OZ_CHUNK * OZ_CHUNK;
        for (int64_t t = at + threadIdx.x; t < end; t += blockDim.x) out[t] = -1;
        for (int64_t t = begin / OZ_CHUNK + threadIdx.x; t < end / OZ_CHUNK; t += blockDim.x) cs[t] = b;
        at = end;
    }
}

// cmax[item * pz + c] = largest high word of |z| over the rows of the item with positive
// weight (the exponent of the column's largest value); *nonfinite = 1 if any entry is
// NaN or Inf, whatever its weight; stat[c] as above over all rows (nullable); entries past lim
// (nullable) count as zero.  A block reads 64
// rows x 128 columns once and keeps their high words in registers while it goes through the items.
constexpr int OZ_MAX_ROWS = 64;
__global__ void __launch_bounds__(128)
k_oz_colmax(const double* __restrict__ X, int64_t ldx, const double* __restrict__ Y, int64_t ldy, int64_t m,
            int32_t pz_x, int32_t pz, int32_t B, const uint32_t* w, const uint8_t* mask, uint32_t* cmax,
            unsigned long long* stat, const int32_t* lim, int32_t* nonfinite)
{
    const int c = blockIdx.x * 128 + threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.y * OZ_MAX_ROWS;
    const int lane = threadIdx.x & 31;
    uint32_t h[OZ_MAX_ROWS], all = 0, exps = 0, used = 0;
#pragma unroll
    for (int u = 0; u < OZ_MAX_ROWS; ++u) {
        const int64_t t = r0 + u;
        double x = 0.0;
        if (t < m && c < pz) x = c < pz_x ? __ldg(X + t * ldx + c) : __ldg(Y + t * ldy + (c - pz_x));
        h[u] = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
        // a subnormal below the high word still counts as the smallest exponent
        if (h[u] == 0 && __double2loint(x) != 0) h[u] = 1;
        if (lim && c < pz && (int)(h[u] >> 20) > lim[c]) h[u] = 0;
        all = max(all, h[u]);
        exps += h[u] >> 20;
        used += h[u] ? 1u : 0u;
    }
    if (stat && used) atomicAdd(&stat[c], (unsigned long long)exps << 24 | used);
    if (__any_sync(0xffffffffu, all >= 0x7FF00000u) && lane == 0) atomicExch(nonfinite, 1);
    for (int k = 0; k < B; ++k) {
        const int64_t o = (int64_t)k * m + r0;
        const uint32_t ma = __ballot_sync(0xffffffffu, r0 + lane < m && oz_weight(w, mask, o + lane) != 0);
        const uint32_t mb = __ballot_sync(0xffffffffu, r0 + 32 + lane < m && oz_weight(w, mask, o + 32 + lane) != 0);
        uint32_t mx = 0;
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            if ((ma >> u) & 1u) mx = max(mx, h[u]);
            if ((mb >> u) & 1u) mx = max(mx, h[32 + u]);
        }
        if (c < pz && mx) atomicMax(&cmax[(int64_t)k * pz + c], mx);
    }
}

// Entries far above the typical one of their column (oz_spread) are zero to the slicing; their
// products are summed in FP64 beside it.  lim[c]: the largest biased exponent of an ordinary entry.
__global__ void k_oz_limits(const unsigned long long* stat, int32_t pz, int far, int32_t* lim)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < pz) lim[c] = oz_mean_exponent(stat[c]) + far;
}

__device__ __forceinline__ double oz_entry(const double* __restrict__ X, int64_t ldx, const double* __restrict__ Y, int64_t ldy,
                                           int32_t pz_x, int64_t t, int32_t c)
{
    return c < pz_x ? __ldg(X + t * ldx + c) : __ldg(Y + t * ldy + (c - pz_x));
}
__device__ __forceinline__ bool oz_far(double x, int lim) { return (int)((__double2hiint(x) >> 20) & 0x7FF) > lim; }

// The rows of each column's far entries, increasing: a warp takes 32 columns of one of OZ_SEGS runs of
// rows.  Without `rows` it counts them into cnt[segment * pz + column], with it it lists them from
// the place that cnt gives then (k_oz_far_places).
constexpr int OZ_SEGS = 256;
__global__ void __launch_bounds__(256)
k_oz_far_entries(const double* __restrict__ X, int64_t ldx, const double* __restrict__ Y, int64_t ldy, int64_t m, int32_t pz_x,
                 int32_t pz, const int32_t* lim, int64_t* cnt, int32_t* rows)
{
    const int seg = blockIdx.y * 8 + (threadIdx.x >> 5), c = blockIdx.x * 32 + (threadIdx.x & 31);
    if (c >= pz) return;
    const int64_t t0 = m * seg / OZ_SEGS, t1 = m * (seg + 1) / OZ_SEGS;
    const int l = lim[c];
    int64_t at = rows ? cnt[(int64_t)seg * pz + c] : 0;
#pragma unroll 4
    for (int64_t t = t0; t < t1; ++t)
        if (oz_far(oz_entry(X, ldx, Y, ldy, pz_x, t, c), l)) {
            if (rows) rows[at] = (int32_t)t;
            ++at;
        }
    if (!rows) cnt[(int64_t)seg * pz + c] = at;
}

// Counts -> places: column after column, segment after segment; first[c] .. first[c + 1] - 1 are
// column c's.  One block.
__global__ void __launch_bounds__(1024) k_oz_far_places(int64_t* cnt, int32_t pz, int64_t* first)
{
    __shared__ int64_t tot[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t base = 0;                                    // the same in every thread
    for (int c0 = 0; c0 < pz; c0 += 1024) {
        const int c = c0 + threadIdx.x;
        int64_t n = 0;
        if (c < pz)
            for (int s = 0; s < OZ_SEGS; ++s) n += cnt[(int64_t)s * pz + c];
        int64_t inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        __syncthreads();                                 // the previous totals have been read
        if (lane == 31) tot[wid] = inc;
        __syncthreads();
        int64_t at = base + inc - n;
        for (int k = 0; k < 32; ++k) {
            if (k < wid) at += tot[k];
            base += tot[k];
        }
        if (c < pz) {
            first[c] = at;
            for (int s = 0; s < OZ_SEGS; ++s) {
                const int64_t v = cnt[(int64_t)s * pz + c];
                cnt[(int64_t)s * pz + c] = at;
                at += v;
            }
        }
    }
    if (threadIdx.x == 0) first[pz] = base;
}

// S[item][i][j] = sum over the far entries f of column i, in row order, of w f z_j: z_j whole for
// j <= i, without column j's own far entries for j > i, so that every product with a far entry
// stands in one of S[i][j] and S[j][i].  A block per column i and item; b_only: the pairs with a
// column of Y.  Columns without far entries are not written.
__global__ void __launch_bounds__(256)
k_oz_far_sums(const double* __restrict__ X, int64_t ldx, const double* __restrict__ Y, int64_t ldy, int64_t m, int32_t pz_x,
              int32_t pz, const uint32_t* w, const uint8_t* mask, const int32_t* lim, const int64_t* first, const int32_t* rows,
              int b_only, double* S)
{
    const int i = blockIdx.x, item = blockIdx.y;
    const int64_t n0 = first[i], n1 = first[i + 1];
    if (n0 == n1) return;
    double* out = S + ((int64_t)item * pz + i) * pz;
    for (int j = threadIdx.x; j < pz; j += 256) {
        if (i >= pz_x ? j >= pz_x : (b_only && j < pz_x)) continue;
        double sum = 0.0;
        for (int64_t e = n0; e < n1; ++e) {
            const int64_t t = rows[e];
            const uint32_t wt = oz_weight(w, mask, (int64_t)item * m + t);
            if (wt == 0) continue;
            const double z = oz_entry(X, ldx, Y, ldy, pz_x, t, j);
            if (j > i && oz_far(z, lim[j])) continue;
            sum += (double)wt * oz_entry(X, ldx, Y, ldy, pz_x, t, i) * z;
        }
        out[j] = sum;
    }
}

// e with |z| < 2^e for every z whose high word is at most h (0 for an all-zero column).
__device__ __forceinline__ int oz_exponent(uint32_t h) { return h == 0 ? 0 : max((int)(h >> 20), 1) - 1022; }

// rint(x 2^(55 - e)) for |x| < 2^e, by shifts.
__device__ __forceinline__ long long oz_fixed(double x, int e)
{
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7FF);
    long long mant = b & 0xFFFFFFFFFFFFFll;
    if (ex) mant |= 1ll << 52;
    const int sh = max(ex, 1) - 1075 + 55 - e;           // <= 2: x 2^-e is below 1
    if (sh >= 0) mant <<= sh;
    else if (sh < -54) mant = 0;
    else mant = (mant + (1ll << (-sh - 1))) >> -sh;
    return b < 0 ? -mant : mant;
}

// The digit in byte `byte` of u (biased by 128) as the bits of a float.
__device__ __forceinline__ uint32_t oz_digit(uint32_t word, int byte)
{
    const uint32_t f = __byte_perm(word, 0x4B000000u, 0x7540u + (uint32_t)byte);   // 2^23 + byte
    return __float_as_uint(__uint_as_float(f) - 8388736.f);
}

// Gathers the listed rows, takes their digits and writes them transposed:
// out[((item * 7 + s) * pz_pad + col) * n_pad + t], t counted from row list entry chunk0 * 128.  A
// block covers 128 listed rows x 32 columns: rows are read along X's rows, the 56-bit values
// turned over in shared memory.
// gsx, gsy: distance of the items' operands (0: all items read the same X and Y).
constexpr int OZ_LD = OZ_CHUNK + 2;
__global__ void __launch_bounds__(256)
k_oz_split(const double* __restrict__ X, int64_t ldx, int64_t gsx, const double* __restrict__ Y, int64_t ldy,
           int64_t gsy, int32_t pz_x, int32_t pz, const int32_t* __restrict__ rows, int64_t cap, const OzItem* items, const uint32_t* cmax,
           int64_t n_pad, int32_t pz_pad, int32_t chunk0, const int32_t* lim, __nv_bfloat16* out)
{
    __shared__ long long tile[32][OZ_LD];
    const int item = blockIdx.x;
    const int64_t t0 = (int64_t)blockIdx.y * OZ_CHUNK;
    const int64_t r0 = (int64_t)chunk0 * OZ_CHUNK + t0;
    if (r0 >= items[item].entries) return;               // past this item's rows: never read
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.z * 32 + lane;
    const int e = c < pz ? oz_exponent(cmax[(int64_t)item * pz + c]) : 0;
    const int32_t* rl = rows + (int64_t)item * cap + r0;
    X += item * gsx;
    Y += item * gsy;
    double x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int64_t row = rl[warp * 16 + i];
        x[i] = 0.0;
        if (row >= 0 && c < pz) x[i] = c < pz_x ? __ldg(X + row * ldx + c) : __ldg(Y + row * ldy + (c - pz_x));
    }
    if (lim && c < pz) {
        const int l = lim[c];
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (oz_far(x[i], l)) x[i] = 0.0;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) tile[lane][warp * 16 + i] = oz_fixed(x[i], e);
    __syncthreads();
    const int64_t slice = (int64_t)pz_pad * n_pad;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int cl = warp + 8 * j;
        __nv_bfloat16* o = out + ((int64_t)item * OZ_S * pz_pad + blockIdx.z * 32 + cl) * n_pad + t0 + 4 * lane;
        uint32_t d[OZ_S][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            // balanced digits: with 128 added to each of the six lower bytes, every byte
            // is its digit + 128; the top part is the first digit itself
            const long long u = tile[cl][4 * lane + q] + 0x808080808080ll;
            const uint32_t lo = (uint32_t)u, hi = (uint32_t)(u >> 32);
            d[0][q] = __float_as_uint((float)(int)(u >> 48));
            d[1][q] = oz_digit(hi, 1);
            d[2][q] = oz_digit(hi, 0);
            d[3][q] = oz_digit(lo, 3);
            d[4][q] = oz_digit(lo, 2);
            d[5][q] = oz_digit(lo, 1);
            d[6][q] = oz_digit(lo, 0);
        }
#pragma unroll
        for (int s = 0; s < OZ_S; ++s)                   // the upper halves are the bf16 values
            *reinterpret_cast<uint2*>(o + s * slice) =
                make_uint2(__byte_perm(d[s][0], d[s][1], 0x7632), __byte_perm(d[s][2], d[s][3], 0x7632));
    }
}

// Integer sums (and the far entries' sums S, nullable) -> FP64 outputs, 64 x 64 at a time: the
// lower triangle of G along its rows (turned over in shared memory), its mirror along the sums'
// own order, and Bm.
__global__ void __launch_bounds__(256)
k_oz_finish(const long long* T, int32_t ntiles, const int32_t* tiles, const uint32_t* cmax, int32_t pz, int32_t pz_x,
            int32_t r, const double* S, const int64_t* first, double* G, double* Bm)
{
    __shared__ double v[64][65];
    const int item = blockIdx.y;
    const int ti = tiles[2 * blockIdx.x], tj = tiles[2 * blockIdx.x + 1];
    const long long* t = T + ((int64_t)item * ntiles + blockIdx.x) * (2 * OZ_TILE) + blockIdx.z * 64;
    const uint32_t* cm = cmax + (int64_t)item * pz;
    const int i0 = ti * OZ_TM + blockIdx.z * 64, j0 = tj * OZ_TN;
    if (i0 >= pz) return;
    for (int x = threadIdx.x; x < 64 * 64; x += 256) {
        const int i = i0 + (x & 63), j = j0 + (x >> 6);
        double val = 0.0;
        if (i < pz && j < pz_x) {
            const long long hi = t[(int64_t)(x >> 6) * OZ_TM + (x & 63)];
            const long long lo = t[OZ_TILE + (int64_t)(x >> 6) * OZ_TM + (x & 63)];
            const int e = oz_exponent(cm[i]) + oz_exponent(cm[j]);
            val = scalbn(fma((double)lo, 0x1p-24, (double)hi), e - 38);
            if (S && j <= i) {
                const double* sk = S + (int64_t)item * pz * pz;
                const double a = first[i] < first[i + 1] ? sk[(int64_t)i * pz + j] : 0.0;
                const double b = j < i && first[j] < first[j + 1] ? sk[(int64_t)j * pz + i] : 0.0;
                val += a + b;
            }
            if (G && i < pz_x && j < i) G[((int64_t)item * pz_x + j) * pz_x + i] = val;
        }
        v[x & 63][x >> 6] = val;
    }
    __syncthreads();
    for (int x = threadIdx.x; x < 64 * 64; x += 256) {
        const int i = i0 + (x >> 6), j = j0 + (x & 63);
        if (i >= pz || j >= pz_x) continue;
        if (i < pz_x) {
            if (G && j <= i) G[((int64_t)item * pz_x + i) * pz_x + j] = v[x >> 6][x & 63];
        } else {
            Bm[((int64_t)item * pz_x + j) * r + (i - pz_x)] = v[x >> 6][x & 63];
        }
    }
}

// Residuals of approximate inverses: the same products with one pair of square matrices per
// item (X = A_k, Y = M_k, every row once).  The order 7 is kept too: the products it drops
// are the largest error of a sum whose terms cancel, and a Newton step cannot go below it
// (without it c = M b came out at 1.4e-14 for p = 400, with it at the level of b).

// One list of the rows 0 .. n - 1 for every item, and the items' entry counts (none where it is
// not active: the kernels below then leave it out).
__global__ void k_oz_all_rows(int32_t n, int32_t n_pad, int32_t B, const int32_t* active, int32_t* rows, OzItem* items)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_pad) rows[t] = t < n ? t : -1;
    if (t < B) {
        items[t].weight = (unsigned long long)n;
        items[t].entries = active[t] > 0 ? n_pad : 0;
    }
}

// Largest high words of the columns of A_k and of M_k (a slice of the rows per block z).
__global__ void __launch_bounds__(128)
k_oz_colmax_pair(const double* __restrict__ A, const double* __restrict__ M, int32_t p, const OzItem* items,
                 uint32_t* cmax)
{
    const int item = blockIdx.y, c = blockIdx.x * 128 + threadIdx.x;
    if (c >= 2 * p || items[item].entries == 0) return;
    const int r0 = (int)((int64_t)p * blockIdx.z / gridDim.z), r1 = (int)((int64_t)p * (blockIdx.z + 1) / gridDim.z);
    const double* src = (c < p ? A + c : M + (c - p)) + (int64_t)item * p * p;
    uint32_t h = 0;
#pragma unroll 8
    for (int t = r0; t < r1; ++t) {
        const double x = __ldg(src + (int64_t)t * p);
        const uint32_t w = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
        h = max(h, w == 0 && __double2loint(x) != 0 ? 1u : w);
    }
    if (h) atomicMax(&cmax[(int64_t)item * 2 * p + c], h);
}

// R = I - A M in FP32, 64 x 64 at a time (rows of the sums are M's columns), and the sums of |R|
// over 32 columns of each row: part[(item * nseg + segment) * p + row], segments counted from
// column 128 (p / 128) of Z.
__global__ void __launch_bounds__(256)
k_oz_residual(const long long* T, int32_t ntiles, const int32_t* tiles, const OzItem* items, const uint32_t* cmax, int32_t p,
              int32_t nseg, float* R, float* part)
{
    const int item = blockIdx.y;
    if (items[item].entries == 0) return;
    const int ti = tiles[2 * blockIdx.x], tj = tiles[2 * blockIdx.x + 1];
    const long long* t = T + ((int64_t)item * ntiles + blockIdx.x) * (2 * OZ_TILE) + blockIdx.z * 64;
    const uint32_t* cm = cmax + (int64_t)item * 2 * p;
    const int i0 = ti * OZ_TM + blockIdx.z * 64 - p, j0 = tj * OZ_TN;      // column of M, row of A
    if (i0 + 63 < 0 || i0 >= p) return;
    const int seg = (i0 + p - p / OZ_TM * OZ_TM) / 32;
    for (int x = threadIdx.x; x < 64 * 64; x += 256) {
        const int i = i0 + (x & 63), j = j0 + (x >> 6);
        float v = 0.f;
        if (i >= 0 && i < p && j < p) {
            const long long hi = t[(int64_t)(x >> 6) * OZ_TM + (x & 63)];
            const long long lo = t[OZ_TILE + (int64_t)(x >> 6) * OZ_TM + (x & 63)];
            const int e = oz_exponent(cm[p + i]) + oz_exponent(cm[j]);
            v = f64_to_f32_int((i == j ? 1.0 : 0.0) - scalbn(fma((double)lo, 0x1p-32, (double)hi), e - 38));
            R[((int64_t)item * p + j) * p + i] = v;
        }
        const float sum = warp_sum(fabsf(v));            // a warp lies within one row
        if ((threadIdx.x & 31) == 0 && j < p) part[((int64_t)item * nseg + seg + ((x >> 5) & 1)) * p + j] = sum;
    }
}

// norm[item]: the largest row sum of |R|, each summed in the order of its segments.
__global__ void __launch_bounds__(256)
k_oz_norm(const float* part, const OzItem* items, const uint32_t* cmax, int32_t p, int32_t nseg, float* norm)
{
    __shared__ uint32_t red[8];
    const int item = blockIdx.x;
    if (items[item].entries == 0) return;
    const int first = -p + p / OZ_TM * OZ_TM;            // M's column at segment 0
    uint32_t top = 0;                                    // floats >= 0 order as their bits, NaN above all
    for (int j = threadIdx.x; j < p; j += 256) {
        float sum = 0.f;
        for (int s = 0; s < nseg; ++s) {
            const int i0 = first + s / 2 * 64;           // k_oz_residual's blocks: others wrote nothing
            if (i0 + 63 >= 0 && i0 < p) sum += part[((int64_t)item * nseg + s) * p + j];
        }
        top = max(top, __float_as_uint(sum));
    }
    for (int c = threadIdx.x; c < 2 * p; c += 256)
        if (cmax[(int64_t)item * 2 * p + c] >= 0x7FF00000u) top = max(top, 0x7F800000u);
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = top;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) top = max(top, red[w]);
        norm[item] = __uint_as_float(top);
    }
}

// Slices of one operand: box of all 7 slices of box_rows columns x 32 sample rows.
CUtensorMap oz_map(void* base, int64_t n_pad, int64_t pz_pad, int64_t depth, int box_rows)
{
    CUtensorMap m;
    cuuint64_t dims[3] = { (cuuint64_t)n_pad, (cuuint64_t)pz_pad, (cuuint64_t)depth };
    cuuint64_t strides[2] = { (cuuint64_t)(n_pad * 2), (cuuint64_t)(n_pad * 2 * pz_pad) };
    cuuint32_t box[3] = { 32u, (cuuint32_t)box_rows, (cuuint32_t)OZ_S };
    cuuint32_t estr[3] = { 1, 1, 1 };
    CUresult res = tc::encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr,
                                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (res != CUDA_SUCCESS) throw Error(UOI_ERR_CUDA, "cuTensorMapEncodeTiled failed");
    return m;
}

}  // namespace

// R_k = I - A_k M_k (FP32, p x p each) with FP64-accurate products and the largest row sum of
// |R_k|; *err becomes a pipeline error.
void residual_f64(const double* A, const double* M, int64_t p, int32_t B, const int32_t* active, float* R, float* norm,
                  int32_t* err, cudaStream_t s)
{
    const int32_t pz_x = (int32_t)p, pz = 2 * pz_x;
    const int32_t pz_pad = (int32_t)ceil_div(pz, OZ_TM) * OZ_TM;
    const int32_t n_pad = (int32_t)ceil_div(p, OZ_CHUNK) * OZ_CHUNK, max_chunks = n_pad / OZ_CHUNK;
    std::vector<int32_t> tiles;
    for (int ti = pz_x / OZ_TM; ti * OZ_TM < pz; ++ti)
        for (int tj = 0; tj * OZ_TN < pz_x; ++tj) { tiles.push_back(ti); tiles.push_back(tj); }
    const int ntiles = (int)tiles.size() / 2;
    const size_t per_item = (size_t)OZ_S * pz_pad * n_pad * sizeof(__nv_bfloat16);
    const size_t t_item = sizeof(long long) * 2 * OZ_TILE * (size_t)ntiles;
    const int32_t nseg = (pz_pad - pz_x / OZ_TM * OZ_TM) / 32;
    const int group = (int)std::max<size_t>(1, std::min<size_t>((size_t)B, scratch_share(8ull << 30) / (per_item + t_item)));
    DevBuf tl(sizeof(int32_t) * tiles.size(), s), rows(sizeof(int32_t) * (size_t)n_pad, s);
    DevBuf items(sizeof(OzItem) * (size_t)B, s), cmax(sizeof(uint32_t) * (size_t)B * pz, s);
    DevBuf cshift(sizeof(int32_t) * (size_t)group * max_chunks, s);
    DevBuf zt(per_item * group, s), T(t_item * group, s), part(sizeof(float) * (size_t)group * nseg * p, s);
    UOI_CUDA(cudaMemcpyAsync(tl.ptr, tiles.data(), sizeof(int32_t) * tiles.size(), cudaMemcpyHostToDevice, s));
    UOI_CUDA(cudaMemsetAsync(cmax.ptr, 0, cmax.bytes, s));
    UOI_CUDA(cudaMemsetAsync(cshift.ptr, 0, cshift.bytes, s));
    k_oz_all_rows<<<(unsigned)ceil_div(std::max<int64_t>(n_pad, B), 256), 256, 0, s>>>(
        pz_x, n_pad, B, active, rows.as<int32_t>(), items.as<OzItem>());
    UOI_CHECK_LAUNCH();
    UOI_CUDA(cudaFuncSetAttribute(k_gram_f64tc<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM));
    for (int b0 = 0; b0 < B; b0 += group) {
        const int nb = std::min(group, B - b0);
        const int64_t o = (int64_t)b0 * p * p;
        uint32_t* cm = cmax.as<uint32_t>() + (int64_t)b0 * pz;
        const unsigned cb = (unsigned)ceil_div(pz, 128);
        k_oz_colmax_pair<<<dim3(cb, (unsigned)nb, (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(p, 32), 1216 / (cb * nb)))),
                           128, 0, s>>>(A + o, M + o, pz_x, items.as<OzItem>() + b0, cm);
        UOI_CHECK_LAUNCH();
        k_oz_split<<<dim3((unsigned)nb, (unsigned)max_chunks, (unsigned)(pz_pad / 32)), 256, 0, s>>>(
            A + o, p, p * p, M + o, p, p * p, pz_x, pz, rows.as<int32_t>(), 0, items.as<OzItem>() + b0, cm, n_pad, pz_pad, 0,
            nullptr, zt.as<__nv_bfloat16>());
        UOI_CHECK_LAUNCH();
        const int splits = (int)std::max<int64_t>(
            1, std::min<int64_t>(max_chunks, 152 / std::max<int64_t>(1, (int64_t)ntiles * nb)));
        if (splits > 1) UOI_CUDA(cudaMemsetAsync(T.ptr, 0, t_item * nb, s));
        OzArgs a;
        a.pz = pz; a.pz_x = pz_x; a.ntiles = ntiles;
        a.tiles = tl.as<int32_t>(); a.items = items.as<OzItem>() + b0;
        a.cshift = cshift.as<int32_t>(); a.max_chunks = a.range = max_chunks;
        a.chunk0 = 0; a.add = splits > 1;
        a.T = T.as<long long>(); a.err = err;
        k_gram_f64tc<8><<<dim3((unsigned)ntiles, (unsigned)nb, (unsigned)splits), OZ_THREADS, OZ_SMEM, s>>>(
            oz_map(zt.ptr, n_pad, pz_pad, (int64_t)OZ_S * nb, OZ_TM),
            oz_map(zt.ptr, n_pad, pz_pad, (int64_t)OZ_S * nb, OZ_TN), a);
        UOI_CHECK_LAUNCH();
        k_oz_residual<<<dim3((unsigned)ntiles, (unsigned)nb, 2), 256, 0, s>>>(T.as<long long>(), ntiles, tl.as<int32_t>(),
                                                                             items.as<OzItem>() + b0, cm, pz_x, nseg, R + o,
                                                                             part.as<float>());
        UOI_CHECK_LAUNCH();
        k_oz_norm<<<(unsigned)nb, 256, 0, s>>>(part.as<float>(), items.as<OzItem>() + b0, cm, pz_x, nseg, norm + b0);
        UOI_CHECK_LAUNCH();
        count_launch(5);
    }
    count_launch();
}

namespace {

constexpr size_t OZ_SCRATCH = 16ull << 30;      // slices and sums in flight
constexpr size_t OZ_SCRATCH_MIN = 16ull << 20;
// One entry in so many may be far above its column's others (each costs p FP64 products per
// item); past that all sums are plain.
constexpr int64_t OZ_FAR_SHARE = 32;

// The sliced moments with at most `budget` bytes of slices and sums (one chunk of rows of one item
// at least); false (nothing usable written) for inputs that it does not take.
bool moments_sliced(const double* X, int64_t ldx, const double* Y, int64_t ldy, int64_t m, int64_t p, int64_t r,
                    const uint32_t* w, const uint8_t* mask, int32_t B, double* G, double* Bm, int b_only,
                    size_t budget, cudaStream_t s)
{
    const int32_t pz_x = (int32_t)p, pz = (int32_t)(p + r);
    const int32_t pz_pad = (int32_t)ceil_div(pz, OZ_TM) * OZ_TM;
    DevBuf items(sizeof(OzItem) * (size_t)B, s), cmax(sizeof(uint32_t) * (size_t)B * pz, s);
    DevBuf flags(3 * sizeof(int32_t), s);                // non-finite input, pipeline error, wide columns
    DevBuf stat(sizeof(unsigned long long) * (size_t)pz, s), lim, first, far_rows;
    std::vector<OzItem> hi((size_t)B);
    int32_t entries = OZ_CHUNK, hf[3] = {};
    unsigned long long weight = 0, least = ~0ull;
    auto look = [&](unsigned long long* st, const int32_t* limits) {
        UOI_CUDA(cudaMemsetAsync(cmax.ptr, 0, cmax.bytes, s));
        UOI_CUDA(cudaMemsetAsync(flags.ptr, 0, flags.bytes, s));
        if (st) UOI_CUDA(cudaMemsetAsync(st, 0, stat.bytes, s));
        k_oz_colmax<<<dim3((unsigned)ceil_div(pz, 128), (unsigned)ceil_div(m, OZ_MAX_ROWS)), 128, 0, s>>>(
            X, ldx, Y, ldy, m, pz_x, pz, B, w, mask, cmax.as<uint32_t>(), st, limits, flags.as<int32_t>());
        UOI_CHECK_LAUNCH();
        k_oz_count<<<B, 1024, 0, s>>>(w, mask, m, items.as<OzItem>(), cmax.as<uint32_t>(), st, pz, flags.as<int32_t>() + 2);
        UOI_CHECK_LAUNCH();
        count_launch(2);
        UOI_CUDA(cudaMemcpyAsync(hi.data(), items.ptr, sizeof(OzItem) * (size_t)B, cudaMemcpyDeviceToHost, s));
        UOI_CUDA(cudaMemcpyAsync(hf, flags.ptr, sizeof(hf), cudaMemcpyDeviceToHost, s));
        UOI_CUDA(cudaStreamSynchronize(s));
        entries = OZ_CHUNK;
        for (const OzItem& it : hi) {
            entries = std::max(entries, it.entries);
            weight = std::max(weight, it.weight);
            if (it.weight) least = std::min(least, it.weight);
        }
    };
    look(stat.as<unsigned long long>(), nullptr);
    // Inf and NaN propagate through the plain sums; heavier weights could pass 2^63
    if (hf[0] || weight > OZ_MAX_WEIGHT) return false;
    const bool far = hf[2] != 0;
    if (far) {
        lim.alloc(sizeof(int32_t) * (size_t)pz, s);
        first.alloc(sizeof(int64_t) * (size_t)(pz + 1), s);
        DevBuf cnt(sizeof(int64_t) * (size_t)OZ_SEGS * pz, s);
        const dim3 grid((unsigned)ceil_div(pz, 32), OZ_SEGS / 8);
        k_oz_limits<<<(unsigned)ceil_div(pz, 256), 256, 0, s>>>(stat.as<unsigned long long>(), pz, oz_spread(least), lim.as<int32_t>());
        UOI_CHECK_LAUNCH();
        k_oz_far_entries<<<grid, 256, 0, s>>>(X, ldx, Y, ldy, m, pz_x, pz, lim.as<int32_t>(), cnt.as<int64_t>(), nullptr);
        UOI_CHECK_LAUNCH();
        k_oz_far_places<<<1, 1024, 0, s>>>(cnt.as<int64_t>(), pz, first.as<int64_t>());
        UOI_CHECK_LAUNCH();
        int64_t n = 0;
        UOI_CUDA(cudaMemcpyAsync(&n, first.as<int64_t>() + pz, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        UOI_CUDA(cudaStreamSynchronize(s));
        count_launch(3);
        if (n > m * (int64_t)pz / OZ_FAR_SHARE) return false;
        far_rows.alloc(sizeof(int32_t) * (size_t)std::max<int64_t>(n, 1), s);
        k_oz_far_entries<<<grid, 256, 0, s>>>(X, ldx, Y, ldy, m, pz_x, pz, lim.as<int32_t>(), cnt.as<int64_t>(),
                                              far_rows.as<int32_t>());
        UOI_CHECK_LAUNCH();
        count_launch();
        look(nullptr, lim.as<int32_t>());
    }
    if (entries / OZ_CHUNK > 65535) return false;
    const int32_t max_chunks = entries / OZ_CHUNK;
    // tiles of the lower triangle of G and of the B block (b_only: those with a row of Y)
    std::vector<int32_t> tiles;
    for (int ti = b_only ? pz_x / OZ_TM : 0; ti * OZ_TM < pz; ++ti) {
        const int last = ti * OZ_TM + OZ_TM - 1 >= pz_x ? pz_x - 1 : ti * OZ_TM + OZ_TM - 1;
        for (int tj = 0; tj * OZ_TN <= last; ++tj) { tiles.push_back(ti); tiles.push_back(tj); }
    }
    const int ntiles = (int)tiles.size() / 2;
    DevBuf tl(sizeof(int32_t) * tiles.size(), s);
    UOI_CUDA(cudaMemcpyAsync(tl.ptr, tiles.data(), sizeof(int32_t) * tiles.size(), cudaMemcpyHostToDevice, s));
    DevBuf rows(sizeof(int32_t) * (size_t)entries * B, s), cshift(sizeof(int32_t) * (size_t)B * max_chunks, s);
    k_oz_lists<<<B, 1024, 0, s>>>(w, mask, m, entries, max_chunks, rows.as<int32_t>(), cshift.as<int32_t>());
    UOI_CHECK_LAUNCH();
    count_launch();
    // as many items at a time as the budget holds; an item that is larger alone in ranges of its
    // rows (integer sums: any split gives the same bits)
    const size_t per_chunk = (size_t)OZ_S * pz_pad * OZ_CHUNK * sizeof(__nv_bfloat16);
    const size_t s_item = far ? sizeof(double) * (size_t)pz * pz : 0;
    const size_t t_item = sizeof(long long) * 2 * OZ_TILE * (size_t)ntiles + s_item;
    const int group = (int)std::max<size_t>(1, std::min<size_t>((size_t)B, budget / (per_chunk * max_chunks + t_item)));
    const int32_t range = (int32_t)std::max<int64_t>(
        1, std::min<int64_t>(max_chunks, ((int64_t)(budget / group) - (int64_t)t_item) / (int64_t)per_chunk));
    const int64_t n_pad = (int64_t)range * OZ_CHUNK;
    DevBuf zt(per_chunk * range * group, s), T((t_item - s_item) * group, s), S;
    if (far) S.alloc(s_item * group, s);
    UOI_CUDA(cudaFuncSetAttribute(k_gram_f64tc<7>, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM));
    for (int b0 = 0; b0 < B; b0 += group) {
        const int nb = std::min(group, B - b0);
        // few tiles: split the rows until every SM has one (integer sums: any split
        // gives the same bits)
        const int splits = (int)std::max<int64_t>(
            1, std::min<int64_t>(range, 152 / std::max<int64_t>(1, (int64_t)ntiles * nb)));
        const bool add = splits > 1 || range < max_chunks;
        if (add) UOI_CUDA(cudaMemsetAsync(T.ptr, 0, (t_item - s_item) * nb, s));
        OzArgs a;
        a.pz = pz; a.pz_x = pz_x; a.ntiles = ntiles;
        a.tiles = tl.as<int32_t>(); a.items = items.as<OzItem>() + b0;
        a.cshift = cshift.as<int32_t>() + (int64_t)b0 * max_chunks; a.max_chunks = max_chunks;
        a.T = T.as<long long>(); a.err = flags.as<int32_t>() + 1;
        a.add = add; a.range = range;
        const CUtensorMap mA = oz_map(zt.ptr, n_pad, pz_pad, (int64_t)OZ_S * nb, OZ_TM);
        const CUtensorMap mB = oz_map(zt.ptr, n_pad, pz_pad, (int64_t)OZ_S * nb, OZ_TN);
        for (a.chunk0 = 0; a.chunk0 < max_chunks; a.chunk0 += range) {
            k_oz_split<<<dim3((unsigned)nb, (unsigned)std::min(range, max_chunks - a.chunk0), (unsigned)(pz_pad / 32)), 256, 0, s>>>(
                X, ldx, 0, Y, ldy, 0, pz_x, pz, rows.as<int32_t>() + (int64_t)b0 * entries, entries, items.as<OzItem>() + b0,
                cmax.as<uint32_t>() + (int64_t)b0 * pz, n_pad, pz_pad, a.chunk0, lim.as<int32_t>(),
                zt.as<__nv_bfloat16>());
            UOI_CHECK_LAUNCH();
            k_gram_f64tc<7><<<dim3((unsigned)ntiles, (unsigned)nb, (unsigned)splits), OZ_THREADS, OZ_SMEM, s>>>(mA, mB, a);
            UOI_CHECK_LAUNCH();
            count_launch(2);
        }
        if (far) {
            k_oz_far_sums<<<dim3((unsigned)pz, (unsigned)nb), 256, 0, s>>>(
                X, ldx, Y, ldy, m, pz_x, pz, w ? w + (int64_t)b0 * m : nullptr, mask ? mask + (int64_t)b0 * m : nullptr,
                lim.as<int32_t>(), first.as<int64_t>(), far_rows.as<int32_t>(), b_only, S.as<double>());
            UOI_CHECK_LAUNCH();
            count_launch();
        }
        k_oz_finish<<<dim3((unsigned)ntiles, (unsigned)nb, 2), 256, 0, s>>>(
            T.as<long long>(), ntiles, tl.as<int32_t>(), cmax.as<uint32_t>() + (int64_t)b0 * pz, pz, pz_x, (int32_t)r,
            S.as<double>(), first.as<int64_t>(), b_only ? nullptr : G + (size_t)b0 * p * p, Bm + (size_t)b0 * p * r);
        UOI_CHECK_LAUNCH();
        count_launch();
    }
    int32_t h = 0;
    UOI_CUDA(cudaMemcpyAsync(&h, flags.as<int32_t>() + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    UOI_CUDA(cudaStreamSynchronize(s));
    if (h) throw Error(h, "tensor-core FP64 Gram: a bounded pipeline wait expired");
    return true;
}

}  // namespace

void moments_f64(const double* X, int64_t ldx, const double* Y, int64_t ldy, int64_t m, int64_t p, int64_t r,
                 const uint32_t* w, const uint8_t* mask, int32_t B, double* G, double* Bm, int b_only,
                 cudaStream_t s)
{
    bool done = false;
    if (gram_tc_available() && m <= 65535ll * OZ_MAX_ROWS) {
        // less scratch where the device has no more, and the sums that need none at the end
        for (size_t budget = std::max(scratch_share(OZ_SCRATCH), OZ_SCRATCH_MIN); budget >= OZ_SCRATCH_MIN; budget /= 4) {
            try {
                done = moments_sliced(X, ldx, Y, ldy, m, p, r, w, mask, B, G, Bm, b_only, budget, s);
                break;
            } catch (const Error& e) {
                if (e.status != UOI_ERR_OOM) throw;
                cudaGetLastError();
            }
        }
    }
    if (!done) moments_fp64(X, ldx, Y, ldy, m, p, r, w, mask, B, G, Bm, b_only, s);
}

}  // namespace uoi
