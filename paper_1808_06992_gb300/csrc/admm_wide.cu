// admm_wide.cu -- G4 for many FP32 chains per group (the equations of a VAR, the lambdas
// of a cold start), 64 < p <= 512: the whole ADMM of a group in one launch, x-updates on the
// tensor cores with the chains as the products' rows.
//
//   x = c + rho M V,  v = x + u,  u' = clamp(v, +-kappa),  z' = v - u',  V' = z' - u'
//
// A cluster of `cs` CTAs iterates 128 chains of one group; CTA `rank` owns F features and
// keeps its rows of M (F x k) in shared memory.  Its product is D (128 chains x F) = V
// (128 x k, all features) times M, both as two scaled fp16 pieces (v = h + l) with the
// three products h.H, h.L, l.H, as in xupdate_tc.cu: h.H goes to one TMEM accumulator per
// 128 k, the small ones to another.  With chains as rows a thread owns one chain: the five
// residual norms are sums in its registers (no shuffles), and thresholds and scales are
// scalars of the thread.  v (which gives z and u) and c stay in TMEM beside the
// accumulators for the whole solve: an iteration moves only V and 5 norms per chain,
// through L2 (stores into the other CTAs' shared memory were slower: their fence waits for
// every store, 3600 clocks against 1200 for p = 90).
//
// One iteration t of a CTA:
//   warps 2-9  decide iteration t - 1 while the products of t run, then update their
//              features, write V' (as the operand blocks the products read) and partial
//              norms to global memory, and arrive on `cbar` of every CTA of the cluster;
//   warp 0     after cbar copies the k blocks of V into a ring (bulk copies);
//   warp 1     issues the products.
// V and the norms have two buffers by the parity of t, so cbar is the only barrier.
// Decisions are taken by every CTA from the same sums in the same order.  A chain that
// ends is replaced by the group's next one; its first product is masked (V = 0).
// Every wait is bounded (one second) and reports UOI_ERR_TIMEOUT.
//
// What bounds it: the length of one iteration, 10.5k clocks at p = 192 (2 CTAs of 96
// features): V's first block 1.0k after cbar, six blocks of products 2.3k, the update
// 4k (about 29 instructions per element on 8 warps), the fences around cbar 1.7k; at
// p = 384 12.5k, at 500 14.6k, where the products (72 clocks each) lead.  One launch per
// step spent 88k clocks per iteration at p = 384, half of them between launches.
// Measured, ADMM stage of a fit (before: the CUDA-core kernel with M in shared memory for
// p <= 192, else k_xupdate_tc once per iteration): VAR p = 192, 30 x 32 46.4 -> 18.7 ms;
// VAR(2) p = 192 (384 regressors), 20 x 16 174 -> 37 ms; VAR p = 500, 8 x 16 174 -> 72 ms.
//
// Precision up to p = 192, where the CUDA-core kernel multiplied in FP32: the tensor cores cut
// off their sums and two fp16 pieces hold 23 bits, and with all of M in the products z was
// 1.1 to 1.7 times as far from FP64 iterates on the same M and c.  M's diagonal, most of a row's
// sum, is therefore left out of the pieces and multiplied in FP32 by the update (FINE): 0.35 to
// 0.6 times as far (p = 65..192, 40 iterations), for 5 % of a VAR p = 192.  Above, the form that
// was replaced had the same pieces.
// At p <= 64 one warp per chain (k_admm_resident) is as quick or quicker: ADMM call of 20 groups,
// r = p, 16 lambdas, here and there: p = 16 1.09 and 0.59 ms, 40 1.21 and 0.85, 64 1.34 and 1.13,
// 72 1.49 and 1.44, 96 1.59 and 1.93; cold starts of 384 chains 0.40 and 0.42 at p = 40.
#include <cuda_fp16.h>

#include <algorithm>

#include "kernels.h"
#include "tc_common.cuh"

namespace uoi {

namespace {
using namespace tc;

constexpr int WD_CHAINS = 128;
constexpr int WD_THREADS = 320;
constexpr int WD_EPI = 256;                    // threads of the epilogue
constexpr int WD_BLOCK = WD_CHAINS * 64;       // one piece of a V block (128 chains x 32 k)
constexpr int WD_KB_MAX = 16;                  // k blocks (p <= 512)
constexpr int WD_CS_MAX = 8;
constexpr int WD_MIN_P = 64;                   // up to here one warp per chain is quicker
constexpr int WD_KAPPA = 256;                  // thresholds kept in shared memory
constexpr int WD_SCALE_EXP = 10;               // scaled magnitudes stay below 2^10

struct WideArgs {
    int32_t G, q, r, p, nchains, warm, W, max_iter;
    int32_t cs, F, kb, nslots, per, tmem_cols;
    float rho, abs_tol, rel_tol, sqrtp;
    const float* c;                 // G x r x p
    const float* cn;                // G x r: norms of c
    const float* row_inv;           // G x (cs F): 1 / scale of the row of M
    const float* diag;              // G x (cs F): M's diagonal (FINE)
    const double* lambdas;
    __half* v;                      // clusters x 2 x kb x 2 pieces x 128 x 32, zero
    float* norms;                   // clusters x 2 x (2 cs) x 5 x 128
    int32_t* chain_next;            // G, zero
    double* beta;
    int32_t* iters;
    uint8_t* conv;
    uint64_t* family;
    unsigned long long* near_count;
    int32_t* err;
    uint64_t wait_ns = tc::kWaitLimitNs;
};

__device__ __forceinline__ float wd_pow2_scale(float bound)
{
    if (!(bound > 0.f) || !(bound < 3.0e38f)) return 1.f;
    int e;
    frexpf(bound, &e);
    return ldexpf(1.f, min(120, max(-120, WD_SCALE_EXP - e)));
}

__device__ __forceinline__ float wd_clamp(float v, float k) { return fminf(fmaxf(v, -k), k); }

// Registers of a warp-wide TMEM load of 16 columns, completed by wd_wait.
__device__ __forceinline__ void wd_ld16(uint32_t taddr, uint32_t (&r)[16]) { tmem_ld16_issue(taddr, r); }

template <int N>
__device__ __forceinline__ void wd_wait(uint32_t (&r)[N][16])
{
    // the first wait completes every load issued before it; the others only tie the
    // registers to it
#pragma unroll
    for (int i = 0; i < N; ++i) tmem_wait16(r[i]);
}

__device__ __forceinline__ void wd_st16(uint32_t taddr, const float (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
        "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15]))
        : "memory");
}

__device__ __forceinline__ void wd_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Address in CTA `rank`'s shared memory of this CTA's shared address `a`.
__device__ __forceinline__ uint32_t wd_map(uint32_t a, int rank)
{
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(rank));
    return d;
}

// 32 bytes to global memory in one store.
__device__ __forceinline__ void wd_store32(void* p, const uint32_t (&v)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// NQ accumulators of h.H (one per 128 k), added with their rounding errors when COMP.  FINE: M's
// diagonal is not in the products; the update multiplies it in FP32.
// TMEM columns: h.H [NQ][F], small products [F], v [F], c [F].
template <int NQ, bool COMP, bool FINE>
__global__ void __launch_bounds__(WD_THREADS, 1)
k_admm_wide(const __grid_constant__ CUtensorMap tmM, WideArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ uint64_t vfull[WD_KB_MAX], vempty[WD_KB_MAX], mfull, accf, cbar;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, s_stop, s_any[2];
    __shared__ __align__(16) float s_rinv[128], s_diag[FINE ? 128 : 4];
    __shared__ float s_kappa[WD_KAPPA];
    __shared__ float s_kst[WD_CHAINS], s_kc[WD_CHAINS], s_vrinv[WD_CHAINS], s_vw[WD_CHAINS];
    __shared__ int s_cid[WD_CHAINS];
    __shared__ int s_e[WD_CHAINS], s_done[WD_CHAINS];   // equation; column index j + 1 finished last, or 0
    __shared__ uint8_t s_fresh[WD_CHAINS];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cs = a.cs, F = a.F, kb = a.kb;
    int rank = 0;
    if (cs > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int g = blockIdx.y, tile = blockIdx.x / cs;
    const int64_t cluster = (int64_t)g * a.per + tile;
    const uint32_t m_piece = (uint32_t)F * 64, m_block = 2 * m_piece;
    const uint32_t sM = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sV = sM + (uint32_t)kb * m_block;      // ring of nslots blocks (two pieces)
    const int64_t v_buf = (int64_t)kb * 2 * (WD_BLOCK / 2);       // halves per buffer
    __half* gv = a.v + cluster * 2 * v_buf;

    if (threadIdx.x == 0) {
        for (int s = 0; s < WD_KB_MAX; ++s) { mbar_init(&vfull[s], 1); mbar_init(&vempty[s], 1); }
        mbar_init(&mfull, 1);
        mbar_init(&accf, 1);
        mbar_init(&cbar, (uint32_t)cs * (WD_EPI / 32));
        abort_flag = 0;
        s_stop = 0;
        s_any[0] = s_any[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    for (int i = threadIdx.x; i < F; i += blockDim.x) s_rinv[i] = a.row_inv[(int64_t)g * cs * F + rank * F + i];
    if constexpr (FINE)
        for (int i = threadIdx.x; i < F; i += blockDim.x) s_diag[i] = a.diag[(int64_t)g * cs * F + rank * F + i];
    for (int i = threadIdx.x; i < min(a.q, WD_KAPPA); i += blockDim.x) s_kappa[i] = (float)a.lambdas[i] / a.rho;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"((uint32_t)a.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    if (cs > 1) cluster_sync();                // every CTA's barriers exist
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    auto fail = [&] {
        abort_flag = 1;
        atomicCAS(a.err, 0, UOI_ERR_TIMEOUT);
    };

    if (warp == 0 && elect_one()) {
        // ---------------- producer: M once, V every iteration ----------------
        mbar_expect_tx(&mfull, (uint32_t)kb * m_block);
        for (int b = 0; b < kb; ++b)
            tma_load_3d(sM + b * m_block, &tmM, &mfull, 0, 0, ((g * cs + rank) * kb + b) * 2);
        bool ok = true;
        // slot of the ring and the parity of its round, counted on (no division per block)
        int s = 0, used = 0;
        uint32_t round = 0;
        for (uint32_t t = 0; ok; ++t) {
            if (t > 0) {
                ok = mbar_wait_cluster(&cbar, (t - 1) & 1u, &abort_flag, a.wait_ns);
                if (!ok || *(volatile int*)&s_stop) break;
                asm volatile("fence.proxy.async.global;" ::: "memory");
            }
            const __half* src = gv + (int64_t)(t & 1u) * v_buf;
            for (int b = 0; b < kb; ++b) {
                // a ring that holds every block is free again once cbar has come
                if (a.nslots < kb && used == a.nslots && !mbar_wait(&vempty[s], round ^ 1u, &abort_flag, a.wait_ns)) {
                    ok = false;
                    break;
                }
                if (used < a.nslots) ++used;
                mbar_expect_tx(&vfull[s], 2 * WD_BLOCK);
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                        sV + (uint32_t)s * 2 * WD_BLOCK),
                    "l"(src + (int64_t)b * WD_BLOCK), "r"(2 * WD_BLOCK), "r"(smem_u32(&vfull[s]))
                    : "memory");
                if (++s == a.nslots) { s = 0; round ^= 1u; }
            }
        }
        if (!ok) {
            fail();
            // copies in flight land before the CTA's memory is given back
            int dummy = 0;
            mbar_wait(&mfull, 0, &dummy, a.wait_ns);
            for (int k = 0; k < used; ++k)           // last round of each slot: this one before s, else the one before
                mbar_wait(&vfull[k], k < s ? round : round ^ 1u, &dummy, a.wait_ns);
        }
    } else if (warp == 1 && elect_one()) {
        // ---------------- MMA issuer ----------------
        const uint32_t idesc = idesc_f16(WD_CHAINS, F);
        const uint32_t small = tmem + (uint32_t)(NQ * F);
        bool ok = mbar_wait(&mfull, 0, &abort_flag, a.wait_ns);
        int s = 0;
        uint32_t round = 0;
        for (uint32_t t = 0; ok; ++t) {
            if (t > 0) {
                ok = mbar_wait_cluster(&cbar, (t - 1) & 1u, &abort_flag, a.wait_ns);
                if (!ok || *(volatile int*)&s_stop) break;
            }
            for (int b = 0; b < kb; ++b) {
                if (!mbar_wait(&vfull[s], round, &abort_flag, a.wait_ns)) { ok = false; break; }
                tc_fence_after();
                const uint32_t va = sV + (uint32_t)s * 2 * WD_BLOCK, mb = sM + (uint32_t)b * m_block;
                const uint64_t Ah = smem_desc_sw64(va), Al = smem_desc_sw64(va + WD_BLOCK);
                const uint64_t Bh = smem_desc_sw64(mb), Bl = smem_desc_sw64(mb + m_piece);
                const uint32_t d1 = tmem + (uint32_t)((b >> 2) * F);       // 4 blocks of 32 k per accumulator
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    const uint64_t adv = (uint64_t)(ks * 32 >> 4);
                    mma_bf16(d1, Ah + adv, Bh + adv, idesc, ((b & 3) > 0 || ks > 0) ? 1u : 0u);
                    mma_bf16(small, Ah + adv, Bl + adv, idesc, (b > 0 || ks > 0) ? 1u : 0u);
                    mma_bf16(small, Al + adv, Bh + adv, idesc, 1u);
                }
                if (a.nslots < kb) mma_commit(&vempty[s]);
                if (++s == a.nslots) { s = 0; round ^= 1u; }
            }
            mma_commit(&accf);
        }
        if (!ok) {
            // after a timeout the products issued finish before TMEM is given back
            fail();
            const uint64_t t0 = now_ns();
            while (now_ns() - t0 < 1000000ull) { }
        }
    } else if (warp >= 2) {
        // ---------------- epilogue ----------------
        const int quad = warp & 3, half = (warp - 2) >> 2;
        const int ch = quad * 32 + lane;                 // chain of this thread
        const int FH = F / 2, f0 = half * FH;            // its features: rank * F + f0 .. + FH - 1
        const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)f0;
        const uint32_t t_small = tl + (uint32_t)(NQ * F), t_v = t_small + (uint32_t)F, t_c = t_v + (uint32_t)F;
        float* nrm = a.norms + cluster * 2 * (2 * cs) * 5 * WD_CHAINS;
        // control state of the chain (threads of half 0; the same in every CTA)
        int status = 0, e = 0, j = 0, jend = 0, it = 0;  // status 0 none, 1 iterating, 2 waiting for the next chain
        float kc = 0.f, kst = 0.f, vw = 0.f, vrinv = 0.f, cnorm = 0.f;
        auto kappa_of = [&](int jj) { return jj < WD_KAPPA ? s_kappa[jj] : (float)a.lambdas[jj] / a.rho; };
        auto start = [&](int cid) {
            status = cid < a.nchains ? 1 : 0;
            if (!status) return;
            if (a.warm) { e = cid; j = 0; jend = a.q; }
            else        { e = cid % a.r; j = cid / a.r; jend = j + 1; }
            it = 0;
            kc = kst = kappa_of(j);
            cnorm = a.cn[(int64_t)g * a.r + e];
            vrinv = 0.f;                                 // the product of the first step is V = 0
            vw = wd_pow2_scale(6.f * cnorm);
        };
        if (half == 0) start(tile * WD_CHAINS + ch);
        const bool more = (int64_t)a.per * WD_CHAINS < a.nchains;
        int done_j = 0;                                  // column finished by this decision + 1
        bool fresh = half == 0;
        for (uint32_t t = 0;; ++t) {
            if (half == 0) {
                if (t > 0) {
                    // ---- decision of iteration t - 1 ----
                    const bool ok = mbar_wait_cluster(&cbar, (t - 1) & 1u, &abort_flag, a.wait_ns);
                    if (!__all_sync(0xffffffffu, ok)) { fail(); }
                    const float* nr = nrm + (int64_t)((t - 1) & 1u) * (2 * cs) * 5 * WD_CHAINS + ch;
                    fresh = false;
                    done_j = 0;
                    kst = kc;
                    vrinv = vw != 0.f ? 1.f / vw : 0.f;
                    if (status == 1) {
                        float tot[5] = { 0.f, 0.f, 0.f, 0.f, 0.f };
#pragma unroll 4
                        for (int k = 0; k < 2 * cs; ++k)
#pragma unroll
                            for (int w = 0; w < 5; ++w) tot[w] += __ldcg(nr + (k * 5 + w) * WD_CHAINS);
                        it += 1;
                        const float xn = sqrtf(tot[2]), zn = sqrtf(tot[3]), un = sqrtf(tot[4]);
                        const float ep = a.sqrtp * a.abs_tol + a.rel_tol * fmaxf(xn, zn);
                        const float ed = a.sqrtp * a.abs_tol + a.rel_tol * a.rho * un;
                        const bool conv = sqrtf(tot[0]) <= ep && a.rho * sqrtf(tot[1]) <= ed;
                        vw = wd_pow2_scale(6.f * (cnorm + zn + 2.f * un));
                        if (conv || it >= a.max_iter) {
                            done_j = j + 1;
                            const int64_t col = ((int64_t)g * a.q + j) * a.r + e;
                            if (rank == 0) {
                                if (a.iters) a.iters[col] = it;
                                if (a.conv) a.conv[col] = conv ? 1 : 0;
                            }
                            if (++j < jend) {
                                it = 0;
                                kc = kappa_of(j);
                            } else {
                                status = more ? 2 : 0;
                                vw = 0.f;
                                if (more && rank == 0) {
                                    const int cid = a.per * WD_CHAINS + atomicAdd(&a.chain_next[g], 1);
                                    for (int k = 0; k < cs; ++k) {
                                        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(
                                                         wd_map(smem_u32(&s_cid[ch]), k)),
                                                     "r"(cid)
                                                     : "memory");
                                    }
                                }
                            }
                        }
                    } else if (status == 2) {
                        start(*(volatile int*)&s_cid[ch]);   // written one iteration ago
                        fresh = status == 1;
                    }
                }
                s_kst[ch] = kst; s_kc[ch] = kc; s_vrinv[ch] = vrinv; s_vw[ch] = status == 1 ? vw : 0.f;
                s_fresh[ch] = fresh ? 1 : 0;
                s_e[ch] = e;
                s_done[ch] = done_j;
                // (after a timeout nobody asks for another iteration, so that all warps stop together)
                if (__any_sync(0xffffffffu, status != 0) && lane == 0 && !*(volatile int*)&abort_flag)
                    s_any[t & 1u] = 1;
            }
            named_barrier_sync(1, WD_EPI);
            const bool go = *(volatile int*)&s_any[t & 1u] != 0;      // the same in all epilogue warps
            if (threadIdx.x == 64) s_any[(t + 1) & 1u] = 0;    // set again only after the next cbar
            const float ks = s_kst[ch], kn = s_kc[ch], vi = s_vrinv[ch], sw = s_vw[ch];
            const int ee = s_e[ch], dj = s_done[ch];
            const bool fr = s_fresh[ch] != 0;
            // ---- output of the columns that finished ----
            if (__any_sync(0xffffffffu, dj != 0)) {
                const int64_t col_je = (int64_t)(dj - 1) * a.r + ee, col = (int64_t)g * a.q * a.r + col_je;
                for (int f = 0; f < FH; f += 16) {
                    uint32_t rv[1][16];
                    wd_ld16(t_v + (uint32_t)f, rv[0]);
                    wd_wait(rv);
                    const int i0 = rank * F + f0 + f;
                    // z = v - clamp(v): zero where |v| <= kappa, and ||v| - kappa| is the margin
                    uint32_t zero = 0;
                    int near = 0;
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const float gap = fabsf(__uint_as_float(rv[0][k])) - ks;
                        if (!(gap > 0.f)) zero |= 1u << k;
                        near += i0 + k < a.p && fabsf(gap) <= (float)kNearThreshold ? 1 : 0;
                    }
                    if (i0 + 16 > a.p) zero &= i0 < a.p ? (1u << (a.p - i0)) - 1u : 0u;
                    if (dj && a.beta) {
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const float v = __uint_as_float(rv[0][k]);
                            const int64_t o = col * a.p + i0 + k;
                            if (i0 + k < a.p && UOI_IN_BOUNDS(o, (int64_t)a.G * a.q * a.r * a.p, 401))
                                a.beta[o] = (double)(v - wd_clamp(v, ks));
                        }
                    }
                    // 16 features from a multiple of 16: within one word
                    if (dj && a.family && zero)
                        atomicAnd((unsigned long long*)&a.family[col_je * a.W + (i0 >> 6)],
                                  ~((unsigned long long)zero << (i0 & 63)));
                    if (dj && a.near_count && near) atomicAdd(a.near_count, (unsigned long long)near);
                }
            }
            // ---- state of a chain that starts: v = 0 and its c ----
            if (__any_sync(0xffffffffu, fr)) {
                for (int f = 0; f < FH; f += 16) {
                    uint32_t rr[2][16];
                    wd_ld16(t_v + (uint32_t)f, rr[0]);
                    wd_ld16(t_c + (uint32_t)f, rr[1]);
                    wd_wait(rr);
                    float nv[16], nc[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const int i = rank * F + f0 + f + k;
                        nv[k] = fr ? 0.f : __uint_as_float(rr[0][k]);
                        nc[k] = !fr ? __uint_as_float(rr[1][k])
                                    : (sw != 0.f && i < a.p ? a.c[((int64_t)g * a.r + ee) * a.p + i] : 0.f);
                    }
                    wd_st16(t_v + (uint32_t)f, nv);
                    wd_st16(t_c + (uint32_t)f, nc);
                    wd_st_wait();
                }
            }
            // ---- update ----
            bool ok = mbar_wait(&accf, t & 1u, &abort_flag, a.wait_ns);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) fail();
            tc_fence_after();
            if (go && ok) {
                float n5[5] = { 0.f, 0.f, 0.f, 0.f, 0.f };
                for (int f = 0; f < FH; f += 16) {
                    uint32_t rr[NQ + 3][16];
#pragma unroll
                    for (int qa = 0; qa < NQ; ++qa) wd_ld16(tl + (uint32_t)(qa * F + f), rr[qa]);
                    wd_ld16(t_small + (uint32_t)f, rr[NQ]);
                    wd_ld16(t_v + (uint32_t)f, rr[NQ + 1]);
                    wd_ld16(t_c + (uint32_t)f, rr[NQ + 2]);
                    wd_wait(rr);
                    float nv[16];
                    uint32_t ph[8], pl[8];
#pragma unroll
                    for (int k = 0; k < 16; k += 2) {
                        float vs[2];
#pragma unroll
                        for (int k2 = 0; k2 < 2; ++k2) {
                            const int kk = k + k2;
                            float hh = __uint_as_float(rr[0][kk]), lo = __uint_as_float(rr[NQ][kk]);
#pragma unroll
                            for (int qa = 1; qa < NQ; ++qa) {
                                const float y = __uint_as_float(rr[qa][kk]);
                                const float s = __fadd_rn(hh, y);
                                if constexpr (COMP) {              // the rounding errors join the small products
                                    const float b = __fsub_rn(s, hh);
                                    lo += __fsub_rn(hh, __fsub_rn(s, b)) + __fsub_rn(y, b);
                                }
                                hh = s;
                            }
                            const float vo = __uint_as_float(rr[NQ + 1][kk]);
                            const float uo = wd_clamp(vo, ks), zp = vo - uo;
                            float prod = (hh + lo) * (s_rinv[f0 + f + kk] * vi);
                            if constexpr (FINE) prod = fmaf(s_diag[f0 + f + kk], zp - uo, prod);
                            const float x = __uint_as_float(rr[NQ + 2][kk]) + a.rho * prod;
                            const float v = x + uo, un = wd_clamp(v, kn), zn = v - un;
                            nv[kk] = v;
                            const float d = x - zn, dz = zn - zp;
                            n5[0] += d * d; n5[1] += dz * dz; n5[2] += x * x; n5[3] += zn * zn; n5[4] += un * un;
                            vs[k2] = (zn - un) * sw;
                        }
                        const __half2 h = __floats2half2_rn(vs[0], vs[1]);
                        const float2 hf = __half22float2(h);
                        const __half2 l = __floats2half2_rn(vs[0] - hf.x, vs[1] - hf.y);
                        ph[k / 2] = *reinterpret_cast<const uint32_t*>(&h);
                        pl[k / 2] = *reinterpret_cast<const uint32_t*>(&l);
                    }
                    wd_st16(t_v + (uint32_t)f, nv);
                    // 32 bytes per piece of row `ch` in this feature's k block (64-byte swizzle: 16-byte
                    // chunk index ^ bits 1-2 of the row, so a pair of chunks stays one sector)
                    const int kf = rank * F + f0 + f, sw2 = (ch >> 1) & 3;
                    unsigned char* blk = reinterpret_cast<unsigned char*>(gv + (int64_t)((t + 1) & 1u) * v_buf) +
                                         (size_t)(kf >> 5) * 2 * WD_BLOCK + ch * 64 + ((((kf & 31) >> 4) ^ (sw2 >> 1)) * 32);
                    uint32_t oh[8], ol[8];
#pragma unroll
                    for (int w = 0; w < 8; ++w) {
                        oh[w] = (sw2 & 1) ? ph[w ^ 4] : ph[w];
                        ol[w] = (sw2 & 1) ? pl[w ^ 4] : pl[w];
                    }
                    wd_store32(blk, oh);
                    wd_store32(blk + WD_BLOCK, ol);
                }
                wd_st_wait();
                float* nw = nrm + ((int64_t)(t & 1u) * (2 * cs) + 2 * rank + half) * 5 * WD_CHAINS + ch;
#pragma unroll
                for (int w = 0; w < 5; ++w) __stcg(nw + w * WD_CHAINS, n5[w]);
                // V' of a chain that has ended is the first operand of the one that takes its lane.  NaN
                // and Inf survive the product with sw = 0: zeros over what was stored (a select
                // per feature in the loop above cost 2.5 % of a fit at p = 192)
                if (__builtin_expect(sw == 0.f && !(n5[2] + n5[3] + n5[4] < 3.0e38f), 0)) {
                    unsigned char* v = reinterpret_cast<unsigned char*>(gv + (int64_t)((t + 1) & 1u) * v_buf) + ch * 64;
#pragma unroll 1
                    for (int x = 0; x < FH / 4; ++x) {       // 16 bytes each: two per piece of 16 features
                        const int k = rank * F + f0 + (x >> 2) * 16;
                        *reinterpret_cast<uint4*>(v + (size_t)((k >> 5) * 2 + ((x >> 1) & 1)) * WD_BLOCK +
                                                  (((k >> 4) ^ (ch >> 2)) & 1) * 32 + (x & 1) * 16) = make_uint4(0u, 0u, 0u, 0u);
                    }
                }
                __syncwarp();
                asm volatile("fence.proxy.async.global;" ::: "memory");    // the bulk copies read V'
            } else if (!go && lane == 0) {
                *(volatile int*)&s_stop = 1;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                // one release fence for the warp, then an arrival per CTA
                asm volatile("fence.acq_rel.cluster;" ::: "memory");
                for (int k = 0; k < cs; ++k)
                    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                                     cluster_addr(&cbar, (uint32_t)k))
                                 : "memory");
            }
            if (!go) break;
        }
    }
    __syncthreads();
    if (cs > 1) cluster_sync();                // no CTA leaves while another may signal it
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)a.tmem_cols));
    }
}

// M_g -> per-row scales and fp16 pieces in blocks [g][rank][k block][piece][F][32] (zero
// padded), one warp per row; the arithmetic is k_scale_split_m's (xupdate_tc.cu).  diag
// (nullable): the diagonal goes there, and zero to the pieces.
__global__ void k_wide_split_m(const float* M, int32_t G, int p, int cs, int F, int kb, float* row_inv, float* diag, __half* out)
{
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, ppad = cs * F;
    if (row >= (int64_t)G * ppad) return;
    const int64_t g = row / ppad;
    const int i = (int)(row % ppad);
    const bool real = i < p;
    const float* mr = M + ((size_t)g * p + (real ? i : 0)) * p;
    float v[WD_KB_MAX], mx = 0.f;
#pragma unroll
    for (int b = 0; b < WD_KB_MAX; ++b) {
        const int k = 32 * b + lane;
        v[b] = real && k < p ? mr[k] : 0.f;
        if (diag && k == i) {
            diag[row] = v[b];
            v[b] = 0.f;
        }
        mx = fmaxf(mx, fabsf(v[b]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const float sc = wd_pow2_scale(mx);
    if (lane == 0) row_inv[row] = 1.f / sc;
    __half* o = out + (((g * cs + i / F) * kb * 2) * (int64_t)F + i % F) * 32 + lane;
#pragma unroll
    for (int b = 0; b < WD_KB_MAX; ++b) {
        if (b >= kb) break;
        const float x = v[b] * sc;
        const __half h = __float2half_rn(x);
        o[(int64_t)(2 * b) * F * 32] = h;
        o[(int64_t)(2 * b + 1) * F * 32] = __float2half_rn(x - __half2float(h));
    }
}

// ||c||_2 of every (group, response), one warp each.
__global__ void k_wide_c_norms(const float* c, int64_t count, int64_t p, float* cn)
{
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= count) return;
    float acc = 0.f;
    for (int64_t i = lane; i < p; i += 32) acc += c[row * p + i] * c[row * p + i];
    acc = warp_sum(acc);
    if (lane == 0) cn[row] = sqrtf(acc);
}

// Blocks of F rows x 32 k of 16-bit values, two consecutive blocks (the pieces) per box.
CUtensorMap wide_map(void* base, int64_t nblocks, int F)
{
    CUtensorMap m;
    cuuint64_t dims[3] = { 32u, (cuuint64_t)F, (cuuint64_t)nblocks };
    cuuint64_t strides[2] = { 64u, 64u * (cuuint64_t)F };
    cuuint32_t box[3] = { 32u, (cuuint32_t)F, 2u };
    cuuint32_t estr[3] = { 1, 1, 1 };
    CUresult res = tc::encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, base, dims, strides, box, estr,
                                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (res != CUDA_SUCCESS) throw Error(UOI_ERR_CUDA, "cuTensorMapEncodeTiled failed");
    return m;
}

using WideKernel = void (*)(CUtensorMap, WideArgs);
// Up to p = WD_FINE_P this form replaces FP32 multiply-adds (k_admm_resident).
constexpr int WD_FINE_P = 192;
WideKernel wide_kernel(int nq, int p)
{
    if (nq == 1) return k_admm_wide<1, false, true>;
    if (nq == 2) return p <= WD_FINE_P ? k_admm_wide<2, false, true> : k_admm_wide<2, true, false>;
    return nq == 3 ? k_admm_wide<3, true, false> : k_admm_wide<4, true, false>;
}

struct WideShape {
    int F = 0, cs = 0, kb = 0, nq = 0, nslots = 0, tmem_cols = 0;
    size_t smem = 0;
};

// The layout for F features per CTA; false where TMEM, shared memory or the cluster is
// too small for it.
bool wide_shape(int p, int F, WideShape& s)
{
    s.F = F;
    s.cs = (int)ceil_div(p, F);
    s.kb = s.cs * F / 32;
    s.nq = (int)ceil_div(s.kb, 4);
    if (s.cs > WD_CS_MAX || s.kb > WD_KB_MAX || (s.nq + 3) * F > 512) return false;
    s.tmem_cols = 32;
    while (s.tmem_cols < (s.nq + 3) * F) s.tmem_cols *= 2;
    constexpr size_t cap = 227 * 1024 - 1024 - 6 * 1024;       // alignment, static arrays
    const size_t m = (size_t)s.kb * F * 128, block = 2 * WD_BLOCK;
    if (m + std::min(4, s.kb) * block > cap) return false;
    s.nslots = (int)std::min<size_t>(s.kb, (cap - m) / block);
    s.smem = m + s.nslots * block + 1024;
    return true;
}

}  // namespace

// Runs the whole solve here if the problem fits; false (nothing launched) otherwise.
bool admm_solve_wide(const AdmmProblem<float>& P, cudaStream_t s)
{
    const int64_t nchains = P.warm ? P.r : P.r * P.q;
    if (P.p <= WD_MIN_P || P.p > 32 * WD_KB_MAX || P.z0 || P.u_out || nchains > (1 << 30) || !gram_tc_available()) return false;
    // Fewest CTAs per chain tile while the tiles fill the device; with fewer tiles, more
    // CTAs each (their epilogues and products shrink with F)
    const int p = (int)P.p;
    const int64_t want = (int64_t)P.G * ceil_div(nchains, WD_CHAINS);
    WideShape sh, best;
    for (int F : { 128, 96, 64, 32 }) {
        if (!wide_shape(p, F, sh)) continue;
        if (best.F && want * sh.cs > 128) break;
        best = sh;
    }
    if (!best.F) return false;
    const int ppad = best.cs * best.F;
    const bool fine = p <= WD_FINE_P;
    const WideKernel kern = wide_kernel(best.nq, p);
    allow_max_dynamic_smem((const void*)kern);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(WD_THREADS);
    cfg.dynamicSmemBytes = best.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)best.cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)best.cs, (unsigned)P.G);
    int resident = 0;
    UOI_CUDA(cudaOccupancyMaxActiveClusters(&resident, kern, &cfg));
    if (resident < 1) return false;
    const int per = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(nchains, WD_CHAINS), resident / P.G));
    DevBuf mp(sizeof(__half) * 2 * (size_t)P.G * ppad * ppad, s), rinv(sizeof(float) * (size_t)P.G * ppad * 2, s);
    DevBuf cn(sizeof(float) * (size_t)P.G * P.r, s);
    DevBuf vb((size_t)P.G * per * 2 * best.kb * 2 * WD_BLOCK, s);
    UOI_CUDA(cudaMemsetAsync(vb.ptr, 0, vb.bytes, s));
    DevBuf nrm(sizeof(float) * (size_t)P.G * per * 2 * 2 * best.cs * 5 * WD_CHAINS, s);
    DevBuf next(sizeof(int32_t) * (size_t)(P.G + 1), s);
    UOI_CUDA(cudaMemsetAsync(next.ptr, 0, next.bytes, s));
    float* diag = rinv.as<float>() + (size_t)P.G * ppad;
    k_wide_split_m<<<(unsigned)ceil_div((int64_t)P.G * ppad * 32, 256), 256, 0, s>>>(
        P.M, P.G, p, best.cs, best.F, best.kb, rinv.as<float>(), fine ? diag : nullptr, mp.as<__half>());
    UOI_CHECK_LAUNCH();
    k_wide_c_norms<<<(unsigned)ceil_div((int64_t)P.G * P.r * 32, 256), 256, 0, s>>>(P.c, (int64_t)P.G * P.r, P.p,
                                                                                    cn.as<float>());
    UOI_CHECK_LAUNCH();
    WideArgs a;
    a.G = P.G; a.q = P.q; a.r = (int32_t)P.r; a.p = p; a.nchains = (int32_t)nchains; a.warm = P.warm;
    a.W = (p + 63) / 64; a.max_iter = P.max_iter;
    a.cs = best.cs; a.F = best.F; a.kb = best.kb; a.nslots = best.nslots; a.per = per;
    a.tmem_cols = best.tmem_cols;
    a.rho = (float)P.rho; a.abs_tol = (float)P.abs_tol; a.rel_tol = (float)P.rel_tol; a.sqrtp = (float)sqrt((double)p);
    a.c = P.c; a.cn = cn.as<float>(); a.row_inv = rinv.as<float>(); a.diag = diag; a.lambdas = P.lambdas;
    a.v = vb.as<__half>(); a.norms = nrm.as<float>(); a.chain_next = next.as<int32_t>();
    a.beta = P.beta; a.iters = P.iters; a.conv = P.conv; a.family = P.family; a.near_count = P.near_count;
    a.err = next.as<int32_t>() + P.G;
    const CUtensorMap mM = wide_map(mp.ptr, (int64_t)P.G * best.cs * best.kb * 2, best.F);
    cfg.gridDim = dim3((unsigned)(best.cs * per), (unsigned)P.G);
    UOI_CUDA(cudaLaunchKernelEx(&cfg, kern, mM, a));
    UOI_CHECK_LAUNCH();
    count_launch(3);
    int32_t* h = pinned_scratch_i32();
    UOI_CUDA(cudaMemcpyAsync(h, a.err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    UOI_CUDA(cudaStreamSynchronize(s));
    if (*h) throw Error(*h, "tensor-core ADMM: a bounded wait expired");
    return true;
}

}  // namespace uoi
