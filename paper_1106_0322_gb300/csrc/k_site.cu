// k_site.cu -- the paper's single-coordinate move cycle (Section 4.1, "Further details").
//
// A cycle of single-coordinate random-walk Metropolis updates, j = 0..p-1 in order, each
// proposing beta_j' = beta_j + sd * xi, repeated M times per step. One warp per particle, one
// launch per step. eta2 = log2(e) X beta is kept per particle (computed from X^T at the start
// of the step) and changes by x_.j delta when an update is accepted, so an update costs O(n):
//   delta l = delta v_j - ln 2 * sum_i [softplus2(eta2_i + x2_ij delta) - softplus2(eta2_i)]
// with the linear half from v = X^T y. softplus2 = max(eta2, 0) + log2(1 + 2^-|eta2|); the
// max parts are summed as differences, the log parts as the base-2 logarithm of the
// product of their factors (each in [1, 2], SITE_CHUNK per product), and each lane keeps
// that log for its individuals at the current state, so a trial needs one ex2 per
// individual. The normal is Box-Muller's cosine branch on words 0 and 1 of the Philox
// block (j, particle, t, TAG_SITE << 16 | m), word 2 the update's uniform.
//
// Lane l owns the individuals l, l + 32, ...: two kernels with the same arithmetic, eta2 in
// registers (n <= 32 SITE_CHUNK) or in shared memory (larger n).
#include "spa_device.cuh"
#include "spa_internal.h"

namespace spa {

namespace {

constexpr int SITE_CHUNK = 64;

// ------------------------------------------------------------ eta2 in registers
// Lane l's KC values eta2[l + 32 k] sit in registers as pairs (k even, odd), and X^T in the
// order the lane reads it, four of its individuals per 16-byte load (k_store_xsite). Padding
// individuals (r >= n) carry x = 0 and eta2 = SITE_PAD, so their terms are exact zeros: the
// max difference is 0 and 2^-|eta2| underflows to 0.
//
// What bounds it (ncu, n = 1859): instruction issue, active 61% of the time at 7.9 instructions
// per individual, and the columns' reads (86% L1 hits, the rest from L2). Per individual a trial is a quarter of a load, half a
// packed FMA, two max, half a packed subtraction, the two serial accumulations and one ex2,
// 6.25 instructions. The p updates' random numbers, log-uniforms and prior terms do not
// depend on the other updates of the cycle, so 32 of them are formed side by side, one per
// lane, and broadcast; one at a time they cost every lane about 300 instructions an update.
// N = 8192, 5 cycles a step, against the shared-memory kernel below: n = 1859, p = 184
// 13.3 -> 4.6 ms; n = 500, p = 50 1.45 -> 0.42 ms; the same bits.
constexpr float SITE_PAD = -1e30f;
constexpr int SITE_WARPS = 4;  // particles per block

// 16-byte loads of the next update's column issued before this update's reduction: 4 where the
// registers allow (n = 1000: 485 -> 370 us a step), none at the widest (n = 1859: 4.55 ms
// without, 4.74 ms with).
__host__ __device__ constexpr int site_prefetch(int KC) { return KC > 48 ? 0 : (KC < 16 ? KC / 4 : 4); }

// Blocks per SM that the register count is held to. More resident warps with fewer registers,
// or 8 to 16 warps a block, measured the same or slower.
constexpr int site_min_blocks(int KC) { return KC <= 16 ? 7 : (KC <= 32 ? 5 : (KC <= 48 ? 4 : 3)); }

template <int KC>
__global__ void __launch_bounds__(32 * SITE_WARPS, site_min_blocks(KC))
    k_move_site_reg(SiteArgs a, int64_t N, int p, int n, PriorArgs pr, const float4* __restrict__ stepk, int t,
                    uint32_t m0, int M, const uint64_t* __restrict__ seedp)
{
    constexpr int K4 = KC / 4;
    constexpr int PF = site_prefetch(KC);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * SITE_WARPS + w;
    int nacc = 0;
    if (i < N) {
        const float4 sk = stepk[t];
        const uint64_t seed = *seedp;
        const float coef = sk.y, inv_ac = sk.w;
        float* bg = a.beta + i * p;
        const float4* X = reinterpret_cast<const float4*>(a.XS) + lane;  // X[(j * K4 + k4) * 32]
        const uint64_t negone = pack2(-1.0f, -1.0f);
        uint64_t eta[KC / 2];
#pragma unroll
        for (int k = 0; k < KC; k += 2)
            eta[k >> 1] = pack2(lane + 32 * k < n ? 0.0f : SITE_PAD, lane + 32 * (k + 1) < n ? 0.0f : SITE_PAD);
        for (int j = 0; j < p; ++j) {  // eta2 = X2 beta, marker by marker
            const float bj = bg[j];
            const uint64_t bb = pack2(bj, bj);
            const float4* xr = X + (size_t)j * K4 * 32;
#pragma unroll
            for (int k4 = 0; k4 < K4; ++k4) {
                const float4 x = __ldg(xr + 32 * k4);
                eta[2 * k4] = fma2(pack2(x.x, x.y), bb, eta[2 * k4]);
                eta[2 * k4 + 1] = fma2(pack2(x.z, x.w), bb, eta[2 * k4 + 1]);
            }
        }
        float lq;  // log2 of the product of the lane's factors at the current state
        {
            float prod = 1.0f;
#pragma unroll
            for (int k = 0; k < KC / 2; ++k) {
                const float2 e = unpack2(eta[k]);
                prod = fmaf(prod, ex2_approx(-fabsf(e.x)), prod);
                prod = fmaf(prod, ex2_approx(-fabsf(e.y)), prod);
            }
            lq = lg2_approx(prod);
        }
        for (int mm = 0; mm < M; ++mm) {
            const uint32_t m = m0 + (uint32_t)mm;
            for (int j0 = 0; j0 < p; j0 += 32) {
                // lane l draws update j0 + l; nothing here depends on the other updates
                const int jl = j0 + lane;
                const bool in = jl < p;
                const uint4 u = philox4x32_10(make_uint4((uint32_t)jl, (uint32_t)i, (uint32_t)t, (TAG_SITE << 16) | m),
                                              seed_key(seed));
                float sn, cs;
                sincospif(2.0f * u01_open_cvt_f(u.y), &sn, &cs);
                const float delta_l = __fmul_rn(a.sd, __fmul_rn(sqrtf(-2.0f * logf(u01_open_cvt_f(u.x))), cs));
                const float lu_l = logf(u01_open_cvt_f(u.z));
                const float b0 = in ? bg[jl] : 0.0f, v_l = in ? a.vy[jl] : 0.0f;
                const float b1 = __fadd_rn(b0, delta_l);
                const float dq_l = prior_term(b1, inv_ac, pr.de) - prior_term(b0, inv_ac, pr.de);
                const int nj = min(32, p - j0);
                uint32_t accm = 0u;
                const float4* xr = X + (size_t)j0 * K4 * 32;
                float4 xn[PF > 0 ? PF : 1];  // the next update's first columns, in flight over this one's reduction
#pragma unroll
                for (int k = 0; k < PF; ++k) xn[k] = __ldg(xr + 32 * k);
                for (int jj = 0; jj < nj; ++jj, xr += K4 * 32) {
                    const float delta = __shfl_sync(0xffffffffu, delta_l, jj);
                    const uint64_t dd = pack2(delta, delta);
                    float d = 0.0f, prod = 1.0f;
#pragma unroll
                    for (int k4 = 0; k4 < K4; ++k4) {
                        const float4 x = k4 < PF ? xn[k4 < PF ? k4 : 0] : __ldg(xr + 32 * k4);
                        const uint64_t x2[2] = {pack2(x.x, x.y), pack2(x.z, x.w)};
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint64_t e0p = eta[2 * k4 + h];
                            const float2 e0 = unpack2(e0p), e1 = unpack2(fma2(x2[h], dd, e0p));
                            const float2 df = unpack2(fma2(pack2(fmaxf(e0.x, 0.0f), fmaxf(e0.y, 0.0f)), negone,
                                                           pack2(fmaxf(e1.x, 0.0f), fmaxf(e1.y, 0.0f))));
                            d += df.x;
                            prod = fmaf(prod, ex2_approx(-fabsf(e1.x)), prod);
                            d += df.y;
                            prod = fmaf(prod, ex2_approx(-fabsf(e1.y)), prod);
                        }
                    }
                    if (PF > 0 && jj + 1 < nj) {
#pragma unroll
                        for (int k = 0; k < PF; ++k) xn[k] = __ldg(xr + K4 * 32 + 32 * k);
                    }
                    const float lq1 = lg2_approx(prod);
                    const float dsp = warp_sum(d + (lq1 - lq));
                    // every lane forms its own update's test with this update's sum; lane jj's counts
                    const float dl = fmaf(delta_l, v_l, -0.69314718f * dsp);
                    const uint32_t bal = __ballot_sync(0xffffffffu, lu_l < fmaf(coef, dq_l, dl));
                    if ((bal >> jj) & 1u) {
#pragma unroll
                        for (int k4 = 0; k4 < K4; ++k4) {
                            const float4 x = __ldg(xr + 32 * k4);
                            eta[2 * k4] = fma2(pack2(x.x, x.y), dd, eta[2 * k4]);
                            eta[2 * k4 + 1] = fma2(pack2(x.z, x.w), dd, eta[2 * k4 + 1]);
                        }
                        lq = lq1;
                        accm |= 1u << jj;
                    }
                }
                if ((accm >> lane) & 1u) bg[jl] = b1;
                nacc += __popc(accm);
                __syncwarp();
            }
        }
        // the MH state at the end of the step, in the units the move kernels keep it:
        // l = beta . v - ln 2 (sum_i max(eta2_i, 0) + sum of the lanes' log products), and the
        // log-prior term sum
        if (a.llq) {
            float mx = 0.0f, yd = 0.0f;
            FSum lt;
#pragma unroll
            for (int k = 0; k < KC / 2; ++k) {
                const float2 e = unpack2(eta[k]);
                mx += fmaxf(e.x, 0.0f);
                mx += fmaxf(e.y, 0.0f);
            }
            for (int j = lane; j < p; j += 32) {
                const float b = bg[j];
                yd = fmaf(b, a.vy[j], yd);
                lt.add(prior_term(b, inv_ac, pr.de));
            }
            const float sp2 = warp_sum(mx + lq);
            yd = warp_sum(yd);
            lt = warp_sum(lt);
            if (lane == 0) {
                a.llq[i] = make_float2((yd - 0.69314718f * sp2) * a.inv_sp_scale, 0.0f);
                a.lpq[i] = make_float2(lt.s, lt.c);
            }
        }
    }
    if (!a.acc_count) return;
    __shared__ int blk[SITE_WARPS];
    if (lane == 0) blk[w] = nacc;
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int k = 0; k < SITE_WARPS; ++k) s += blk[k];
        if (s) atomicAdd(a.acc_count, (unsigned long long)s);
    }
}

// XS[j][k / 4][lane][k % 4] = x_ij log2(e) of individual i = lane + 32 k (0 for i >= n), from
// X^T log2(e) [p][n]: each lane's individuals in the order and width it loads them.
__global__ void k_store_xsite(const float* __restrict__ XT2, int64_t n, int64_t p, int64_t KC, float* __restrict__ XS)
{
    const int64_t per = 32 * KC, total = p * per;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = e / per, o = e - j * per;
        const int64_t k4 = o >> 7, lane = (o >> 2) & 31, q = o & 3;
        const int64_t i = lane + 32 * (4 * k4 + q);
        XS[e] = i < n ? XT2[j * n + i] : 0.0f;
    }
}

// --------------------------------------------------------- eta2 in shared memory
// Per-lane: sum over the lane's individuals r = lane + 32k of max(eta2', 0) - max(eta2, 0)
// (dm) and log2 of the product of (1 + 2^-|eta2'|) (returned), eta2' = eta2 + x2 delta.
__device__ __forceinline__ float site_trial(const float* __restrict__ eta, const float* __restrict__ xr, int n,
                                            int lane, float delta, float& dm)
{
    float lq = 0.0f, d = 0.0f;
    for (int k0 = 0; 32 * k0 < n; k0 += SITE_CHUNK) {
        float prod = 1.0f;
        const int r1 = min(n, 32 * (k0 + SITE_CHUNK));
        for (int r = lane + 32 * k0; r < r1; r += 32) {
            const float e0 = eta[r];
            const float e1 = fmaf(xr[r], delta, e0);
            d += fmaxf(e1, 0.0f) - fmaxf(e0, 0.0f);
            prod = fmaf(prod, ex2_approx(-fabsf(e1)), prod);
        }
        lq += lg2_approx(prod);
    }
    dm = d;
    return lq;
}

__global__ void k_move_site(SiteArgs a, int64_t N, int p, int n, PriorArgs pr, const float4* __restrict__ stepk, int t,
                            uint32_t m0, int M, const uint64_t* __restrict__ seedp)
{
    extern __shared__ float site_sm[];
    __shared__ int blk;
    const int wpc = blockDim.x >> 5;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) blk = 0;
    __syncthreads();
    const float4 sk = stepk[t];
    float* eta = site_sm + (size_t)w * (size_t)(n + p);
    float* brow = eta + n;
    const int64_t i = (int64_t)blockIdx.x * wpc + w;
    if (i < N) {
        const uint64_t seed = *seedp;
        const float coef = sk.y, inv_ac = sk.w;
        float* bg = a.beta + i * p;
        for (int j = lane; j < p; j += 32) brow[j] = bg[j];
        for (int r = lane; r < n; r += 32) eta[r] = 0.0f;
        __syncwarp();
        for (int j = 0; j < p; ++j) {  // eta2 = X2 beta, marker by marker (coalesced rows of X^T)
            const float bj = brow[j];
            const float* xr = a.XT2 + (size_t)j * n;
            for (int r = lane; r < n; r += 32) eta[r] = fmaf(xr[r], bj, eta[r]);
        }
        float dm;
        float lq = site_trial(eta, a.XT2, n, lane, 0.0f, dm);  // delta = 0: the current state
        int nacc = 0;
        for (int mm = 0; mm < M; ++mm) {
            const uint32_t m = m0 + (uint32_t)mm;
            for (int j = 0; j < p; ++j) {
                const uint4 u = philox4x32_10(make_uint4((uint32_t)j, (uint32_t)i, (uint32_t)t, (TAG_SITE << 16) | m),
                                              seed_key(seed));
                float sn, cs;
                sincospif(2.0f * u01_open_cvt_f(u.y), &sn, &cs);
                const float delta = a.sd * (sqrtf(-2.0f * logf(u01_open_cvt_f(u.x))) * cs);
                const float* xr = a.XT2 + (size_t)j * n;
                const float lq1 = site_trial(eta, xr, n, lane, delta, dm);
                const float dsp = warp_sum(dm + (lq1 - lq));
                const float b0 = brow[j], b1 = b0 + delta;
                const float dlp = coef * (prior_term(b1, inv_ac, pr.de) - prior_term(b0, inv_ac, pr.de));
                const float dl = fmaf(delta, a.vy[j], -0.69314718f * dsp);
                int acc = logf(u01_open_cvt_f(u.z)) < dl + dlp;
                acc = __shfl_sync(0xffffffffu, acc, 0);
                if (acc) {
                    for (int r = lane; r < n; r += 32) eta[r] = fmaf(xr[r], delta, eta[r]);
                    lq = lq1;
                    if (lane == 0) brow[j] = b1;
                    ++nacc;
                }
                __syncwarp();
            }
        }
        for (int j = lane; j < p; j += 32) bg[j] = brow[j];
        if (lane == 0 && nacc) atomicAdd(&blk, nacc);
        // the MH state at the end of the step, in the units the move kernels keep it:
        // l = beta . v - ln 2 (sum_i max(eta2_i, 0) + sum of the lanes' log products), and the
        // log-prior term sum
        if (a.llq) {
            float mx = 0.0f, yd = 0.0f;
            FSum lt;
            for (int r = lane; r < n; r += 32) mx += fmaxf(eta[r], 0.0f);
            for (int j = lane; j < p; j += 32) {
                yd = fmaf(brow[j], a.vy[j], yd);
                lt.add(prior_term(brow[j], inv_ac, pr.de));
            }
            const float sp2 = warp_sum(mx + lq);
            yd = warp_sum(yd);
            lt = warp_sum(lt);
            if (lane == 0) {
                a.llq[i] = make_float2((yd - 0.69314718f * sp2) * a.inv_sp_scale, 0.0f);
                a.lpq[i] = make_float2(lt.s, lt.c);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && blk && a.acc_count) atomicAdd(a.acc_count, (unsigned long long)blk);
}

}  // namespace

// Individuals per lane of the register kernel (a multiple of 4), or 0 when n is too large for it.
static int site_kc(int64_t n)
{
    const int64_t k = (n + 31) / 32;
    return k <= SITE_CHUNK ? (int)((k + 3) / 4 * 4) : 0;
}

int64_t site_xs_floats(int64_t n, int64_t p) { return p * 32 * (int64_t)site_kc(n); }

cudaError_t launch_store_xsite(const float* XT2, int64_t n, int64_t p, float* XS, cudaStream_t st)
{
    const int64_t total = site_xs_floats(n, p);
    const unsigned blocks = (unsigned)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
    k_store_xsite<<<blocks, 256, 0, st>>>(XT2, n, p, site_kc(n), XS);
    return cudaGetLastError();
}

int site_warps_per_block(int64_t n, int p)
{
    const int64_t per = (n + p) * (int64_t)sizeof(float);
    int64_t w = (int64_t)SITE_SMEM_MAX / (per > 0 ? per : 1);
    if (w > 8) w = 8;
    return (int)w;
}

cudaError_t site_init_attributes()
{
    return cudaFuncSetAttribute(k_move_site, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SITE_SMEM_MAX);
}

template <int KC>
static cudaError_t launch_site_reg(int kc, const SiteArgs& a, int64_t N, int p, int64_t n, PriorArgs pr,
                                   const float4* stepk, int t, uint32_t m0, int M, const uint64_t* seed, cudaStream_t st)
{
    if constexpr (KC < SITE_CHUNK) {
        if (kc != KC) return launch_site_reg<KC + 4>(kc, a, N, p, n, pr, stepk, t, m0, M, seed, st);
    }
    k_move_site_reg<KC><<<(unsigned)((N + SITE_WARPS - 1) / SITE_WARPS), 32 * SITE_WARPS, 0, st>>>(a, N, p, (int)n, pr,
                                                                                                  stepk, t, m0, M, seed);
    return cudaGetLastError();
}

cudaError_t launch_move_site(const SiteArgs& a, int64_t N, int p, int64_t n, PriorArgs pr, const float4* stepk, int t,
                             uint32_t m0, int M, const uint64_t* seed, cudaStream_t st)
{
    if (M <= 0) return cudaSuccess;
    const int kc = site_kc(n);
    if (kc > 0 && a.XS) return launch_site_reg<4>(kc, a, N, p, n, pr, stepk, t, m0, M, seed, st);
    const int wpc = site_warps_per_block(n, p);
    if (wpc < 1) return cudaErrorInvalidValue;
    const size_t smem = (size_t)wpc * (size_t)(n + p) * sizeof(float);
    k_move_site<<<(unsigned)((N + wpc - 1) / wpc), 32 * wpc, smem, st>>>(a, N, p, (int)n, pr, stepk, t, m0, M, seed);
    return cudaGetLastError();
}

}  // namespace spa
