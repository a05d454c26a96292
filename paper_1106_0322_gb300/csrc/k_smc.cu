// k_smc.cu -- the per-step kernels of the SMC sampler over the prior scale (Section 4).
//
// Particle state: beta [N][p] FP32 (particle-major); the log-likelihood and the log-prior
// term sum as compensated FP32 pairs (llq, lpq; the log-prior without the constant
// -p log(2c), which cancels in every ratio taken at one scale; the change of scale is
// handled by the incremental weight in FP64); normalised log-weights and weights
// (WeightArrays).
//
// Precision plan for GB300: the CUDA-core FP64 rate is a small fraction of FP32 and an
// FP64 warp instruction costs a full warp's issue time even with one lane active. So sums
// over markers run in FP32 with compensated (TwoSum) accumulation, the Metropolis-Hastings
// ratios are formed in FP32 from compensated pairs, and FP64 appears only in the weights
// (incremental weight, log-sum-exp, ESS, log-evidence; one thread per particle) and in the
// resampling cumulative sum, whose association order is specified.
#include <cfloat>
#include <cmath>

#include "spa_device.cuh"
#include "spa_internal.h"

namespace spa {

namespace {

constexpr int BLOCK = 256;
constexpr int WARPS = BLOCK / 32;

__device__ __forceinline__ int64_t warp_global_id()
{
    return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
}

// The log prior's coefficient of its term sum (prior_term, spa_device.cuh), FP64.
__device__ __forceinline__ double prior_coef(PriorArgs pr, double c) { return pr.de ? -1.0 / c : -((double)pr.a + 1.0); }

// MALA's drift is (h^2/2) D_j times the slope of the log posterior: g = grad l plus the prior's part,
// -(a+1) sgn(b)/(a c + |b|) or, for the double exponential, -sgn(b)/c. The quotient is the product with
// the approximate reciprocal (rcp.approx.ftz.f32, 1 ulp): the drift may be any fixed function of the
// state. Every operation is rounded as written, so that the slope does not depend on how the compiler
// joins it to the code around, which differs between the kernels. The forward density rounds the prior's
// part before the sum, the reverse density (slope_reverse) adds it in one rounding: the two are within
// 2^-24 of the prior's part of each other, which enters log alpha as the FP32 roundings of the two
// residual sums do. One rounding in both would be the cleaner rule, but gives every sweep whose a + 1 is
// not a power of two other bits.
__device__ __forceinline__ float slope_sign(float b, float v) { return b > 0.0f ? -v : (b < 0.0f ? v : 0.0f); }
__device__ __forceinline__ float slope_forward(float g, float b, float a1, float ac, float inv_c, int de)
{
    return __fadd_rn(g, de ? __fmul_rn(slope_sign(b, 1.0f), inv_c)
                           : __fmul_rn(slope_sign(b, a1), rcp_approx(__fadd_rn(ac, fabsf(b)))));
}
__device__ __forceinline__ float slope_reverse(float g, float b, float a1, float ac, float inv_c, int de)
{
    return de ? __fmaf_rn(slope_sign(b, 1.0f), inv_c, g)
              : __fmaf_rn(slope_sign(b, a1), rcp_approx(__fadd_rn(ac, fabsf(b))), g);
}

// ------------------------------------------------------------------- init (t = 0)
__global__ void k_init_prior(float* __restrict__ beta, int64_t N, int p, PriorArgs pr, const double* __restrict__ sched,
                             int t0, const uint64_t* __restrict__ seedp)
{
    const uint64_t seed = *seedp;
    const float c = (float)sched[t0];
    const int64_t total = N * (int64_t)p;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / p;
        const int j = (int)(e - i * p);
        beta[e] = prior_draw(seed, (uint32_t)i, (uint32_t)j, pr.a, c, pr.de != 0);
    }
}

// Split-BF16 GEMM row of one coordinate: bt = b log2(e)/s_j. Returns m_j bt for the offset.
__device__ __forceinline__ float pack_coord(__nv_bfloat16* __restrict__ Arow, int Kp, int j, float b,
                                            const float* __restrict__ l2e_over_s, const float* __restrict__ mean_f)
{
    const float bt = b * l2e_over_s[j];
    __nv_bfloat16 hi, lo;
    split_bf16(bt, hi, lo);
    Arow[j] = hi;
    Arow[Kp + j] = lo;
    return mean_f[j] * bt;
}

__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// Four consecutive coordinates j..j+3 (j a multiple of 4): two 8-byte stores per half.
__device__ __forceinline__ float pack_coord4(__nv_bfloat16* __restrict__ Arow, int Kp, int j, float4 b, float4 l2e,
                                             float4 mf)
{
    const float bt[4] = {b.x * l2e.x, b.y * l2e.y, b.z * l2e.z, b.w * l2e.w};
    // split_bf16, two at a time: a pair's BF16 values as FP32 are the word's halves shifted up
    uint32_t hi[2], lo[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        hi[k] = bf16x2_bits(bt[2 * k], bt[2 * k + 1]);
        lo[k] = bf16x2_bits(bt[2 * k] - __uint_as_float(hi[k] << 16), bt[2 * k + 1] - __uint_as_float(hi[k] & 0xFFFF0000u));
    }
    *reinterpret_cast<uint2*>(Arow + j) = make_uint2(hi[0], hi[1]);
    *reinterpret_cast<uint2*>(Arow + Kp + j) = make_uint2(lo[0], lo[1]);
    return mf.x * bt[0] + mf.y * bt[1] + mf.z * bt[2] + mf.w * bt[3];
}

__device__ __forceinline__ void pack_offset(__nv_bfloat16* __restrict__ Arow, int Kp, int p, float off)
{
    __nv_bfloat16 hi, lo;
    split_bf16(-off, hi, lo);
    Arow[p] = hi;
    Arow[Kp + p] = lo;
}

// ------------------------------------------------------------ Metropolis-Hastings test
// The log-likelihood of particle i is sp_scale * (sum of the GEMM partials + ydq[i]), kept
// as a compensated FP32 pair (s, c) in partial units; the log-prior is coef(c_t) * (sum of
// log1p(|b|/(a c_t)) or |b|), kept as the pair of that sum. At one scale both differences
// of the MH ratio are between nearby values, so they are formed in FP32 from the pairs:
// s' - s is exact when the two are within a factor of two, and the c parts carry the rest.

// The block's proposals' softplus partials, gathered for the MH tests (one warp per particle,
// WARPS particles per block): thread t adds the chunks q = t / WARPS, t / WARPS + 32, ... of
// particle WARPS blockIdx.x + t % WARPS, so the WARPS threads of a group read one 32-byte
// sector per chunk, where a warp per particle touches one sector per lane. Slice s of a
// particle is exactly the compensated partial sum that lane s of a warp-per-particle loop
// over q = s, s + 32, ... forms, so the warp's tree over the slices gives the same bits.
struct PartSlices {
    float2 v[32][WARPS];
};
__device__ __forceinline__ void gather_partials(const MhState& s, int64_t N, PartSlices& sh)
{
    const int k = threadIdx.x % WARPS, slice = threadIdx.x / WARPS;
    const int64_t i = (int64_t)blockIdx.x * WARPS + k;
    FSum L;
    if (i < N)
        for (int q = slice; q < s.n_parts; q += 32) L.add(s.partial[(int64_t)q * s.ld_part + i]);
    sh.v[slice][k] = make_float2(L.s, L.c);
}

// The same for the residuals' chunk sums of a gradient evaluation, into one sum a particle: the 32
// slices in order, by the first threads of the block. Two barriers after the caller's gather.
struct RsumSlices {
    float2 v[32][WARPS];
    float sum[WARPS];
};
__device__ __forceinline__ void gather_rsum(const MhState& s, const GradParts& gp, int64_t N, RsumSlices& sh)
{
    const int k = threadIdx.x % WARPS, slice = threadIdx.x / WARPS;
    const int64_t i = (int64_t)blockIdx.x * WARPS + k;
    FSum r;
    if (i < N)
        for (int q = slice; q < s.n_parts; q += 32) r.add(gp.rsum[(int64_t)q * s.ld_part + i]);
    sh.v[slice][k] = make_float2(r.s, r.c);
}
__device__ __forceinline__ void sum_rsum(RsumSlices& sh)
{
    if (threadIdx.x < WARPS) {
        FSum r;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const float2 v = sh.v[k][threadIdx.x];
            r.add(v.x);
            r.c += v.y;
        }
        sh.sum[threadIdx.x] = (float)r.value();
    }
    __syncthreads();
}

// grad l of four coordinates of particle i, `stride` apart from j0 (those beyond p are 0), as
// k_grad_finish forms it (rs: the sum of its residuals). The products are rounded by themselves:
// what is added to them does not join in. Two K-split partials of each at a time are in flight.
template <int STRIDE>
__device__ __forceinline__ void finish_gradient4(const MoveArgs& a, int64_t i, int p, int j0, float rs, float (&out)[4])
{
    const GradParts& gp = a.gp;
    const int64_t step = a.mh.ld_part * p;
    const float* c = gp.gpart + i * p + j0;
    FSum g[4];
    for (int q = 0; q < gp.ksplit; q += 2, c += 2 * step) {
        float x[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const bool in = q + u < gp.ksplit;
            if (STRIDE == 1) {
                const float4 v = in ? ld4(c + u * step) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int k = 0; k < 4; ++k) x[u][k] = comp(v, k);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) x[u][k] = in && j0 + STRIDE * k < p ? c[u * step + STRIDE * k] : 0.0f;
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int k = 0; k < 4; ++k) g[k].add(x[u][k]);
    }
    float m[4], d[4];
    if (STRIDE == 1) {
        const float4 m4 = ldg4(a.mean_f + j0), d4 = ldg4(gp.inv_sd + j0);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            m[k] = comp(m4, k);
            d[k] = comp(d4, k);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool in = j0 + STRIDE * k < p;
            m[k] = in ? a.mean_f[j0 + STRIDE * k] : 0.0f;
            d[k] = in ? gp.inv_sd[j0 + STRIDE * k] : 0.0f;
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = __fmul_rn(fmaf(-m[k], rs, (float)g[k].value()), d[k]);
}

// The proposal's log-likelihood pair: the warp sums the slices, then adds y . eta.
__device__ __forceinline__ FSum proposal_loglik(const MhState& s, const PartSlices& sh, int64_t i, int lane)
{
    FSum L;
    const float2 v = sh.v[lane][threadIdx.x >> 5];
    L.s = v.x;
    L.c = v.y;
    L = warp_sum(L);
    const float2 yd = s.ydq[i];
    L.add(yd.x);
    L.add(yd.y);
    return L;
}

// ---- the block's sums at once
// A block's warps each hold one particle's 32 lane partials of several sums. Reduced by the
// warp that holds them, a compensated sum is 5 shuffled additions, made by 8 warps for 8
// sums; here one warp reduces all 8: lane 4 k + s first adds the partials s, s + 4, ... of
// particle k in the order in which lane s of the warp tree would, then two shuffles end the
// tree. The lanes 4 k have the results: the bits that lane 0 of warp_sum has.
constexpr int LANES_LD = WARPS + 1;  // (an odd stride keeps a warp's column off one bank)
struct LaneSums {
    float2 v[32][LANES_LD];
};
template <int LD>
__device__ __forceinline__ FSum block_fsum(const float2 (&v)[32][LD])
{
    const int lane = threadIdx.x & 31, k = lane >> 2, s = lane & 3;
    FSum a[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 x = v[s + 4 * j][k], y = v[s + 4 * j + 16][k];
        FSum o;
        a[j].s = x.x;
        a[j].c = x.y;
        o.s = y.x;
        o.c = y.y;
        a[j].add(o);
    }
    a[0].add(a[2]);
    a[1].add(a[3]);
    a[0].add(a[1]);
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
        FSum w;
        w.s = __shfl_xor_sync(0xffffffffu, a[0].s, o);
        w.c = __shfl_xor_sync(0xffffffffu, a[0].c, o);
        a[0].add(w);
    }
    return a[0];
}
// The same of two plain sums.
__device__ __forceinline__ float2 block_sum2(const float2 (&v)[32][LANES_LD])
{
    const int lane = threadIdx.x & 31, k = lane >> 2, s = lane & 3;
    float2 a[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 x = v[s + 4 * j][k], y = v[s + 4 * j + 16][k];
        a[j] = make_float2(x.x + y.x, x.y + y.y);
    }
    float2 r = make_float2((a[0].x + a[2].x) + (a[1].x + a[3].x), (a[0].y + a[2].y) + (a[1].y + a[3].y));
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
        r.x += __shfl_xor_sync(0xffffffffu, r.x, o);
        r.y += __shfl_xor_sync(0xffffffffu, r.y, o);
    }
    return r;
}

// log U of the MH test of move m for the block's particles (one warp per particle, so
// blockDim.x / 32 of them), by the kernel that proposes move m: lanes 0.. of warp 0 draw
// them side by side instead of lane 0 of every warp one at a time in the test.
__device__ __forceinline__ void draw_accept_logu(const MhState& s, int64_t N, int t, uint32_t m, uint64_t seed)
{
    const int lane = threadIdx.x & 31;
    if (!s.lu || threadIdx.x >= 32 || lane >= (int)(blockDim.x >> 5)) return;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + lane;
    if (i >= N) return;
    const uint4 u = philox4x32_10(make_uint4(0u, (uint32_t)i, (uint32_t)t, (TAG_ACCEPT << 16) | m), seed_key(seed));
    s.lu[(int64_t)(m & 1u) * s.ld_lu + i] = logf(u01_open_f(u.x));
}

// MH test of particle i's pending proposal, by one lane: L is the proposal's log-likelihood, `extra`
// the MALA q-correction. It decides with the accept uniform of move m_prev (drawn by the kernel that
// proposed it) and, on acceptance, moves the proposal's log-likelihood and log-prior into the
// current state.
__device__ __forceinline__ bool mh_test(const MhState& s, const FSum& L, int64_t i, float coef, float extra, uint32_t m_prev,
                                        uint32_t* err)
{
    const float2 L0 = s.llq[i];
    const float2 Q1 = s.lpt_p[i], Q0 = s.lpq[i];
    // written two launches back, by the kernel that proposed (read from L2)
    const float lu = __ldcg(s.lu + (int64_t)(m_prev & 1u) * s.ld_lu + i);
    const float dL = (L.s - L0.x) + (L.c - L0.y);
    const float dQ = (Q1.x - Q0.x) + (Q1.y - Q0.y);
    // rounded as written (no contraction), so that the decision does not depend on
    // how the compiler schedules the surrounding code
    const float log_alpha = __fadd_rn(__fadd_rn(__fmul_rn(s.sp_scale, dL), __fmul_rn(coef, dQ)), extra);
    if (!isfinite(L.s)) atomicOr(err, DERR_NONFINITE);
    const bool accept = lu < log_alpha;
    if (accept) {
        s.llq[i] = make_float2(L.s, L.c);
        s.lpq[i] = Q1;
    }
    return accept;
}
// The tests of all the block's particles, by one warp: lane 4 k decides for particle k, into acc[k].
// MALA: with the lane partials of the reverse moves' residual sums (mala_reverse) in bwd.
template <bool MALA>
__device__ __forceinline__ void mh_decide_block(const MoveArgs& a, const PartSlices& sh, const LaneSums& bwd, int64_t N,
                                                float coef, uint32_t m_prev, int* acc, uint32_t* err)
{
    const MhState& s = a.mh;
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * WARPS + (lane >> 2);
    FSum L = block_fsum(sh.v), B;
    if (MALA) B = block_fsum(bwd.v);
    if (lane & 3) return;
    int accept = 0;
    if (i < N) {
        const float2 yd = s.ydq[i];
        L.add(yd.x);
        L.add(yd.y);
        float extra = 0.0f;
        if (MALA) {
            const float2 fw = a.fwd[i];
            const float h = *a.h;
            extra = -((B.s - fw.x) + (B.c - fw.y)) / (2.0f * h * h);
        }
        accept = mh_test(s, L, i, coef, extra, m_prev, err);
    }
    acc[lane >> 2] = accept;
}


// A step's first move after a resampling: the gather left particle i's row in beta_p (and its
// gradient in gl_p), so the move reads it there and writes it back as the state, as it does with
// an accepted proposal; here its MH state and the uniform weights follow. Returns whether the
// step resampled.
__device__ __forceinline__ bool take_resampled(const MoveArgs& a, int64_t i, int lane)
{
    if (!a.rs.flag || *a.rs.flag == 0) return false;
    if (lane == 0) {
        a.mh.llq[i] = a.rs.llq_tmp[i];
        a.mh.lpq[i] = a.rs.lpq_tmp[i];
        a.rs.w.logw[i] = a.rs.lw;
        a.rs.w.W[i] = a.rs.wi;
        a.rs.w.Wf[i] = (float)a.rs.wi;
        a.rs.w.wfix[i] = a.rs.wf;
    }
    return true;
}

// ------------------------------------------------------------ RW move kernel
// One warp per particle. With DECIDE, the warp first runs the MH test of the proposal
// left by the previous move (its log-likelihood partials are complete, the GEMM having run
// in between) and, on acceptance, writes that proposal back as the particle's state while
// reading it. Then it draws the next random-walk proposal beta' = beta + sigma xi from the
// (possibly just accepted) state: beta' to beta_p, the compensated log-prior term sum to
// lpt_p, y . eta' = beta' . v to ydq and (A != NULL) the split-BF16 GEMM row
// [hi(bt) | lo(bt)] with bt_j = beta'_j log2(e)/s_j and the offset o = -sum_j m_j bt_j in
// column p. noise = 0 packs beta unchanged (log-likelihood entry points, t = 0).
// Lane l handles the 4-coordinate groups g = l, l+32, ... (one Philox block of normals).

// One 4-coordinate group of a random-walk proposal (VEC: p % 4 == 0, float4 access).
// `live` masks the memory traffic of a lane whose group lies beyond p.
template <bool VEC>
__device__ __forceinline__ void rw_group(const MoveArgs& a, int p, int g, bool live, bool acc, int noise, float4 z,
                                         float inv_ac, int de, const float* src, float* dst, float* cur,
                                         __nv_bfloat16* Arow, FSum& lt, float& yd, float& off)
{
    const int j0 = 4 * g;
    if (VEC) {
        if (!live) return;
        const float4 b0 = ld4(src + j0);
        if (acc) st4(cur + j0, b0);
        const float4 sg = ld4(a.sigma + j0);
        const float4 b = noise ? make_float4(fmaf(sg.x, z.x, b0.x), fmaf(sg.y, z.y, b0.y), fmaf(sg.z, z.z, b0.z),
                                             fmaf(sg.w, z.w, b0.w))
                               : b0;
        st4(dst + j0, b);
        const float4 v = ld4(a.vy + j0);
        if (de) {
#pragma unroll
            for (int k = 0; k < 4; ++k) lt.add(fabsf(comp(b, k)));
        } else {
            lt.add(prior_terms4(b, inv_ac));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) yd = fmaf(comp(b, k), comp(v, k), yd);
        if (Arow) off += pack_coord4(Arow, a.Kp, j0, b, ld4(a.l2e_over_s + j0), ld4(a.mean_f + j0));
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int j = j0 + k;
            if (live && j < p) {
                const float b0 = src[j];
                if (acc) cur[j] = b0;
                const float b = noise ? fmaf(a.sigma[j], comp(z, k), b0) : b0;
                dst[j] = b;
                lt.add(prior_term(b, inv_ac, de));
                yd = fmaf(b, a.vy[j], yd);
                if (Arow) off += pack_coord(Arow, a.Kp, j, b, a.l2e_over_s, a.mean_f);
            }
        }
    }
}

// The scale constants of every step of a schedule, formed once per sweep, so that the move
// kernels read their step's float4 instead of redoing FP64 arithmetic in every block:
// x = a c_t (FP64 product), y = the log-prior coefficient (-(a+1), or -1/c_t for the double
// exponential), z = 1/c_t, w = 1/(a c_t) (FP64 quotient).
__global__ void k_step_constants(PriorArgs pr, const double* __restrict__ sched, int T, int p, float4* __restrict__ out,
                                 ReweightK* __restrict__ rk)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const double c = sched[t];
    float4 k;
    k.x = (float)((double)pr.a * c);
    k.z = 1.0f / (float)c;
    k.y = pr.de ? -k.z : -(pr.a + 1.0f);
    k.w = (float)(1.0 / ((double)pr.a * c));
    out[t] = k;
    if (rk) {
        ReweightK r{};
        if (t > 0) {
            const double cp = sched[t - 1];
            r.k1 = (float)(cp - c);
            r.kc = (float)c;
            r.kac = (float)((double)pr.a * cp);
            r.inv_ac = (float)(1.0 / ((double)pr.a * c));
            r.lbase = -(double)p * log(c / cp);
            r.dinv = 1.0 / c - 1.0 / cp;
        }
        rk[t] = r;
    }
}

// Accepted proposals of a block, from its particles' decisions (one warp, after the barrier that
// follows them): one global atomic.
__device__ __forceinline__ void count_accepts(unsigned long long* acc_count, const int* accw)
{
    const int lane = threadIdx.x & 31;
    const int n = __popc(__ballot_sync(0xffffffffu, lane < WARPS && accw[lane % WARPS] != 0));
    if (lane == 0 && acc_count && n) atomicAdd(acc_count, (unsigned long long)n);
}

template <bool DECIDE, bool VEC>
__global__ void __launch_bounds__(BLOCK, 5) k_move_rw(MoveArgs a, int64_t N, int p, PriorArgs pr,
                                                  const float4* __restrict__ stepk, int t, uint32_t m, uint32_t m_prev,
                                                  const uint64_t* __restrict__ seedp, int noise, uint32_t* err)
{
    __shared__ int accw[BLOCK / 32];
    __shared__ PartSlices parts;
    __shared__ LaneSums lts, yos;
    const int w = threadIdx.x >> 5;
    const int64_t i = warp_global_id();
    const int lane = threadIdx.x & 31, groups = (p + 3) >> 2;
    // The first group's normals depend on nothing that the previous kernel writes: drawn by blocks that
    // are resident before it ends. RW step of 10 moves at n = 2000, p = 200, N = 8192: 331 -> 328 us;
    // 5 moves at n = 1859, p = 183, N = 5003: 190 -> 187.
    float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    if (noise && i < N && lane < groups) z = normals4(*seedp, (uint32_t)lane, (uint32_t)i, (uint32_t)t, m);
    grid_dependency_wait();  // the previous kernel (the likelihood GEMM) has finished
    grid_launch_dependents();
    if (DECIDE) {
        gather_partials(a.mh, N, parts);
        __syncthreads();
    }
    const float4 sk = stepk[t];
    if (DECIDE) {
        if (w == 0) mh_decide_block<false>(a, parts, lts, N, sk.y, m_prev, accw, err);
        __syncthreads();
    }
    FSum lt;
    float yd = 0.0f, off = 0.0f;
    bool acc = false;  // the state is the row in beta_p: an accepted proposal, or a resampled particle
    if (i < N) {
        const uint64_t seed = (noise || DECIDE) ? *seedp : 0ull;
        if (DECIDE)
            acc = accw[w] != 0;
        else
            acc = take_resampled(a, i, lane);
        const float* src = (acc ? a.beta_p : a.beta) + i * p;
        float* dst = a.beta_p + i * p;
        float* cur = a.beta + i * p;
        __nv_bfloat16* Arow = a.A ? a.A + i * (int64_t)a.ldA : nullptr;
        for (int g = lane; g < groups; g += 32) {
            if (noise && g >= 32) z = normals4(seed, (uint32_t)g, (uint32_t)i, (uint32_t)t, m);
            rw_group<VEC>(a, p, g, true, acc, noise, z, sk.w, pr.de, src, dst, cur, Arow, lt, yd, off);
        }
    }
    lts.v[lane][w] = make_float2(lt.s, lt.c);
    yos.v[lane][w] = make_float2(yd, off);
    __syncthreads();
    const int64_t ib = (int64_t)blockIdx.x * WARPS + (lane >> 2);
    const bool mine = (lane & 3) == 0 && ib < N;
    if (w == 0) {
        const FSum q = block_fsum(lts.v);
        if (mine) a.lpt_p[ib] = make_float2(q.s, q.c);
    } else if (w == 1) {
        const float2 q = block_sum2(yos.v);
        if (mine) {
            a.ydq[ib] = make_float2(q.x, 0.0f);
            if (a.A) pack_offset(a.A + ib * (int64_t)a.ldA, a.Kp, p, q.y);
        }
    }
    if (noise) draw_accept_logu(a.mh, N, t, m, *seedp);
    if (DECIDE && w == 2) count_accepts(a.mh.acc_count, accw);
}

// ------------------------------------------------------------ MALA move kernel
// The reverse move's residual sum of particle i's pending proposal (lane partial, before the
// warp sum): sum_j (beta_j - beta'_j - (h^2/2) D_j g'_j)^2 / D_j, g' = grad l' + the prior
// gradient at beta'. VEC (p % 4 == 0): lane l takes the 4-coordinate groups l, l + 32, ...
// with float4 loads; else coordinates l, l + 32, ...
template <bool VEC, bool PARTS>
__device__ __forceinline__ FSum mala_reverse(const MoveArgs& a, int64_t i, int p, int lane, float h2, float a1, float ac,
                                             float inv_c, int de, float rs)
{
    FSum bwd;
    const float* b0 = a.beta + i * p;
    const float* b1 = a.beta_p + i * p;
    float* g1 = a.gl_p + i * p;
    if (VEC) {
        for (int j0 = 4 * lane; j0 < p; j0 += 128) {
            const float4 x0 = ld4(b0 + j0), x1 = ld4(b1 + j0);
            float4 gg;
            if (PARTS) {
                float o[4];
                finish_gradient4<1>(a, i, p, j0, rs, o);
                gg = make_float4(o[0], o[1], o[2], o[3]);
                st4(g1 + j0, gg);
            } else {
                gg = ld4(g1 + j0);
            }
            const float4 Dv = ldg4(a.sigma + j0), iD = ldg4(a.inv_D + j0);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float drift = h2 * comp(Dv, k) * slope_reverse(comp(gg, k), comp(x1, k), a1, ac, inv_c, de);
                const float d = (comp(x0, k) - comp(x1, k)) - drift;
                bwd.add(d * d * comp(iD, k));
            }
        }
    } else if (PARTS) {
        for (int j0 = lane; j0 < p; j0 += 128) {
            float g4[4];
            finish_gradient4<32>(a, i, p, j0, rs, g4);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = j0 + 32 * k;
                if (j >= p) break;
                g1[j] = g4[k];
                const float drift = h2 * a.sigma[j] * slope_reverse(g4[k], b1[j], a1, ac, inv_c, de);
                const float d = (b0[j] - b1[j]) - drift;
                bwd.add(d * d * a.inv_D[j]);
            }
        }
        // k_move_mala reads an accepted row back by fours, from other lanes than stored it here
        __syncwarp();
    } else {
        const float* g = a.gl_p + i * p;
        for (int j = lane; j < p; j += 32) {
            const float drift = h2 * a.sigma[j] * slope_reverse(g[j], b1[j], a1, ac, inv_c, de);
            const float d = (b0[j] - b1[j]) - drift;
            bwd.add(d * d * a.inv_D[j]);
        }
    }
    return bwd;
}

// beta' = beta + (h^2/2) D grad log pi_t(beta) + h D^{1/2} xi with D = diag(D_j) and
// h = lambda p^{-1/6} (written by the column-statistics kernel); grad log pi_t = grad l
// (stored per particle) + the prior gradient -(a+1) sgn(beta)/(a c + |beta|) (double
// exponential: -sgn(beta)/c). The forward density is evaluated at the proposal as
// written (rounded to FP32): fwd = sum_j (beta'_j - beta_j - (h^2/2) D_j g_j)^2 / D_j, so
// log q(beta'|beta) = -fwd/(2h^2) + const, the same formula as the reverse term. With
// DECIDE the warp first forms the reverse term of the pending proposal,
// bwd = sum_j (beta_j - beta'_j - (h^2/2) D_j g'_j)^2 / D_j, and runs its MH test with
// log alpha = l' + lp' - l - lp - (bwd - fwd)/(2h^2); an accepted proposal and its gradient
// are written back as the state while being read. At most 64 registers, so that 4 blocks
// fit an SM (1.68 waves of 8192 particle warps; the test variant would take 74 and 3 blocks).
template <bool DECIDE, bool VEC, bool PARTS>
__global__ void __launch_bounds__(BLOCK, 4) k_move_mala(MoveArgs a, int64_t N, int p, PriorArgs pr,
                                                    const float4* __restrict__ stepk, int t, uint32_t m,
                                                    uint32_t m_prev, const uint64_t* __restrict__ seedp, uint32_t* err)
{
    __shared__ int accw[BLOCK / 32];
    __shared__ PartSlices parts;
    __shared__ RsumSlices rsum;
    __shared__ LaneSums lts, fws, yos;  // (lts: the reverse sums first)
    const int w = threadIdx.x >> 5;
    const int64_t i = warp_global_id();
    const int lane = threadIdx.x & 31, groups = (p + 3) >> 2;
    float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);  // (as in k_move_rw)
    if (VEC && i < N && lane < groups) z4 = normals4(*seedp, (uint32_t)lane, (uint32_t)i, (uint32_t)t, m);
    grid_dependency_wait();  // the previous kernel (the gradient finish, or the step's proposal scales) has finished
    grid_launch_dependents();
    if (DECIDE) {
        gather_partials(a.mh, N, parts);
        if (PARTS) gather_rsum(a.mh, a.gp, N, rsum);
        __syncthreads();
        if (PARTS) sum_rsum(rsum);
    }
    const float4 sk = stepk[t];
    bool acc = false;
    const uint64_t seed = *seedp;
    const float ac = sk.x, a1 = pr.a + 1.0f, inv_c = sk.z;
    const float h = *a.h, h2 = 0.5f * h * h;
    const float* D = a.sigma;
    if (DECIDE) {
        // (each warp by itself: two more barriers here cost as much as the block's way saves)
        int accept = 0;
        if (i < N) {
            const FSum bwd = warp_sum(mala_reverse<VEC, PARTS>(a, i, p, lane, h2, a1, ac, inv_c, pr.de, PARTS ? rsum.sum[w] : 0.0f));
            const FSum L = proposal_loglik(a.mh, parts, i, lane);
            if (lane == 0) {
                const float2 fq = a.fwd[i];
                accept = mh_test(a.mh, L, i, sk.y, -((bwd.s - fq.x) + (bwd.c - fq.y)) / (2.0f * h * h), m_prev, err);
            }
        }
        if (lane == 0) accw[w] = accept;
        acc = __shfl_sync(0xffffffffu, accept, 0) != 0;
    } else if (i < N) {
        acc = take_resampled(a, i, lane);
    }
    FSum lt, fw;
    float yd = 0.0f, off = 0.0f;
    if (i < N) {
        const float* src = (acc ? a.beta_p : a.beta) + i * p;
        const float* gsrc = (acc ? a.gl_p : a.gl) + i * p;
        float* cur = a.beta + i * p;
        float* gcur = a.gl + i * p;
        float* dst = a.beta_p + i * p;
        __nv_bfloat16* Arow = a.A ? a.A + i * (int64_t)a.ldA : nullptr;
        const bool grouped = (p & 3) == 0 && !pr.de;  // the four-coordinate prior term
        if (VEC) {
            // p % 4 == 0: the same per-coordinate arithmetic on float4 groups, the state's and
            // the gradient's rows read and written 16 bytes at a time, the GEMM row 8
            for (int g = lane; g < groups; g += 32) {
                if (g >= 32) z4 = normals4(seed, (uint32_t)g, (uint32_t)i, (uint32_t)t, m);
                const int j0 = 4 * g;
                const float4 x0 = ld4(src + j0), g0 = ld4(gsrc + j0);
                if (acc) {
                    st4(cur + j0, x0);
                    st4(gcur + j0, g0);
                }
                const float4 Dv = ldg4(D + j0), sD = ldg4(a.sqrt_D + j0), iD = ldg4(a.inv_D + j0);
                const float4 v = ldg4(a.vy + j0);
                float bq[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float b0 = comp(x0, k);
                    const float drift = h2 * comp(Dv, k) * slope_forward(comp(g0, k), b0, a1, ac, inv_c, pr.de);
                    const float b = (b0 + drift) + h * comp(sD, k) * comp(z4, k);
                    const float d = (b - b0) - drift;
                    fw.add(d * d * comp(iD, k));
                    bq[k] = b;
                    yd = fmaf(b, comp(v, k), yd);
                }
                const float4 b4 = make_float4(bq[0], bq[1], bq[2], bq[3]);
                st4(dst + j0, b4);
                if (grouped) {
                    lt.add(prior_terms4(b4, sk.w));
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) lt.add(prior_term(bq[k], sk.w, pr.de));
                }
                if (Arow) off += pack_coord4(Arow, a.Kp, j0, b4, ldg4(a.l2e_over_s + j0), ldg4(a.mean_f + j0));
            }
        }
        for (int g = VEC ? groups : lane; g < groups; g += 32) {
            const float4 z4 = normals4(seed, (uint32_t)g, (uint32_t)i, (uint32_t)t, m);
            float bq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = 4 * g + k;
                if (j < p) {
                    const float b0 = src[j];
                    const float g0 = gsrc[j];
                    if (acc) {
                        cur[j] = b0;
                        gcur[j] = g0;
                    }
                    const float drift = h2 * D[j] * slope_forward(g0, b0, a1, ac, inv_c, pr.de);
                    const float b = (b0 + drift) + h * a.sqrt_D[j] * comp(z4, k);
                    dst[j] = b;
                    const float d = (b - b0) - drift;
                    fw.add(d * d * a.inv_D[j]);
                    bq[k] = b;
                    if (!grouped) lt.add(prior_term(b, sk.w, pr.de));
                    yd = fmaf(b, a.vy[j], yd);
                    if (Arow) off += pack_coord(Arow, a.Kp, j, b, a.l2e_over_s, a.mean_f);
                }
            }
            if (grouped) lt.add(prior_terms4(make_float4(bq[0], bq[1], bq[2], bq[3]), sk.w));
        }
    }
    lts.v[lane][w] = make_float2(lt.s, lt.c);
    fws.v[lane][w] = make_float2(fw.s, fw.c);
    yos.v[lane][w] = make_float2(yd, off);
    __syncthreads();
    const int64_t ib = (int64_t)blockIdx.x * WARPS + (lane >> 2);
    const bool mine = (lane & 3) == 0 && ib < N;
    if (w == 0) {
        const FSum q = block_fsum(lts.v);
        if (mine) a.lpt_p[ib] = make_float2(q.s, q.c);
    } else if (w == 1) {
        const float2 q = block_sum2(yos.v);
        if (mine) {
            a.ydq[ib] = make_float2(q.x, 0.0f);
            if (a.A) pack_offset(a.A + ib * (int64_t)a.ldA, a.Kp, p, q.y);
        }
    } else if (w == 2) {
        const FSum q = block_fsum(fws.v);
        if (mine) a.fwd[ib] = make_float2(q.s, q.c);
    }
    draw_accept_logu(a.mh, N, t, m, *seedp);
    if (DECIDE && w == 3) count_accepts(a.mh.acc_count, accw);
}

// ------------------------------------------------------------ last move of a step
// MH test of the pending proposals (RW, or MALA with the reverse term), then accepted
// proposals (and their gradients) are copied into the state rows, so that between steps
// beta and gl hold the particles.
// The block's tests: accw[k] = the decision on its particle k, for all threads on return.
template <bool MALA, bool VEC, bool PARTS>
__device__ __forceinline__ void commit_tests(const MoveArgs& a, const PartSlices& parts, const RsumSlices& rsum, LaneSums& bwds,
                                             int64_t N, int p, PriorArgs pr, float4 sk, uint32_t m_prev, int* accw,
                                             uint32_t* err)
{
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (MALA) {
        const int64_t i = warp_global_id();
        const float ac = sk.x, a1 = pr.a + 1.0f, inv_c = sk.z;
        const float h = *a.h, h2 = 0.5f * h * h;
        FSum bwd;
        if (i < N) bwd = mala_reverse<VEC, PARTS>(a, i, p, lane, h2, a1, ac, inv_c, pr.de, PARTS ? rsum.sum[w] : 0.0f);
        bwds.v[lane][w] = make_float2(bwd.s, bwd.c);
        __syncthreads();
    }
    if (w == 0) mh_decide_block<MALA>(a, parts, bwds, N, sk.y, m_prev, accw, err);
    __syncthreads();
}

template <bool MALA, bool VEC>
__device__ __forceinline__ void commit_row(const MoveArgs& a, int64_t i, int p, int lane)
{
    const float* src = a.beta_p + i * p;
    float* dst = a.beta + i * p;
    if (VEC) {
        for (int j = 4 * lane; j < p; j += 128) st4(dst + j, ld4(src + j));
        if (MALA)
            for (int j = 4 * lane; j < p; j += 128) st4(a.gl + i * p + j, ld4(a.gl_p + i * p + j));
    } else {
        for (int j = lane; j < p; j += 32) dst[j] = src[j];
        if (MALA)
            for (int j = lane; j < p; j += 32) a.gl[i * p + j] = a.gl_p[i * p + j];
    }
}

template <bool MALA, bool VEC, bool PARTS>
__global__ void __launch_bounds__(BLOCK) k_move_commit(MoveArgs a, int64_t N, int p, PriorArgs pr,
                                                      const float4* __restrict__ stepk, int t, uint32_t m_prev,
                                                      const uint64_t* __restrict__ seedp, uint32_t* err)
{
    __shared__ int accw[BLOCK / 32];
    __shared__ PartSlices parts;
    __shared__ RsumSlices rsum;
    __shared__ LaneSums bwds;
    grid_dependency_wait();
    gather_partials(a.mh, N, parts);
    if (PARTS) gather_rsum(a.mh, a.gp, N, rsum);
    __syncthreads();
    if (PARTS) sum_rsum(rsum);
    const float4 sk = stepk[t];
    const int64_t i = warp_global_id();
    const int lane = threadIdx.x & 31;
    commit_tests<MALA, VEC, PARTS>(a, parts, rsum, bwds, N, p, pr, sk, m_prev, accw, err);
    if (accw[threadIdx.x >> 5]) commit_row<MALA, VEC>(a, i, p, lane);
    if (threadIdx.x < 32) count_accepts(a.mh.acc_count, accw);
}

// ------------------------------------------------------------ log-likelihood finish
// The packed particles' log-likelihood as the state: llq (pair), lpq = lpt_p, and in FP64
// l = sp_scale (s + c) to logw (prior-IS weights at t = 0) and/or ll_out.
__global__ void __launch_bounds__(BLOCK) k_finish_loglik(MhState s, int64_t N, double* __restrict__ logw,
                                                        double* __restrict__ ll_out, uint32_t* __restrict__ err)
{
    __shared__ PartSlices parts;
    gather_partials(s, N, parts);
    __syncthreads();
    const int64_t i = warp_global_id();
    const int lane = threadIdx.x & 31;
    if (i >= N) return;
    const FSum L = proposal_loglik(s, parts, i, lane);
    if (lane != 0) return;
    if (!isfinite(L.s)) atomicOr(err, DERR_NONFINITE);
    s.llq[i] = make_float2(L.s, L.c);
    s.lpq[i] = s.lpt_p[i];
    const double l = s.sp_scale_d * ((double)L.s + (double)L.c);
    if (logw) logw[i] = l;
    if (ll_out) ll_out[i] = l;
}

// ------------------------------------------------------------------ reweighting
// log w_i = sum_j log p(beta_ij | c_t) - log p(beta_ij | c_{t-1}) in the form without
// cancellation: -log(c_t/c_{t-1}) - (a+1) log1p(x (c_{t-1} - c_t) / (c_t (a c_{t-1} + x))),
// x = |beta_ij| (double exponential: -log(c_t/c_{t-1}) - x (1/c_t - 1/c_{t-1})).
// A block handles 8 particles: its warps form the FP32 row sums, then warp 0 finishes them in FP64. The step's constants come from the per-sweep table.
constexpr int RW_PER_BLOCK = 8;
constexpr int RW_THREADS = 32 * RW_PER_BLOCK;

// The row sums of particle i (row b): the incremental weight's and the log-prior's at c_t.
__device__ __forceinline__ void reweight_row(const float* b, int p, PriorArgs pr, const ReweightK& rk, int lane, FSum& sdiff,
                                             FSum& snew)
{
    const float k1 = rk.k1, kc = rk.kc, kac = rk.kac, inv_ac = rk.inv_ac;
    const bool grouped = (p & 3) == 0 && !pr.de;  // the moves' four-coordinate prior term
    for (int j = lane; j < p; j += 32) {
        const float x = fabsf(b[j]);
        sdiff.add(pr.de ? x : log1pf(x * k1 / (kc * (kac + x))));
        if (!grouped) snew.add(prior_term(x, inv_ac, pr.de));
    }
    if (grouped)
        for (int g = lane; 4 * g < p; g += 32) snew.add(prior_terms4(ld4(b + 4 * g), inv_ac));
}

// The block's particles' log-weights from the lane partials of their row sums (one warp; lane 4 k
// finishes particle k in FP64).
__device__ __forceinline__ void reweight_block(const LaneSums& diffs, const LaneSums& news, int64_t N, PriorArgs pr,
                                               const ReweightK& rk, double* __restrict__ logw, float2* __restrict__ lpq,
                                               uint32_t* err)
{
    static_assert(RW_PER_BLOCK == WARPS, "one warp per particle");
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * WARPS + (lane >> 2);
    const FSum ds = block_fsum(diffs.v), q = block_fsum(news.v);
    if ((lane & 3) || i >= N) return;
    const double sd = (double)ds.s + (double)ds.c;
    const double d = pr.de ? rk.lbase - sd * rk.dinv : rk.lbase - ((double)pr.a + 1.0) * sd;
    const double nl = logw[i] + d;
    if (!isfinite(nl)) atomicOr(err, DERR_NONFINITE);
    logw[i] = nl;
    lpq[i] = make_float2(q.s, q.c);
}

__global__ void __launch_bounds__(RW_THREADS) k_reweight(const float* __restrict__ beta, double* __restrict__ logw,
                                                   float2* __restrict__ lpq, int64_t N, int p, PriorArgs pr,
                                                   const ReweightK* __restrict__ rkp, int t, uint32_t* __restrict__ err)
{
    grid_dependency_wait();
    __shared__ LaneSums diffs, news;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t base = (int64_t)blockIdx.x * RW_PER_BLOCK;
    const ReweightK rk = rkp[t];
    FSum sdiff, snew;
    if (base + w < N) reweight_row(beta + (base + w) * p, p, pr, rk, lane, sdiff, snew);
    diffs.v[lane][w] = make_float2(sdiff.s, sdiff.c);
    news.v[lane][w] = make_float2(snew.s, snew.c);
    __syncthreads();
    if (w == 0) reweight_block(diffs, news, N, pr, rk, logw, lpq, err);
}

// The step's last MH test with its commit (k_move_commit), then the reweighting to the next
// scale of the row just settled, in one launch: one kernel boundary less a step, and the row is
// read once.
template <bool MALA, bool VEC, bool PARTS>
__global__ void __launch_bounds__(BLOCK) k_commit_reweight(MoveArgs a, int64_t N, int p, PriorArgs pr,
                                                          const float4* __restrict__ stepk, int t, uint32_t m_prev,
                                                          double* __restrict__ logw, const ReweightK* __restrict__ rkp,
                                                          uint32_t* err)
{
    __shared__ int accw[BLOCK / 32];
    __shared__ PartSlices parts;
    __shared__ RsumSlices rsum;
    __shared__ LaneSums diffs, news;  // (diffs: the reverse moves' sums first)
    grid_dependency_wait();
    gather_partials(a.mh, N, parts);
    if (PARTS) gather_rsum(a.mh, a.gp, N, rsum);
    __syncthreads();
    if (PARTS) sum_rsum(rsum);
    const float4 sk = stepk[t];
    const ReweightK rk = rkp[t + 1];
    const int64_t i = warp_global_id();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    commit_tests<MALA, VEC, PARTS>(a, parts, rsum, diffs, N, p, pr, sk, m_prev, accw, err);
    FSum sdiff, snew;
    if (i < N) {
        const bool acc = accw[w] != 0;
        if (acc) commit_row<MALA, VEC>(a, i, p, lane);
        reweight_row((acc ? a.beta_p : a.beta) + i * p, p, pr, rk, lane, sdiff, snew);
    }
    diffs.v[lane][w] = make_float2(sdiff.s, sdiff.c);
    news.v[lane][w] = make_float2(snew.s, snew.c);
    __syncthreads();
    if (w == 1) count_accepts(a.mh.acc_count, accw);
    if (w == 0) reweight_block(diffs, news, N, pr, rk, logw, a.mh.lpq, err);
}

// ---------------------------------------------------------- log-sum-exp and ESS
// Order-preserving integer of a double (NaN apart): the maximum runs on the integer units, where an
// FP64 comparison costs a warp 16 issue cycles.
__device__ __forceinline__ long long f64_key(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double key_f64(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}
__device__ __forceinline__ long long warp_max(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Each block: (m_b, sum e^{x - m_b}, sum e^{2(x - m_b)}) over its elements, combined by
// k_normalise. FP64 latency bounds it: one exp (about 40 dependent operations) and two sums whose
// trees run side by side.
constexpr int LSE_THREADS = 128;  // one weight per thread up to 128 x LSE_BLOCKS particles

__global__ void __launch_bounds__(LSE_THREADS) k_lse_partial(const double* __restrict__ logw, int64_t N,
                                                      double* __restrict__ scratch)
{
    grid_dependency_wait();
    constexpr int W = LSE_THREADS / 32;
    __shared__ long long shm[W];
    __shared__ double sh1[W], sh2[W];
    const int w = threadIdx.x >> 5;
    const int64_t stride = (int64_t)gridDim.x * LSE_THREADS, i0 = (int64_t)blockIdx.x * LSE_THREADS + threadIdx.x;
    const double x0 = i0 < N ? logw[i0] : -DBL_MAX;
    long long mk = max(f64_key(x0), f64_key(-DBL_MAX));
    for (int64_t i = i0 + stride; i < N; i += stride) mk = max(mk, f64_key(logw[i]));
    mk = warp_max(mk);
    if ((threadIdx.x & 31) == 0) shm[w] = mk;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < W; ++k) mk = max(mk, shm[k]);
    const double mb = key_f64(mk);
    double s1 = 0.0, s2 = 0.0;
    for (int64_t i = i0; i < N; i += stride) {
        const double e = exp((i == i0 ? x0 : logw[i]) - mb);
        s1 += e;
        s2 += e * e;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double v1 = __shfl_xor_sync(0xffffffffu, s1, o), v2 = __shfl_xor_sync(0xffffffffu, s2, o);
        s1 += v1;
        s2 += v2;
    }
    if ((threadIdx.x & 31) == 0) {
        sh1[w] = s1;
        sh2[w] = s2;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    s1 = sh1[0];
    s2 = sh2[0];
#pragma unroll
    for (int k = 1; k < W; ++k) {
        s1 += sh1[k];
        s2 += sh2[k];
    }
    const int B = gridDim.x;
    scratch[blockIdx.x] = mb;
    scratch[B + blockIdx.x] = s1;
    scratch[2 * B + blockIdx.x] = s2;
}

// lambda exp(acceptance - 0.574), the acceptance being acc of denom proposals.
__device__ __forceinline__ double adapted_lambda(double lam, unsigned long long acc, double denom)
{
    return denom > 0.0 ? lam * exp((double)acc / denom - 0.574) : lam;
}

__device__ __forceinline__ uint32_t weight_fix(double W) { return (uint32_t)__double2ull_rn(W * 2147483648.0); }

// The log-sum-exp of B <= LSE_BLOCKS block partials and the weights normalised by it. Every block
// combines the partials itself, lane l of warp 0 taking blocks l, l + 32, ... and then a
// fixed-order warp tree; block 0 publishes ESS, log Z and the resampling flag, from another warp
// while warp 0 takes the logarithm. A combining last block of the first kernel (a fence, a
// counter, a second read) and this pass took 12 + 5 us cold at N = 4096 as at N = 8192.
// With lam (MALA), block 0 also adapts the step size to the last block of moves' acceptance.
constexpr int NORM_THREADS = 64;

__global__ void __launch_bounds__(NORM_THREADS) k_normalise(WeightArrays w, int64_t N, const double* __restrict__ scratch, int B,
                                                            LseOut o, double* __restrict__ lam,
                                                            const unsigned long long* __restrict__ acc, double denom)
{
    grid_dependency_wait();
    __shared__ double sh_lse;
    const int lane = threadIdx.x & 31;
    double m, S1 = 0.0, S2 = 0.0;
    {
        constexpr int K = LSE_BLOCKS / 32;
        double x[K], a[K], c[K];
        long long mk = f64_key(-DBL_MAX);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int b = lane + 32 * k;
            const bool in = b < B;
            x[k] = in ? scratch[b] : -DBL_MAX;
            a[k] = in ? scratch[B + b] : 0.0;
            c[k] = in ? scratch[2 * B + b] : 0.0;
            mk = max(mk, f64_key(x[k]));
        }
        m = key_f64(warp_max(mk));
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (lane + 32 * k >= B) break;
            const double f = (a[k] > 0.0) ? exp(x[k] - m) : 0.0;
            S1 += a[k] * f;
            S2 += c[k] * f * f;
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
            const double v1 = __shfl_xor_sync(0xffffffffu, S1, s), v2 = __shfl_xor_sync(0xffffffffu, S2, s);
            S1 += v1;
            S2 += v2;
        }
    }
    if (threadIdx.x == 0) {
        const double lse = m + log(S1);
        sh_lse = lse;
        if (blockIdx.x == 0) {
            if (!isfinite(lse)) atomicOr(o.err, DERR_NONFINITE);
            if (o.logz) o.logz[o.t] = (o.mode == 0) ? lse : lse - log((double)N);
            if (lam) *lam = adapted_lambda(*lam, *acc, denom);
        }
    } else if (threadIdx.x == 32 && blockIdx.x == 0) {
        const double ess = (S1 * S1) / S2;
        if (!(ess >= 1.0 - 1e-9)) atomicOr(o.err, isfinite(S1) && S1 > 0.0 ? DERR_ESS : DERR_NONFINITE);
        const int res = (o.mode == 2) ? 1 : (ess < o.ess_frac * (double)N);
        *o.flag = res;
        if (o.mode != 2) {
            if (o.ess) o.ess[o.t] = ess;
            if (o.resampled) o.resampled[o.t] = (uint8_t)res;
        }
    }
    __syncthreads();
    const double lse = sh_lse;
    for (int64_t i = (int64_t)blockIdx.x * NORM_THREADS + threadIdx.x; i < N; i += (int64_t)gridDim.x * NORM_THREADS) {
        const double l = w.logw[i] - lse;
        const double W = exp(l);
        w.logw[i] = l;
        w.W[i] = W;
        w.Wf[i] = (float)W;
        w.wfix[i] = weight_fix(W);
    }
}

__global__ void k_weight_forms(const double* __restrict__ W, int64_t N, float* __restrict__ Wf,
                               uint32_t* __restrict__ wfix)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        Wf[i] = (float)W[i];
        wfix[i] = weight_fix(W[i]);
    }
}

__global__ void k_mark_uniform(int64_t N, int t, double* ess_out, uint8_t* res_out, int* flag)
{
    if (threadIdx.x == 0) {
        *flag = 0;
        if (ess_out) ess_out[t] = (double)N;
        if (res_out) res_out[t] = 0;
    }
}

// ------------------------------------------------------------ systematic resampling
// The cumulative sum C of W in the specified order: a running sum inside each 256-block
// in index order, a running sum of the block totals, C_i = carry(block) + local_i. cum holds
// N + ceil(N/256) + 1 doubles: the block-local running sums, then one carry per block, then u.
// Three kernels spread it over the SMs: the local sums (a warp per block), the carries (one
// warp, in block order), and the search, which forms C_i = carry + local_i as it reads it. A sweep of
// up to 64 blocks takes the local sums alone, the rest in its gather (k_resample_gather).
// Every bit of C is that of additions in the definition's order (running_sums).
constexpr int RS_BLOCK = 256;  // cumulative-sum block of the specified association order
constexpr int RS_CHUNKS = 4;   // 256-blocks (warps) per CTA of the local pass
constexpr int RS_CARRY_GROUPS = 8;  // block totals a lane of the carry kernel reads ahead

// The 32 running sums S + w_0, (S + w_0) + w_1, ... of a warp's values, each rounded as that chain
// of FP64 additions rounds; lane l's in r, the last returned.
//
// The chain itself is 32 additions of about 110 cycles, one after the other. But as long as the sum
// keeps its exponent e, an addition adds to its 53-bit integer mantissa M the addend's mantissa
// shifted right, rounded to nearest, a tie to the even sum: M + d0 if M is even, M + d1 if it is
// odd, integers that each lane knows by itself. Such pairs compose associatively (the first
// step's sum decides which of the second's is taken), so one scan gives all 32 sums. The lanes
// before the first whose sum leaves the exponent, or whose addend is above it, have their
// result; that one lane's is an FP64 addition, and the scan begins again behind it. A sum of
// n terms of one size changes its exponent about log2 n times. The local pass, 256 additions in a
// row: 19 -> 10 us at N = 1024 and 8192. A whole resampling of 10^5 weights: 62 -> 43 us.
// Negative, infinite and NaN addends take the addition (their exponent field reads as larger).
__device__ __forceinline__ double running_sums(double S, double w, double& r)
{
    constexpr unsigned long long TOP = 1ull << 52, HALF = 1ull << 63;
    const int lane = threadIdx.x & 31;
    const unsigned long long wb = (unsigned long long)__double_as_longlong(w);
    const int ew = max((int)(wb >> 52), 1);  // (a subnormal has exponent 1 and no leading one)
    const unsigned long long mw = (wb & (TOP - 1)) | (wb >= TOP ? TOP : 0ull);
    int first = 0;  // the lanes before it are done
    if (S == 0.0) {  // the first few sums change their exponent most often
        for (; first < 8; ++first) {
            S = __dadd_rn(S, __shfl_sync(0xffffffffu, w, first));
            if (lane == first) r = S;
        }
    }
    for (;;) {
        const unsigned long long sb = (unsigned long long)__double_as_longlong(S);
        const int e = max((int)(sb >> 52), 1), sh = e - ew;
        const unsigned long long M = (sb & (TOP - 1)) | (sb >= TOP ? TOP : 0ull);
        const bool chain = e < 0x7ff && sh >= 0;
        unsigned long long d0 = 0, d1 = 0;
        if (lane >= first && chain && sh < 64) {
            const unsigned long long q = mw >> sh, rest = sh ? mw << (64 - sh) : 0ull;
            const unsigned long long up = rest > HALF ? 1ull : 0ull, tie = rest == HALF ? 1ull : 0ull;
            d0 = q + up + (tie & q & 1ull);
            d1 = q + up + (tie & ~q & 1ull);
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long p0 = __shfl_up_sync(0xffffffffu, d0, o), p1 = __shfl_up_sync(0xffffffffu, d1, o);
            if (lane >= o) {
                const unsigned long long n0 = p0 + (p0 & 1ull ? d1 : d0), n1 = p1 + (p1 & 1ull ? d0 : d1);
                d0 = n0;
                d1 = n1;
            }
        }
        const unsigned long long sum = M + (M & 1ull ? d1 : d0);
        const unsigned int out = __ballot_sync(0xffffffffu, lane >= first && (!chain || sum >= 2 * TOP));
        const int f = out ? __ffs(out) - 1 : 32;
        const double v = __longlong_as_double((long long)(((unsigned long long)(e - 1) << 52) + sum));
        if (lane >= first && lane < f) r = v;
        const double before = f > first ? __shfl_sync(0xffffffffu, v, f - 1) : S;
        if (f == 32) return before;
        S = __dadd_rn(before, __shfl_sync(0xffffffffu, w, f));
        if (lane == f) r = S;
        first = f + 1;
        if (first == 32) return S;
    }
}

__global__ void __launch_bounds__(32 * RS_CHUNKS) k_resample_local(const double* __restrict__ W, int64_t N,
                                                                   double* __restrict__ cum,
                                                                   const int* __restrict__ flag)
{
    grid_dependency_wait();
    if (flag && *flag == 0) return;
    const int64_t b = (int64_t)blockIdx.x * RS_CHUNKS + (threadIdx.x >> 5), i0 = b * RS_BLOCK + (threadIdx.x & 31);
    if (b * RS_BLOCK >= N) return;
    double w[RS_BLOCK / 32];
#pragma unroll
    for (int g = 0; g < RS_BLOCK / 32; ++g) w[g] = i0 + 32 * g < N ? W[i0 + 32 * g] : 0.0;
    double local = 0.0;
#pragma unroll 1
    for (int g = 0; g < RS_BLOCK / 32; ++g) {
        double r, x = w[0];  // (shifted along, so that the loop's body stands once)
        local = running_sums(local, x, r);
        if (i0 + 32 * g < N) cum[i0 + 32 * g] = r;
#pragma unroll
        for (int k = 0; k + 1 < RS_BLOCK / 32; ++k) w[k] = w[k + 1];
    }
    // the block total, turned into the block's carry by k_resample_carry
    if ((threadIdx.x & 31) == 0) cum[N + b] = local;
}

// carry[b] = total_0 + ... + total_{b-1} in block order (the totals are read from the carry
// slots and replaced), then the resampling uniform after the carries. One warp.
__global__ void __launch_bounds__(32) k_resample_carry(int64_t N, double* __restrict__ cum,
                                                       const int* __restrict__ flag, int t,
                                                       const uint64_t* __restrict__ seedp, double u_override)
{
    grid_dependency_wait();
    if (flag && *flag == 0) return;
    const int tid = threadIdx.x;
    const int64_t nblk = (N + RS_BLOCK - 1) / RS_BLOCK;
    double* carry = cum + N;
    double run = 0.0;
    for (int64_t b0 = 0; b0 < nblk; b0 += 32 * RS_CARRY_GROUPS) {
        double w[RS_CARRY_GROUPS];
#pragma unroll
        for (int g = 0; g < RS_CARRY_GROUPS; ++g) w[g] = b0 + 32 * g + tid < nblk ? carry[b0 + 32 * g + tid] : 0.0;
#pragma unroll 1
        for (int g = 0; g < RS_CARRY_GROUPS; ++g) {
            const int64_t b = b0 + 32 * g + tid;
            double r;
            const double next = running_sums(run, w[0], r);
            const double prev = __shfl_up_sync(0xffffffffu, r, 1);
            if (b < nblk) carry[b] = tid == 0 ? run : prev;
            run = next;
#pragma unroll
            for (int k = 0; k + 1 < RS_CARRY_GROUPS; ++k) w[k] = w[k + 1];
        }
    }
    if (tid == 0) {
        if (seedp) {
            const uint4 u = philox4x32_10(make_uint4(0u, 0u, (uint32_t)t, TAG_RESAMPLE << 16), seed_key(*seedp));
            carry[nblk] = u01_d(u.x);
        } else {
            carry[nblk] = u_override;
        }
    }
}

// A_k = min{i : C_i > (k + u)/N}, clamped to N - 1, with C_i = carry(i / 256) + local_i (the
// first block's carry is 0 and its C_i is local_i, as in the definition). C is non-negative
// and non-decreasing, and for non-negative doubles the order of the bit patterns as signed
// integers is the numeric order, so the search compares integers.
__device__ __forceinline__ long long resample_c_bits(const double* __restrict__ cum, int64_t N, int64_t i)
{
    const double c = (i < RS_BLOCK) ? cum[i] : __dadd_rn(cum[N + i / RS_BLOCK], cum[i]);
    return __double_as_longlong(c);
}

__global__ void k_resample_search(const double* __restrict__ cum, int64_t N, int32_t* __restrict__ idx,
                                  const int* __restrict__ flag)
{
    grid_dependency_wait();
    if (flag && *flag == 0) return;
    const int64_t nblk = (N + RS_BLOCK - 1) / RS_BLOCK;
    const double u = cum[N + nblk];
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += (int64_t)gridDim.x * blockDim.x) {
        const long long target = __double_as_longlong(__ddiv_rn(__dadd_rn((double)k, u), (double)N));
        int64_t lo = 0, hi = N;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (resample_c_bits(cum, N, mid) > target)
                hi = mid;
            else
                lo = mid + 1;
        }
        idx[k] = (int32_t)(lo < N ? lo : N - 1);
    }
}

// Ancestor rows into the scratch buffers, one warp per new particle k: beta_tmp[k] =
// beta[idx[k]] (and the gradient rows for MALA), with the log-likelihood and log-prior pairs.
template <bool VEC>
__global__ void __launch_bounds__(BLOCK) k_gather(const int32_t* __restrict__ idx, const float* __restrict__ beta,
                                                 float* __restrict__ beta_tmp, const float2* __restrict__ llq,
                                                 const float2* __restrict__ lpq, float2* __restrict__ llq_tmp,
                                                 float2* __restrict__ lpq_tmp, const float* __restrict__ g,
                                                 float* __restrict__ g_tmp, int64_t N, int p, const int* __restrict__ flag)
{
    grid_dependency_wait();
    if (*flag == 0) return;
    const int64_t k = warp_global_id();
    const int lane = threadIdx.x & 31;
    if (k >= N) return;
    const int64_t a = idx[k];
    const float* src = beta + a * p;
    float* dst = beta_tmp + k * p;
    if (VEC) {
        for (int j = 4 * lane; j < p; j += 128) st4(dst + j, ld4(src + j));
        if (g)
            for (int j = 4 * lane; j < p; j += 128) st4(g_tmp + k * p + j, ld4(g + a * p + j));
    } else {
        for (int j = lane; j < p; j += 32) dst[j] = src[j];
        if (g)
            for (int j = lane; j < p; j += 32) g_tmp[k * p + j] = g[a * p + j];
    }
    if (lane == 0) {
        llq_tmp[k] = llq[a];
        lpq_tmp[k] = lpq[a];
    }
}

// The same from the local sums alone, for N <= RG_MAX_BLOCKS blocks of 256: every block of the
// gather forms the carries itself (one thread, in block order), and every warp finds its ancestor
// by a 32-way search, the smallest i with C_i > (k + u)/N as in k_resample_search. Two kernel
// boundaries less than carries, search and gather apart. The line lies at 16384 particles: at
// 30000 every block's 118 additions cost more than the boundaries (a sweep 1.60 against 1.50 ms).
constexpr int RG_MAX_BLOCKS = 64;

template <bool VEC>
__global__ void __launch_bounds__(BLOCK) k_resample_gather(const double* __restrict__ cum, int t,
                                                          const uint64_t* __restrict__ seedp, const float* __restrict__ beta,
                                                          float* __restrict__ beta_tmp, const float2* __restrict__ llq,
                                                          const float2* __restrict__ lpq, float2* __restrict__ llq_tmp,
                                                          float2* __restrict__ lpq_tmp, const float* __restrict__ g,
                                                          float* __restrict__ g_tmp, int64_t N, int p, const int* __restrict__ flag)
{
    grid_dependency_wait();
    if (*flag == 0) return;
    __shared__ double tot[RG_MAX_BLOCKS], carry[RG_MAX_BLOCKS], us;
    const int nblk = (int)((N + RS_BLOCK - 1) / RS_BLOCK);
    if ((int)threadIdx.x < nblk) tot[threadIdx.x] = cum[N + threadIdx.x];
    if (threadIdx.x == 32) {
        const uint4 x = philox4x32_10(make_uint4(0u, 0u, (uint32_t)t, TAG_RESAMPLE << 16), seed_key(*seedp));
        us = u01_d(x.x);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        double run = 0.0;
        for (int b0 = 0; b0 < nblk; b0 += 32) {
            const int b = b0 + (int)threadIdx.x;
            double r;
            const double next = running_sums(run, b < nblk ? tot[b] : 0.0, r);
            const double prev = __shfl_up_sync(0xffffffffu, r, 1);
            if (b < nblk) carry[b] = threadIdx.x == 0 ? run : prev;
            run = next;
        }
    }
    __syncthreads();
    const int64_t k = warp_global_id();
    const int lane = threadIdx.x & 31;
    if (k >= N) return;
    const long long target = __double_as_longlong(__ddiv_rn(__dadd_rn((double)k, us), (double)N));
    int lo = 0, hi = (int)N;  // the answer is in [lo, hi), or hi = N if no C_i exceeds the target
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) / 32;
        const int i = min(lo + (lane + 1) * step, hi) - 1;
        const double c = (i < RS_BLOCK) ? cum[i] : __dadd_rn(carry[i / RS_BLOCK], cum[i]);
        const unsigned int gt = __ballot_sync(0xffffffffu, __double_as_longlong(c) > target);
        if (gt == 0u) {  // only in the first round: rounding left C below the target
            lo = (int)N - 1;
            break;
        }
        const int f = __ffs(gt) - 1;
        hi = min(lo + (f + 1) * step, hi);
        lo = min(lo + f * step, hi - 1);
    }
    const int64_t a = lo;
    const float* src = beta + a * p;
    float* dst = beta_tmp + k * p;
    if (VEC) {
        for (int j = 4 * lane; j < p; j += 128) st4(dst + j, ld4(src + j));
        if (g)
            for (int j = 4 * lane; j < p; j += 128) st4(g_tmp + k * p + j, ld4(g + a * p + j));
    } else {
        for (int j = lane; j < p; j += 32) dst[j] = src[j];
        if (g)
            for (int j = lane; j < p; j += 32) g_tmp[k * p + j] = g[a * p + j];
    }
    if (lane == 0) {
        llq_tmp[k] = llq[a];
        lpq_tmp[k] = lpq[a];
    }
}

// The resampled particles back into the state, with uniform weights (log(1/N), 1/N and
// round(2^31/N), formed on the host).
template <bool VEC>
__global__ void __launch_bounds__(BLOCK) k_copyback(float* __restrict__ beta, const float* __restrict__ beta_tmp,
                                                   float2* __restrict__ llq, float2* __restrict__ lpq,
                                                   const float2* __restrict__ llq_tmp, const float2* __restrict__ lpq_tmp,
                                                   float* __restrict__ g, const float* __restrict__ g_tmp, WeightArrays w,
                                                   int64_t N, int p, const int* __restrict__ flag, double lw, double wi,
                                                   uint32_t wf)
{
    grid_dependency_wait();
    if (*flag == 0) return;
    const int64_t k = warp_global_id();
    const int lane = threadIdx.x & 31;
    if (k >= N) return;
    const int64_t o = k * p;
    if (VEC) {
        for (int j = 4 * lane; j < p; j += 128) st4(beta + o + j, ld4(beta_tmp + o + j));
        if (g)
            for (int j = 4 * lane; j < p; j += 128) st4(g + o + j, ld4(g_tmp + o + j));
    } else {
        for (int j = lane; j < p; j += 32) beta[o + j] = beta_tmp[o + j];
        if (g)
            for (int j = lane; j < p; j += 32) g[o + j] = g_tmp[o + j];
    }
    if (lane == 0) {
        llq[k] = llq_tmp[k];
        lpq[k] = lpq_tmp[k];
        w.logw[k] = lw;
        w.W[k] = wi;
        w.Wf[k] = (float)wi;
        w.wfix[k] = wf;
    }
}

// -------------------------------------------------------------- column moments
constexpr int CS_ROWS = 8;

// With rs_flag set (a step that resampled, its rows still in beta_rs): those rows, weights wi.
__global__ void k_colstats_partial(const float* __restrict__ beta_state, const float* __restrict__ Wf, int64_t N, int p,
                                   float4* __restrict__ part, const float* __restrict__ beta_rs,
                                   const int* __restrict__ rs_flag, float wi)
{
    grid_dependency_wait();
    const bool rs = rs_flag && *rs_flag != 0;
    const float* __restrict__ beta = rs ? beta_rs : beta_state;
    __shared__ float4 sh[CS_ROWS][32];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int j = blockIdx.x * 32 + tx;
    FSum s1, s2;
    if (j < p) {
        const int64_t step = (int64_t)CS_ROWS * gridDim.y;
        int64_t i = (int64_t)blockIdx.y * CS_ROWS + ty;
        for (; i + 3 * step < N; i += 4 * step) {  // four rows in flight
            float b[4], wv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                b[u] = beta[(i + u * step) * p + j];
                wv[u] = rs ? wi : Wf[i + u * step];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float wb = wv[u] * b[u];
                s1.add(wb);
                s2.add(wb * b[u]);
            }
        }
        for (; i < N; i += step) {
            const float b = beta[i * p + j];
            const float wb = (rs ? wi : Wf[i]) * b;
            s1.add(wb);
            s2.add(wb * b);
        }
    }
    sh[ty][tx] = make_float4(s1.s, s1.c, s2.s, s2.c);
    __syncthreads();
    if (ty == 0 && j < p) {
        for (int r = 1; r < CS_ROWS; ++r) {
            const float4 o = sh[r][tx];
            s1.add(o.x);
            s1.c += o.y;
            s2.add(o.z);
            s2.c += o.w;
        }
        part[(int64_t)blockIdx.y * p + j] = make_float4(s1.s, s1.c, s2.s, s2.c);
    }
}

// One warp per coordinate: lane s takes split s (fixed order), then a warp tree.
__global__ void k_colstats_finish(const float4* __restrict__ part, int p, int splits, float* __restrict__ scale_out,
                                  int kind, double rw_factor, const double* __restrict__ lam_dev, double sd_floor,
                                  const double* __restrict__ sched, int t, float* __restrict__ h_out, double p_pow)
{
    grid_dependency_wait();
    const int j = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (j >= p) return;
    double s1 = 0.0, s2 = 0.0;
    for (int s = lane; s < splits; s += 32) {
        const float4 q = part[(int64_t)s * p + j];
        s1 += (double)q.x + (double)q.y;
        s2 += (double)q.z + (double)q.w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (lane != 0) return;
    if (j == 0 && h_out) *h_out = (float)(*lam_dev * p_pow);
    const double var = fmax(s2 - s1 * s1, 0.0);
    const double fl = sd_floor * sched[t];
    if (kind == 0) {
        scale_out[j] = (float)(rw_factor * fmax(sqrt(var), fl));
    } else {
        // MALA's D_j, and beside it sqrt(D_j) and 1/D_j for the proposal and its densities
        const double D = fmax(var, fl * fl);
        scale_out[j] = (float)D;
        scale_out[p + j] = (float)sqrt(D);
        scale_out[2 * p + j] = (float)(1.0 / D);
    }
}

// ------------------------------------------------------------------ summaries
// One CTA per marker j. Weighted mean (FP32 weights, compensated sum) and concentrations
// 1 - sum_{|beta| < Delta} W (Delta passed as the smallest float >= Delta, which makes the
// float comparison equal to the exact one). Weighted quantiles Q_q = the smallest value v
// with sum_{beta_i <= v} W_i >= q, by a three-pass radix select (11, 11, 10 bits) over the
// order-preserving 32-bit key of v. Weights enter the histograms as the integers
// round(W 2^31), so every cumulative sum is exact and independent of the order of the
// atomic additions.
constexpr int SUM_THREADS = 512;

__device__ __forceinline__ uint32_t float_key(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k)
{
    const uint32_t u = (k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k;
    return __uint_as_float(u);
}

// First bin of hist[0..nbins) (weights) at which *below + the cumulative weight reaches
// target; one warp. Adds the weight of the bins before it to *below. Returns -1 if no bin
// reaches the target. Lane l owns bins l*per .. l*per+per-1 and sums them starting at a
// lane-dependent offset, so the 32 lanes hit 32 different shared-memory banks.
__device__ int warp_find_bin(const uint32_t* hist, int nbins, unsigned long long target, unsigned long long* below)
{
    const int lane = threadIdx.x & 31;
    const int per = nbins / 32;
    const uint32_t* mine_p = hist + lane * per;
    unsigned long long mine = 0;
#pragma unroll 16
    for (int k = 0; k < per; ++k) mine += mine_p[(k + lane) & (per - 1)];
    unsigned long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const unsigned long long base = *below;
    const unsigned int hit = __ballot_sync(0xffffffffu, base + incl >= target);
    if (hit == 0u) return -1;
    const int L = __ffs(hit) - 1;
    // inside lane L's range: the whole warp scans its `per` bins, `per / 32` per lane
    const unsigned long long start = __shfl_sync(0xffffffffu, base + incl - mine, L);
    const int sub = per / 32;  // bins per lane (per is a multiple of 32)
    const uint32_t* rng = hist + L * per + lane * sub;
    unsigned long long part = 0;
    for (int k = 0; k < sub; ++k) part += rng[k];
    unsigned long long inc2 = part;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long v = __shfl_up_sync(0xffffffffu, inc2, o);
        if (lane >= o) inc2 += v;
    }
    const unsigned int hit2 = __ballot_sync(0xffffffffu, start + inc2 >= target);
    const int L2 = __ffs(hit2) - 1;  // lane L's total reaches the target, so some lane does
    int bin = -1;
    unsigned long long cum = 0;
    if (lane == L2) {
        cum = start + inc2 - part;
        for (int k = 0; k < sub; ++k) {
            const unsigned long long h = rng[k];
            if (cum + h >= target) {
                bin = L * per + L2 * sub + k;
                break;
            }
            cum += h;
        }
    }
    bin = __shfl_sync(0xffffffffu, bin, L2);
    cum = __shfl_sync(0xffffffffu, cum, L2);
    if (bin >= 0) *below = cum;
    return bin;
}

// keysT[j][i] = float_key(beta[i][j]): the particles' values marker-major as
// order-preserving integer keys, so each summaries CTA streams its marker's column with
// coalesced loads. 32 x 32 tiles through shared memory. With WfS != NULL the weights (Wf,
// wfix) are copied beside them, so that the summaries read nothing the next step rewrites.
__global__ void k_keys_transpose(const float* __restrict__ beta, int64_t N, int p, uint32_t* __restrict__ keysT,
                                 const float* __restrict__ Wf, const uint32_t* __restrict__ wfix,
                                 float* __restrict__ WfS, uint32_t* __restrict__ wfixS)
{
    grid_dependency_wait();
    __shared__ uint32_t tile[32][33];
    const int64_t i0 = (int64_t)blockIdx.x * 32;
    const int j0 = blockIdx.y * 32;
    if (WfS && blockIdx.y == 0 && threadIdx.y == 0) {
        const int64_t i = i0 + threadIdx.x;
        if (i < N) {
            WfS[i] = Wf[i];
            wfixS[i] = wfix[i];
        }
    }
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int64_t i = i0 + r;
        const int j = j0 + threadIdx.x;
        tile[r][threadIdx.x] = (i < N && j < p) ? float_key(beta[i * p + j]) : 0u;
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int j = j0 + r;
        const int64_t i = i0 + threadIdx.x;
        if (i < N && j < p) keysT[(int64_t)j * N + i] = tile[threadIdx.x][r];
    }
}

// Two compensated sums at once, in packed operations (each rounds as its scalar form).
struct FSum2 {
    static __device__ __forceinline__ void add(FSum& a, FSum& b, float xa, float xb)
    {
        const uint64_t neg = pack2(-1.0f, -1.0f);
        const uint64_t s = pack2(a.s, b.s), x = pack2(xa, xb);
        const uint64_t t = add2(s, x);
        const uint64_t z = fma2(s, neg, t);                                       // t - s
        const uint64_t e = add2(fma2(fma2(z, neg, t), neg, s), fma2(z, neg, x));  // (s - (t - z)) + (x - z)
        const uint64_t c = add2(pack2(a.c, b.c), e);
        const float2 t2 = unpack2(t), c2 = unpack2(c);
        a.s = t2.x;
        b.s = t2.y;
        a.c = c2.x;
        b.c = c2.y;
    }
};

constexpr int SUM_SUB = 4;     // sub-histograms of the first radix digit (by lane % 4)
constexpr int SUM_BINS = 2048;  // bins of an 11-bit digit

// Per coordinate j (one CTA): the weighted mean and the concentrations (compensated FP32
// sums), and the weighted quantiles by an exact radix select on the fixed-point weights
// round(W 2^31) over the order-preserving integer keys of the values: digits of 11, 11 and
// 10 bits from the top. The first digit's histogram is built while the values are loaded,
// in SUM_SUB copies that are merged before the search: particles cluster in a few top-digit
// bins, and neighbouring copies in neighbouring banks spread a warp's atomics. The later digits'
// passes read the keys again (from L2), and the weights of those in a selected bin only: kept in
// shared memory instead, keys and weights took 8 N bytes, one CTA an SM from N = 12000 on.
// At most NQ levels and ND thresholds; the usual few take less work a value. Bound by instructions
// and the latency of the reads; it runs beside the next step and keeps the likelihood kernel off the
// SMs it holds. n = 2000, p = 200, N = 8192: 34 -> 20 us, a RW step of 10 moves 333 -> 328;
// n = 5000, p = 500, N = 16384: 143 -> 56 us, step 1479 -> 1395.
template <int NQ, int ND>
__global__ void __launch_bounds__(SUM_THREADS, 2) k_summaries(const uint32_t* __restrict__ keysT, const float* __restrict__ Wf,
                                                               const uint32_t* __restrict__ wfix, int64_t N, int p,
                                                               SummaryArgs sa, int t, double* __restrict__ mean,
                                                               double* __restrict__ quant, double* __restrict__ conc)
{
    grid_dependency_wait();
    extern __shared__ __align__(16) uint32_t hist[];  // max(SUM_SUB, nq) * SUM_BINS words
    __shared__ float red_s[SUM_THREADS / 32][9], red_c[SUM_THREADS / 32][9];
    __shared__ unsigned long long shu[SUM_THREADS / 32];
    __shared__ uint32_t shk[SUM_THREADS / 32];
    __shared__ int bins[8][3];
    __shared__ unsigned long long below[8];
    const int j = blockIdx.x;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int nq = (quant && sa.nq > 0) ? sa.nq : 0, nd = sa.nd;
    if (nq > 0) {
        for (int e = tid; e < SUM_SUB * SUM_BINS / 4; e += SUM_THREADS)
            reinterpret_cast<uint4*>(hist)[e] = make_uint4(0u, 0u, 0u, 0u);
        if (tid < 8) below[tid] = 0ull;
        __syncthreads();
    }
    uint32_t* hsub = hist + (lane & (SUM_SUB - 1));
    // ---- mean, concentrations, top-digit histogram
    FSum msum;
    FSum cs[ND];
    uint32_t kmax = 0;
    unsigned long long tot = 0;
    const uint32_t* kcol = keysT + (int64_t)j * N;
    auto take = [&](uint32_t k, uint32_t wv, float wf) {
        const float b = key_float(k);
        msum.add(wf * b);
        if (ND == 2) {  // a zero term leaves a compensated sum as it is
            FSum2::add(cs[0], cs[1], fabsf(b) < sa.dthr[0] ? wf : 0.0f, fabsf(b) < sa.dthr[1] ? wf : 0.0f);
        } else {
#pragma unroll
            for (int d = 0; d < ND; ++d)
                if (d < nd && fabsf(b) < sa.dthr[d]) cs[d].add(wf);
        }
        kmax = k > kmax ? k : kmax;
        tot += wv;
        if (nq > 0 && wv != 0u) atomicAdd(&hsub[(k >> 21) * SUM_SUB], wv);
    };
    constexpr int U = 4;  // elements a thread has in flight
    int64_t i = tid;
    for (; i + (U - 1) * SUM_THREADS < N; i += U * SUM_THREADS) {
        uint32_t k[U], wv[U];
        float wf[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            k[u] = kcol[i + u * SUM_THREADS];
            wv[u] = wfix[i + u * SUM_THREADS];
            wf[u] = Wf[i + u * SUM_THREADS];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) take(k[u], wv[u], wf[u]);
    }
    for (; i < N; i += SUM_THREADS) take(kcol[i], wfix[i], Wf[i]);
    // ---- one block reduction for every scalar
    msum = warp_sum(msum);
#pragma unroll
    for (int d = 0; d < ND; ++d)
        if (d < nd) cs[d] = warp_sum(cs[d]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        tot += __shfl_xor_sync(0xffffffffu, tot, o);
        kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
    }
    if (lane == 0) {
        red_s[w][0] = msum.s;
        red_c[w][0] = msum.c;
#pragma unroll
        for (int d = 0; d < ND; ++d)
            if (d < nd) {
                red_s[w][1 + d] = cs[d].s;
                red_c[w][1 + d] = cs[d].c;
            }
        shu[w] = tot;
        shk[w] = kmax;
    }
    __syncthreads();
    if (w == 0) {
        // lane v < 1 + nd finishes scalar v: the mean (v = 0) or concentration v - 1
        if (lane < 1 + nd) {
            FSum r;
            for (int k = 0; k < SUM_THREADS / 32; ++k) {
                r.add(red_s[k][lane]);
                r.c += red_c[k][lane];
            }
            const double val = (double)r.s + (double)r.c;
            if (lane == 0) {
                if (mean) mean[(int64_t)t * p + j] = val;
            } else if (conc) {
                conc[((int64_t)t * p + j) * nd + (lane - 1)] = 1.0 - val;
            }
        }
    }
    if (nq == 0) return;
    tot = 0;
    kmax = 0;
    for (int k = 0; k < SUM_THREADS / 32; ++k) {
        tot += shu[k];
        kmax = max(kmax, shk[k]);
    }
    // merge the top-digit copies: bin b's in words SUM_SUB b .., their sum in word b
    static_assert(SUM_SUB == 4 && SUM_BINS % SUM_THREADS == 0, "one uint4 a bin");
    uint32_t merged[SUM_BINS / SUM_THREADS];
#pragma unroll
    for (int u = 0; u < SUM_BINS / SUM_THREADS; ++u) {
        const uint4 v = reinterpret_cast<const uint4*>(hist)[tid + u * SUM_THREADS];
        merged[u] = v.x + v.y + v.z + v.w;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < SUM_BINS / SUM_THREADS; ++u) hist[tid + u * SUM_THREADS] = merged[u];
    __syncthreads();
    // ---- digit searches: the top digit on the merged histogram, then bits 10..20 and 0..9
    // of the keys that share the selected prefix, one histogram per quantile level
    for (int pass = 0; pass < 3; ++pass) {
        const int bits = (pass == 2) ? 10 : 11;
        const int shift = (pass == 0) ? 21 : ((pass == 1) ? 10 : 0);
        const int nb = 1 << bits;
        if (pass > 0) {
            uint32_t want[NQ];  // (no key has the prefix ~0)
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                want[q] = q < nq && bins[q][0] >= 0
                              ? ((pass == 1) ? (uint32_t)bins[q][0] : (((uint32_t)bins[q][0] << 11) | (uint32_t)bins[q][1]))
                              : ~0u;
            for (int e = tid; e < nq * nb; e += SUM_THREADS) hist[e] = 0u;
            __syncthreads();
            auto look = [&](uint32_t k, int64_t at) {
                const uint32_t pre = k >> (shift + bits);
                bool any = false;
#pragma unroll
                for (int q = 0; q < NQ; ++q) any |= pre == want[q];
                if (!any) return;
                const uint32_t wv = wfix[at];
                if (wv == 0u) return;
                const uint32_t dig = (k >> shift) & (uint32_t)(nb - 1);
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (pre == want[q]) atomicAdd(&hist[q * nb + dig], wv);
            };
            int64_t at = tid;
            for (; at + (2 * U - 1) * SUM_THREADS < N; at += 2 * U * SUM_THREADS) {
                uint32_t k[2 * U];
#pragma unroll
                for (int u = 0; u < 2 * U; ++u) k[u] = kcol[at + u * SUM_THREADS];
#pragma unroll
                for (int u = 0; u < 2 * U; ++u) look(k[u], at + u * SUM_THREADS);
            }
            for (; at < N; at += SUM_THREADS) look(kcol[at], at);
            __syncthreads();
        }
        if (w < nq) {
            const int q = w;
            const unsigned long long target = sa.target[q];
            int b = -1;
            if (tot >= target && (pass == 0 || bins[q][0] >= 0)) {
                unsigned long long bl = below[q];
                b = warp_find_bin(hist + (pass == 0 ? 0 : q * nb), nb, target, &bl);
                if (lane == 0) below[q] = bl;
            }
            if (lane == 0) {
                if (pass == 0)
                    bins[q][0] = b;
                else if (bins[q][0] >= 0)
                    bins[q][pass] = b;
            }
        }
        __syncthreads();
    }
    if (tid < nq) {
        const int q = tid;
        uint32_t key;
        if (bins[q][0] < 0 || bins[q][1] < 0 || bins[q][2] < 0)
            key = kmax;  // rounding left the total below q: the largest value, as in the definition
        else
            key = ((uint32_t)bins[q][0] << 21) | ((uint32_t)bins[q][1] << 10) | (uint32_t)bins[q][2];
        quant[((int64_t)t * p + j) * nq + q] = (double)key_float(key);
    }
}

// ------------------------------------------------ scale-marginalised summaries
// Section 4, eq. all_particles: with a uniform prior on log b over the log-spaced
// schedule, the particle systems of all steps mix with weights Z_t / Z_1, each the running
// product of the Z_t / Z_{t-1} estimates: w_t = exp(L_t - max L) / sum_s exp(L_s - max L),
// L_t = sum_{s=1..t} inc_s (the t = 0 evidence is common to every L_t). One thread, in
// step order (T is a few hundred).
__global__ void k_marginal_weights(const double* __restrict__ log_z_inc, int64_t T, double* __restrict__ post_c)
{
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    double acc = 0.0, m = -DBL_MAX;
    for (int64_t t = 0; t < T; ++t) {
        if (t > 0) acc += log_z_inc[t];
        post_c[t] = acc;
        m = fmax(m, acc);
    }
    double s = 0.0;
    for (int64_t t = 0; t < T; ++t) s += exp(post_c[t] - m);
    for (int64_t t = 0; t < T; ++t) post_c[t] = exp(post_c[t] - m) / s;
}

// Mixture of the per-step summaries: thread (j, v) sums w_t * mean[t][j] (v = 0) or
// w_t * conc[t][j][v - 1] over t in order.
__global__ void k_marginal_apply(const double* __restrict__ post_c, const double* __restrict__ mean,
                                 const double* __restrict__ conc, int64_t T, int64_t p, int D,
                                 double* __restrict__ mean_out, double* __restrict__ conc_out)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= p * (1 + D)) return;
    const int64_t j = e / (1 + D);
    const int v = (int)(e - j * (1 + D));
    double acc = 0.0;
    if (v == 0) {
        for (int64_t t = 0; t < T; ++t) acc += post_c[t] * mean[t * p + j];
        mean_out[j] = acc;
    } else {
        for (int64_t t = 0; t < T; ++t) acc += post_c[t] * conc[(t * p + j) * D + (v - 1)];
        conc_out[j * D + (v - 1)] = acc;
    }
}

__global__ void k_accept_rate(const unsigned long long* acc, int T, double denom, double* rate)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < T) rate[t] = denom > 0.0 ? (double)acc[t] / denom : 0.0;
}

__global__ void k_adapt_lambda(double* lam, const unsigned long long* acc, double denom)
{
    if (threadIdx.x == 0) *lam = adapted_lambda(*lam, *acc, denom);
}

__global__ void k_set_f64(double* ptr, double v)
{
    if (threadIdx.x == 0) *ptr = v;
}

// ------------------------------------------------------------ stream-test kernels
__global__ void k_philox(const uint32_t* ctr, uint2 key, int64_t count, uint32_t* out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const uint4 r = philox4x32_10(make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]), key);
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
}

__global__ void k_normals(uint64_t seed, uint32_t particle, uint32_t t, uint32_t m, int64_t p, float* out)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (4 * g >= p) return;
    const float4 z = normals4(seed, (uint32_t)g, particle, t, m);
    const float zz[4] = {z.x, z.y, z.z, z.w};
    for (int k = 0; k < 4 && 4 * g + k < p; ++k) out[4 * g + k] = zz[k];
}

__global__ void k_prior_sample(uint64_t seed, PriorArgs pr, float c, int64_t N, int64_t p, float* out)
{
    const int64_t total = N * p;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / p;
        out[e] = prior_draw(seed, (uint32_t)i, (uint32_t)(e - i * p), pr.a, c, pr.de != 0);
    }
}

// The full log density, -log(2c) included.
__global__ void k_prior_logpdf(PriorArgs pr, double c, const float* beta, int64_t k, double* out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= k) return;
    const float inv_ac = (float)(1.0 / ((double)pr.a * c));
    out[i] = -log(2.0 * c) + prior_coef(pr, c) * (double)prior_term(beta[i], inv_ac, pr.de);
}

}  // namespace

// ======================================================================= launchers
// Launch configuration with programmatic stream serialization (programmatic dependent
// launch): the kernel may be scheduled while its predecessor drains and waits for it with
// grid_dependency_wait before reading anything the predecessor wrote.
static cudaLaunchConfig_t pdl_config(unsigned grid, unsigned block, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    return cfg;
}
static void pdl_attr(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[1])
{
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// A launch with programmatic stream serialization: the kernels of the sweep's chain begin
// with grid_dependency_wait, so each may be scheduled while its predecessor drains.
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

static int64_t lse_blocks(int64_t N)
{
    const int64_t blocks = (N + LSE_THREADS - 1) / LSE_THREADS;
    return blocks < LSE_BLOCKS ? blocks : LSE_BLOCKS;
}
static unsigned warps_grid(int64_t N) { return (unsigned)((N + WARPS - 1) / WARPS); }
static unsigned elem_grid(int64_t total)
{
    int64_t b = (total + 255) / 256;
    if (b < 1) b = 1;
    return (unsigned)(b < 8192 ? b : 8192);
}

cudaError_t smc_init_attributes()
{
    return cudaFuncSetAttribute(k_summaries<8, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                8 * SUM_BINS * (int)sizeof(uint32_t));
}

cudaError_t launch_init_prior(float* beta, int64_t N, int p, PriorArgs pr, const double* sched, int t0,
                              const uint64_t* seed, cudaStream_t st)
{
    k_init_prior<<<elem_grid(N * p), 256, 0, st>>>(beta, N, p, pr, sched, t0, seed);
    return cudaGetLastError();
}

cudaError_t launch_step_constants(PriorArgs pr, const double* sched, int T, int p, float4* out, ReweightK* rk,
                                  cudaStream_t st)
{
    k_step_constants<<<(T + 127) / 128, 128, 0, st>>>(pr, sched, T, p, out, rk);
    return cudaGetLastError();
}

cudaError_t launch_move_rw(const MoveArgs& a, bool decide, int64_t N, int p, PriorArgs pr, const float4* stepk, int t,
                           uint32_t m, uint32_t m_prev, const uint64_t* seed, int noise, uint32_t* err, cudaStream_t st)
{
    const bool vec = (p & 3) == 0;
    const unsigned grid = warps_grid(N);
    if (decide) {  // follows the likelihood GEMM: programmatic dependent launch
        cudaLaunchConfig_t cfg = pdl_config(grid, BLOCK, st);
        cudaLaunchAttribute attr[1];
        pdl_attr(cfg, attr);
        if (vec)
            return cudaLaunchKernelEx(&cfg, k_move_rw<true, true>, a, N, p, pr, stepk, t, m, m_prev, seed, noise, err);
        return cudaLaunchKernelEx(&cfg, k_move_rw<true, false>, a, N, p, pr, stepk, t, m, m_prev, seed, noise, err);
    } else {
        if (vec)
            { const cudaError_t e_ = launch_pdl(k_move_rw<false, true>, dim3(grid), dim3(BLOCK), (size_t)(0), st, a, N, p, pr, stepk, t, m, m_prev, seed, noise, err); if (e_ != cudaSuccess) return e_; }
        else
            { const cudaError_t e_ = launch_pdl(k_move_rw<false, false>, dim3(grid), dim3(BLOCK), (size_t)(0), st, a, N, p, pr, stepk, t, m, m_prev, seed, noise, err); if (e_ != cudaSuccess) return e_; }
    }
    return cudaGetLastError();
}

cudaError_t launch_move_mala(const MoveArgs& a, bool decide, int64_t N, int p, PriorArgs pr, const float4* stepk, int t,
                             uint32_t m, uint32_t m_prev, const uint64_t* seed, uint32_t* err, cudaStream_t st)
{
    const bool vec = (p & 3) == 0;
    cudaLaunchConfig_t cfg = pdl_config(warps_grid(N), BLOCK, st);  // follows the gradient finish or the scales
    cudaLaunchAttribute attr[1];
    pdl_attr(cfg, attr);
    const bool parts = a.gp.gpart != nullptr;
    auto* kern = vec ? k_move_mala<false, true, false> : k_move_mala<false, false, false>;
    if (decide && parts)
        kern = vec ? k_move_mala<true, true, true> : k_move_mala<true, false, true>;
    else if (decide)
        kern = vec ? k_move_mala<true, true, false> : k_move_mala<true, false, false>;
    return cudaLaunchKernelEx(&cfg, kern, a, N, p, pr, stepk, t, m, m_prev, seed, err);
}

cudaError_t launch_move_commit(const MoveArgs& a, bool mala, int64_t N, int p, PriorArgs pr, const float4* stepk, int t,
                               uint32_t m_prev, const uint64_t* seed, uint32_t* err, cudaStream_t st)
{
    const bool vec = (p & 3) == 0;
    cudaLaunchConfig_t cfg = pdl_config(warps_grid(N), BLOCK, st);  // follows the likelihood GEMM
    cudaLaunchAttribute attr[1];
    pdl_attr(cfg, attr);
    const bool parts = mala && a.gp.gpart != nullptr;
    auto* kern = vec ? k_move_commit<false, true, false> : k_move_commit<false, false, false>;
    if (parts)
        kern = vec ? k_move_commit<true, true, true> : k_move_commit<true, false, true>;
    else if (mala)
        kern = vec ? k_move_commit<true, true, false> : k_move_commit<true, false, false>;
    return cudaLaunchKernelEx(&cfg, kern, a, N, p, pr, stepk, t, m_prev, seed, err);
}

cudaError_t launch_finish_loglik(const MhState& s, int64_t N, double* logw, double* ll_out, uint32_t* err,
                                 cudaStream_t st)
{
    k_finish_loglik<<<warps_grid(N), BLOCK, 0, st>>>(s, N, logw, ll_out, err);
    return cudaGetLastError();
}

cudaError_t launch_commit_reweight(const MoveArgs& a, bool mala, int64_t N, int p, PriorArgs pr, const float4* stepk, int t,
                                   uint32_t m_prev, double* logw, const ReweightK* rk, uint32_t* err, cudaStream_t st)
{
    const bool vec = (p & 3) == 0;
    const dim3 grid(warps_grid(N)), block(BLOCK);
    const bool parts = mala && a.gp.gpart != nullptr;
    auto* kern = vec ? k_commit_reweight<false, true, false> : k_commit_reweight<false, false, false>;
    if (parts)
        kern = vec ? k_commit_reweight<true, true, true> : k_commit_reweight<true, false, true>;
    else if (mala)
        kern = vec ? k_commit_reweight<true, true, false> : k_commit_reweight<true, false, false>;
    return launch_pdl(kern, grid, block, (size_t)0, st, a, N, p, pr, stepk, t, m_prev, logw, rk, err);
}

cudaError_t launch_reweight(const float* beta, double* logw, float2* lpq, int64_t N, int p, PriorArgs pr,
                            const ReweightK* rk, int t, uint32_t* err, cudaStream_t st)
{
    { const cudaError_t e_ = launch_pdl(k_reweight, dim3((unsigned)((N + RW_PER_BLOCK - 1) / RW_PER_BLOCK)), dim3(RW_THREADS), (size_t)(0), st, beta, logw, lpq, N, p, pr, rk,
                                                                                         t, err); if (e_ != cudaSuccess) return e_; }
    return cudaGetLastError();
}

cudaError_t launch_lse(const double* logw, int64_t N, double* scratch, cudaStream_t st)
{
    return launch_pdl(k_lse_partial, dim3((unsigned)lse_blocks(N)), dim3(LSE_THREADS), (size_t)0, st, logw, N, scratch);
}

cudaError_t launch_normalise(const WeightArrays& w, int64_t N, const double* scratch, const LseOut& out, double* lam,
                             const unsigned long long* acc, double denom, cudaStream_t st)
{
    // one FP64 exp per weight: blocks of 64 spread them over the SMs' FP64 units; no more blocks than
    // fill them, since each combines the partials first
    const unsigned nb = (unsigned)std::min<int64_t>((N + NORM_THREADS - 1) / NORM_THREADS, 1024);
    return launch_pdl(k_normalise, dim3(nb), dim3(NORM_THREADS), (size_t)0, st, w, N, scratch, (int)lse_blocks(N), out, lam, acc,
                      denom);
}

cudaError_t launch_weight_forms(const double* W, int64_t N, float* Wf, uint32_t* wfix, cudaStream_t st)
{
    k_weight_forms<<<elem_grid(N), 256, 0, st>>>(W, N, Wf, wfix);
    return cudaGetLastError();
}

cudaError_t launch_mark_uniform(int64_t N, int t, double* ess_out, uint8_t* resampled_out, int* flag, cudaStream_t st)
{
    k_mark_uniform<<<1, 32, 0, st>>>(N, t, ess_out, resampled_out, flag);
    return cudaGetLastError();
}

cudaError_t launch_resample_index(const double* W, int64_t N, double* cum, int32_t* idx, const int* flag, int t,
                                  const uint64_t* seed, double u_override, cudaStream_t st)
{
    const int64_t chunks = (N + RS_BLOCK - 1) / RS_BLOCK;
    const unsigned local_grid = (unsigned)((chunks + RS_CHUNKS - 1) / RS_CHUNKS);
    cudaError_t e = launch_pdl(k_resample_local, dim3(local_grid), dim3(32 * RS_CHUNKS), (size_t)0, st, W, N, cum,
                               flag);
    if (e == cudaSuccess)
        e = launch_pdl(k_resample_carry, dim3(1), dim3(32), (size_t)0, st, N, cum, flag, t, seed,
                       u_override);
    if (e == cudaSuccess)
        e = launch_pdl(k_resample_search, dim3(elem_grid(N)), dim3(256), (size_t)0, st, cum, N, idx, flag);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

bool resample_gather_fits(int64_t N) { return (N + RS_BLOCK - 1) / RS_BLOCK <= RG_MAX_BLOCKS; }

cudaError_t launch_resample_gather(const double* W, int64_t N, double* cum, const int* flag, int t, const uint64_t* seed,
                                   const float* beta, float* beta_tmp, const float2* llq, const float2* lpq, float2* llq_tmp,
                                   float2* lpq_tmp, const float* g, float* g_tmp, int p, cudaStream_t st)
{
    const int64_t chunks = (N + RS_BLOCK - 1) / RS_BLOCK;
    const cudaError_t e = launch_pdl(k_resample_local, dim3((unsigned)((chunks + RS_CHUNKS - 1) / RS_CHUNKS)),
                                     dim3(32 * RS_CHUNKS), (size_t)0, st, W, N, cum, flag);
    if (e != cudaSuccess) return e;
    const dim3 grid(warps_grid(N)), block(BLOCK);
    if ((p & 3) == 0)
        return launch_pdl(k_resample_gather<true>, grid, block, (size_t)0, st, cum, t, seed, beta, beta_tmp, llq, lpq, llq_tmp,
                          lpq_tmp, g, g_tmp, N, p, flag);
    return launch_pdl(k_resample_gather<false>, grid, block, (size_t)0, st, cum, t, seed, beta, beta_tmp, llq, lpq, llq_tmp,
                      lpq_tmp, g, g_tmp, N, p, flag);
}

cudaError_t launch_gather(const int32_t* idx, const float* beta, float* beta_tmp, const float2* llq, const float2* lpq,
                          float2* llq_tmp, float2* lpq_tmp, const float* g, float* g_tmp, int64_t N, int p,
                          const int* flag, cudaStream_t st)
{
    if ((p & 3) == 0)
        { const cudaError_t e_ = launch_pdl(k_gather<true>, dim3(warps_grid(N)), dim3(BLOCK), (size_t)(0), st, idx, beta, beta_tmp, llq, lpq, llq_tmp, lpq_tmp, g, g_tmp, N, p,
                                                        flag); if (e_ != cudaSuccess) return e_; }
    else
        { const cudaError_t e_ = launch_pdl(k_gather<false>, dim3(warps_grid(N)), dim3(BLOCK), (size_t)(0), st, idx, beta, beta_tmp, llq, lpq, llq_tmp, lpq_tmp, g, g_tmp, N, p,
                                                         flag); if (e_ != cudaSuccess) return e_; }
    return cudaGetLastError();
}

// uniform weights after resampling: log(1/N), 1/N and round(2^31 / N), formed on the host
UniformWeights uniform_weights(int64_t N)
{
    const double wi = 1.0 / (double)N;
    return UniformWeights{-std::log((double)N), wi, (uint32_t)std::llrint(wi * 2147483648.0)};
}

cudaError_t launch_copyback(float* beta, const float* beta_tmp, float2* llq, float2* lpq, const float2* llq_tmp,
                            const float2* lpq_tmp, float* g, const float* g_tmp, const WeightArrays& w, int64_t N, int p,
                            const int* flag, cudaStream_t st)
{
    const UniformWeights u = uniform_weights(N);
    const double wi = u.wi, lw = u.lw;
    const uint32_t wf = u.wf;
    if ((p & 3) == 0)
        { const cudaError_t e_ = launch_pdl(k_copyback<true>, dim3(warps_grid(N)), dim3(BLOCK), (size_t)(0), st, beta, beta_tmp, llq, lpq, llq_tmp, lpq_tmp, g, g_tmp, w, N, p,
                                                          flag, lw, wi, wf); if (e_ != cudaSuccess) return e_; }
    else
        { const cudaError_t e_ = launch_pdl(k_copyback<false>, dim3(warps_grid(N)), dim3(BLOCK), (size_t)(0), st, beta, beta_tmp, llq, lpq, llq_tmp, lpq_tmp, g, g_tmp, w, N, p,
                                                           flag, lw, wi, wf); if (e_ != cudaSuccess) return e_; }
    return cudaGetLastError();
}

cudaError_t launch_colstats(const float* beta, const float* Wf, int64_t N, int p, float4* part, float* scale_out,
                            int kind, double lam_const, const double* lam_dev, double sd_floor, const double* sched,
                            int t, float* h_out, cudaStream_t st, const float* beta_rs, const int* rs_flag)
{
    const float wi = (float)uniform_weights(N).wi;
    const double rw_factor = lam_const / std::sqrt((double)p);  // the same FP64 quotient on the host
    dim3 block(32, CS_ROWS);
    dim3 grid((unsigned)((p + 31) / 32), COLSTAT_SPLITS);
    { const cudaError_t e_ = launch_pdl(k_colstats_partial, dim3(grid), dim3(block), (size_t)(0), st, beta, Wf, N, p, part, beta_rs, rs_flag, wi); if (e_ != cudaSuccess) return e_; }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // one warp (and block) per coordinate: its FP64 sums and square roots on their own SM
    { const cudaError_t e_ = launch_pdl(k_colstats_finish, dim3((unsigned)p), dim3(32), (size_t)(0), st, part, p, COLSTAT_SPLITS, scale_out, kind, rw_factor,
                                                               lam_dev, sd_floor, sched, t, h_out,
                                                               std::pow((double)p, -1.0 / 6.0)); if (e_ != cudaSuccess) return e_; }
    return cudaGetLastError();
}

cudaError_t launch_keys(const float* beta, const float* Wf, const uint32_t* wfix, int64_t N, int p, uint32_t* keysT,
                        float* WfS, uint32_t* wfixS, bool pdl, cudaStream_t st)
{
    const dim3 grid((unsigned)((N + 31) / 32), (unsigned)((p + 31) / 32)), block(32, 8);
    if (pdl) return launch_pdl(k_keys_transpose, grid, block, (size_t)0, st, beta, N, p, keysT, Wf, wfix, WfS, wfixS);
    k_keys_transpose<<<grid, block, 0, st>>>(beta, N, p, keysT, Wf, wfix, WfS, wfixS);
    return cudaGetLastError();
}

cudaError_t launch_summaries_keys(const uint32_t* keysT, const float* Wf, const uint32_t* wfix, int64_t N, int p,
                                  const SummaryArgs& s, int t, double* mean, double* quant, double* conc, bool pdl,
                                  cudaStream_t st)
{
    SummaryArgs a = s;
    // host-side constants: the smallest float >= Delta (the open interval |b| < Delta tested
    // in FP32) and the fixed-point quantile targets ceil(q 2^31)
    for (int d = 0; d < 8; ++d) {
        float f = (float)a.delta[d];
        if ((double)f < a.delta[d]) f = std::nextafter(f, INFINITY);
        a.dthr[d] = f;
    }
    for (int q = 0; q < 8; ++q) a.target[q] = (unsigned long long)std::ceil(a.q[q] * 2147483648.0);
    const int nh = (quant && s.nq > 0) ? (s.nq > SUM_SUB ? s.nq : SUM_SUB) : 0;
    const size_t bytes = (size_t)nh * SUM_BINS * sizeof(uint32_t);
    auto* kern = (s.nq <= 4 && s.nd <= 2) ? k_summaries<4, 2> : k_summaries<8, 8>;
    if (pdl)
        return launch_pdl(kern, dim3((unsigned)p), dim3(SUM_THREADS), bytes, st, keysT, Wf, wfix, N, p, a, t, mean, quant,
                          conc);
    kern<<<(unsigned)p, SUM_THREADS, bytes, st>>>(keysT, Wf, wfix, N, p, a, t, mean, quant, conc);
    return cudaGetLastError();
}

cudaError_t launch_summaries(const float* beta, const float* Wf, const uint32_t* wfix, int64_t N, int p,
                             const SummaryArgs& s, int t, double* mean, double* quant, double* conc, uint32_t* keysT,
                             cudaStream_t st)
{
    const cudaError_t e = launch_keys(beta, Wf, wfix, N, p, keysT, nullptr, nullptr, true, st);
    if (e != cudaSuccess) return e;
    return launch_summaries_keys(keysT, Wf, wfix, N, p, s, t, mean, quant, conc, true, st);
}

cudaError_t launch_marginal(const double* log_z_inc, const double* mean, const double* conc, int64_t T, int64_t p,
                            int D, double* post_c, double* mean_out, double* conc_out, cudaStream_t st)
{
    k_marginal_weights<<<1, 32, 0, st>>>(log_z_inc, T, post_c);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t work = p * (1 + D);
    k_marginal_apply<<<(unsigned)((work + 127) / 128), 128, 0, st>>>(post_c, mean, conc, T, p, D, mean_out, conc_out);
    return cudaGetLastError();
}

cudaError_t launch_accept_rate(const unsigned long long* acc, int T, double denom, double* rate, cudaStream_t st)
{
    k_accept_rate<<<(T + 127) / 128, 128, 0, st>>>(acc, T, denom, rate);
    return cudaGetLastError();
}

cudaError_t launch_adapt_lambda(double* lam, const unsigned long long* acc, double denom, cudaStream_t st)
{
    k_adapt_lambda<<<1, 32, 0, st>>>(lam, acc, denom);
    return cudaGetLastError();
}

cudaError_t launch_set_f64(double* ptr, double v, cudaStream_t st)
{
    k_set_f64<<<1, 32, 0, st>>>(ptr, v);
    return cudaGetLastError();
}

cudaError_t launch_philox(const uint32_t* ctr, uint2 key, int64_t count, uint32_t* out, cudaStream_t st)
{
    k_philox<<<(unsigned)((count + 127) / 128), 128, 0, st>>>(ctr, key, count, out);
    return cudaGetLastError();
}

cudaError_t launch_normals(uint64_t seed, uint32_t particle, uint32_t t, uint32_t m, int64_t p, float* out,
                           cudaStream_t st)
{
    const int64_t groups = (p + 3) / 4;
    k_normals<<<(unsigned)((groups + 127) / 128), 128, 0, st>>>(seed, particle, t, m, p, out);
    return cudaGetLastError();
}

cudaError_t launch_prior_sample(uint64_t seed, PriorArgs pr, double c, int64_t N, int64_t p, float* out,
                                cudaStream_t st)
{
    k_prior_sample<<<elem_grid(N * p), 256, 0, st>>>(seed, pr, (float)c, N, p, out);
    return cudaGetLastError();
}

cudaError_t launch_prior_logpdf(PriorArgs pr, double c, const float* beta, int64_t k, double* out, cudaStream_t st)
{
    k_prior_logpdf<<<(unsigned)((k + 255) / 256), 256, 0, st>>>(pr, c, beta, k, out);
    return cudaGetLastError();
}

}  // namespace spa
