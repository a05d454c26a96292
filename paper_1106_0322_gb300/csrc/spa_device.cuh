// spa_device.cuh -- device helpers shared by the library's kernels (sm_103a).
//
// Random numbers: Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11), one round
// (x0,x1,x2,x3) -> (hi(B x2) ^ x1 ^ k0, lo(B x2), hi(A x0) ^ x3 ^ k1, lo(A x0)),
// A = 0xD2511F53, B = 0xCD9E8D57, key bumped by (0x9E3779B9, 0xBB67AE85) between
// rounds. The stream layout (counter = what is drawn) is a specification:
//   init prior draws   (j/2, particle, 0, 1<<16)      u[2(j%2)] -> V_j, u[2(j%2)+1] bit 31 -> sign
//   move normals       (j/4, particle, t, 2<<16 | m)  Box-Muller on (u0,u1), (u2,u3)
//   MH uniform         (0,   particle, t, 3<<16 | m)  u0
//   resampling uniform (0,   0,        t, 4<<16)      u0
// key = (seed & 0xffffffff, seed >> 32). Open uniforms are (k + 1/2) 2^-23 with k the
// top 23 bits (exact in FP32); the resampling uniform is (top 24 bits) 2^-24 in [0,1).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cfloat>

namespace spa {

// ------------------------------------------------------------------ error word bits
enum : uint32_t {
    DERR_NONFINITE = 1u,  // non-finite log-likelihood or log-weight
    DERR_TIMEOUT = 2u,    // a bounded wait gave up
    DERR_INPUT = 4u,      // invalid input data found on the device
    DERR_ESS = 8u,        // ESS < 1 (all weights non-finite)
};

constexpr uint32_t TAG_INIT = 1u, TAG_NORMAL = 2u, TAG_ACCEPT = 3u, TAG_RESAMPLE = 4u, TAG_SITE = 5u;

// ---------------------------------------------------------------------- Philox
__device__ __forceinline__ uint4 philox4x32_10(uint4 x, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const uint32_t hiA = __umulhi(0xD2511F53u, x.x), loA = 0xD2511F53u * x.x;
        const uint32_t hiB = __umulhi(0xCD9E8D57u, x.z), loB = 0xCD9E8D57u * x.z;
        x = make_uint4(hiB ^ x.y ^ k.x, loB, hiA ^ x.w ^ k.y, loA);
    }
    return x;
}

__device__ __forceinline__ uint2 seed_key(uint64_t seed)
{
    return make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
}

// (k + 1/2) 2^-23, k = top 23 bits: exact in single precision, in (0,1). As 1 + k 2^-23, whose bits are
// those of 1 with k in the mantissa, less 1 - 2^-24 (exact: the difference has 24 bits); no
// conversion, which the units for logarithms and roots would have to make. With the packed split of
// pack_coord4, the RW move kernel at p = 200, N = 8192: 1233 -> 1148 instructions a warp, 16.6 -> 15.7 us
// alone.
__device__ __forceinline__ float u01_open_f(uint32_t u) { return __uint_as_float((u >> 9) + 0x3F800000u) - 0.999999940395355224609375f; }
// The same by conversion, for the single-coordinate kernel: one lane per update converts there, and at
// that kernel's register limit the other form cost more (23.8 against 22.5 ms for 5 steps at n = 1859,
// p = 184).
__device__ __forceinline__ float u01_open_cvt_f(uint32_t u) { return ((float)(u >> 9) + 0.5f) * 1.1920928955078125e-7f; }
// twice that, in (0,2)
__device__ __forceinline__ float u02_open_f(uint32_t u) { return __uint_as_float((u >> 9) + 0x40000000u) - 1.99999988079071044921875f; }
__device__ __forceinline__ double u01_open_d(uint32_t u) { return ((double)(u >> 9) + 0.5) * 1.1920928955078125e-7; }
// top 24 bits / 2^24 in [0,1)
__device__ __forceinline__ double u01_d(uint32_t u) { return (double)(u >> 8) * 5.9604644775390625e-8; }

// Four standard normals (Box-Muller) of one Philox block.
__device__ __forceinline__ float4 normals4(uint64_t seed, uint32_t blk, uint32_t particle, uint32_t t, uint32_t m)
{
    const uint4 u = philox4x32_10(make_uint4(blk, particle, t, (TAG_NORMAL << 16) | m), seed_key(seed));
    float s0, c0, s1, c1;
    const float r0 = sqrtf(-2.0f * logf(u01_open_f(u.x)));
    const float r1 = sqrtf(-2.0f * logf(u01_open_f(u.z)));
    sincospif(u02_open_f(u.y), &s0, &c0);
    sincospif(u02_open_f(u.w), &s1, &c1);
    return make_float4(r0 * c0, r0 * s0, r1 * c1, r1 * s1);
}

// One draw from Gt(a, c) (a = +inf: double exponential) by inversion of the tail
// P(|beta| > x) = (1 + x/(a c))^-a: |beta| = a c (V^{-1/a} - 1) = a c expm1(-log(V)/a).
__device__ __forceinline__ float prior_draw(uint64_t seed, uint32_t particle, uint32_t j, float a, float c, bool de)
{
    const uint4 u = philox4x32_10(make_uint4(j >> 1, particle, 0u, TAG_INIT << 16), seed_key(seed));
    const uint32_t uv = (j & 1u) ? u.z : u.x;
    const uint32_t us = (j & 1u) ? u.w : u.y;
    const float lv = logf(u01_open_f(uv));
    const float mag = de ? -c * lv : a * c * expm1f(-lv / a);
    return (us >> 31) ? -mag : mag;
}

// ------------------------------------------------- compensated FP32 summation
// A float pair (s, c) whose value is s + c. Each addition uses the error-free TwoSum
// transformation (Knuth; Moller), so a sum of k terms carries an error of about
// 2^-24 |sum| + k 2^-48 sum|x|: double-like accuracy at FP32 cost. On GB300 the
// CUDA-core FP64 rate is a small fraction of FP32, so per-element sums use this.
struct FSum {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        const float t = s + x;
        const float z = t - s;
        c += (s - (t - z)) + (x - z);
        s = t;
    }
    __device__ __forceinline__ void add(FSum o)
    {
        add(o.s);
        c += o.c;
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

__device__ __forceinline__ FSum warp_sum(FSum v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        FSum w;
        w.s = __shfl_xor_sync(0xffffffffu, v.s, o);
        w.c = __shfl_xor_sync(0xffffffffu, v.c, o);
        v.add(w);
    }
    return v;
}

// ---------------------------------------------------------- reductions / helpers
template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16& hi, __nv_bfloat16& lo)
{
    hi = __float2bfloat16_rn(x);
    lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// Programmatic dependent launch: a kernel launched with programmatic stream serialization
// may start before its predecessor finishes; this waits until the predecessor grid has
// completed and its memory is visible (a no-op for kernels launched without the attribute).
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's blocks be scheduled once every block of this grid has passed here
// (they still wait for this grid's completion before reading its results).
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// -------------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// The default limit of a bounded wait (a context can set another, spa_set_wait_limit).
constexpr uint64_t WAIT_LIMIT_DEFAULT_NS = 4000000000ull;
// The limit of a drain: the wait for a CTA's own copies and MMAs in flight before it frees
// TMEM and exits.
constexpr uint64_t DRAIN_LIMIT_NS = 100000000ull;

// Wait until the phase with the given parity of barrier `bar` has completed. Gives up
// after `limit_ns` (setting DERR_TIMEOUT) or as soon as another thread has given up.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint32_t* err,
                                                  uint64_t limit_ns = WAIT_LIMIT_DEFAULT_NS)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t spin = 1;; ++spin) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((spin & 63u) == 0u) {
            if (*reinterpret_cast<volatile uint32_t*>(err) & DERR_TIMEOUT) return false;
            if (globaltimer_ns() - t0 > limit_ns) {
                atomicOr(err, DERR_TIMEOUT);
                return false;
            }
        }
    }
}

// The drain before a CTA frees TMEM or exits: wait for this CTA's own asynchronous work
// (TMA copies into its shared memory, its MMAs) to complete. Unlike mbar_wait_bounded it does
// not stop when another thread has given up -- that is exactly when the work in flight must
// still land -- and only its own limit (DRAIN_LIMIT_NS) ends it.
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity, uint32_t* err)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t spin = 1;; ++spin) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((spin & 63u) == 0u && globaltimer_ns() - t0 > DRAIN_LIMIT_NS) {
            atomicOr(err, DERR_TIMEOUT);
            return false;
        }
    }
}

// ------------------------------------------------------------------------- TMA
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// 2-D tiled load of the box at element coordinates (x = innermost, y) into shared memory,
// completing `bytes` on barrier `bar`. x * element size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t x, int32_t y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// An L2 cache policy under which the lines an access touches become the first candidates
// for eviction (for data read for the last time).
__device__ __forceinline__ uint64_t l2_policy_evict_first()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// tma_load_2d with an L2 cache-policy hint for the lines it reads.
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int32_t x, int32_t y,
                                                 uint64_t pol)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar), "l"(pol)
        : "memory");
}

// --------------------------------------------------------------------- tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor (sm_100 format) of a K-major BF16 operand tile whose rows are
// one swizzle span of row_bytes: 128 (64 columns, 128-byte swizzle), 64 (64-byte) or 32 (32-byte):
//   [0,14) start address >> 4, [16,30) leading byte offset >> 4 (unused here),
//   [32,46) stride byte offset >> 4 (8 rows), [46,48) = 1, [61,64) layout = 2, 4 or 6.
// The tile base must be 1024-byte aligned. Kept as two words: the low one (start address)
// advances with the operand (2 per K = 16 step), the high one is fixed by the row size.
__device__ __forceinline__ uint32_t sdesc_lo(uint32_t smem_addr) { return ((smem_addr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ uint32_t sdesc_hi(uint32_t row_bytes)
{
    const uint32_t layout = row_bytes == 128u ? 2u : (row_bytes == 64u ? 4u : 6u);
    return ((8u * row_bytes) >> 4) | (1u << 14) | (layout << 29);
}
__device__ __forceinline__ uint64_t sdesc_make(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }

// Instruction descriptor of kind::f16 with BF16 A and B (both K-major), FP32 accumulate:
//   [4,6) D format = 1 (F32), [7,10) A = 1 (BF16), [10,13) B = 1 (BF16),
//   [15] A major = 0 (K), [16] B major = 0 (K), [17,23) N >> 3, [24,29) M >> 4.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(uint32_t M, uint32_t N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem]^T for one K = 16 slice; accumulate != 0 adds to D. For a whole
// warp in step: only the lane with `issue` set issues. With the loop and
// its operands uniform over the warp the descriptors stay in uniform registers; inside an
// `if (lane == 0)` each MMA first moves them there one by one, and the issue, not the tensor
// core, sets the pace.
__device__ __forceinline__ void umma_bf16_if(uint32_t issue, uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(issue)
        : "memory");
}

// One lane of a converged warp. In an `if (elect_one())` block the compiler knows that a single
// lane runs and that the block's operands are uniform: a run of unrolled MMAs there issues every
// 47 cycles, against 71 to 77 predicated one by one (umma_bf16_if) and 92 to 103 in a loop inside
// `if (lane == 0)` (128 x 128 x 16, measured with a stand-alone issue loop; the tensor core takes 65).
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}
// D[tmem] (+)= A[smem] * B[smem]^T, or A[tmem], for one K = 16 slice, issued by the calling lane.
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive once on `bar` when every tcgen05.mma issued so far by the calling lane has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem]^T for one K = 16 slice, A read from tensor memory: row m of
// A in lane m, K packed two BF16 per 32-bit column (even k in the low half), 8 columns per slice.
// Issued as umma_bf16_if.
__device__ __forceinline__ void umma_bf16_ta_if(uint32_t issue, uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc,
                                                uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(issue)
        : "memory");
}

// Each thread of the warp writes 4 consecutive 32-bit columns of its TMEM lane (the warp's
// 32 lanes start at taddr's lane field); tmem_wait_st() before the writes are relied on.
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint4 v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(v.x), "r"(v.y),
                 "r"(v.z), "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Arrive once on `bar` when every tcgen05.mma issued so far by the lane with `issue` set has
// completed (a whole warp in step).
__device__ __forceinline__ void umma_commit_if(uint32_t issue, uint32_t bar)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar),
        "r"(issue)
        : "memory");
}

// Each thread of the warp reads 32 consecutive 32-bit columns of its TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Asynchronous form: issue the load into r, then tmem_wait_ld(r) before reading r. The
// wait names r as in/out operands so the compiler cannot move reads of r above it.
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

// ------------------------------------------------------------ fast base-2 math
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// softplus in base-2 units: log2(1 + 2^x) = max(x, 0) + log2(1 + 2^-|x|).
__device__ __forceinline__ float softplus2(float x)
{
    return fmaxf(x, 0.0f) + lg2_approx(1.0f + ex2_approx(-fabsf(x)));
}

// ------------------------------------------------------- packed FP32 pairs
// Two FP32 operations in one instruction, each rounded as its scalar form rounds.
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
// Two FP32 fused multiply-adds in one instruction, each rounded as fmaf rounds.
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// A sum tree over 32 columns as 16 column pairs (2q, 2q + 1): column k is added to k + 16, then
// k + 8, 4, 2 and 1. Pairs are produced in bit-reversed order, so that each level's two terms
// follow each other and at most five partial sums are live; all levels but the last are
// packed additions.
__host__ __device__ constexpr int tree_pair(int j)
{
    return ((j & 1) << 3) | ((j & 2) << 1) | ((j & 4) >> 1) | ((j & 8) >> 3);
}
struct PairTree {
    uint64_t part[5];
    // the j-th pair produced (j a compile-time constant after unrolling)
    __device__ __forceinline__ void add(int j, uint64_t v)
    {
        int level = 0;
#pragma unroll
        for (int m = j; m & 1; m >>= 1) {
            v = add2(part[level], v);
            ++level;
        }
        part[level] = v;
    }
    __device__ __forceinline__ float sum() const
    {
        const float2 r = unpack2(part[4]);
        return r.x + r.y;
    }
};

// Sum over the first `valid` of 32 columns of softplus2(eta2) = log2(1 + 2^eta2): 32
// independent ex2/lg2 pairs, then a tree. The SFU bounds it: two operations a column, 16 lanes a
// cycle and SM, 2.0 us per 128 x 256 tile. (Packed additions in PairTree's order save 1.5
// instructions a column but were 1.5% slower over a sweep, n = 5000, p = 500: the independent
// pairs keep the SFU busier. One lg2 of the product of the (1 + 2^-|eta2|) factors was slower too,
// as a running product and as a product tree.)
__device__ __forceinline__ float sum_sp2_32(const uint32_t (&r)[32], int valid)
{
    float t[32];
    if (valid >= 32) {
#pragma unroll
        for (int k = 0; k < 32; ++k) t[k] = softplus2(__uint_as_float(r[k]));
    } else {
#pragma unroll
        for (int k = 0; k < 32; ++k) t[k] = (k < valid) ? softplus2(__uint_as_float(r[k])) : 0.0f;
    }
#pragma unroll
    for (int w = 16; w > 0; w >>= 1)
#pragma unroll
        for (int k = 0; k < w; ++k) t[k] += t[k + w];
    return t[0];
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The residual pass's work on a chunk of 32 individuals of one particle: the softplus sum
// (returned), and r = y - logit^{-1}(eta) as BF16 hi and lo pairs (column 2q in the low half of
// word q) and its sum. eta2 = eta log2(e): with e = 2^-|eta2|, softplus2 = max(eta2, 0) +
// log2(1 + e) and logit^{-1}(eta) = 1/(1 + e) for eta >= 0, e/(1 + e) otherwise (one ex2 shared).
// FULL: all 32 columns are individuals (every chunk but the last of a region's row), so no
// column needs the valid-count test. YV: the phenotypes come as floats (yv, 16-byte aligned, FULL
// only), else from the bits of ybits.
template <bool FULL, bool YV = false>
__device__ __forceinline__ float resid_chunk(const uint32_t (&x2)[32], int valid, uint32_t ybits, const float* yv,
                                             uint32_t (&hi2)[16], uint32_t (&lo2)[16], float& rsum)
{
    const uint64_t one = pack2(1.0f, 1.0f), negone = pack2(-1.0f, -1.0f);
    PairTree ts, tr;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int q = tree_pair(j), k = 2 * q;
        const float x0 = __uint_as_float(x2[k]), x1 = __uint_as_float(x2[k + 1]);
        const float e0 = ex2_approx(-fabsf(x0)), e1 = ex2_approx(-fabsf(x1));
        const float2 o = unpack2(add2(one, pack2(e0, e1)));
        // sigma: the numerator is 1 or e, so the product with 1/(1 + e) rounds as the two cases do
        const uint64_t sig = mul2(pack2(x0 >= 0.0f ? 1.0f : e0, x1 >= 0.0f ? 1.0f : e1), pack2(rcp_approx(o.x), rcp_approx(o.y)));
        uint64_t y;
        if (YV) {
            const float2 yf = __ldg(reinterpret_cast<const float2*>(yv + k));
            y = pack2(yf.x, yf.y);
        } else {
            y = pack2((ybits >> k) & 1u ? 1.0f : 0.0f, (ybits >> (k + 1)) & 1u ? 1.0f : 0.0f);
        }
        uint64_t r = fma2(sig, negone, y);
        uint64_t sp = add2(pack2(fmaxf(x0, 0.0f), fmaxf(x1, 0.0f)), pack2(lg2_approx(o.x), lg2_approx(o.y)));
        if (!FULL) {
            const bool in0 = k < valid, in1 = k + 1 < valid;
            const float2 rf = unpack2(r), sf = unpack2(sp);
            r = pack2(in0 ? rf.x : 0.0f, in1 ? rf.y : 0.0f);
            sp = pack2(in0 ? sf.x : 0.0f, in1 ? sf.y : 0.0f);
        }
        ts.add(j, sp);
        tr.add(j, r);
        const float2 rf = unpack2(r);
        const __nv_bfloat162 h = __floats2bfloat162_rn(rf.x, rf.y);
        const float2 hf = __bfloat1622float2(h);
        const float2 lf = unpack2(fma2(pack2(hf.x, hf.y), negone, r));
        const __nv_bfloat162 l = __floats2bfloat162_rn(lf.x, lf.y);
        hi2[q] = *reinterpret_cast<const uint32_t*>(&h);
        lo2[q] = *reinterpret_cast<const uint32_t*>(&l);
    }
    rsum = tr.sum();
    return ts.sum();
}

// ------------------------------------------------------------------- log prior
// One coordinate's term of the log prior (the -log(2c) constant dropped): Gt sums
// log1p(|b|/(a c)) and multiplies by -(a+1); the double exponential sums |b| and
// multiplies by -1/c.
__device__ __forceinline__ float prior_term(float b, float inv_ac, int de)
{
    const float x = fabsf(b);
    return de ? x : log1pf(x * inv_ac);
}

// The Gt terms of four coordinates at once: log1p(x0) + ... + log1p(x3) with x = |b|/(a c),
// as the logarithm of the product of the factors 1 + x_k (one logarithm instead of four).
// Each factor and product carries a relative rounding of 2^-24, so the sum is accurate to
// a few 1e-7 in absolute terms, about the same as four rounded log1p terms of moderate size.
// Products beyond FP32 range (factors near 1e9) take the four logarithms instead. Every
// kernel that forms a state's log-prior sum for the MH test (the moves, and the reweighting's
// sum at the new scale) uses this grouping when p % 4 == 0, so that the test compares one
// function of the state.
__device__ __forceinline__ float prior_terms4(float4 b, float inv_ac)
{
    const float f0 = fmaf(fabsf(b.x), inv_ac, 1.0f), f1 = fmaf(fabsf(b.y), inv_ac, 1.0f);
    const float f2 = fmaf(fabsf(b.z), inv_ac, 1.0f), f3 = fmaf(fabsf(b.w), inv_ac, 1.0f);
    const float q = (f0 * f1) * (f2 * f3);
    if (q <= FLT_MAX) return logf(q);
    return log1pf(fabsf(b.x) * inv_ac) + log1pf(fabsf(b.y) * inv_ac) + log1pf(fabsf(b.z) * inv_ac) +
           log1pf(fabsf(b.w) * inv_ac);
}

// ----------------------------------------------------------- float4 groups
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
// read-only path: per-coordinate constants no thread writes while the kernel runs
__device__ __forceinline__ float4 ldg4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ float comp(const float4& v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w)); }

}  // namespace spa
