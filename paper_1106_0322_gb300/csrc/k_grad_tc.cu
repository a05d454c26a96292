// k_grad_tc.cu -- log-likelihood and C = R G of one particle tile without R in memory.
//
// The gradient needs r = y - logit^{-1}(eta) contracted with the genotypes again:
// C[k, j] = sum_i r_ki g_ij. Written to memory and read back by a second GEMM (k_loglik_tc's
// residual mode, then k_adjoint_tc), r is N x 2 n BF16, 67 MB at N = 8192 and n = 2000. Here
// both contractions run in one CTA and r stays in tensor memory:
//
//   S  = A_tile [G, 1]^T   (tcgen05.mma, A and G in shared memory, 128 particles x 128 individuals)
//   r  = y - sigma(S)      (epilogue warps: also the softplus and residual sums per 32 individuals);
//                          the BF16 hi | lo split of r overwrites S in tensor memory
//   C += [r_hi | r_lo] G   (tcgen05.mma, r from tensor memory, G^T in shared memory)
//
// A unit is one particle tile against one K-split of the individuals (the adjoint's split, in
// 64-individual k-blocks, hi before lo in each), so C's partial sums, and with k_grad_finish
// the gradient, are bit for bit those of the two kernels. Two S buffers: while the epilogue
// turns tile i into r, the tensor core forms S of tile i + 1 and then adds tile i to C.
//
// What bounds it (n = 2000, p = 200, N = 8192; cycles of one CTA, 8 tiles): about 5500 a tile.
// S takes 3300 (26 MMAs of 65 to 77 and their waits), the epilogue 4000 (three SFU operations an
// element, 16 lanes a cycle, are 3070), C 1800, and a buffer goes round S, epilogue and C; before
// the first tile 6000 (A from L2), after the last 7000 (C to L2). With k_grad_finish 38.5 us, the
// two kernels and the finish 51.2; n = 3000, p = 128, N = 6000: 31.8 against 48.9 us.
#include "spa_device.cuh"
#include "spa_internal.h"

namespace spa {

namespace {

constexpr int GM = 128;                 // particles: TMEM lanes
constexpr int GT_N = 128;               // individuals per tile
constexpr int GK = 64;                  // individuals, or operand columns, per k-block
constexpr int G_EPI = 16;               // epilogue warps, four per lane quadrant: one per 32 individuals of a tile
constexpr int G_THREADS = 32 * (4 + G_EPI);  // warps: operand and G loads, S, epilogue, G^T loads, C
constexpr int G_MAX_STAGES = 6;
constexpr int G_T_STAGES = 2;
constexpr uint32_t G_STAGE = GT_N * 128u;               // one k-block of a G tile
constexpr uint32_t G_KB_BYTES = 2u * GM * 128u;         // A_hi and A_lo of a full k-block
constexpr uint32_t G_S_COL = 256;                       // TMEM columns: C from 0, S from 256 and 384
constexpr uint32_t G_XPOSE = 32 * 17 * 4;               // an epilogue warp's transpose buffer
constexpr int G_NBARS = 2 * G_MAX_STAGES + 2 * G_T_STAGES + 4 + 1 + 2 + 2 + 2 + 2 + 2 + 2;

// 16 consecutive 32-bit columns of each thread's TMEM lane.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// The MMAs of one k-block of S (the calling lane issues): A_hi, then A_lo, against the G tile.
__device__ __forceinline__ void s_block(const GradArgs& g, uint32_t d, uint32_t a, uint32_t gt, int kb, uint32_t hi128,
                                        uint32_t hi_tail, uint32_t half_tail)
{
    constexpr uint32_t IDESC_S = idesc_bf16_f32(GM, GT_N);
    const uint32_t a_lo = sdesc_lo(a), g_lo = sdesc_lo(gt);
    const int nks = g.ksteps - 4 * kb;
    if (nks >= 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            umma_bf16(d, sdesc_make(a_lo + 2u * q, hi128), sdesc_make(g_lo + 2u * q, hi128), IDESC_S, (kb | q) != 0 ? 1u : 0u);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            umma_bf16(d, sdesc_make(a_lo + GM * 8u + 2u * q, hi128), sdesc_make(g_lo + 2u * q, hi128), IDESC_S, 1u);
    } else {
        for (int q = 0; q < nks; ++q)
            umma_bf16(d, sdesc_make(a_lo + 2u * q, hi_tail), sdesc_make(g_lo + 2u * q, hi_tail), IDESC_S, (kb | q) != 0 ? 1u : 0u);
        for (int q = 0; q < nks; ++q)
            umma_bf16(d, sdesc_make(a_lo + half_tail + 2u * q, hi_tail), sdesc_make(g_lo + 2u * q, hi_tail), IDESC_S, 1u);
    }
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                   "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])::"memory");
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

__global__ void __launch_bounds__(G_THREADS, 1)
    k_grad_tc(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapAt,
              const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapBt,
              const __grid_constant__ CUtensorMap mapT, const GradArgs g)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;  // warp-uniform
    const uint32_t gst0 = sbase + g.a_bytes;                                 // G stages
    const uint32_t tst0 = gst0 + (uint32_t)g.stages * G_STAGE;               // G^T stages; C leaves through them or after them
    const uint32_t t_stage = (uint32_t)g.N2 * 128u;
    const uint32_t bar0 = tst0 + g.t_bytes;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + (bar0 - sbase) + 8 * G_NBARS);
    // barriers
    const uint32_t gfull = bar0, gempty = gfull + 8u * G_MAX_STAGES, tfull = gempty + 8u * G_MAX_STAGES;
    const uint32_t tempty = tfull + 8u * G_T_STAGES, afull = tempty + 8u * G_T_STAGES, aempty = afull + 32u;
    const uint32_t sfull = aempty + 8u, pfull = sfull + 16u, pfree = pfull + 16u, cfull = pfree + 16u, cempty = cfull + 16u;
    const uint32_t drain_bar = cempty + 16u;
    const int kb_last = g.kblocks - 1;
    const uint32_t tail_row = g.tw ? (uint32_t)g.tw * 2u : 128u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) {
            mbar_init(gfull + 8u * s, 1);
            mbar_init(gempty + 8u * s, 1);
        }
        for (int s = 0; s < G_T_STAGES; ++s) {
            mbar_init(tfull + 8u * s, 1);
            mbar_init(tempty + 8u * s, 1);
        }
        for (int k = 0; k < 4; ++k) mbar_init(afull + 8u * k, 1);
        mbar_init(aempty, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(sfull + 8u * b, 1);
            mbar_init(pfull + 8u * b, G_EPI);
            mbar_init(pfree + 8u * b, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(cfull + 8u * b, 1);
            mbar_init(cempty + 8u * b, G_EPI);
        }
        mbar_init(drain_bar, 1);
        mbar_init(drain_bar + 8u, 1);
        mbar_fence_init();
        tma_prefetch_desc(&mapA);
        tma_prefetch_desc(&mapB);
        tma_prefetch_desc(&mapT);
        if (g.tw) {
            tma_prefetch_desc(&mapAt);
            tma_prefetch_desc(&mapBt);
        }
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // unit u = (particle tile, K-split), the split fastest; its k-blocks [k0, k1) of individuals.
    // A CTA takes a contiguous range of units, and A stays while the particle tile does.
    const int units = g.m_tiles * g.ksplit;
    const int u0 = (int)((int64_t)units * blockIdx.x / gridDim.x), u1 = (int)((int64_t)units * (blockIdx.x + 1) / gridDim.x);
    auto split = [&](int u, int& mt, int& ks, int& k0, int& k1) {
        ks = u % g.ksplit;
        mt = u / g.ksplit;
        k0 = (int)((int64_t)g.kb_n * ks / g.ksplit);
        k1 = (int)((int64_t)g.kb_n * (ks + 1) / g.ksplit);
    };

    if (warp == 0) {
        // ------------------------------------------- particle operand and G tiles
        if (lane == 0) {
            // G's k-blocks in the order the units need them; the genotypes were there before the
            // sweep, so the first ones go out before the previous kernel (which writes A) is done
            uint32_t it = 0, s = 0, ph = 1u;
            int done = 0;
            int a_mt = -1, a_tiles = 0, a_issued = 0;  // particle tiles whose A was sent out; the last one's k-blocks
            bool ok = true;
            auto load_g = [&](int k, int kb) {
                const bool tail = g.tw && kb == kb_last;
                if (!mbar_wait_bounded(gempty + 8u * s, ph, g.err, g.wait_ns)) {
                    ok = false;
                    return;
                }
                mbar_arrive_expect_tx(gfull + 8u * s, GT_N * (tail ? tail_row : 128u));
                tma_load_2d(gst0 + s * G_STAGE, tail ? &mapBt : &mapB, gfull + 8u * s, kb * GK, k * GK);
                ++it;
                if (++s == (uint32_t)g.stages) {
                    s = 0;
                    ph ^= 1u;
                }
            };
            const int early = min(g.stages, g.kblocks);
            if (u0 < u1) {
                int mt, ks, k0, k1;
                split(u0, mt, ks, k0, k1);
                for (int kb = 0; kb < early && ok; ++kb) load_g(k0, kb);
            }
            grid_dependency_wait();
            for (int u = u0; u < u1 && ok; ++u) {
                int mt, ks, k0, k1;
                split(u, mt, ks, k0, k1);
                if (mt != a_mt) {
                    // the S of the previous particle tile are done with A
                    if (a_tiles > 0 && !mbar_wait_bounded(aempty, (uint32_t)((a_tiles - 1) & 1), g.err, g.wait_ns)) break;
                    a_mt = mt;
                    ++a_tiles;
                    a_issued = 0;
                    for (int kb = 0; kb < g.kblocks; ++kb) {
                        const bool tail = g.tw && kb == kb_last;
                        const uint32_t a = sbase + (uint32_t)kb * G_KB_BYTES, half = GM * (tail ? tail_row : 128u);
                        const CUtensorMap* ma = tail ? &mapAt : &mapA;
                        mbar_arrive_expect_tx(afull + 8u * kb, 2u * half);
                        tma_load_2d(a, ma, afull + 8u * kb, kb * GK, mt * GM);
                        tma_load_2d(a + half, ma, afull + 8u * kb, g.Kp + kb * GK, mt * GM);
                        ++a_issued;
                    }
                }
                for (int k = k0; k < k1 && ok; k += 2)
                    for (int kb = (done == 0 && k == k0) ? early : 0; kb < g.kblocks && ok; ++kb) load_g(k, kb);
                ++done;
            }
            // never leave with a copy in flight
            const uint32_t last = it < (uint32_t)g.stages ? it : (uint32_t)g.stages;
            for (uint32_t q = 1; q <= last; ++q) {
                const uint32_t i2 = it - q;
                mbar_drain(gfull + 8u * (i2 % (uint32_t)g.stages), (i2 / (uint32_t)g.stages) & 1u, g.err);
            }
            for (int kb = 0; kb < a_issued; ++kb) mbar_drain(afull + 8u * kb, (uint32_t)((a_tiles - 1) & 1), g.err);
        }
    } else if (warp == 2 + G_EPI) {
        // ------------------------------------------------------------- G^T tiles
        if (lane == 0) {
            uint32_t it = 0, s = 0, ph = 1u;
            int done = 0;
            bool ok = true;
            for (int u = u0; u < u1 && ok; ++u, ++done) {
                int mt, ks, k0, k1;
                split(u, mt, ks, k0, k1);
                // with one C buffer, the previous unit's C leaves through this memory
                if (g.c_bufs == 1 && done > 0 && !mbar_wait_bounded(cempty, (uint32_t)((done - 1) & 1), g.err, g.wait_ns))
                    break;
                for (int k = k0; k < k1; ++k) {
                    if (!mbar_wait_bounded(tempty + 8u * s, ph, g.err, g.wait_ns)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(tfull + 8u * s, t_stage);
                    tma_load_2d(tst0 + s * t_stage, &mapT, tfull + 8u * s, k * GK, 0);
                    ++it;
                    if (++s == G_T_STAGES) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            const uint32_t last = it < (uint32_t)G_T_STAGES ? it : (uint32_t)G_T_STAGES;
            for (uint32_t q = 1; q <= last; ++q) {
                const uint32_t i2 = it - q;
                mbar_drain(tfull + 8u * (i2 % G_T_STAGES), (i2 / G_T_STAGES) & 1u, g.err);
            }
        }
    } else if (warp == 1) {
        // --------------------------------------------------------------------- S
        // Each of the two MMA warps walks its loop in step and one elected lane issues.
        const uint32_t hi128 = sdesc_hi(128u), hi_tail = sdesc_hi(tail_row), half_tail = GM * tail_row / 16u;
        uint32_t gs = 0, gph = 0;
        uint32_t t = 0;  // tiles so far (S buffer t & 1)
        int a_mt = -1, a_tiles = 0;
        bool ok = true;
        auto wait = [&](uint32_t bar, uint32_t parity) {
            const bool w = mbar_wait_bounded(bar, parity, g.err, g.wait_ns);
            ok = ok && __all_sync(0xffffffffu, w) != 0;
            return ok;
        };
        // Injected stall (tests of the timeout path), as in the likelihood kernel
        if (g.stall) wait(drain_bar, 0u);
        for (int u = u0; u < u1 && ok; ++u) {
            int mt, ks, k0, k1;
            split(u, mt, ks, k0, k1);
            const bool a_first = mt != a_mt;  // wait for A's k-blocks in the first tile
            if (a_first) {
                a_mt = mt;
                ++a_tiles;
            }
            for (int k = k0; k < k1 && ok; k += 2, ++t) {
                const uint32_t b = t & 1u;
                // C has taken the tile that was in this buffer
                if (t >= 2u && !wait(pfree + 8u * b, ((t >> 1) - 1u) & 1u)) break;
                tc_fence_after();
                const uint32_t d = tmem + G_S_COL + b * (uint32_t)GT_N;
                // two k-blocks at a time: the waits and the set-up take as long as four MMAs
                for (int kb = 0; kb < g.kblocks; kb += 2) {
                    const int nkb = min(2, g.kblocks - kb);
                    const uint32_t gs1 = gs + 1u == (uint32_t)g.stages ? 0u : gs + 1u, gph1 = gs1 == 0u ? gph ^ 1u : gph;
                    if (a_first && k == k0) {
                        if (!wait(afull + 8u * kb, (uint32_t)((a_tiles - 1) & 1))) break;
                        if (nkb > 1 && !wait(afull + 8u * (kb + 1), (uint32_t)((a_tiles - 1) & 1))) break;
                    }
                    if (!wait(gfull + 8u * gs, gph)) break;
                    if (nkb > 1 && !wait(gfull + 8u * gs1, gph1)) break;
                    tc_fence_after();
                    if (elect_one()) {
                        s_block(g, d, sbase + (uint32_t)kb * G_KB_BYTES, gst0 + gs * G_STAGE, kb, hi128, hi_tail, half_tail);
                        umma_commit(gempty + 8u * gs);
                        if (nkb > 1) {
                            s_block(g, d, sbase + (uint32_t)(kb + 1) * G_KB_BYTES, gst0 + gs1 * G_STAGE, kb + 1, hi128, hi_tail,
                                    half_tail);
                            umma_commit(gempty + 8u * gs1);
                        }
                        if (kb + nkb == g.kblocks) umma_commit(sfull + 8u * b);
                    }
                    __syncwarp();
                    gs = nkb > 1 ? gs1 : gs;
                    gph = nkb > 1 ? gph1 : gph;
                    if (++gs == (uint32_t)g.stages) {
                        gs = 0;
                        gph ^= 1u;
                    }
                }
            }
            // A is free once these S are done, if the next unit is of another particle tile
            if (ok && u + 1 < u1 && (u + 1) / g.ksplit != mt && elect_one()) umma_commit(aempty);
            __syncwarp();
        }
        if (elect_one()) umma_commit(drain_bar);
        __syncwarp();
        mbar_drain(drain_bar, 0u, g.err);
    } else if (warp == 3 + G_EPI) {
        // --------------------------------------------------------------------- C
        const uint32_t idesc_c = idesc_bf16_f32(GM, (uint32_t)g.N2), hi128 = sdesc_hi(128u);
        uint32_t ts = 0, tph = 0, t = 0;
        int done = 0;
        bool ok = true;
        auto wait = [&](uint32_t bar, uint32_t parity) {
            const bool w = mbar_wait_bounded(bar, parity, g.err, g.wait_ns);
            ok = ok && __all_sync(0xffffffffu, w) != 0;
            return ok;
        };
        for (int u = u0; u < u1 && ok; ++u, ++done) {
            int mt, ks, k0, k1;
            split(u, mt, ks, k0, k1);
            // the unit that used this C buffer has left
            const uint32_t cb = (uint32_t)(done % g.c_bufs), c_col = tmem + 128u * cb;
            if (done >= g.c_bufs && !wait(cempty + 8u * cb, (uint32_t)((done / g.c_bufs - 1) & 1))) break;
            for (int k = k0; k < k1 && ok; k += 2, ++t) {
                const uint32_t b = t & 1u;
                if (!wait(pfull + 8u * b, (t >> 1) & 1u)) break;
                const int nsb = min(2, k1 - k);
                for (int sb = 0; sb < nsb; ++sb) {
                    if (!wait(tfull + 8u * ts, tph)) break;
                    tc_fence_after();
                    if (elect_one()) {
                        // r of individuals 64 sb .. +63: chunk c of 32 is hi in 16 columns from 32 c, then lo
                        const uint32_t r0 = tmem + G_S_COL + b * (uint32_t)GT_N + 64u * (uint32_t)sb;
                        const uint32_t t_lo = sdesc_lo(tst0 + ts * t_stage);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            umma_bf16_ta(c_col, r0 + 32u * (q >> 1) + 8u * (q & 1), sdesc_make(t_lo + 2u * q, hi128), idesc_c,
                                         (k > k0 || sb || q) ? 1u : 0u);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            umma_bf16_ta(c_col, r0 + 16u + 32u * (q >> 1) + 8u * (q & 1), sdesc_make(t_lo + 2u * q, hi128), idesc_c,
                                         1u);
                        umma_commit(tempty + 8u * ts);
                        if (sb + 1 == nsb) umma_commit(pfree + 8u * b);
                    }
                    __syncwarp();
                    if (++ts == G_T_STAGES) {
                        ts = 0;
                        tph ^= 1u;
                    }
                }
            }
            if (ok && elect_one()) umma_commit(cfull + 8u * cb);
            __syncwarp();
        }
        if (elect_one()) umma_commit(drain_bar + 8u);
        __syncwarp();
        mbar_drain(drain_bar + 8u, 0u, g.err);
    } else {
        // --------------------------------------------------------------- epilogue
        grid_dependency_wait();  // the previous kernel read the partial sums written here
        grid_launch_dependents();
        const int quad = warp & 3, grp = (warp - 2) >> 2;  // lane quadrant; 32-individual chunk of a tile
        const int row = quad * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        float* xp = reinterpret_cast<float*>(smem + (tst0 - sbase) + (g.c_bufs == 2 ? G_T_STAGES * t_stage : 0u)) +
                    (warp - 2) * (int)(G_XPOSE / 4);
        uint32_t tile = 0;
        int done = 0;
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u, ++done) {
            int mt, ks, k0, k1;
            split(u, mt, ks, k0, k1);
            const int64_t prow = (int64_t)mt * GM + row;
            const int tiles = (k1 - k0 + 1) / 2;
            for (int i = 0; i < tiles; ++i, ++tile) {
                const uint32_t b = tile & 1u;
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(sfull + 8u * b, (tile >> 1) & 1u, g.err, g.wait_ns)) != 0;
                if (!ok) break;
                tc_fence_after();
                const int i0 = (k0 + 2 * i) * GK + 32 * grp;  // the chunk's first individual
                if (i0 < k1 * GK) {
                    const uint32_t col = tmem + lane_addr + G_S_COL + b * (uint32_t)GT_N + 32u * (uint32_t)grp;
                    const int valid = g.n - i0;
                    uint32_t hi2[16], lo2[16];
                    if (valid > 0) {
                        uint32_t x[32];
                        tmem_ld32_async(col, x);
                        tmem_wait_ld(x);
                        float rs, sp;
                        if (valid >= 32)
                            sp = resid_chunk<true, true>(x, valid, 0u, g.yv + i0, hi2, lo2, rs);
                        else
                            sp = resid_chunk<false>(x, valid, __ldg(g.ybits + (i0 >> 5)), nullptr, hi2, lo2, rs);
                        const int64_t o = (int64_t)(i0 >> 5) * g.N_pad + prow;
                        g.partial[o] = -sp;
                        g.rsum_part[o] = rs;
                    } else {
#pragma unroll
                        for (int q = 0; q < 16; ++q) hi2[q] = lo2[q] = 0u;
                    }
                    tmem_st16(col, hi2);
                    tmem_st16(col + 16u, lo2);
                    tmem_wait_st();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(pfull + 8u * b);
            }
            if (!ok) break;
            // C leaves through a shared-memory transpose, so that the stores write row segments
            const uint32_t cb = (uint32_t)(done % g.c_bufs);
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(cfull + 8u * cb, (uint32_t)((done / g.c_bufs) & 1), g.err, g.wait_ns)) != 0;
            if (!ok) break;
            tc_fence_after();
            // 16 columns at a time: a lane holds 16 of its row's, a store then writes two rows' 64 bytes
            float* out0 = g.gpart + ((int64_t)ks * g.N_pad + (int64_t)mt * GM + quad * 32 + (lane >> 4)) * g.p + (lane & 15);
#pragma unroll 1
            for (int c = 16 * grp; c < g.p; c += 16 * (G_EPI / 4)) {
                float v[16];
                tmem_ld16(tmem + lane_addr + 128u * cb + (uint32_t)c, v);
#pragma unroll
                for (int k = 0; k < 16; ++k) xp[lane * 17 + k] = v[k];
                __syncwarp();
                if (c + (lane & 15) < g.p) {
#pragma unroll
                    for (int r = 0; r < 32; r += 2) out0[(int64_t)r * g.p + c] = xp[(r + (lane >> 4)) * 17 + (lane & 15)];
                }
                __syncwarp();
            }
            tc_fence_before();
            asm volatile("fence.proxy.async;" ::: "memory");  // before the next unit's copies into this memory
            __syncwarp();
            if (lane == 0) mbar_arrive(cempty + 8u * cb);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace

cudaError_t grad_tc_init_attributes()
{
    return cudaFuncSetAttribute(k_grad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
}

bool grad_tc_plan(GradPlan& pl, int64_t n, int p, const AdjPlan& adj, int max_ctas)
{
    if (p + 1 > 256 || adj.p_tiles != 1) return false;
    pl.ksteps = (p + 1 + 15) / 16;
    pl.kblocks = (pl.ksteps + 3) / 4;
    const int last = pl.ksteps - 4 * (pl.kblocks - 1);
    pl.tw = last <= 2 ? 16 * last : 0;
    pl.N2 = (p + 15) / 16 * 16;
    pl.a_bytes = (uint32_t)(pl.kblocks - 1) * G_KB_BYTES + (pl.tw ? 2u * GM * (uint32_t)pl.tw * 2u : G_KB_BYTES);
    const uint32_t t = (uint32_t)G_T_STAGES * (uint32_t)pl.N2 * 128u, x = (uint32_t)G_EPI * G_XPOSE;
    // markers for two C buffers (128 columns each): the next unit's C starts while one leaves, through
    // memory of its own; else C leaves through the G^T stages
    pl.c_bufs = pl.N2 <= 128 ? 2 : 1;
    pl.t_bytes = ((pl.c_bufs == 2 ? t + x : (t > x ? t : x)) + 1023u) / 1024u * 1024u;
    const uint32_t fixed = pl.a_bytes + pl.t_bytes + 8u * G_NBARS + 16u;
    pl.stages = 0;
    while (pl.stages < G_MAX_STAGES && fixed + (uint32_t)(pl.stages + 1) * G_STAGE <= 232448u - 1024u) ++pl.stages;
    pl.smem = fixed + (uint32_t)pl.stages * G_STAGE + 1024u;
    const int units = adj.m_tiles * adj.ksplit;
    pl.grid = units < max_ctas ? units : max_ctas;
    return pl.stages >= 2;
}

bool grad_tc_make_maps(GradMaps& m, const __nv_bfloat16* Gbf, const __nv_bfloat16* GT, int64_t n, int p, int Kp, int64_t n_r,
                       const GradPlan& pl)
{
    if (!tc_make_map_B(&m.B, Gbf, n, Kp, GT_N)) return false;
    m.Bt = m.B;
    if (pl.tw && !tc_make_map_B_tail(&m.Bt, Gbf, n, Kp, GT_N, pl.tw)) return false;
    return adj_make_map_GT(&m.T, GT, p, n_r, pl.N2);
}

cudaError_t launch_grad_tc(const CUtensorMap& A, const CUtensorMap& At, const GradMaps& m, const GradPlan& pl,
                           const AdjPlan& adj, GradArgs g, cudaStream_t st)
{
    g.m_tiles = adj.m_tiles;
    g.ksplit = adj.ksplit;
    g.kb_n = adj.kblocks;
    g.ksteps = pl.ksteps;
    g.kblocks = pl.kblocks;
    g.tw = pl.tw;
    g.N2 = pl.N2;
    g.c_bufs = pl.c_bufs;
    g.stages = pl.stages;
    g.a_bytes = pl.a_bytes;
    g.t_bytes = pl.t_bytes;
    if (g.wait_ns == 0) g.wait_ns = WAIT_LIMIT_DEFAULT_NS;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)pl.grid);
    cfg.blockDim = dim3(G_THREADS);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_grad_tc, A, pl.tw ? At : A, m.B, m.Bt, m.T, g);
}

}  // namespace spa
