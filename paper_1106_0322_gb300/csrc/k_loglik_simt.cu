// k_loglik_simt.cu -- the plain FP32 path: the same log-likelihood on CUDA cores (FFMA).
//
// eta = X beta with the standardised FP32 X (Section 3) and FP32 accumulation, then
// softplus(eta) = max(eta, 0) + log1p(exp(-|eta|)) with the accurate FP32 functions, summed
// per particle over each 64-individual tile (the linear half sum_i y_i eta_i = beta . X^T y
// is a p-length dot product the move kernels form). The gradient path (mode 1) keeps the
// full y eta - softplus(eta) per tile for its log-likelihood output, and the residuals for the
// adjoint. This is the comparator the split-BF16 tensor-core path is measured against; it is also the gradient (adjoint) kernel pair
// behind spa_grad: grad l = X^T (y - logit^{-1}(eta)).
#include "spa_device.cuh"
#include "spa_internal.h"

namespace spa {

namespace {

constexpr int TK = 16;     // k-chunk
constexpr int STAGES = 3;  // chunks in shared memory

// One CTA's tile of a product C = A B^T: TY x 16 threads, thread (ty, tx) owning rows ty NA .. + NA - 1
// and columns 64 h + 4 tx .. + 3 of each h < HB. Every entry is one chain of FP32 FMAs in the order of
// k from 0, whatever the tile.
//
// Bound by the FMA pipe, its register reads and shared-memory reads together (each about 60% busy at
// 8 x 8 entries a thread). So: packed pairs of FMAs, which halve the issue slots and need each row's
// value twice (two moves, cheaper than reading it twice); 8 rows x 4 columns a thread or more, 12
// values read for 32 FMAs; chunks of 16 k three deep by cp.async, no registers on the way; and a
// k's values read while the previous ones are multiplied. Against a 64 x 64 tile of 256 threads,
// 4 x 4 entries each, one chunk at a time: loglik 1222 -> 893 us at n = 5000, p = 500, N = 8192
// (23 TFMA/s), 39 -> 31 us at 1000, 100, 4096; gradient (wall) 4049 -> 2093 and 296 -> 146 us.
template <int NA, int HB, int TY>
struct Tile {
    static constexpr int ROWS = TY * NA, COLS = 64 * HB, THREADS = 16 * TY;
    float a[STAGES][TK][ROWS + 4];
    float b[STAGES][TK][COLS + 4];
};

constexpr int tile_blocks(int na, int hb, int ty) { return (na * hb == 16 ? 32 : 48) / ty; }  // resident on an SM

// an operand: element (i, k) at base[i * si + k * sk], i < m (0 outside)
struct Operand {
    const float* base;
    int64_t m, si, sk;
};

__device__ __forceinline__ void cp_async4(float* dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Chunk k0 of an operand's R rows from row r0 into s[k][row]; K_NEXT: consecutive k are
// neighbours in memory (8 lanes a row, which keeps the transposed stores off each other's
// banks), otherwise consecutive rows are.
template <int R, bool K_NEXT, int THREADS, int LD>
__device__ __forceinline__ void fetch_chunk(float (&s)[TK][LD], const Operand& o, int64_t r0, int64_t k0, int64_t K)
{
    constexpr int U = R * TK / THREADS, RS = THREADS / 8;  // (RS rows at once)
    const int r = K_NEXT ? threadIdx.x >> 3 : threadIdx.x % R, k = K_NEXT ? threadIdx.x & 7 : threadIdx.x / R;
    const float* src = o.base + (r0 + r) * o.si + (k0 + k) * o.sk;
    float* dst = &s[k][r];
    const bool inside = r0 + R <= o.m && k0 + TK <= K;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int dr = K_NEXT ? RS * (u % (R / RS)) : 0, dk = K_NEXT ? 8 * (u / (R / RS)) : u * (THREADS / R);
        const float* from = src + dr * o.si + dk * o.sk;
        float* to = dst + dk * LD + dr;
        if (inside || (r0 + r + dr < o.m && k0 + k + dk < K))
            cp_async4(to, from);
        else
            *to = 0.0f;
    }
}

// The operands of one k: NA values of rows, 4 HB of columns in pairs.
template <int NA, int HB, int TY>
struct Fragment {
    float4 a[NA / 4];
    ulonglong2 b[HB];
    __device__ __forceinline__ void load(const Tile<NA, HB, TY>& t, int stage, int kk)
    {
        const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
        for (int q = 0; q < NA / 4; ++q) a[q] = *reinterpret_cast<const float4*>(&t.a[stage][kk][NA * ty + 4 * q]);
#pragma unroll
        for (int h = 0; h < HB; ++h) b[h] = *reinterpret_cast<const ulonglong2*>(&t.b[stage][kk][64 * h + 4 * tx]);
    }
    // acc[x][y]: columns 2y, 2y + 1 (of the thread's 4 HB) of its row x
    __device__ __forceinline__ void multiply(uint64_t (&acc)[NA][2 * HB]) const
    {
        uint64_t aa[NA];
#pragma unroll
        for (int q = 0; q < NA / 4; ++q) {
            aa[4 * q] = pack2(a[q].x, a[q].x);
            aa[4 * q + 1] = pack2(a[q].y, a[q].y);
            aa[4 * q + 2] = pack2(a[q].z, a[q].z);
            aa[4 * q + 3] = pack2(a[q].w, a[q].w);
        }
#pragma unroll
        for (int y = 0; y < 2 * HB; ++y)
#pragma unroll
            for (int x = 0; x < NA; ++x) acc[x][y] = fma2(y & 1 ? b[y / 2].y : b[y / 2].x, aa[x], acc[x][y]);
    }
};

template <int NA, int HB, int TY, bool B_K_NEXT>
__device__ __forceinline__ void tile_product(Tile<NA, HB, TY>& t, int64_t K, uint64_t (&acc)[NA][2 * HB], const Operand& A,
                                             const Operand& B, int64_t i0, int64_t j0)
{
    using T = Tile<NA, HB, TY>;
#pragma unroll
    for (int x = 0; x < NA; ++x)
#pragma unroll
        for (int y = 0; y < 2 * HB; ++y) acc[x][y] = 0;
    auto fetch = [&](int stage, int64_t k0) {
        if (k0 < K) {
            fetch_chunk<T::ROWS, true, T::THREADS>(t.a[stage], A, i0, k0, K);
            fetch_chunk<T::COLS, B_K_NEXT, T::THREADS>(t.b[stage], B, j0, k0, K);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(0, 0);
    fetch(1, TK);
    int stage = 0;
    for (int64_t k0 = 0; k0 < K; k0 += TK) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();  // chunk k0 is there, and every thread has done with the one before it
        fetch(stage == 0 ? 2 : stage - 1, k0 + 2 * TK);
        Fragment<NA, HB, TY> f[2];  // the next k's operands are read while this one's are multiplied
        f[0].load(t, stage, 0);
        if (K - k0 >= TK) {
#pragma unroll
            for (int kk = 0; kk < TK; ++kk) {
                if (kk + 1 < TK) f[(kk + 1) & 1].load(t, stage, kk + 1);
                f[kk & 1].multiply(acc);
            }
        } else {
#pragma unroll 1
            for (int kk = 0; kk < (int)(K - k0); ++kk) {
                f[1].load(t, stage, kk + 1);  // (a row of zeros or of the stage after it at the end)
                f[0].multiply(acc);
                f[0] = f[1];
            }
        }
        stage = stage == 2 ? 0 : stage + 1;
    }
}

__device__ __forceinline__ float softplus_acc(float x) { return fmaxf(x, 0.0f) + log1pf(expf(-fabsf(x))); }

// Rows: particles, columns: individuals. mode 0: partial = -sum over 64 individuals of
// softplus(eta); mode 1: partial = sum of y eta - softplus(eta), and the residuals y -
// logit^{-1}(eta) stored to resid [N][n].
template <int MODE, int NA, int HB, int TY>
__global__ void __launch_bounds__(16 * TY, tile_blocks(NA, HB, TY))
    k_eta_tile(const float* __restrict__ B, const float* __restrict__ Xf, const uint8_t* __restrict__ y, int64_t N,
               int64_t n, int p, float* __restrict__ partial, int64_t N_pad, float* __restrict__ resid)
{
    using T = Tile<NA, HB, TY>;
    extern __shared__ __align__(16) float simt_sm[];
    T& t = *reinterpret_cast<T*>(simt_sm);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t i0 = (int64_t)blockIdx.x * T::ROWS;  // particle tile
    const int64_t r0 = (int64_t)blockIdx.y * T::COLS;  // individual tile
    uint64_t acc[NA][2 * HB];
    tile_product<NA, HB, TY, true>(t, p, acc, Operand{B, N, p, 1}, Operand{Xf, n, p, 1}, i0, r0);
#pragma unroll
    for (int x = 0; x < NA; ++x) {
        const int64_t gi = i0 + ty * NA + x;
#pragma unroll
        for (int h = 0; h < HB; ++h) {
            float e[4], sp[4], s = 0.0f;  // (all four computed, also beyond n: no branch between them)
#pragma unroll
            for (int z = 0; z < 4; ++z) {
                const float2 v = unpack2(acc[x][2 * h + z / 2]);
                e[z] = z & 1 ? v.y : v.x;
                sp[z] = softplus_acc(e[z]);
            }
#pragma unroll
            for (int z = 0; z < 4; ++z) {
                const int64_t gr = r0 + 64 * h + 4 * tx + z;
                if (MODE == 0) {
                    s = gr < n ? s - sp[z] : s;
                } else {
                    const float sig = 1.0f / (1.0f + expf(-e[z]));
                    if (gr < n) {
                        s += (y[gr] ? e[z] : 0.0f) - sp[z];
                        if (gi < N) resid[gi * n + gr] = (y[gr] ? 1.0f : 0.0f) - sig;
                    }
                }
            }
            // reduce over the 16 threads (tx) that share these particles: lanes differ in bits 0..3
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (tx == 0 && gi < N && r0 + 64 * h < n) partial[((int64_t)blockIdx.y * HB + h) * N_pad + gi] = s;
        }
    }
}

// grad[i, j] = sum_r x_rj resid[i, r] (+ prior gradient at scale c).
// Rows: particles, columns: markers.
template <int NA, int HB, int TY>
__global__ void __launch_bounds__(16 * TY, tile_blocks(NA, HB, TY))
    k_grad_tile(const float* __restrict__ resid, const float* __restrict__ Xf, const float* __restrict__ B, int64_t N,
                int64_t n, int p, float* __restrict__ grad, PriorArgs pr, double c)
{
    using T = Tile<NA, HB, TY>;
    extern __shared__ __align__(16) float simt_sm[];
    T& t = *reinterpret_cast<T*>(simt_sm);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t i0 = (int64_t)blockIdx.x * T::ROWS;  // particle tile
    const int j0 = blockIdx.y * T::COLS;               // marker tile
    uint64_t acc[NA][2 * HB];
    tile_product<NA, HB, TY, false>(t, n, acc, Operand{resid, N, n, 1}, Operand{Xf, p, 1, p}, i0, j0);
#pragma unroll
    for (int x = 0; x < NA; ++x) {
        const int64_t gi = i0 + ty * NA + x;
#pragma unroll
        for (int y = 0; y < 4 * HB; ++y) {
            const int gj = j0 + 64 * (y / 4) + 4 * tx + y % 4;
            if (gi < N && gj < p) {
                const float2 v = unpack2(acc[x][y / 2]);
                float g = y & 1 ? v.y : v.x;
                if (c > 0.0) {
                    const float b = B[gi * p + gj];
                    const float sg = (b > 0.0f) ? 1.0f : ((b < 0.0f) ? -1.0f : 0.0f);
                    g += pr.de ? (float)(-sg / c) : (float)(-((double)pr.a + 1.0) * sg / ((double)pr.a * c + fabs((double)b)));
                }
                grad[gi * p + gj] = g;
            }
        }
    }
}

__global__ void k_sum_partials(const float* __restrict__ partial, int n_parts, int64_t N_pad, int64_t N,
                               double* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double s = 0.0;
    for (int k = 0; k < n_parts; ++k) s += (double)partial[(int64_t)k * N_pad + i];
    out[i] = s;
}

}  // namespace

namespace {

// The tiles, <NA, HB, TY>, by the product's rows and columns: the one whose busiest SM has least to
// do. Costs are the times of a tile at n = 5000, p = 500, N = 8192 (loglik 893, 1086 and 1568 us).
// Larger tiles read less shared memory per FMA; smaller ones spread small products over the SMs and
// leave less of a last wave: N = 1024, n = 5000, p = 500: 166, 155, 207 us; N = 64, n = 1000, p = 300:
// 41, 19, 14 us; N = 4096, n = 1000, p = 100: 31, 33, 43 us.
enum { TILE_128x128, TILE_64x64, TILE_32x64 };
int pick_tile(int64_t rows, int64_t cols, int num_sms)
{
    const int64_t r[3] = {128, 64, 32}, c[3] = {128, 64, 64}, cost[3] = {26, 8, 6};
    int best = 0;
    int64_t least = 0;
    for (int k = 0; k < 3; ++k) {
        const int64_t ctas = ((rows + r[k] - 1) / r[k]) * ((cols + c[k] - 1) / c[k]);
        const int64_t t = (ctas + num_sms - 1) / num_sms * cost[k];
        if (k == 0 || t < least) {
            best = k;
            least = t;
        }
    }
    return best;
}

template <int MODE, int NA, int HB, int TY>
cudaError_t eta_tile(const float* B, const float* Xf, const uint8_t* y, int64_t N, int64_t n, int p, float* partial,
                     int64_t N_pad, float* resid, cudaStream_t st)
{
    using T = Tile<NA, HB, TY>;
    dim3 grid((unsigned)((N + T::ROWS - 1) / T::ROWS), (unsigned)((n + T::COLS - 1) / T::COLS));
    k_eta_tile<MODE, NA, HB, TY><<<grid, T::THREADS, sizeof(T), st>>>(B, Xf, y, N, n, p, partial, N_pad, resid);
    return cudaGetLastError();
}

template <int MODE>
cudaError_t enq_eta(int num_sms, const float* B, const float* Xf, const uint8_t* y, int64_t N, int64_t n, int p,
                    float* partial, int64_t N_pad, float* resid, cudaStream_t st)
{
    switch (pick_tile(N, n, num_sms)) {
        case TILE_128x128: return eta_tile<MODE, 8, 2, 16>(B, Xf, y, N, n, p, partial, N_pad, resid, st);
        case TILE_64x64: return eta_tile<MODE, 8, 1, 8>(B, Xf, y, N, n, p, partial, N_pad, resid, st);
        default: return eta_tile<MODE, 4, 1, 8>(B, Xf, y, N, n, p, partial, N_pad, resid, st);
    }
}

template <int NA, int HB, int TY>
cudaError_t grad_tile(const float* resid, const float* Xf, const float* B, int64_t N, int64_t n, int p,
                      float* grad, PriorArgs pr, double c, cudaStream_t st)
{
    using T = Tile<NA, HB, TY>;
    dim3 grid((unsigned)((N + T::ROWS - 1) / T::ROWS), (unsigned)((p + T::COLS - 1) / T::COLS));
    k_grad_tile<NA, HB, TY><<<grid, T::THREADS, sizeof(T), st>>>(resid, Xf, B, N, n, p, grad, pr, c);
    return cudaGetLastError();
}

}  // namespace

cudaError_t simt_init_attributes()
{
    const int bytes = (int)sizeof(Tile<8, 2, 16>);
    cudaError_t e = cudaFuncSetAttribute(k_eta_tile<0, 8, 2, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_eta_tile<1, 8, 2, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_grad_tile<8, 2, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e;
}

cudaError_t launch_loglik_simt(const float* beta_p, const float* Xf, const uint8_t* y, int64_t N, int64_t n, int p,
                               float* partial, int64_t N_pad, int num_sms, cudaStream_t st)
{
    return enq_eta<0>(num_sms, beta_p, Xf, y, N, n, p, partial, N_pad, nullptr, st);
}

cudaError_t launch_grad_simt(const float* B, const float* Xf, const uint8_t* y, int64_t N, int64_t n, int p,
                             float* eta_scratch, float* grad, double* ll, PriorArgs pr, double c, int num_sms,
                             cudaStream_t st)
{
    // the log-likelihood partials live in the tail of the eta scratch (allocated N*n + n_tiles*N)
    const int n_tiles = (int)((n + SIMT_TILE_N - 1) / SIMT_TILE_N);
    float* partial = eta_scratch + N * n;
    cudaError_t e = enq_eta<1>(num_sms, B, Xf, y, N, n, p, partial, N, eta_scratch, st);
    if (e != cudaSuccess) return e;
    switch (pick_tile(N, p, num_sms)) {
        case TILE_128x128: e = grad_tile<8, 2, 16>(eta_scratch, Xf, B, N, n, p, grad, pr, c, st); break;
        case TILE_64x64: e = grad_tile<8, 1, 8>(eta_scratch, Xf, B, N, n, p, grad, pr, c, st); break;
        default: e = grad_tile<4, 1, 8>(eta_scratch, Xf, B, N, n, p, grad, pr, c, st);
    }
    if (e != cudaSuccess || !ll) return e;
    k_sum_partials<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(partial, n_tiles, N, N, ll);
    return cudaGetLastError();
}

}  // namespace spa
