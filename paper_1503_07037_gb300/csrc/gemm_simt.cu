// CUDA-core GEMM D = alpha X Y^T + beta C + gamma I (FFMA for float, DFMA for
// double): an independent cross-check of the tcgen05 engines, and the engine of small FP64
// products (k_gemm_small_f64).
#include <cuda_runtime.h>

#include <string>

#include "epilogue.cuh"
#include "internal.cuh"

namespace cdmpt {

namespace {

constexpr int BM = 64, BN = 64, BK = 16;

template <typename T>
__global__ void __launch_bounds__(256) k_gemm_simt(const T* __restrict__ X, int ldx,
                                                   const T* __restrict__ Y, int ldy, int K,
                                                   EpiParams<T> p, const double* skip) {
    if (skip && *skip != 0.0) return;
    __shared__ T Xs[BK][BM + 4];
    __shared__ T Ys[BK][BN + 4];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    // loader mapping: 64 rows x 16 k = 1024 elements, 4 per thread
    const int lr = threadIdx.x >> 2, lk = (threadIdx.x & 3) * 4;
    T acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = T(0);

    for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = k0 + lk + q;
            const int mx = m0 + lr, ny = n0 + lr;
            Xs[lk + q][lr] = (mx < p.M && k < K) ? X[(size_t)mx * ldx + k] : T(0);
            Ys[lk + q][lr] = (ny < p.N && k < K) ? Y[(size_t)ny * ldy + k] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = Xs[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Ys[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }

    double dsum = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty + 16 * i;
        if (m >= p.M) continue;
        T local = T(0);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx + 16 * j;
            if (n < p.N) local += epi_apply(p, m, n, acc[i][j]);
        }
        dsum += (double)local;
    }
    if (p.dot) {
        __shared__ double part[8];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dsum += __shfl_down_sync(0xffffffffu, dsum, o);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = dsum;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < 8; ++w) s += part[w];
            if (s != 0.0) atomicAdd(p.dot, s);
        }
    }
}

// FP64 product of small matrices: one 8 x 8 output tile per CTA. The FP64 pipe of an SM takes
// two FMAs per clock, so a product is short only if every SM gets a share: N = 120 has 225 such
// tiles (120 of a symmetric result) against four of 64 x 64, which took 135 us. The rows of
// both operands are staged in shared memory in chunks of 256 k (odd row pitch: the eight rows
// a warp reads fall into different banks); four groups of 64 threads take a quarter of the
// chunk each, so that the FMAs of several warps overlap, and their sums meet in shared memory.
constexpr int SM_T = 8, SM_KC = 256, SM_G = 4;

__global__ void __launch_bounds__(SM_G* SM_T* SM_T) k_gemm_small_f64(
    const double* __restrict__ X, int ldx, const double* __restrict__ Y, int ldy, int K,
    EpiParams<double> p, int nt, const double* skip) {
    // programmatic dependent launch: the next product's blocks may take their places while this
    // one runs, and this one touches memory only once its predecessor has finished
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (skip && *skip != 0.0) return;
    __shared__ double rows[2 * SM_T][SM_KC + 1];
    __shared__ double part[SM_G - 1][SM_T * SM_T];
    const int tid = threadIdx.x, g = tid / (SM_T * SM_T), e = tid % (SM_T * SM_T);
    const int i = e / SM_T, j = e % SM_T;
    int bm, bn;
    if (p.sym) {   // tiles of the upper triangle, column by column: bn + 1 of them in column bn
        bn = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
        while (bn * (bn + 1) / 2 > (int)blockIdx.x) --bn;
        while ((bn + 1) * (bn + 2) / 2 <= (int)blockIdx.x) ++bn;
        bm = (int)blockIdx.x - bn * (bn + 1) / 2;
    } else {
        bn = (int)blockIdx.x % nt;
        bm = (int)blockIdx.x / nt;
    }
    const int m0 = bm * SM_T, n0 = bn * SM_T;
    const int lr = tid >> 4, lc = tid & 15;   // loader: 16 threads per row
    const bool is_x = lr < SM_T;
    const int row = is_x ? m0 + lr : n0 + lr - SM_T;
    const bool row_ok = row < (is_x ? p.M : p.N);
    const double* src = is_x ? X + (size_t)row * ldx : Y + (size_t)row * ldy;
    double acc = 0.0;
    for (int k0 = 0; k0 < K; k0 += SM_KC) {
        const int kc = min(SM_KC, K - k0);
        if (k0) __syncthreads();
#pragma unroll 4
        for (int k = lc; k < kc; k += 16) rows[lr][k] = row_ok ? src[k0 + k] : 0.0;
        __syncthreads();
        const int q = (kc + SM_G - 1) / SM_G, kb = g * q, ke = min(kc, kb + q);
#pragma unroll 4
        for (int k = kb; k < ke; ++k) acc = fma(rows[i][k], rows[SM_T + j][k], acc);
    }
    if (g > 0) part[g - 1][e] = acc;
    __syncthreads();
    if (g > 0) return;
#pragma unroll
    for (int w = 0; w < SM_G - 1; ++w) acc += part[w][e];
    const int m = m0 + i, n = n0 + j;
    double d = 0.0;
    if (m < p.M && n < p.N)
        d = p.sym ? epi_apply_sym(p, m, n, acc, bm == bn) : epi_apply(p, m, n, acc);
    if (p.dot) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
        if ((tid & 31) == 0 && d != 0.0) atomicAdd(p.dot, d);
    }
}

}  // namespace

// An FP64 product takes M N K / 304 clocks on the FP64 pipes of 152 SMs, 1.7 us per 10^6; the
// tensor-core engine takes about 45 us plus two slicing passes for any product up to N = 400
// (measured, DFMA against tensor cores: N = 120 11 and 52 us, 256 37 and 60, 343 78 and 66;
// half of the DFMA time for a symmetric result). The line is drawn where both take 60 us:
// N = 324 for a full product, 408 for a symmetric one.
bool small_f64(int M, int N, int K, bool sym) {
    return (sym ? 0.5 : 1.0) * M * (double)N * K <= 3.4e7;
}

bool dfma_small_tiles(int M, int N) {
    return (size_t)((M + BM - 1) / BM) * ((N + BN - 1) / BN) < 304;
}

template <typename T>
cdmpt_status gemm_simt(int M, int N, int K, const T* X, int ldx, const T* Y, int ldy, T* D,
                       int ldd, const Epilogue<T>& ep, const double* skip, cudaStream_t s) {
    if (M <= 0 || N <= 0) return CDMPT_OK;
    EpiParams<T> p;
    p.alpha = (T)ep.alpha;
    p.beta = (T)ep.beta;
    p.gamma = (T)ep.gamma;
    p.C = ep.C;
    p.ldc = ep.ldc;
    p.D = D;
    p.ldd = ldd;
    p.M = M;
    p.N = N;
    p.diag_block = ep.diag_block > 0 ? ep.diag_block : M;
    p.trans_block = ep.trans_block;
    p.dot = ep.dot;
    p.E = ep.E;
    p.lde = ep.lde;
    p.Dhi = ep.Dhi;
    p.Dlo = ep.Dlo;
    p.sym = 0;   // every element is computed here
    if constexpr (sizeof(T) == 8) {
        // small matrices: 8 x 8 tiles until the 64 x 64 tiles fill the SMs
        if (dfma_small_tiles(M, N)) {
            const int mt = (M + SM_T - 1) / SM_T, nt = (N + SM_T - 1) / SM_T;
            p.sym = (ep.sym && M == N && p.trans_block <= 0) ? 1 : 0;
            const int tiles = p.sym ? nt * (nt + 1) / 2 : mt * nt;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(tiles);
            cfg.blockDim = dim3(SM_G * SM_T * SM_T);
            cfg.stream = s;
            cudaLaunchAttribute a;
            a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
            a.val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = &a;
            cfg.numAttrs = 1;
            cudaError_t e = cudaLaunchKernelEx(&cfg, k_gemm_small_f64, X, ldx, Y, ldy, K, p, nt, skip);
            count_launch();
            if (e == cudaSuccess) e = cudaGetLastError();
            if (e != cudaSuccess) {
                set_error(std::string("gemm_simt launch: ") + cudaGetErrorString(e));
                return CDMPT_ERR_CUDA;
            }
            return CDMPT_OK;
        }
    }
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
    k_gemm_simt<T><<<grid, 256, 0, s>>>(X, ldx, Y, ldy, K, p, skip);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error(std::string("gemm_simt launch: ") + cudaGetErrorString(e));
        return CDMPT_ERR_CUDA;
    }
    return CDMPT_OK;
}

template cdmpt_status gemm_simt<float>(int, int, int, const float*, int, const float*, int,
                                       float*, int, const Epilogue<float>&, const double*,
                                       cudaStream_t);
template cdmpt_status gemm_simt<double>(int, int, int, const double*, int, const double*, int,
                                        double*, int, const Epilogue<double>&, const double*,
                                        cudaStream_t);

}  // namespace cdmpt
