// C = X U for the FP64 path's sums over hidden variables and auxiliary fields
// (S_p = sum_k x_pk U_k, the field planes sum_g y_wg L_g) in fixed point: 32-bit
// integer multiply-adds with 64-bit sums, which issue at some eight times the rate
// of FP64 ones here (15 against 2 per clock and SM measured), three to a product.
//
// A row of X and a column of U (one entry of every matrix) each share an exponent, so an
// element keeps the digits that matter to its own sum.  Values become
// integers of 28 + b bits, h 2^28 + l with |l| <= 2^27, and a product
// h h' 2^56 + (h l' + l h') 2^28; the dropped l l' is below 2^-(b + b') of the two
// largest entries' product.  b + b' = 62 - log2 K keeps the sums of h h' within 63 bits
// (56 bits of each operand at K = 50, 55 at 250): each product is off by 2^-56 (2^-55)
// of the largest entries' product at most, of either sign, where an FP64 sum rounds its
// partial sums at 2^-53.
//
// What bounds it: that pipe (15 multiply-adds per clock and SM), 3 R^2 of them a thread and k for
// 2 R shared-memory reads; few rows, whose tiles of 64 x 64 leave SMs idle, take smaller ones (the sums are
// integers: the same for every tile).  Against the FP64 GEMM (0.8 of the FP64 pipe) on one GB300:
// S of 16384 paths, 50 orbitals and variables 4.42 -> 1.27 ms, of 4096 1.11 -> 0.33; the planes of
// 512 walkers, 250 fields 1.30 -> 0.37.
#include <algorithm>

#include "digits64.cuh"
#include "kernels.cuh"

namespace afq {

namespace {

constexpr int GF_K = 16;

// exponent e with |m| 2^-e < 1 of the largest |entry| m
__device__ __forceinline__ int gf_exp(double m) { return m > 0.0 ? ilogb(m) + 1 : 0; }

__device__ __forceinline__ int2 gf_split(double x, int e) {
    const long long v = dg64_fix(x, e);
    const int l = ((int)v << 4) >> 4;
    return make_int2((int)((v - l) >> 28), l);
}

__global__ void gf_colexp_kernel(int K, long long Nc, const double* __restrict__ U, int* __restrict__ uexp) {
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < Nc; c += (long long)gridDim.x * blockDim.x) {
        double m = 0.0;
        bool bad = false;
        for (int k = 0; k < K; ++k) {
            const double v = fabs(U[(long long)k * Nc + c]);
            bad |= !isfinite(v);
            m = fmax(m, v);
        }
        uexp[c] = bad ? DG64_NAN : gf_exp(m);
    }
}

// 16 R x 16 R output tile per block, R x R per thread.
template <int R>
__global__ void __launch_bounds__(256) gemm_fix_kernel(int M, long long Nc, int K, const double* __restrict__ X,
                                                       const double* __restrict__ U, const int* __restrict__ uexp,
                                                       double* __restrict__ C, int bx, int bu) {
    constexpr int T = 16 * R, TPR = 256 / T;
    __shared__ int2 Xs[GF_K][T + 1], Us[GF_K][T];
    __shared__ int xe[T], ue[T];
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    const long long row0 = (long long)blockIdx.y * T, col0 = (long long)blockIdx.x * T;
    // a k tile's values, one R-th of X's and U's each; small tiles load the next one ahead, the first beside the exponents
    double xv[R], uv[R];
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int e = tid + q * 256;
            const int r = e / GF_K, kk = e % GF_K;              // X tile: T rows x 16 k
            const int kb = e / T, c = e % T;                    // U tile: 16 k x T columns
            xv[q] = row0 + r < M && k0 + kk < K ? X[(row0 + r) * K + k0 + kk] : 0.0;
            uv[q] = col0 + c < Nc && k0 + kb < K ? U[(long long)(k0 + kb) * Nc + col0 + c] : 0.0;
        }
    };
    if (R < 4) load(0);
    {   // exponents of the tile's rows: TPR threads a row
        const long long r = row0 + tid / TPR;
        double m = 0.0;
        bool bad = false;
        if (r < M)
            for (int k = tid % TPR; k < K; k += TPR) {
                const double v = fabs(X[r * K + k]);
                bad |= !isfinite(v);
                m = fmax(m, v);
            }
#pragma unroll
        for (int o = 1; o < TPR; o <<= 1) {
            m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
            bad |= __shfl_xor_sync(0xffffffffu, (int)bad, o) != 0;
        }
        if (tid % TPR == 0) xe[tid / TPR] = bad ? DG64_NAN : gf_exp(m);
        if (tid < T) ue[tid] = col0 + tid < Nc ? uexp[col0 + tid] : 0;
    }
    __syncthreads();
    long long h[R][R] = {}, x[R][R] = {};
    for (int k0 = 0; k0 < K; k0 += GF_K) {
        if (R == 4) load(k0);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int e = tid + q * 256;
            Xs[e % GF_K][e / GF_K] = gf_split(xv[q], 28 + bx - xe[e / GF_K]);
            Us[e / T][e % T] = gf_split(uv[q], 28 + bu - ue[e % T]);
        }
        __syncthreads();
        if (R < 4 && k0 + GF_K < K) load(k0 + GF_K);
#pragma unroll
        for (int kk = 0; kk < GF_K; ++kk) {
            int2 a[R], b[R];
#pragma unroll
            for (int i = 0; i < R; ++i) a[i] = Xs[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < R; ++j) b[j] = Us[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    h[i][j] += (long long)a[i].x * b[j].x;
                    x[i][j] += (long long)a[i].x * b[j].y;
                    x[i][j] += (long long)a[i].y * b[j].x;
                }
        }
        if ((k0 & 48) == 48)                                    // 64 terms: the cross sums stay below 2^62
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    h[i][j] += x[i][j] >> 28;
                    x[i][j] &= (1 << 28) - 1;
                }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int rl = ty + 16 * i;
        if (row0 + rl >= M) continue;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int cl = tx + 16 * j;
            if (col0 + cl >= Nc) continue;
            const int er = xe[rl], ec = ue[cl];
            double v = __longlong_as_double(0x7FF8000000000000LL);
            if (er != DG64_NAN && ec != DG64_NAN)
                v = ldexp((double)(h[i][j] + ((x[i][j] + (1 << 27)) >> 28)), er + ec - bx - bu);
            C[(row0 + rl) * Nc + col0 + cl] = v;
        }
    }
}

}  // namespace

// By the length of the sums alone: a row's arithmetic does not depend on how many rows a call holds, so blocks of
// walkers and parts of a batch give the bits of the whole.  A few rows of the smallest systems lose 2 us to the second
// pass over them (8 orbitals and variables, up to 256 rows: 4.2 us in FP64, 6.2 here), 16384 rows gain (39 -> 23).
bool gemm_fix_supported(int K) { return K >= 1 && K <= 4096; }

cudaError_t gemm_fix_prepare(cudaStream_t s, int K, long long Nc, const double* U, int* uexp) {
    if (Nc <= 0 || K <= 0) return cudaSuccess;
    gf_colexp_kernel<<<(unsigned)std::min<long long>((Nc + 255) / 256, 1024), 256, 0, s>>>(K, Nc, U, uexp);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t gemm_fix(cudaStream_t s, int M, long long Nc, int K, const double* X, const double* U, const int* uexp, double* C) {
    if (!gemm_fix_supported(K)) return cudaErrorInvalidValue;
    if (M <= 0 || Nc <= 0) return cudaSuccess;
    int lg = 0;
    while ((1 << lg) < K) ++lg;
    const int b = std::min(58, 62 - lg), bx = b / 2, bu = b - bx;
    auto tiles = [&](int t) { return (long long)((Nc + t - 1) / t) * ((M + t - 1) / t); };
    auto grid = [&](int t) { return dim3((unsigned)((Nc + t - 1) / t), (unsigned)((M + t - 1) / t)); };
    if (tiles(64) >= 152) gemm_fix_kernel<4><<<grid(64), 256, 0, s>>>(M, Nc, K, X, U, uexp, C, bx, bu);
    else if (tiles(32) >= 152) gemm_fix_kernel<2><<<grid(32), 256, 0, s>>>(M, Nc, K, X, U, uexp, C, bx, bu);
    else gemm_fix_kernel<1><<<grid(16), 256, 0, s>>>(M, Nc, K, X, U, uexp, C, bx, bu);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace afq
