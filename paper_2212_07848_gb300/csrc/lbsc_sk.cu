// Density structure factor S(k) = <|delta n(k)|^2> (defined after Eq. (12)
// of arXiv:2212.07848) accumulated on the device.
//
// One sample: delta rho [ny][nx] (written by the step kernel on sampling
// steps) -> row FFTs (two real rows packed into one complex transform) ->
// half spectrum [ny][ldx] -> column FFTs over tiles of adjacent columns ->
// acc[ky][kx] += |X(k)|^2 / (nx ny) in FP64.  The transforms are iterative
// radix-2 decimation-in-time FFTs in shared memory over power-of-two sizes,
// with twiddle tables computed once in FP64.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "lbsc_fft.cuh"
#include "lbsc_internal.cuh"

namespace lbsc {

// Twiddles e^{-2 pi i m / n}, m < n/2, evaluated in FP64.
template <typename T>
__global__ void twiddle_kernel(typename C2<T>::t *tw, int n) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= n / 2) return;
    double s, c;
    sincospi(2.0 * (double)m / (double)n, &s, &c);
    typename C2<T>::t v;
    v.x = (T)c;
    v.y = (T)(-s);
    tw[m] = v;
}

cudaError_t launch_twiddles(int precision, void *tw, int n, cudaStream_t s) {
    const int blocks = (n / 2 + 255) / 256;
    if (precision == 0)
        twiddle_kernel<float><<<blocks, 256, 0, s>>>((float2 *)tw, n);
    else
        twiddle_kernel<double><<<blocks, 256, 0, s>>>((double2 *)tw, n);
    return cudaGetLastError();
}

template <typename T>
__global__ void sk_rows_kernel(const T *__restrict__ drho, typename C2<T>::t *__restrict__ spec,
                               const typename C2<T>::t *__restrict__ tw, int nx, int log2nx,
                               int ldx) {
    sk_rows_block<T>(drho, spec, tw, nx, log2nx, ldx, blockIdx.x);
}

template <typename T>
__global__ void sk_cols_kernel(const typename C2<T>::t *__restrict__ spec, double *__restrict__ acc,
                               const typename C2<T>::t *__restrict__ tw, int nx, int ny,
                               int log2ny, int ldx, int cpb, double inv_n) {
    sk_cols_block<T>(spec, acc, tw, nx, ny, log2ny, ldx, cpb, inv_n, blockIdx.x * cpb);
}

template <typename T>
static cudaError_t sk_sample_t(const SkArgs &a, cudaStream_t s) {
    using CT = typename C2<T>::t;
    const int lx = ilog2(a.nx), ly = ilog2(a.ny);
    const size_t row_smem = (size_t)a.nx * sizeof(CT);
    const int cpb = cols_per_block(a.ny, sizeof(CT));
    const size_t col_smem = (size_t)cpb * a.ny * sizeof(CT);
    cudaError_t e;
    e = cudaFuncSetAttribute(sk_rows_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)row_smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(sk_cols_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)col_smem);
    if (e != cudaSuccess) return e;
    const int rthreads = a.nx / 2 < 512 ? (a.nx / 2 < 32 ? 32 : a.nx / 2) : 512;
    sk_rows_kernel<T><<<a.ny / 2, rthreads, row_smem, s>>>(
        (const T *)a.drho, (CT *)a.spec, (const CT *)a.tw_x, a.nx, lx, a.ldx);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int hx = a.nx / 2 + 1;
    const int cblocks = (hx + cpb - 1) / cpb;
    sk_cols_kernel<T><<<cblocks, 512, col_smem, s>>>((const CT *)a.spec, a.acc,
                                                     (const CT *)a.tw_y, a.nx, a.ny, ly,
                                                     a.ldx, cpb, 1.0 / ((double)a.nx * a.ny));
    return cudaGetLastError();
}

cudaError_t launch_sk_sample(int precision, const SkArgs &a, cudaStream_t s) {
    return precision == 0 ? sk_sample_t<float>(a, s) : sk_sample_t<double>(a, s);
}

// Mean over samples on the half plane, host layout [ny][nx/2+1]; k = 0 -> 0.
__global__ void sk_readout_kernel(const double *__restrict__ acc, double inv_count,
                                  double *__restrict__ out, int nx, int ny, int ldx) {
    const int hx = nx / 2 + 1;
    const size_t total = (size_t)hx * ny;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        const int ky = (int)(e / hx), kx = (int)(e % hx);
        out[e] = (kx == 0 && ky == 0) ? 0.0 : acc[(size_t)ky * ldx + kx] * inv_count;
    }
}

cudaError_t launch_sk_readout(const double *acc, double inv_count, double *out, int nx, int ny,
                              int ldx, cudaStream_t s) {
    const size_t total = (size_t)(nx / 2 + 1) * ny;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 152 * 16) blocks = 152 * 16;
    sk_readout_kernel<<<blocks, 256, 0, s>>>(acc, inv_count, out, nx, ny, ldx);
    return cudaGetLastError();
}

// Radial bins over the full plane: bin b = round(|k| / dk), dk = 2 pi / max(nx, ny);
// a half-plane column 0 < kx < nx/2 stands for two modes (k and -k).
//
// One block per bin gathers the modes of its annulus.  The sides are powers of
// two, so |k|^2 / dk^2 = m is an integer and round(sqrt(m)) = b is exactly
// b^2 - b < m <= b^2 + b: no square root, no atomics, no counters to clear, and
// a fixed summation order.  Where |kx| >= |ky| (in units of dk) a thread takes a
// row and the one or two columns of it inside the annulus, elsewhere a column
// and its rows.  The means and the context's status flag go straight to mapped
// host memory, so a read-out is one launch and one wait.  4096^2, 2048 bins:
// 55 us against 284 us for FP64 atomics per mode; bound by the gather's 32-byte
// sectors (a part of each is used).
__device__ __forceinline__ int first_at_least(int v, int s) {   // least k >= 0: (k s)^2 >= v
    if (v <= 0) return 0;
    int k = (int)(sqrtf((float)v) / (float)s);
    while (k * s * (k * s) < v) ++k;
    while (k > 0 && (k - 1) * s * ((k - 1) * s) >= v) --k;
    return k;
}

constexpr int kBinThreads = 256;

__global__ void __launch_bounds__(kBinThreads)
sk_bins_kernel(const double *__restrict__ acc, double inv_count, double *__restrict__ out,
               const int *__restrict__ flag, int *__restrict__ flag_out, int nx, int ny, int ldx) {
    const int b = blockIdx.x;
    const int L = max(nx, ny), sx = L / nx, sy = L / ny;
    const int lo2 = b * b - b + 1, hi2 = b * b + b;
    double s = 0.0;
    int cnt = 0;
    // rows: |my| sy <= kx sx
    const int ra = min(ny / 2, b / sy);
    for (int j = threadIdx.x; j <= 2 * ra; j += kBinThreads) {
        const int my = j - ra;
        if (2 * my == -ny) continue;             // the row ny/2 counts once
        const int qy = abs(my) * sy, qy2 = qy * qy;
        if (2 * qy2 > hi2) continue;
        const double *row = acc + (size_t)(my < 0 ? my + ny : my) * ldx;
        for (int kx = max((qy + sx - 1) / sx, first_at_least(lo2 - qy2, sx));
             kx <= nx / 2 && kx * sx * (kx * sx) + qy2 <= hi2; ++kx) {
            const bool once = kx == 0 || 2 * kx == nx;
            s += once ? row[kx] : 2.0 * row[kx];
            cnt += once ? 1 : 2;
        }
    }
    // columns: kx sx < |my| sy
    const int rb = min(nx / 2, b / sx);
    for (int kx = threadIdx.x; kx <= rb; kx += kBinThreads) {
        const int qx = kx * sx, qx2 = qx * qx;
        if (2 * qx2 >= hi2) continue;
        const bool once = kx == 0 || 2 * kx == nx;
        for (int my = max(qx / sy + 1, first_at_least(lo2 - qx2, sy));
             my <= ny / 2 && my * sy * (my * sy) + qx2 <= hi2; ++my) {
            double v = acc[(size_t)my * ldx + kx];
            int c = 1;
            if (2 * my != ny) {
                v += acc[(size_t)(ny - my) * ldx + kx];
                c = 2;
            }
            s += once ? v : 2.0 * v;
            cnt += once ? c : 2 * c;
        }
    }
    __shared__ double sh[kBinThreads / 32];
    __shared__ int shc[kBinThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, o);
        cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sh[threadIdx.x >> 5] = s;
        shc[threadIdx.x >> 5] = cnt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kBinThreads / 32; ++w) {
            s += sh[w];
            cnt += shc[w];
        }
        out[b] = cnt > 0 ? s * inv_count / (double)cnt : __longlong_as_double(0x7ff8000000000000ll);
        if (b == 0) *flag_out = *flag;
    }
}

cudaError_t launch_sk_bins(const double *acc, double inv_count, double *out, const int *flag,
                           int *flag_out, int nbins, int nx, int ny, int ldx, cudaStream_t s) {
    sk_bins_kernel<<<nbins, kBinThreads, 0, s>>>(acc, inv_count, out, flag, flag_out, nx, ny, ldx);
    return cudaGetLastError();
}

// First moments of the mean S(k) over the full plane (k = 0 excluded):
// out = (sum_k S(k), sum_k |k| S(k)), |k| = 2 pi sqrt((kx/nx)^2 + (ky/ny)^2)
// with folded indices; a half-plane column 0 < kx < nx/2 counts twice.  Two
// passes with a fixed launch shape and summation order: blocks over the rows
// my = 0 .. ny/2 (the rows my and -my share one square root of the integer
// |k|^2 in units of dk^2, the FP64 square root being what bounds the pass),
// then one block over their partial sums.  4096^2: 120 us for the two
// against 75.3 ms for one block of 256 threads over the whole plane.
constexpr int kMomThreads = 256;

__device__ __forceinline__ void block_sum2(double &a, double &b) {   // valid in thread 0
    __shared__ double sh[2][kMomThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = a;
        sh[1][threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kMomThreads / 32; ++w) {
            a += sh[0][w];
            b += sh[1][w];
        }
}

__global__ void __launch_bounds__(kMomThreads)
sk_moments_kernel(const double *__restrict__ acc, int nx, int ny, int ldx,
                  double *__restrict__ part) {
    const int hx = nx / 2 + 1;
    const int L = max(nx, ny), sx = L / nx, sy = L / ny;
    double s0 = 0.0, s1 = 0.0;
    for (int my = blockIdx.x; my <= ny / 2; my += gridDim.x) {
        const int qy2 = my * sy * (my * sy);
        const double *up = acc + (size_t)my * ldx, *dn = acc + (size_t)(ny - my) * ldx;
        const bool two = my > 0 && 2 * my < ny;
        for (int kx = threadIdx.x; kx < hx; kx += kMomThreads) {
            if (kx == 0 && my == 0) continue;
            double S = two ? up[kx] + dn[kx] : up[kx];
            if (kx > 0 && 2 * kx < nx) S += S;
            s0 += S;
            s1 += S * sqrt((double)(kx * sx * (kx * sx) + qy2));
        }
    }
    block_sum2(s0, s1);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = s0;
        part[2 * blockIdx.x + 1] = s1;
    }
}

__global__ void __launch_bounds__(kMomThreads)
sk_moments_final_kernel(const double *__restrict__ part, int nblocks, double inv_count, int L,
                        double *__restrict__ out, const int *__restrict__ flag,
                        int *__restrict__ flag_out) {
    double s0 = 0.0, s1 = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kMomThreads) {
        s0 += part[2 * b];
        s1 += part[2 * b + 1];
    }
    block_sum2(s0, s1);
    if (threadIdx.x == 0) {
        out[0] = s0 * inv_count;
        out[1] = s1 * inv_count * (6.283185307179586 / L);
        *flag_out = *flag;
    }
}

cudaError_t launch_sk_moments(const double *acc, double inv_count, int nx, int ny, int ldx,
                              double *part, int nblocks, double *out2, const int *flag,
                              int *flag_out, cudaStream_t s) {
    const int nb = nblocks < ny / 2 + 1 ? nblocks : ny / 2 + 1;
    sk_moments_kernel<<<nb, kMomThreads, 0, s>>>(acc, nx, ny, ldx, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sk_moments_final_kernel<<<1, kMomThreads, 0, s>>>(part, nb, inv_count, nx > ny ? nx : ny, out2,
                                                      flag, flag_out);
    return cudaGetLastError();
}

}  // namespace lbsc
