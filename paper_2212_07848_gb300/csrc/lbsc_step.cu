// Fused fluctuating Shan-Chen D2Q9 time step (Eq. (12) of arXiv:2212.07848):
// pull streaming -> density -> pseudopotential on the tile and its halo ->
// Shan-Chen force, Eq. (1) -> moments -> BGK + Guo source -> Philox noise on
// the non-conserved moments -> inverse transform -> store.
//
// Layout: populations are stored as deviations delta f_i = f_i - w_i rho0,
// structure of arrays [9][ny][nx] (x fastest), two buffers swapped per step.
// Storing deviations keeps the relative precision of density fluctuations of
// size sqrt(kT) in FP32.
//
// Three kernels, the same arithmetic per site and so the same bits:
//
// step_kernel_pair (FP32, large lattices): a group of NT threads owns a strip of
// columns, two to a thread, and sweeps strip_h rows (step_pair).  Each iteration
// pulls one new row, writes its pseudopotential deviation into a shared-memory
// ring of rows, and collides the row H above it, whose 2H+1 pseudopotential rows
// are then complete; what the collision needs of the last rows stays in
// registers and the next row's loads are prefetched, so every population is read
// from DRAM once per step.  Bound by DRAM at 4096^2 (188 us = 89 GLUPS at 72
// B/site, 0.95 of the measured copy rate; one column per thread in 128-column
// strips with scalar arithmetic took 220 us, bound by issue: 391 instructions a
// site against 280 now (2048^2, bands of 44 rows), by the packed FP32 instructions,
// the shared addresses and the 8-byte accesses) and by latency below that (2048^2:
// 61% of the issue slots, 17 warps an SM, 64% of the DRAM peak).
// 96 registers (ten 64-thread groups an SM) is the fewest without spills on the
// unit-relaxation path: eleven and more groups measured 237-290 us, eight 217.
//
// step_kernel_pair_tile (FP32, smaller lattices): one thread per pair of sites of a
// 32 x 8 tile, all rows at once.  A strip sweep is one long dependent program
// per thread (about 1 us a row), which a lattice of a few hundred thousand sites
// cannot hide; the tile trades a ring of recomputed halo pseudopotentials (36% of
// the sites for E4) for a single barrier and many more warps in flight.  us per
// step, old strips -> this: 64^2 6.8 -> 2.7, 512^2 9.7 -> 5.2, 1024^2 17.9 -> 14.4.
// Tiles of 32 x 4, 32 x 12, 32 x 16, 16 x 16, 64 x 8 and 64 x 16 measured 0-25% slower.
//
// step_kernel_tile (FP64): one thread per site of a tile.  FP64 is bound by the FP64
// pipe (about 390 FP64 instructions a site at two a clock and SM) wherever the
// lattice fills the chip; 128^2 takes 16.1 us in 128 tiles of 16 x 8 (121 us in
// sixteen strips of 8 rows, the default before), 1024^2 681 us (762 us in strips).
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbsc_collide.cuh"
#include "lbsc_device.cuh"
#include "lbsc_internal.cuh"
#include "lbsc_strip.cuh"

namespace lbsc {

// Resident threads per SM that the strip kernel is compiled for: the most without
// spilled registers on the unit path; the general path keeps all nine populations
// of its rows and measured fastest at 512 (2048^2, tau 0.8: 67 us against 69-95).
__host__ __device__ constexpr int kPairThreads(bool unit) { return unit ? 640 : 512; }

// FP32: a group of NT threads, two columns each (step_pair).
template <int ORDER, bool SAMPLE, bool UNIT, int NT>
__global__ void __launch_bounds__(NT, kPairThreads(UNIT) / NT)
step_kernel_pair(const KParams<float> p, const PairShape shape) {
    const int y0 = blockIdx.y * p.strip_h * shape.bands;
    step_pair<ORDER, SAMPLE, false, UNIT, NT>(p, p.rk, shape, blockIdx.x * shape.cols, y0,
                                              p.strip_h, p.ny);
}

// FP64: one thread per site of a TX x TY tile, every row at once.  The tile's ring
// of halo pseudopotentials, H wide, is recomputed by the CTA's first threads; one
// barrier, no row loop.
// TALL: one of several launches over a lattice of more rows of tiles than a grid's
// second dimension holds; its first row is row0.
constexpr int kGridRows = 65535;
template <typename T, int ORDER, bool SAMPLE, bool UNIT, int TX, int TY, bool TALL>
__global__ void __launch_bounds__(TX *TY) step_kernel_tile(const KParams<T> p, const int row0) {
    constexpr int H = Stencil<ORDER>::H, W = TX + 2 * H, NT = TX * TY;
    constexpr int kRing = W * (TY + 2 * H) - NT;   // rows above and below, then the sides
    __shared__ T s_psi[TY + 2 * H][W];
    const int nx = p.nx, ny = p.ny;
    const size_t plane = (size_t)nx * ny;
    const int x0 = blockIdx.x * TX, y0 = (TALL ? row0 : 0) + blockIdx.y * TY;
    // populations of the site (x0 + i, y0 + j), -H <= i < TX + H, periodic (a tile
    // may reach past the lattice's edge by more than its size)
    auto pull_at = [&](int i, int j, T g[9], int &x, int &y) {
        x = x0 + i;
        y = y0 + j;
        while (x < 0) x += nx;
        while (x >= nx) x -= nx;
        while (y < 0) y += ny;
        while (y >= ny) y -= ny;
        pull(p.src, plane, nx, x, x == 0 ? nx - 1 : x - 1, x == nx - 1 ? 0 : x + 1, y,
             y == 0 ? ny - 1 : y - 1, y == ny - 1 ? 0 : y + 1, g);
    };
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    T g[9];
    int x, y;
    pull_at(tx, ty, g, x, y);
    for (int e = tid; e < kRing; e += NT) {
        int i, j;
        if (e < 2 * H * W) {
            const int r = e / W;
            i = e % W - H;
            j = r < H ? r - H : TY + r - H;
        } else {
            const int f = e - 2 * H * W, c = f % (2 * H);
            i = c < H ? c - H : TX + c - H;
            j = f / (2 * H);
        }
        T gh[9];
        int xh, yh;
        pull_at(i, j, gh, xh, yh);
        s_psi[j + H][i + H] = delta_psi(sum9(gh), p.psi_kind, p.rho0, p.psi_c, p.psi_b);
    }
    s_psi[ty + H][tx + H] = delta_psi(sum9(g), p.psi_kind, p.rho0, p.psi_c, p.psi_b);
    __syncthreads();
    if (x0 + tx >= nx || y0 + ty >= ny) return;
    auto at = [&](int ex, int ey) { return s_psi[ty + H + ey][tx + H + ex]; };
    T sx, sy;
    force_sums<ORDER>(at, sx, sy);
    const T pf = vmul(p.force_pref, vadd(p.psi0, at(0, 0)));
    const T Fx = vmul(pf, sx), Fy = vmul(pf, sy);
    const uint32_t site = (uint32_t)y * (uint32_t)nx + (uint32_t)x, step = step_of(p);
    T f[9];
    if constexpr (UNIT) {
        T drho, m1, m2;
        unit_moments(g, drho, m1, m2);
        collide_unit_m(drho, m1, m2, Fx, Fy, p, p.rk, site, step, f);
    } else {
        collide<T>(g, Fx, Fy, p, p.rk, site, step, f);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) p.dst[i * plane + site] = f[i];
    if (SAMPLE) p.drho_out[site] = sum9(g);
    if (!isfinite(f[1] + f[5])) atomicOr(p.flag, LB_STEP_NONFINITE);
}

template <typename T, int ORDER, int TX, int TY, bool TALL = false>
static cudaError_t launch_tile_t(const StepArgs &a, cudaStream_t s, int row0 = 0) {
    const KParams<T> k = make_params<T>(a);
    const int rows = (a.ny - row0 + TY - 1) / TY;
    const dim3 grid((a.nx + TX - 1) / TX, rows < kGridRows ? rows : kGridRows);
#define TILE(SAMPLE, UNIT)                                                                   \
    step_kernel_tile<T, ORDER, SAMPLE, UNIT, TX, TY, TALL><<<grid, TX * TY, 0, s>>>(k, row0)
    if (k.unit) {
        if (a.drho_out) TILE(true, true);
        else TILE(false, true);
    } else {
        if (a.drho_out) TILE(true, false);
        else TILE(false, false);
    }
#undef TILE
    return cudaGetLastError();
}

// The same tile in packed FP32: TX x TY sites by TX / 2 x TY threads, two neighbouring
// columns each; the halo ring is two columns wide on both sides whatever H.
template <int ORDER, bool SAMPLE, bool UNIT, int TX, int TY>
__global__ void __launch_bounds__(TX / 2 * TY, ORDER == 4 ? 8 : 10)
step_kernel_pair_tile(const KParams<float> p) {
    constexpr int H = Stencil<ORDER>::H, W = TX + 4, NT = TX / 2 * TY;
    constexpr int kRing = W / 2 * (TY + 2 * H) - NT;   // pairs above and below, then the sides
    // delta psi: s_a[.][i] is column i - 2, s_b[.][i] column i - 3 (see step_pair)
    __shared__ __align__(8) float s_a[TY + 2 * H][W], s_b[TY + 2 * H][W];
    const int nx = p.nx, ny = p.ny;
    const size_t pl = (size_t)nx * ny;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    // populations of the sites (x0 + i, y0 + j) and (x0 + i + 1, y0 + j), periodic
    auto pull_at = [&](int i, int j, float2 g[9], int &x, int &y) {
        x = x0 + i;
        y = y0 + j;
        while (x < 0) x += nx;
        while (x >= nx) x -= nx;
        while (y < 0) y += ny;
        while (y >= ny) y -= ny;
        const uint32_t r1 = (uint32_t)y * (uint32_t)nx;
        const uint32_t r0 = y == 0 ? (uint32_t)(ny - 1) * nx : r1 - nx;
        const uint32_t r2 = y == ny - 1 ? 0u : r1 + nx;
        pull2<false>(p.src, pl, r0, r1, r2, x, x == 0 ? nx - 1 : x - 1, x + 2 == nx ? 0 : x + 2, g);
    };
    auto put = [&](int i, int j, float2 d) {
        *reinterpret_cast<float2 *>(&s_a[j + H][i + 2]) = d;
        s_b[j + H][i + 3] = d.x;
        if (i + 4 < W) s_b[j + H][i + 4] = d.y;
    };
    const int tid = threadIdx.x, tx = 2 * (tid % (TX / 2)), ty = tid / (TX / 2);
    float2 g[9];
    int x, y;
    pull_at(tx, ty, g, x, y);
    for (int e = tid; e < kRing; e += NT) {
        int i, j;
        if (e < H * W) {
            const int r = e / (W / 2);
            i = 2 * (e % (W / 2)) - 2;
            j = r < H ? r - H : TY + r - H;
        } else {
            const int f = e - H * W;
            i = f & 1 ? TX : -2;
            j = f >> 1;
        }
        float2 gh[9];
        int xh, yh;
        pull_at(i, j, gh, xh, yh);
        put(i, j, delta_psi(sum9(gh), p.psi_kind, p.rho0, p.psi_c, p.psi_b));
    }
    put(tx, ty, delta_psi(sum9(g), p.psi_kind, p.rho0, p.psi_c, p.psi_b));
    __syncthreads();
    if (x0 + tx >= nx || y0 + ty >= ny) return;
    auto at = [&](int ex, int ey) {
        const float *a = s_a[ty + H + ey] + tx + 2, *b = s_b[ty + H + ey] + tx + 2;
        return *reinterpret_cast<const float2 *>(ex == 1 ? b + 2 : ex == -1 ? b : a + ex);
    };
    float2 sx, sy;
    force_sums<ORDER>(at, sx, sy);
    const float2 pf = vmul(bc<float2>(p.force_pref), vadd(bc<float2>(p.psi0), at(0, 0)));
    const float2 Fx = vmul(pf, sx), Fy = vmul(pf, sy);
    const uint32_t o = (uint32_t)y * (uint32_t)nx + (uint32_t)x, step = step_of(p);
    float2 f[9];
    if constexpr (UNIT) {
        float2 drho, m1, m2;
        unit_moments(g, drho, m1, m2);
        collide_unit_m(drho, m1, m2, Fx, Fy, p, p.rk, o, step, f);
    } else {
        collide<float2>(g, Fx, Fy, p, p.rk, o, step, f);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) st_off(p.dst + i * pl, o, f[i]);
    if (SAMPLE) st_off(p.drho_out, o, sum9(g));
    const float2 chk = vadd(f[1], f[5]);
    if (!(fabsf(chk.x) <= 3.402823466e38f && fabsf(chk.y) <= 3.402823466e38f))
        atomicOr(p.flag, LB_STEP_NONFINITE);
}

template <int ORDER, int TX, int TY>
static cudaError_t launch_pair_tile_t(const StepArgs &a, cudaStream_t s) {
    const KParams<float> k = make_params<float>(a);
    const dim3 grid((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY);
    constexpr int N = TX / 2 * TY;
    if (k.unit) {
        if (a.drho_out) step_kernel_pair_tile<ORDER, true, true, TX, TY><<<grid, N, 0, s>>>(k);
        else step_kernel_pair_tile<ORDER, false, true, TX, TY><<<grid, N, 0, s>>>(k);
    } else {
        if (a.drho_out) step_kernel_pair_tile<ORDER, true, false, TX, TY><<<grid, N, 0, s>>>(k);
        else step_kernel_pair_tile<ORDER, false, false, TX, TY><<<grid, N, 0, s>>>(k);
    }
    return cudaGetLastError();
}

template <int ORDER, int NT>
static cudaError_t launch_pair_t(const StepArgs &a, cudaStream_t s) {
    const KParams<float> k = make_params<float>(a);
    const PairShape shape = pair_shape(a.nx, NT);
    const int rows = a.strip_h * shape.bands;
    const dim3 grid(shape.strips, (a.ny + rows - 1) / rows);
    if (k.unit) {
        if (a.drho_out) step_kernel_pair<ORDER, true, true, NT><<<grid, NT, 0, s>>>(k, shape);
        else step_kernel_pair<ORDER, false, true, NT><<<grid, NT, 0, s>>>(k, shape);
    } else {
        if (a.drho_out) step_kernel_pair<ORDER, true, false, NT><<<grid, NT, 0, s>>>(k, shape);
        else step_kernel_pair<ORDER, false, false, NT><<<grid, NT, 0, s>>>(k, shape);
    }
    return cudaGetLastError();
}

template <int ORDER>
static cudaError_t launch_f32(const StepArgs &a, cudaStream_t s) {
    if (a.layout == kLayoutTile) return launch_pair_tile_t<ORDER, 32, 8>(a, s);
    return a.layout == kLayoutWide ? launch_pair_t<ORDER, 128>(a, s) : launch_pair_t<ORDER, 64>(a, s);
}

// Small FP64 lattices take the smaller tile, which spreads them over more SMs
// (128^2: 16 against 27 us; 1024^2: 1% slower).  A lattice of more than 524280 rows
// takes a launch for each kGridRows rows of tiles.
template <int ORDER>
static cudaError_t launch_f64(const StepArgs &a, cudaStream_t s) {
    if (a.ny > 8 * kGridRows) {
        cudaError_t e = cudaSuccess;
        for (int r = 0; r < a.ny && e == cudaSuccess; r += 8 * kGridRows)
            e = launch_tile_t<double, ORDER, 16, 8, true>(a, s, r);
        return e;
    }
    return (size_t)a.nx * a.ny < (1u << 17) ? launch_tile_t<double, ORDER, 16, 8>(a, s)
                                            : launch_tile_t<double, ORDER, 32, 8>(a, s);
}

// FP32, no strip height or wide strips asked for: tiles up to the size where the
// strips have caught up.  us per step, tiles / strips: unit rates E4 1024^2 14.4 /
// 15.4, 1500 x 1000 22.0 / 22.5, 2048^2 59.9 / 52.8; general rates E4 708 x 452 6.1 /
// 8.0, 2048^2 62 / 67, 4096^2 238 / 234; E8 general 512^2 5.9 / 9.1, 2048^2 66 / 74,
// 4096^2 255 / 234.  Never for more rows of tiles than a grid has.
bool tile_is_faster(int nx, int ny, bool unit) {
    return ny <= 8 * kGridRows &&
           (size_t)nx * ny <= (unit ? (size_t)3 << 19 : (size_t)1 << 23);
}

// Rows per band of a strip: the fewest waves of resident groups whose bands are at
// most 128 rows high, filled evenly (4096^2, 128-thread groups: one wave of 88 rows
// 188 us, two of 44 191, three of 30 201; a partly filled second wave of 64 225).
int strip_rows(int nx, int ny, int layout, bool unit) {
    const int nt = layout == kLayoutWide ? 128 : 64;
    const PairShape shape = pair_shape(nx, nt);
    const long slots = 152L * kPairThreads(unit) / nt;
    for (long waves = 1;; ++waves) {
        const long groups = waves * slots / shape.strips;   // per strip of columns
        if (groups < 1) continue;
        const long rows = (ny + groups - 1) / groups;       // of a group, over its bands
        const long h = (rows + shape.bands - 1) / shape.bands;
        if (h <= 128) return (int)h;
    }
}

cudaError_t launch_step(int precision, int stencil, const StepArgs &a, cudaStream_t s) {
    if (precision == 0) {
        if (stencil == 4) return launch_f32<4>(a, s);
        if (stencil == 6) return launch_f32<6>(a, s);
        if (stencil == 8) return launch_f32<8>(a, s);
    } else {
        if (stencil == 4) return launch_f64<4>(a, s);
        if (stencil == 6) return launch_f64<6>(a, s);
        if (stencil == 8) return launch_f64<8>(a, s);
    }
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Initial state: delta f_i = w_i * amp * z(site), z from Philox block 2 of
// step 0 (amp = 0: the homogeneous state at rest).
// ---------------------------------------------------------------------------
struct InitKeys {
    uint32_t rk[20];
};

template <typename T>
__global__ void init_kernel(T *__restrict__ df, int nx, int ny, T amp, InitKeys keys,
                            uint32_t replica) {
    const size_t plane = (size_t)nx * ny;
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < plane;
         s += (size_t)gridDim.x * blockDim.x) {
        T d = T(0);
        if (amp != T(0)) {
            uint4 r = philox4x32_10(make_uint4((uint32_t)s, 0u, replica, 2u), keys.rk);
            T z0, z1;
            box_muller(uniform01<T>(r.x), uniform01<T>(r.y), z0, z1);
            d = amp * z0;
        }
        df[0 * plane + s] = T(4.0 / 9.0) * d;
#pragma unroll
        for (int i = 1; i < 5; ++i) df[i * plane + s] = T(1.0 / 9.0) * d;
#pragma unroll
        for (int i = 5; i < 9; ++i) df[i * plane + s] = T(1.0 / 36.0) * d;
    }
}

cudaError_t launch_init(int precision, void *df, int nx, int ny, double amp,
                        const uint32_t round_keys[20], uint32_t replica, cudaStream_t s) {
    InitKeys k;
    for (int i = 0; i < 20; ++i) k.rk[i] = round_keys[i];
    const size_t plane = (size_t)nx * ny;
    int blocks = (int)((plane + 255) / 256);
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (precision == 0)
        init_kernel<float><<<blocks, 256, 0, s>>>((float *)df, nx, ny, (float)amp, k, replica);
    else
        init_kernel<double><<<blocks, 256, 0, s>>>((double *)df, nx, ny, amp, k, replica);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Density of the stored state: rho = rho0 + sum_i delta f_i (FP64 output),
// and the delta rho field in storage precision for an unscheduled S(k) sample.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void density_kernel(const T *__restrict__ df, double rho0, double *__restrict__ out,
                               size_t plane) {
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < plane;
         s += (size_t)gridDim.x * blockDim.x) {
        T g[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = df[i * plane + s];
        out[s] = rho0 + (double)sum9(g);
    }
}

template <typename T>
__global__ void drho_kernel(const T *__restrict__ df, T *__restrict__ out, size_t plane) {
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < plane;
         s += (size_t)gridDim.x * blockDim.x) {
        T g[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = df[i * plane + s];
        out[s] = sum9(g);
    }
}

cudaError_t launch_density(int precision, const void *df, double rho0, double *out, int nx,
                           int ny, cudaStream_t s) {
    const size_t plane = (size_t)nx * ny;
    int blocks = (int)((plane + 255) / 256);
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (precision == 0)
        density_kernel<float><<<blocks, 256, 0, s>>>((const float *)df, rho0, out, plane);
    else
        density_kernel<double><<<blocks, 256, 0, s>>>((const double *)df, rho0, out, plane);
    return cudaGetLastError();
}

cudaError_t launch_drho(int precision, const void *df, void *drho, int nx, int ny,
                        cudaStream_t s) {
    const size_t plane = (size_t)nx * ny;
    int blocks = (int)((plane + 255) / 256);
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (precision == 0)
        drho_kernel<float><<<blocks, 256, 0, s>>>((const float *)df, (float *)drho, plane);
    else
        drho_kernel<double><<<blocks, 256, 0, s>>>((const double *)df, (double *)drho, plane);
    return cudaGetLastError();
}

}  // namespace lbsc
