// Shared-memory-resident replicas of a batched ensemble.
//
// A replica of up to 4096 sites (64^2 FP32: 147 KB of populations) lives in
// one CTA's shared memory for a whole window of steps; a taller one (128^2)
// is split by rows over a cluster of C CTAs that read each other's boundary
// rows through distributed shared memory.  HBM is touched to load the state
// at the start of the window, to store it at the end and to write delta rho
// at a sampling step: a window of n steps moves 72 B per site once instead
// of n times.
//
// Layout of one CTA (rows [rank R, rank R + R) of its replica, R = ny / C): the nine
// population planes [9][R][nx] and the pseudopotential deviations of its rows with
// H halo rows and two halo columns on each side, kept twice (see step_pair).  A
// step is two phases with a barrier after each.  First every thread pulls its
// pairs of neighbouring sites, writes their delta psi (and the copies of it that
// the halo of its own or a neighbouring CTA needs) and keeps of the populations what
// the collision reads: mass and momentum on the unit-relaxation path, all nine
// otherwise.  Every read of the old state is then done, so the second phase
// collides and writes the new populations in place.  No site is computed twice and
// nothing is copied.  With C > 1 the rows beyond the CTA's are read, and the halo rows
// written, through distributed shared memory, and the barriers are the cluster's.
// The arithmetic, summation order and Philox counters are those of the tile path,
// so a resident replica evolves bit-identically to a single lattice with the same
// seed and replica index.
//
// Bound by latency: 64^2 on the unit path runs 32 warps an SM at 64 registers, 214
// instructions a site update, 46% of the issue slots busy; its warps wait for spilled
// registers and the shared-memory pipe.  1024 x 64^2: 81 GLUPS (56 with bands of rows
// swept in lock step, one column per thread at 16 warps an SM, 418 instructions, which
// pulled ten rows for eight and copied the boundary rows every step); 4096 x 32^2: 93 (60).
// 512 and 768 threads of more registers measured 74; the general path is faster at
// 512 (63) than at 384 (51).  One CTA a replica (C = 1), whose shared-memory loads the
// compiler interleaves over a thread's pairs, spills 208 bytes a thread at E4 and 256 to
// 272 at E6 and E8 (general path 480 to 612); the cluster forms none, or 112 to 116.
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbsc.h"
#include "lbsc_ens.cuh"

namespace lbsc {
namespace {

// Most sites per CTA, threads per CTA and pairs per thread of a path: the unit path
// holds three values of a pair across the barrier, the general path eighteen.
constexpr int kResMaxSites = 4096;
__host__ __device__ constexpr int res_threads(bool unit) { return unit ? 1024 : 512; }

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The float at the offset of `p` in the shared memory of cluster CTA `rank`.
__device__ __forceinline__ uint32_t map_cluster(const float *p, uint32_t rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    return ra;
}
__device__ __forceinline__ float ld_cluster(const float *p, uint32_t rank) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(map_cluster(p, rank))
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(float *p, uint32_t rank, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(map_cluster(p, rank)), "f"(v) : "memory");
}
template <int C>
__device__ __forceinline__ void sync_all() {
    if constexpr (C > 1) cluster_sync();
    else __syncthreads();
}

// `nsteps` steps of every replica in `list` (one shape, all of them on the unit
// path or none), C CTAs per replica.
template <int ORDER, int C, bool UNIT>
__global__ void __launch_bounds__(res_threads(UNIT))
ens_resident_kernel(const EnsRep *__restrict__ reps, const int *__restrict__ list,
                    const EnsClock *__restrict__ clk, int *flag, const EnsKeys keys, int nsteps,
                    int sample) {
    constexpr int H = Stencil<ORDER>::H;
    constexpr int NP = (kResMaxSites / 2 + res_threads(UNIT) - 1) / res_threads(UNIT);   // pairs a thread
    constexpr int NQ = UNIT ? 3 : 9;
    extern __shared__ __align__(16) float sm[];
    __shared__ KParams<float> sp;
    __shared__ uint32_t s_t0;
    __shared__ int s_cur;
    const uint32_t rank = C > 1 ? cluster_rank() : 0u;
    const EnsRep &R = reps[list[blockIdx.x / C]];
    const int nx = R.nx, ny = R.ny;
    const int rows = ny / C, ybase = (int)rank * rows;
    const uint32_t P = (uint32_t)rows * nx;                    // plane stride
    const int W = nx + 4;
    float *sa = sm + 9 * P, *sb = sa + (rows + 2 * H) * W;     // rows -H .. rows + H - 1
    if (threadIdx.x == 0) {
        s_t0 = __ldcg(&clk->t);
        s_cur = __ldcg(&clk->cur);
        fill_tile_params(sp, R, EnsTile(), s_t0, s_cur, false, flag);
    }
    __syncthreads();
    const uint32_t t0 = s_t0;
    const int cur = s_cur;
    const uint32_t gplane = (uint32_t)nx * ny;
    const uint32_t n4 = P / 4;   // float4 of a plane's own rows
    {
        const float4 *src = reinterpret_cast<const float4 *>(R.buf[cur]);
        for (uint32_t k = threadIdx.x; k < 9 * n4; k += blockDim.x) {
            const uint32_t i = k / n4, e = k - i * n4;
            reinterpret_cast<float4 *>(sm + i * P)[e] =
                __ldcg(src + (i * gplane + (uint32_t)ybase * nx) / 4 + e);
        }
    }
    const int npair = (int)P / 2, lg = __ffs(nx) - 2;          // nx / 2 = 1 << lg
    const uint32_t prev = (rank + C - 1) % C, next = (rank + 1) % C;
    sync_all<C>();
    for (int s = 0; s < nsteps; ++s) {
        float *drho = (sample && s == nsteps - 1) ? R.drho : nullptr;
        float2 q[NP][NQ];
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int idx = threadIdx.x + k * blockDim.x;
            if (idx >= npair) continue;
            const int y = idx >> lg, x = 2 * (idx & (nx / 2 - 1));
            const int xm = (x - 1) & (nx - 1), xq = (x + 2) & (nx - 1);
            // element (row yy, column c) of plane i, -1 <= yy <= rows
            auto ld = [&](int i, int yy, int c) {
                const float *pl = sm + i * P + c;
                if (C > 1 && yy < 0) return ld_cluster(pl + (rows - 1) * nx, prev);
                if (C > 1 && yy >= rows) return ld_cluster(pl, next);
                return pl[(yy < 0 ? rows - 1 : yy >= rows ? 0 : yy) * nx];
            };
            auto mid = [&](int i, int yy) {
                if (C > 1 && (yy < 0 || yy >= rows))
                    return make_float2(ld(i, yy, x), ld(i, yy, x + 1));
                return *reinterpret_cast<const float2 *>(
                    sm + i * P + (yy < 0 ? rows - 1 : yy >= rows ? 0 : yy) * nx + x);
            };
            auto plus = [&](int i, int yy) { return make_float2(ld(i, yy, xm), ld(i, yy, x)); };
            auto minus = [&](int i, int yy) {
                return make_float2(ld(i, yy, x + 1), ld(i, yy, xq));
            };
            const float2 g[9] = {mid(0, y),      plus(1, y),      mid(2, y - 1),
                                 minus(3, y),    mid(4, y + 1),   plus(5, y - 1),
                                 minus(6, y - 1), minus(7, y + 1), plus(8, y + 1)};
            const float2 s9 = sum9(g);
            const float2 d = delta_psi(s9, sp.psi_kind, sp.rho0, sp.psi_c, sp.psi_b);
            // delta psi into row r of the CTA `to`, with the periodic columns
            auto put = [&](int r, uint32_t to, bool remote) {
                float *a = sa + (r + H) * W + 2, *b = sb + (r + H) * W + 3;
                auto st = [&](float *q_, float v) {
                    if (remote) st_cluster(q_, to, v);
                    else *q_ = v;
                };
                st(a + x, d.x);
                st(a + x + 1, d.y);
                st(b + x, d.x);
                st(b + x + 1, d.y);
                if (x == 0) {
                    st(a + nx, d.x);
                    st(a + nx + 1, d.y);
                    st(b + nx, d.x);
                }
                if (x == nx - 2) {
                    st(a - 2, d.x);
                    st(a - 1, d.y);
                    st(b - 1, d.y);
                }
            };
            put(y, rank, false);
            if (y < H) put(rows + y, prev, C > 1);
            if (y >= rows - H) put(y - rows, next, C > 1);
            if constexpr (UNIT) {
                unit_moments(g, q[k][0], q[k][1], q[k][2]);
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) q[k][i] = g[i];
            }
            if (drho)
                *reinterpret_cast<float2 *>(drho + (uint32_t)(ybase + y) * nx + x) = s9;
        }
        sync_all<C>();   // delta psi is complete and the old state has been read
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int idx = threadIdx.x + k * blockDim.x;
            if (idx >= npair) continue;
            const int y = idx >> lg, x = 2 * (idx & (nx / 2 - 1));
            const float *a = sa + (y + H) * W + 2 + x, *b = sb + (y + H) * W + 2 + x;
            auto at = [&](int ex, int ey) {
                return *reinterpret_cast<const float2 *>(
                    ex == 1 ? b + ey * W + 2 : ex == -1 ? b + ey * W : a + ey * W + ex);
            };
            float2 sx, sy;
            force_sums<ORDER>(at, sx, sy);
            const float2 pf = vmul(bc<float2>(sp.force_pref), vadd(bc<float2>(sp.psi0), at(0, 0)));
            const float2 Fx = vmul(pf, sx), Fy = vmul(pf, sy);
            float2 f[9];
            const uint32_t site = (uint32_t)(ybase + y) * nx + x;
            if constexpr (UNIT)
                collide_unit_m(q[k][0], q[k][1], q[k][2], Fx, Fy, sp, keys.rk, site,
                               t0 + (uint32_t)s, f);
            else collide<float2>(q[k], Fx, Fy, sp, keys.rk, site, t0 + (uint32_t)s, f);
            float *w = sm + y * nx + x;
#pragma unroll
            for (int i = 0; i < 9; ++i) *reinterpret_cast<float2 *>(w + i * P) = f[i];
            const float2 chk = vadd(f[1], f[5]);
            if (!(fabsf(chk.x) <= 3.402823466e38f && fabsf(chk.y) <= 3.402823466e38f))
                atomicOr(flag, LB_STEP_NONFINITE);
        }
        sync_all<C>();   // the new state is complete
    }
    {
        float4 *dst = reinterpret_cast<float4 *>(R.buf[cur ^ (nsteps & 1)]);
        for (uint32_t k = threadIdx.x; k < 9 * n4; k += blockDim.x) {
            const uint32_t i = k / n4, e = k - i * n4;
            dst[(i * gplane + (uint32_t)ybase * nx) / 4 + e] =
                reinterpret_cast<const float4 *>(sm + i * P)[e];
        }
    }
}

template <int ORDER, int C>
const void *res_fn_u(bool unit) {
    return unit ? (const void *)ens_resident_kernel<ORDER, C, true>
                : (const void *)ens_resident_kernel<ORDER, C, false>;
}
template <int ORDER>
const void *res_fn_o(int C, bool unit) {
    switch (C) {
    case 1: return res_fn_u<ORDER, 1>(unit);
    case 2: return res_fn_u<ORDER, 2>(unit);
    case 4: return res_fn_u<ORDER, 4>(unit);
    case 8: return res_fn_u<ORDER, 8>(unit);
    default: return nullptr;
    }
}
const void *res_fn(int stencil, int C, bool unit) {
    return stencil == 4   ? res_fn_o<4>(C, unit)
           : stencil == 6 ? res_fn_o<6>(C, unit)
                          : res_fn_o<8>(C, unit);
}

// Threads of a CTA of `rows` rows: a pair of sites each, as far as they go.  On the
// general path (128 registers) one CTA of 32^2 then fills an SM, so with more CTAs
// than SMs (`many`) a thread takes two pairs and two CTAs overlap: 4096 x 32^2, tau
// 0.9, 54.8 us a step against 73.3 (four pairs 58.8); 152 replicas 4.3 against 4.4.
int res_block(int nx, int rows, bool unit, bool many) {
    const int pairs = rows * nx / (many && !unit ? 4 : 2);
    return pairs < res_threads(unit) ? (pairs + 31) / 32 * 32 : res_threads(unit);
}

}  // namespace

size_t resident_smem(int nx, int rows, int stencil) {
    const int H = stencil == 4 ? 1 : 2;
    if ((nx != 32 && nx != 64 && nx != 128) || rows < 8 || rows % 8 || rows * nx > kResMaxSites)
        return 0;
    return ((size_t)9 * rows * nx + (size_t)2 * (rows + 2 * H) * (nx + 4)) * sizeof(float);
}

cudaError_t resident_prepare(int stencil, int C, size_t smem) {
    for (bool unit : {false, true}) {
        const void *fn = res_fn(stencil, C, unit);
        if (!fn) return cudaErrorInvalidValue;
        const cudaError_t e =
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int resident_max_clusters(int stencil, int C, int nx, int rows, bool unit, bool many,
                          size_t smem) {
    const void *fn = res_fn(stencil, C, unit);
    if (!fn) return 0;
    const int threads = res_block(nx, rows, unit, many);
    if (C == 1) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem) != cudaSuccess)
            return 0;
        return n;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = C;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) return 0;
    return n;
}

cudaError_t launch_ens_resident(const ResLaunch &a, cudaStream_t s) {
    const void *fn = res_fn(a.stencil, a.C, a.unit);
    if (!fn || a.nres < 1) return cudaErrorInvalidValue;
    const int rows = a.ny / a.C;
    const size_t smem = resident_smem(a.nx, rows, a.stencil);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.nres * a.C);
    cfg.blockDim = dim3(res_block(a.nx, rows, a.unit, a.many));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = a.C;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = a.C > 1 ? 1 : 0;
    const EnsRep *reps = a.reps;
    const int *list = a.list;
    const EnsClock *clk = a.clk;
    int *flag = a.flag;
    const EnsKeys keys = a.keys;
    int nsteps = a.nsteps, sample = a.sample;
    void *args[] = {(void *)&reps, (void *)&list,   (void *)&clk,   (void *)&flag,
                    (void *)&keys, (void *)&nsteps, (void *)&sample};
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace lbsc
