// The fused D2Q9 step of FP32 lattices for one strip of columns (shared by the
// single-lattice kernel and the batched ensemble kernels).  See lbsc_step.cu for
// the design.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbsc_collide.cuh"
#include "lbsc_device.cuh"
#include "lbsc_internal.cuh"

namespace lbsc {

// ---------------------------------------------------------------------------
// FP32: two neighbouring columns per thread, so that the floating-point work
// of both runs in packed two-site instructions (float2), the populations of
// c_x = 0 and all stores move 8 bytes, and the address, loop and barrier
// instructions are shared.
//
// A group of NT threads sweeps a strip of up to 2 NT columns.  Lattices wider than
// that are cut into strips of equal width; then one warp also recomputes the
// pseudopotential of the strip's 2H halo columns, one lane per (column,
// population): a single load and four shuffle-adds a row, in the summation order
// of sum9.  A lattice that fits one strip needs no halo columns (the edge
// threads store their values a second time), and one of at most NT columns
// leaves room for several bands of rows side by side.
// ---------------------------------------------------------------------------
constexpr int kMaxBands = 8;

// How a lattice nx wide is cut for groups of nt threads: columns per strip (the
// last may be narrower), strips, and bands of rows per group.
struct PairShape {
    int cols, strips, bands;
};
__host__ __device__ inline PairShape pair_shape(int nx, int nt) {
    PairShape s;
    const int n = (nx + 2 * nt - 1) / (2 * nt);
    s.cols = ((nx + n - 1) / n + 1) / 2 * 2;
    s.strips = (nx + s.cols - 1) / s.cols;
    const int b = 2 * nt / s.cols;
    s.bands = s.strips > 1 ? 1 : (b < kMaxBands ? b : kMaxBands);
    return s;
}

// Address of element `o` of a plane: one widening multiply-add from the plane's
// uniform start, so that one 32-bit offset a thread serves every plane.
__device__ __forceinline__ uint64_t at_elem(const float *plane, uint32_t o) {
    uint64_t a;
    asm("mad.wide.u32 %0, %1, 4, %2;" : "=l"(a) : "r"(o), "l"(plane));
    return a;
}
template <typename V, bool CG>
__device__ __forceinline__ V ld_off(const float *plane, uint32_t o) {
    const V *q = reinterpret_cast<const V *>(at_elem(plane, o));
    if constexpr (CG) return __ldcg(q);
    else return __ldg(q);
}
__device__ __forceinline__ void st_off(float *plane, uint32_t o, float2 v) {
    *reinterpret_cast<float2 *>(at_elem(plane, o)) = v;
}

// Pull streaming of the sites x, x + 1 (x even): r0, r1, r2 are the offsets of the
// rows y - 1, y, y + 1; xm = x - 1 and xq = x + 2, wrapped.
template <bool CG>
__device__ __forceinline__ void pull2(const float *__restrict__ src, size_t pl, uint32_t r0,
                                      uint32_t r1, uint32_t r2, uint32_t x, uint32_t xm,
                                      uint32_t xq, float2 g[9]) {
    auto mid = [&](int i, uint32_t r) { return ld_off<float2, CG>(src + i * pl, r + x); };
    auto plus = [&](int i, uint32_t r) {    // c_x = 1
        return make_float2(ld_off<float, CG>(src + i * pl, r + xm),
                           ld_off<float, CG>(src + i * pl, r + x));
    };
    auto minus = [&](int i, uint32_t r) {   // c_x = -1
        return make_float2(ld_off<float, CG>(src + i * pl + 1, r + x),
                           ld_off<float, CG>(src + i * pl, r + xq));
    };
    g[0] = mid(0, r1);
    g[1] = plus(1, r1);
    g[2] = mid(2, r0);
    g[3] = minus(3, r1);
    g[4] = mid(4, r2);
    g[5] = plus(5, r0);
    g[6] = minus(6, r0);
    g[7] = minus(7, r2);
    g[8] = plus(8, r2);
}

// One group's work: the strip of columns [x0, x0 + ncol) of `shape`, rows
// [y0, yend) in bands of `h` rows (band b starts at y0 + b h).
template <int ORDER, bool SAMPLE, bool CG, bool UNIT, int NT>
__device__ __forceinline__ void step_pair(const KParams<float> &p,
                                          const uint32_t *__restrict__ rk, const PairShape shape,
                                          int x0, int y0, int h, int yend) {
    constexpr int H = Stencil<ORDER>::H;
    constexpr int RING = (H == 1) ? 4 : 8;   // >= 2H + 2 rows, power of two
    constexpr int SW = 2 * NT + 4 * kMaxBands;
    // delta psi of the last rows, twice: s_a[j] is column j, s_b[j] column j - 1, so
    // that the pairs (x, x + 1), (x - 1, x) and (x + 1, x + 2) are all aligned
    __shared__ __align__(8) float s_a[RING][SW], s_b[RING][SW];

    const int nx = p.nx, ny = p.ny;
    const size_t pl = (size_t)nx * ny;
    const int tid = threadIdx.x, tb = shape.cols / 2;
    const int band = shape.bands > 1 ? tid / tb : 0, c = 2 * (tid - band * tb);
    const int ncol = min(shape.cols, nx - x0);
    const int yb = y0 + band * h, hb = min(h, yend - yb);
    const bool active = band < shape.bands && c < ncol && hb > 0;
    const int base = band * (shape.cols + 4);
    const int j = base + 2 + c;   // this pair's slot in a ring row
    const bool whole = shape.strips == 1;
    const bool first = active && whole && c == 0, last = active && whole && c == ncol - 2;

    const uint32_t x = active ? (uint32_t)(x0 + c) : 0u;
    const uint32_t xm = x == 0u ? (uint32_t)nx - 1u : x - 1u;   // idle threads pull column 0
    const uint32_t xq = x + 2u == (uint32_t)nx ? 0u : x + 2u;

    // halo columns of a strip (shape.bands == 1): 16 lanes a column, lane k < 9 of
    // them loads population k.  H = 1: the two columns by one warp, the warps in
    // turn; H = 2: the left two by warp 0, the right two by warp 1.
    constexpr int kWarps = NT / 32;
    const int lane = tid & 31, warp = tid >> 5, k = lane & 15, u = lane >> 4;
    const bool side = !whole && (H == 1 || warp < 2);
    const int hc = H == 1 ? (u ? ncol : -1) : (warp == 0 ? u - 2 : ncol + u);   // column
    const uint32_t cxm = 0x122u, cxp = 0x0c8u;   // lanes (c_x = 1 at k 1, 5, 8; -1 at 3, 6, 7)
    const int ecx = (cxm >> k) & 1u ? 1 : ((cxp >> k) & 1u ? -1 : 0);
    const int ecy = k == 2 || k == 5 || k == 6 ? 1 : (k == 4 || k == 7 || k == 8 ? -1 : 0);
    const float *hp = p.src;
    if (side) hp += (k < 9 ? k : 0) * pl + wrap_once(wrap_once(x0 + hc, nx) - ecx, nx);

    const float rho0 = p.rho0;
    const uint32_t step = step_of(p);

    // what a row keeps for its collision H rows later: the nine pulled populations,
    // or on the unit-relaxation path only their mass and momentum
    // (and their sum, where the sample is written)
    constexpr int NQ = UNIT ? (SAMPLE ? 4 : 3) : 9;
    float2 q[H + 1][NQ];
#pragma unroll
    for (int r = 0; r <= H; ++r)
#pragma unroll
        for (int i = 0; i < NQ; ++i) q[r][i] = make_float2(0.f, 0.f);

    const int it_end = min(h, yend - y0) + 2 * H;   // the same for every band of the group
    int yn = hb > 0 ? wrap_once(yb - H, ny) : 0;     // the row being prefetched
    uint32_t r1 = (uint32_t)yn * (uint32_t)nx;
    uint32_t r0 = (uint32_t)(yn == 0 ? ny - 1 : yn - 1) * (uint32_t)nx;
    yn = yn == ny - 1 ? 0 : yn + 1;
    uint32_t r2 = (uint32_t)yn * (uint32_t)nx;
    float2 gn[9];
    float hn = 0.f;
    pull2<CG>(p.src, pl, r0, r1, r2, x, xm, xq, gn);
    if (side && (H > 1 || warp == 0)) hn = ld_off<float, CG>(hp, ecy > 0 ? r0 : ecy < 0 ? r2 : r1);
#pragma unroll 2
    for (int it = 0; it < it_end; ++it) {
        const int slot = it & (RING - 1);
        float2 g[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = gn[i];
        const float hv = hn;
        // Register prefetch: the next row's loads are in flight during this
        // row's arithmetic (the last row's are repeated, from L1)
        if (it + 1 < it_end) {
            r0 = r1;
            r1 = r2;
            yn = yn == ny - 1 ? 0 : yn + 1;
            r2 = yn == 0 ? 0u : r2 + (uint32_t)nx;
        }
        pull2<CG>(p.src, pl, r0, r1, r2, x, xm, xq, gn);
        if (side && (H > 1 || (it + 1) % kWarps == warp))
            hn = ld_off<float, CG>(hp, ecy > 0 ? r0 : ecy < 0 ? r2 : r1);
        const float2 s9 = sum9(g);
        if (active) {
            const float2 d = delta_psi(s9, p.psi_kind, rho0, p.psi_c, p.psi_b);
            *reinterpret_cast<float2 *>(&s_a[slot][j]) = d;
            s_b[slot][j + 1] = d.x;
            s_b[slot][j + 2] = d.y;
            if (first) {   // columns ncol, ncol + 1
                *reinterpret_cast<float2 *>(&s_a[slot][j + ncol]) = d;
                s_b[slot][j + ncol + 1] = d.x;
            }
            if (last) {    // columns -2, -1
                *reinterpret_cast<float2 *>(&s_a[slot][base]) = d;
                s_b[slot][base + 2] = d.y;
            }
        }
        if (side && (H > 1 || it % kWarps == warp)) {
            // sum9 over the lanes: (1 + 3), (2 + 4), (5 + 7), (6 + 8) are two lanes apart
            const unsigned full = 0xffffffffu;
            const float s2 = vadd(hv, __shfl_down_sync(full, hv, 2));
            const float s3 = vadd(k == 0 ? hv : s2, __shfl_down_sync(full, s2, 1));
            const float s4 = vadd(s3, __shfl_down_sync(full, s2, 2));
            const float hs = vadd(s4, __shfl_down_sync(full, s3, 5));
            if (k == 0) {
                const float d = delta_psi(hs, p.psi_kind, rho0, p.psi_c, p.psi_b);
                s_a[slot][2 + hc] = d;
                s_b[slot][3 + hc] = d;
            }
        }
#pragma unroll
        for (int r = 0; r < H; ++r)
#pragma unroll
            for (int i = 0; i < NQ; ++i) q[r][i] = q[r + 1][i];
        if constexpr (UNIT) {
            unit_moments(g, q[H][0], q[H][1], q[H][2]);
            if (SAMPLE) q[H][NQ - 1] = s9;
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) q[H][i] = g[i];
        }
        __syncthreads();
        if (it < 2 * H || !active || it >= hb + 2 * H) continue;

        // ---- collide row yr, H rows behind: Shan-Chen force, Eq. (1) ---------
        const int yr = yb + it - 2 * H;
        auto at = [&](int ex, int ey) {
            const float *a = s_a[(it - H + ey) & (RING - 1)], *b = s_b[(it - H + ey) & (RING - 1)];
            return *reinterpret_cast<const float2 *>(ex == 1    ? b + j + 2
                                                     : ex == -1 ? b + j
                                                                : a + j + ex);
        };
        float2 sx, sy;
        force_sums<ORDER>(at, sx, sy);
        const float2 pf = vmul(bc<float2>(p.force_pref), vadd(bc<float2>(p.psi0), at(0, 0)));
        const float2 Fx = vmul(pf, sx), Fy = vmul(pf, sy);

        float2 f[9];
        const uint32_t o = (uint32_t)yr * (uint32_t)nx + x;   // the first site's number
        if constexpr (UNIT) collide_unit_m(q[0][0], q[0][1], q[0][2], Fx, Fy, p, rk, o, step, f);
        else collide<float2>(q[0], Fx, Fy, p, rk, o, step, f);
#pragma unroll
        for (int i = 0; i < 9; ++i) st_off(p.dst + i * pl, o, f[i]);
        if (SAMPLE) {
            float2 s;
            if constexpr (UNIT) s = q[0][NQ - 1];
            else s = sum9(q[0]);
            st_off(p.drho_out, o, s);
        }
        const float2 chk = vadd(f[1], f[5]);
        if (!(fabsf(chk.x) <= 3.402823466e38f && fabsf(chk.y) <= 3.402823466e38f))
            atomicOr(p.flag, LB_STEP_NONFINITE);
    }
}

}  // namespace lbsc
