// Per-site arithmetic of the fused D2Q9 step shared by the step kernels:
// kernel parameters, pull streaming from global memory, and the
// moment-space collision with Guo forcing and Philox noise (Eq. (12)).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbsc_device.cuh"
#include "lbsc_internal.cuh"

namespace lbsc {

template <typename T> struct KParams {
    const T *__restrict__ src;
    T *__restrict__ dst;
    T *__restrict__ drho_out;
    int *__restrict__ flag;
    int nx, ny, strip_h, psi_kind, noise;
    uint32_t step, replica;
    T rho0, force_pref, psi_c, psi_b, psi0;
    T gamma_b, gamma, gamma_g;        // 1 - 1/tau of the bulk, shear and ghost modes
    T c3a, c3b, c4a, c4b, c5a, c5b;   // folded relaxation/source constants
    T amp[6];                         // minus the noise amplitudes (ring_polar)
    int unit;                         // every relaxation rate is 1 (see collide)
    uint32_t rk[20];
    // when not null, the step counter of the noise is *clock + step (a
    // captured window of steps replays for any starting step)
    const uint32_t *__restrict__ clock;
};

__device__ __forceinline__ int wrap_once(int a, int n) {
    return a < 0 ? a + n : (a >= n ? a - n : a);
}

// Pull streaming of one site: g_i(x) = f*_i(x - c_i).  32-bit element
// indices (the context requires 9 nx ny < 2^32).  CG: load through L2 only
// (ld.global.cg) instead of the read-only path, for kernels in which the
// source buffer was written earlier in the same launch.
template <bool CG = false, typename T>
__device__ __forceinline__ T ldsrc(const T *p) {
    if constexpr (CG) return __ldcg(p);
    else return __ldg(p);
}
template <bool CG = false, typename T>
__device__ __forceinline__ void pull(const T *__restrict__ src, size_t plane_, int nx, int xc,
                                     int xm, int xp, int yc, int ym, int yp, T g[9]) {
    const uint32_t plane = (uint32_t)plane_;
    const uint32_t rc = (uint32_t)yc * nx, rm = (uint32_t)ym * nx, rp = (uint32_t)yp * nx;
    g[0] = ldsrc<CG>(src + (0u * plane + rc + xc));
    g[1] = ldsrc<CG>(src + (1u * plane + rc + xm));
    g[2] = ldsrc<CG>(src + (2u * plane + rm + xc));
    g[3] = ldsrc<CG>(src + (3u * plane + rc + xp));
    g[4] = ldsrc<CG>(src + (4u * plane + rp + xc));
    g[5] = ldsrc<CG>(src + (5u * plane + rm + xm));
    g[6] = ldsrc<CG>(src + (6u * plane + rm + xp));
    g[7] = ldsrc<CG>(src + (7u * plane + rp + xp));
    g[8] = ldsrc<CG>(src + (8u * plane + rp + xm));
}

// 1/rho: FP32 from the reciprocal square root squared (NaN for a negative
// density, which the step then reports); FP64 correctly rounded.
__device__ __forceinline__ float inv_rho_of(float rho) {
    const float r = hw_rsqrt(rho);
    return __fmul_rn(r, r);
}
__device__ __forceinline__ float2 inv_rho_of(float2 rho) {
    const float2 r = make_float2(hw_rsqrt(rho.x), hw_rsqrt(rho.y));
    return vmul(r, r);
}
__device__ __forceinline__ double inv_rho_of(double rho) { return 1.0 / rho; }

template <typename V>
__device__ __forceinline__ V sum9(const V g[9]) {
    return vadd(vadd(vadd(g[0], vadd(g[1], g[3])), vadd(g[2], g[4])),
                vadd(vadd(g[5], g[7]), vadd(g[6], g[8])));
}

// The step counter of the noise for a kernel launched with params p.
template <typename T>
__device__ __forceinline__ uint32_t step_of(const KParams<T> &p) {
    return p.clock ? p.step + __ldg(p.clock) : p.step;
}

// Mass and momentum deviations of the pulled populations (the mass in the order of
// the forward transform, which is not that of sum9).
template <typename V>
__device__ __forceinline__ void unit_moments(const V g[9], V &drho, V &m1, V &m2) {
    const V t1 = vadd(vsub(g[5], g[7]), vsub(g[8], g[6]));
    const V t2 = vsub(vsub(g[5], g[7]), vsub(g[8], g[6]));
    drho = vadd(g[0], vadd(vadd(vadd(g[1], g[3]), vadd(g[2], g[4])),
                           vadd(vadd(g[5], g[7]), vadd(g[6], g[8]))));
    m1 = vadd(vsub(g[1], g[3]), t1);
    m2 = vadd(vsub(g[2], g[4]), t2);
}

// The three ring pairs of a site (or of the sites `site` and `site + 1`): radii
// with sqrt(rho) folded in, cosines and sines.  One Philox call a site and step:
// radius words r.x, r.y, r.z and three 10-bit angle indices of r.w.
template <typename T>
__device__ __forceinline__ void ring_noise(T rho, const KParams<T> &p,
                                           const uint32_t *__restrict__ rk, uint32_t site,
                                           uint32_t step, T rad[3], T c[3], T s[3]) {
    const uint4 r = philox4x32_10(make_uint4(site, step, p.replica, 0u), rk);
    ring_polar(uniform01<T>(r.x), r.w & 1023u, rho, rad[0], c[0], s[0]);
    ring_polar(uniform01<T>(r.y), (r.w >> 10) & 1023u, rho, rad[1], c[1], s[1]);
    ring_polar(uniform01<T>(r.z), (r.w >> 20) & 1023u, rho, rad[2], c[2], s[2]);
}
__device__ __forceinline__ void ring_noise(float2 rho, const KParams<float> &p,
                                           const uint32_t *__restrict__ rk, uint32_t site,
                                           uint32_t step, float2 rad[3], float2 c[3],
                                           float2 s[3]) {
    const uint4 r0 = philox4x32_10(make_uint4(site, step, p.replica, 0u), rk);
    const uint4 r1 = philox4x32_10(make_uint4(site + 1u, step, p.replica, 0u), rk);
    const uint32_t w0[3] = {r0.x, r0.y, r0.z}, w1[3] = {r1.x, r1.y, r1.z};
    const float2 k = vmul(bc<float2>(-1.3862943611198906f), rho);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float2 u = vfma(make_float2(__uint2float_rn(w0[j]), __uint2float_rn(w1[j])),
                              bc<float2>(2.3283064365386963e-10f),
                              bc<float2>(1.1641532182693481e-10f));
        const float2 x = vmul(k, make_float2(hw_log2(u.x), hw_log2(u.y)));
        const float2 h = make_float2(hw_rsqrt(fmaxf(x.x, 1e-30f)), hw_rsqrt(fmaxf(x.y, 1e-30f)));
        rad[j] = vmul(x, h);
        const uint32_t a0 = (r0.w >> (10 * j)) & 1023u, a1 = (r1.w >> (10 * j)) & 1023u;
        const float2 th = vfma(make_float2(__uint2float_rn(a0), __uint2float_rn(a1)),
                               bc<float2>(6.1359231515425647e-3f),
                               bc<float2>(-3.1385246920140220f));
        c[j] = make_float2(hw_cos(th.x), hw_cos(th.y));
        s[j] = make_float2(hw_sin(th.x), hw_sin(th.y));
    }
}

// Everything after the forward transform: Guo velocity, relaxation with the
// source, noise, inverse transform delta f_i = w_i sum_k e_ki m_k / b_k, factored
// into symmetric sums and differences.  m: the raw moments 3 .. 8 (general path
// only).
template <bool UNIT, typename V>
__device__ __forceinline__ void collide_tail(V drho, V m1, V m2, const V m[6], V Fx, V Fy,
                                             const KParams<scalar_t<V>> &p,
                                             const uint32_t *__restrict__ rk, uint32_t site,
                                             uint32_t step, V f[9]) {
    using T = scalar_t<V>;
    const V rho = vadd(bc<V>(p.rho0), drho);
    const V inv_rho = inv_rho_of(rho);
    const V jxh = vfma(bc<V>(T(0.5)), Fx, m1), jyh = vfma(bc<V>(T(0.5)), Fy, m2);   // rho u
    const V ux = vmul(jxh, inv_rho), uy = vmul(jyh, inv_rho), nuy = vneg(uy);
    // sums and differences of rho u u (q) and u F (p), each with one rounding of
    // its x part
    const V qs = vfma(jxh, ux, vmul(jyh, uy)), qd = vfma(jxh, ux, vmul(jyh, nuy));
    const V ps = vfma(ux, Fx, vmul(uy, Fy)), pd = vfma(ux, Fx, vmul(nuy, Fy));
    const V qxy = vmul(jxh, uy), pxy = vfma(ux, Fy, vmul(uy, Fx));
    V m3, m4, m5, m6, m7, m8;
    if (UNIT) {   // the general expressions with gamma = 0
        m3 = vfma(bc<V>(T(3)), qs, vmul(bc<V>(T(3)), ps));
        m4 = vadd(qd, pd);
        m5 = vfma(bc<V>(T(0.5)), pxy, qxy);
        m6 = m7 = m8 = bc<V>(T(0));
    } else {
        m3 = vfma(bc<V>(p.gamma_b), m[0], vfma(bc<V>(p.c3a), qs, vmul(bc<V>(p.c3b), ps)));
        m4 = vfma(bc<V>(p.gamma), m[1], vfma(bc<V>(p.c4a), qd, vmul(bc<V>(p.c4b), pd)));
        m5 = vfma(bc<V>(p.gamma), m[2], vfma(bc<V>(p.c5a), qxy, vmul(bc<V>(p.c5b), pxy)));
        m6 = vmul(bc<V>(p.gamma_g), m[3]);
        m7 = vmul(bc<V>(p.gamma_g), m[4]);
        m8 = vmul(bc<V>(p.gamma_g), m[5]);
    }
    if (p.noise) {
        V rad[3], c[3], s[3];
        ring_noise(rho, p, rk, site, step, rad, c, s);
        m3 = vfma(vmul(bc<V>(p.amp[0]), rad[0]), c[0], m3);
        m4 = vfma(vmul(bc<V>(p.amp[1]), rad[0]), s[0], m4);
        m5 = vfma(vmul(bc<V>(p.amp[2]), rad[1]), c[1], m5);
        m6 = vfma(vmul(bc<V>(p.amp[3]), rad[1]), s[1], m6);
        m7 = vfma(vmul(bc<V>(p.amp[4]), rad[2]), c[2], m7);
        m8 = vfma(vmul(bc<V>(p.amp[5]), rad[2]), s[2], m8);
    }
    const V jx = vadd(m1, Fx), jy = vadd(m2, Fy);

    f[0] = vfma(bc<V>(T(1.0 / 18.0)), m8,
                vfma(bc<V>(T(-2.0 / 9.0)), m3, vmul(bc<V>(T(4.0 / 9.0)), drho)));
    const V B = vfma(bc<V>(T(1.0 / 36.0)), vsub(m3, m8), vmul(bc<V>(T(1.0 / 9.0)), drho));
    const V P = vfma(bc<V>(T(0.25)), m4, B), R = vfma(bc<V>(T(-0.25)), m4, B);
    const V Q = vfma(bc<V>(T(-1.0 / 6.0)), m6, vmul(bc<V>(T(1.0 / 3.0)), jx));
    const V Sq = vfma(bc<V>(T(-1.0 / 6.0)), m7, vmul(bc<V>(T(1.0 / 3.0)), jy));
    f[1] = vadd(P, Q);
    f[3] = vsub(P, Q);
    f[2] = vadd(R, Sq);
    f[4] = vsub(R, Sq);
    const V D = vfma(bc<V>(T(1.0 / 72.0)), m8, vmul(bc<V>(T(1.0 / 36.0)), vadd(drho, m3)));
    const V U = vfma(bc<V>(T(0.25)), m5, D), W = vfma(bc<V>(T(-0.25)), m5, D);
    const V A = vadd(jx, m6), C = vadd(jy, m7);
    const V X = vfma(bc<V>(T(1.0 / 12.0)), A, vmul(bc<V>(T(1.0 / 12.0)), C));
    const V Y = vfma(bc<V>(T(1.0 / 12.0)), A, vmul(bc<V>(T(-1.0 / 12.0)), C));
    f[5] = vadd(U, X);
    f[7] = vsub(U, X);
    f[6] = vsub(W, Y);
    f[8] = vadd(W, Y);
}

// The unit-relaxation collision from the mass and momentum deviations alone.
template <typename V>
__device__ __forceinline__ void collide_unit_m(V drho, V m1, V m2, V Fx, V Fy,
                                               const KParams<scalar_t<V>> &p,
                                               const uint32_t *__restrict__ rk, uint32_t site,
                                               uint32_t step, V f[9]) {
    collide_tail<true, V>(drho, m1, m2, nullptr, Fx, Fy, p, rk, site, step, f);
}

// Collision of one site in the Hermite moment basis, Eq. (12):
// moments of the pulled deviations g -> Guo velocity u = (j + F/2)/rho ->
// relaxation of the stress modes towards rho u u with the Guo source
// (1 - 1/2tau_k)(u F + F u) (BGK when every rate is 1/tau; bulk mode 3,
// shear modes 4-5 and ghosts 6-8 may relax at their own rates), ghost modes
// relaxed towards zero, momentum j + F
// -> noise sqrt(mu rho b_k (1 - gamma^2)) z_k on modes 3..8 -> inverse
// transform.  FP32 kernels take collide_unit_m where p.unit (every relaxation
// rate is 1: the non-conserved moments of the pulled populations are not
// needed), this one elsewhere.
template <typename V>
__device__ __forceinline__ void collide(const V g[9], V Fx, V Fy, const KParams<scalar_t<V>> &p,
                                        const uint32_t *__restrict__ rk, uint32_t site,
                                        uint32_t step, V f[9]) {
    using T = scalar_t<V>;
    // forward transform (integer coefficients, shared subexpressions)
    const V e13 = vsub(g[1], g[3]), e24 = vsub(g[2], g[4]);
    const V s13 = vadd(g[1], g[3]), s24 = vadd(g[2], g[4]);
    const V d57 = vsub(g[5], g[7]), d86 = vsub(g[8], g[6]);
    const V s57 = vadd(g[5], g[7]), s68 = vadd(g[6], g[8]);
    const V sa = vadd(s13, s24), sd = vadd(s57, s68);
    const V drho = vadd(g[0], vadd(sa, sd));
    const V t1 = vadd(d57, d86), t2 = vsub(d57, d86);
    const V m1 = vadd(e13, t1);                                              // j_x
    const V m2 = vadd(e24, t2);                                              // j_y
    V m[6];
    m[0] = vfma(bc<V>(T(4)), sd, vfma(bc<V>(T(-2)), g[0], sa));              // 3c^2 - 2
    m[1] = vsub(s13, s24);                                                   // cx^2 - cy^2
    m[2] = vsub(s57, s68);                                                   // cx cy
    m[3] = vfma(bc<V>(T(2)), t1, vneg(e13));                                 // (3c^2 - 4) cx
    m[4] = vfma(bc<V>(T(2)), t2, vneg(e24));                                 // (3c^2 - 4) cy
    m[5] = vfma(bc<V>(T(8)), sd, vfma(bc<V>(T(-4)), sa, vadd(g[0], g[0])));  // 9c^4 - 15c^2 + 2
    collide_tail<false, V>(drho, m1, m2, m, Fx, Fy, p, rk, site, step, f);
}

// Folded constants of KParams (any struct with its members) from the rates
// 1 - 1/tau of the bulk, shear and ghost modes and the noise amplitudes:
// m3: (1-gb) 3 rho u^2 + hb 6 u.F ; m4: (1-gs) rho (ux^2-uy^2) + hs 2 (uxFx-uyFy)
// m5: (1-gs) rho ux uy + hs (ux Fy + uy Fx), h = (1 + gamma)/2 = 1 - 1/(2 tau).
template <typename T, typename K>
inline void fold_rates(K &k, double gb, double gs, double gg, const double amp[6]) {
    k.unit = gb == 0.0 && gs == 0.0 && gg == 0.0;
    k.gamma_b = (T)gb;
    k.gamma = (T)gs;
    k.gamma_g = (T)gg;
    k.c3a = (T)(3.0 * (1.0 - gb));
    k.c3b = (T)(3.0 * (1.0 + gb));
    k.c4a = (T)(1.0 - gs);
    k.c4b = (T)(1.0 + gs);
    k.c5a = (T)(1.0 - gs);
    k.c5b = (T)(0.5 * (1.0 + gs));
    for (int i = 0; i < 6; ++i) k.amp[i] = (T)-amp[i];
}

template <typename T>
inline KParams<T> make_params(const StepArgs &a) {
    KParams<T> k;
    k.src = (const T *)a.src;
    k.dst = (T *)a.dst;
    k.drho_out = (T *)a.drho_out;
    k.flag = a.flag;
    k.nx = a.nx;
    k.ny = a.ny;
    k.strip_h = a.strip_h;
    k.psi_kind = (int)a.psi_kind;
    k.noise = a.noise;
    k.step = a.step;
    k.clock = a.clock;
    k.replica = a.replica;
    k.rho0 = (T)a.rho0;
    k.force_pref = (T)a.force_pref;
    k.psi_c = (T)a.psi_c;
    k.psi_b = (T)a.psi_b;
    k.psi0 = (T)a.psi0;
    fold_rates<T>(k, a.gamma_b, a.gamma, a.gamma_g, a.noise_amp);
    for (int i = 0; i < 20; ++i) k.rk[i] = a.round_keys[i];
    return k;
}

}  // namespace lbsc
