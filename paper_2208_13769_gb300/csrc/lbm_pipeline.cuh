// lbm_pipeline.cuh -- device helpers shared by the fused step kernels:
// bulk-copy and mbarrier wrappers, boundary data, the ghost-rule differences,
// lattice-unit constants and the storage geometry.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_device.cuh"

namespace lbm {

namespace {

constexpr uint32_t kSpinLimit = 1u << 22;  // bounded mbarrier polling

__device__ __forceinline__ int wrap_coord(int g, int n) {
    int w = g % n;
    return w < 0 ? w + n : w;
}

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: false if the phase did not complete within `limit` polls.
__device__ __forceinline__ bool mbar_wait_n(uint64_t* bar, uint32_t parity, uint32_t limit) {
    for (uint32_t it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    return mbar_wait_n(bar, parity, kSpinLimit);
}

// Tiled global -> shared copy of a 3-D box (x, row, plane) by a tensor map;
// dst is 128-byte aligned, x times the element size a multiple of 16.
__device__ __forceinline__ void tensor_load(uint32_t dst, const void* map, int x, int row, int plane, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(dst),
        "l"(map), "r"(x), "r"(row), "r"(plane), "r"(bar)
        : "memory");
}
// This thread's stores to tensor maps in global memory, for the kernels after
// this one that acquire them.
__device__ __forceinline__ void release_tensor_maps() {
    asm volatile("fence.proxy.tensormap::generic.release.sys;" ::: "memory");
}
// A tensor map that the host or an earlier kernel wrote to global memory, before
// this thread's first copy by it.
__device__ __forceinline__ void acquire_tensor_map(const void* map) {
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}

// A launch chained to its predecessor (programmatic stream serialization):
// lets the next one's CTAs start, and waits until the previous one is
// complete and its writes are visible.  Both do nothing in other launches.
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// T*(t) of a Neumann edge: T0 outside [t_on, t_off), ramping to T1 over t_ramp.
__device__ __forceinline__ void traction(const EdgeBC& e, double t, double& tx, double& ty) {
    double s;
    if (t < e.times[0] || t >= e.times[2])
        s = 0.0;
    else if (e.times[1] > 0.0)
        s = fmin(1.0, (t - e.times[0]) / e.times[1]);
    else
        s = 1.0;
    tx = e.value[0] + (e.rate[0] - e.value[0]) * s;
    ty = e.value[1] + (e.rate[1] - e.value[1]) * s;
}

// Boundary data of one edge at the collision time of a launch, evaluated once
// per CTA (in FP64, then rounded): the Dirichlet displacement u*(t) and wall
// momentum j*/c in lattice units, the Neumann traction T*(t).
template <class TC, class UT>
struct EdgeNow {
    int kind;
    UT us[2];
    TC jh[2];
    TC T[2];
};

template <class TC, class UT>
__device__ __forceinline__ void edge_now(EdgeNow<TC, UT>& out, const EdgeBC& e, double t, double rho0_over_c) {
    out.kind = e.kind;
    for (int c = 0; c < 2; ++c) {
        out.us[c] = UT::from_double(e.value[c] + e.rate[c] * t);
        out.jh[c] = TC(e.rate[c] * rho0_over_c);
    }
    double tx, ty;
    traction(e, t, tx, ty);
    out.T[0] = TC(tx);
    out.T[1] = TC(ty);
}

// u(+1) - u(-1) along one axis around u0 with the ghost rules of bounded
// edges (Dirichlet: u_g = 2 u*(t) - u0; Neumann: linear extrapolation,
// u_g = 2 u0 - u1).  um, up: neighbours below/above; u1: the inward
// neighbour (read only when a ghost is needed); u2 is not used by these
// rules.
template <class TC, class UT>
__device__ __forceinline__ TC du_axis(const UT& um, const UT& u0, const UT& up, const UT& u1, const UT& u2,
                                      bool ghost_lo, bool ghost_hi, const EdgeNow<TC, UT>& e, int comp) {
    if (!ghost_lo && !ghost_hi) return up.minus(um);
    if (e.kind == kDirichlet) {
        const TC v = u0.minus(e.us[comp]) + u1.minus(e.us[comp]);
        return ghost_hi ? -v : v;
    }
    const TC v = TC(2) * u1.minus(u0);
    return ghost_hi ? -v : v;
}

// Q(+1) - Q(-1) with the linear ghost of bounded edges, Q_g = 2 Q0 - Q1.
template <class TC>
__device__ __forceinline__ TC dq_axis(TC qm, TC q0, TC qp, TC q1, TC q2, bool ghost_lo, bool ghost_hi) {
    if (!ghost_lo && !ghost_hi) return qp - qm;
    const TC v = TC(2) * (q1 - q0);
    return ghost_hi ? -v : v;
}

// Lattice constants of a launch in the arithmetic type, read from the
// host-computed table (no FP64 arithmetic on the device: its FP64 units are
// slow on this part).
template <class TC>
__device__ __forceinline__ TC lat_const(const StepParams& p, int k);
template <>
__device__ __forceinline__ float lat_const<float>(const StepParams& p, int k) {
    return p.lat_f[k];
}
template <>
__device__ __forceinline__ double lat_const<double>(const StepParams& p, int k) {
    return p.lat_d[k];
}

template <class TC>
struct LatConsts {
    TC omega, one_m_omega, force_pref, ku, inv_2dx, sq_scale, sb0, sb1, lam, mu, inv_c2, c_over_rho0,
        rho0_over_c, rho0;
    TC omega18, omega12, omega4, omega3, force3, half_one_m_omega, omega18_lo, omega3_lo, force3_lo;
    __device__ __forceinline__ void load(const StepParams& p) {
        omega = lat_const<TC>(p, kLatOmega);
        one_m_omega = lat_const<TC>(p, kLatOneMOmega);
        force_pref = lat_const<TC>(p, kLatForcePref);
        ku = lat_const<TC>(p, kLatKu);
        inv_2dx = lat_const<TC>(p, kLatInv2dX);
        sq_scale = lat_const<TC>(p, kLatSqScale);
        sb0 = lat_const<TC>(p, kLatSb0);
        sb1 = lat_const<TC>(p, kLatSb1);
        lam = lat_const<TC>(p, kLatLambda);
        mu = lat_const<TC>(p, kLatMu);
        inv_c2 = lat_const<TC>(p, kLatInvC2);
        c_over_rho0 = lat_const<TC>(p, kLatCOverRho0);
        rho0_over_c = lat_const<TC>(p, kLatRho0OverC);
        rho0 = lat_const<TC>(p, kLatRho0);
        omega18 = lat_const<TC>(p, kLatOmega18);
        omega12 = lat_const<TC>(p, kLatOmega12);
        omega4 = lat_const<TC>(p, kLatOmega4);
        omega3 = lat_const<TC>(p, kLatOmega3);
        force3 = lat_const<TC>(p, kLatForce3);
        half_one_m_omega = lat_const<TC>(p, kLatHalfOneMOmega);
        omega18_lo = lat_const<TC>(p, kLatOmega18Lo);
        omega3_lo = lat_const<TC>(p, kLatOmega3Lo);
        force3_lo = lat_const<TC>(p, kLatForce3Lo);
    }
};

// Two FP32 operations in one instruction (fma.rn.f32x2 and its kin), which
// halves what the two cost of the issue slots that bound the interior kernel
// with 16-bit storage: 1000 x 777 FP16 20.3 us a step and 19.2 so, 3000 x 2900
// 147.8 and 143.3; FP32 waits for memory (800 x 700 16.1 and 15.8, 4096 x 2048
// 162.4 and 161.9).  Each half is rounded as the scalar instruction is.  The
// forms below spell out which products are fused with an addition, so that
// the kernel keeps the bits of the scalar code (the edge kernel's).
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, f2(-b.x, -b.y)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a b rounded on its own, for add2: a mul2 is fused with the add2 that takes
// it, in spite of the rounding modifiers of both
__device__ __forceinline__ float2 product2(float2 a, float2 b) {
    return f2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}
// the nine populations times their scales (one for each weight)
__device__ __forceinline__ void scale9(float* f, const float* scale) {
    f[0] = __fmul_rn(f[0], scale[0]);
#pragma unroll
    for (int i = 1; i < 9; i += 2) {
        const float2 v = mul2(f2(f[i], f[i + 1]), f2(scale[i < 5 ? 1 : 5]));
        f[i] = v.x;
        f[i + 1] = v.y;
    }
}
// UPair::renorm of both components: hi the high words, lo the low ones
__device__ __forceinline__ void renorm2(float2& hi, float2& lo) {
    const float2 s = add2(hi, lo), b = sub2(s, hi);
    lo = add2(sub2(hi, sub2(s, b)), sub2(lo, b));
    hi = s;
}
// Equilibrium, He forcing and BGK collision in FP32, by pairs: directions (1,
// 2) and their opposites (3, 4), (5, 6) and (7, 8); j, s: jh and s.
template <class TS>
__device__ __forceinline__ void collide2(const float* f, float r, float pxx, float pyy, float pxy, float2 j, float2 s,
                                         const LatConsts<float>& k, float* fc) {
    const float tr = __fadd_rn(pxx, pyy), hr = __fmul_rn(0.5f, r);
    const float E0 = __fmaf_rn(-1.5f, tr, __fmul_rn(2.0f, r));
    const float2 Exy = fma2(f2(-1.5f), f2(tr), add2(f2(hr), product2(f2(4.5f), f2(pxx, pyy))));
    const float Ed = __fmaf_rn(-1.5f, tr, __fmaf_rn(4.5f, tr, -r));
    const float2 Epm = f2(__fmaf_rn(9.0f, pxy, Ed), __fmaf_rn(-9.0f, pxy, Ed));
    const float w0 = wgt<float>(0), w1 = wgt<float>(1), w5 = wgt<float>(5);
    const float2 om = f2(k.omega), o1 = f2(k.one_m_omega);
    const float2 b = mul2(f2(3.0f), fma2(f2(k.force_pref), s, mul2(om, j)));
    const float2 bd = f2(__fadd_rn(b.x, b.y), __fsub_rn(b.y, b.x));
    const float2 e1 = mul2(om, Exy), e5 = mul2(om, Epm);
    const float e0 = __fmul_rn(k.omega, E0);
    float2 p1, q1, p5, q5;  // w (omega E + b) and w (omega E - b)
    if constexpr (sizeof(TS) == 4) {
        auto wm = [](float w, float2 x) { return fma2(f2(w), x, mul2(f2(-w * 0x1p-27f), x)); };  // wmul
        const float2 a1 = wm(w1, e1), a5 = wm(w5, e5), b1 = wm(w1, b), b5 = wm(w5, bd);
        p1 = add2(a1, b1);
        q1 = sub2(a1, b1);
        p5 = add2(a5, b5);
        q5 = sub2(a5, b5);
        fc[0] = __fmaf_rn(k.one_m_omega, f[0], wmul<TS>(w0, e0));
    } else {
        const float2 b1 = mul2(f2(w1), b), b5 = mul2(f2(w5), bd);
        p1 = fma2(f2(w1), e1, b1);
        q1 = fma2(f2(w1), e1, f2(-b1.x, -b1.y));
        p5 = fma2(f2(w5), e5, b5);
        q5 = fma2(f2(w5), e5, f2(-b5.x, -b5.y));
        fc[0] = __fmaf_rn(w0, e0, __fmul_rn(k.one_m_omega, f[0]));
    }
    const float2 c12 = fma2(o1, f2(f[1], f[2]), p1), c34 = fma2(o1, f2(f[3], f[4]), q1);
    const float2 c56 = fma2(o1, f2(f[5], f[6]), p5), c78 = fma2(o1, f2(f[7], f[8]), q5);
    fc[1] = c12.x;
    fc[2] = c12.y;
    fc[3] = c34.x;
    fc[4] = c34.y;
    fc[5] = c56.x;
    fc[6] = c56.y;
    fc[7] = c78.x;
    fc[8] = c78.y;
}

// The FP64 collision on sums and differences of opposite populations, g =
// {f0, f1 + f3, f2 + f4, f5 + f7, f6 + f8, f1 - f3, f2 - f4, f5 - f7, f6 -
// f8}: the moments, equilibrium and forcing need only these, each pair's
// even and odd part relax separately, and omega times the lattice weights
// come from the constants (stage C in 64 FP64 operations against about 95).
// Mass and momentum are what a step must keep: there the constants' rounding
// errors (2^-54, of the same sign at every node and step) are made good.
__device__ __forceinline__ void pairs64(const double* f, double* g) {
    g[0] = f[0];
    g[1] = f[1] + f[3];
    g[2] = f[2] + f[4];
    g[3] = f[5] + f[7];
    g[4] = f[6] + f[8];
    g[5] = f[1] - f[3];
    g[6] = f[2] - f[4];
    g[7] = f[5] - f[7];
    g[8] = f[6] - f[8];
}
__device__ __forceinline__ void momentum64(const double* g, double& m0, double& m1) {
    m0 = g[5] + (g[7] - g[8]);
    m1 = g[6] + (g[7] + g[8]);
}
// fc: the post-collision populations; j, s: jh and s; dg, r: the diagonals'
// sum and the zeroth moment.
__device__ __forceinline__ void collide64(const double* g, double j0, double j1, double s0, double s1,
                                          const LatConsts<double>& k, double* fc, double& dg, double& r) {
    dg = g[3] + g[4];
    const double ax = g[1] + g[2];
    r = (g[0] + ax) + dg;
    const double q = k.omega12 * fma(2.0, dg, ax);  // omega / 12 tr Pf
    const double pd = k.omega4 * (g[1] - g[2]), pxy = k.omega4 * (g[3] - g[4]);
    const double er = fma(k.omega18, r, k.omega18_lo * r);
    const double e1 = er + q, e5 = fma(-0.5, er, q);
    fc[0] = fma(k.one_m_omega, g[0], fma(16.0, er, -8.0 * q));
    const double bx = fma(k.omega3, j0, fma(k.force3, s0, fma(k.omega3_lo, j0, k.force3_lo * s0)));
    const double by = fma(k.omega3, j1, fma(k.force3, s1, fma(k.omega3_lo, j1, k.force3_lo * s1)));
    const double h = k.half_one_m_omega;
    const double p1 = fma(h, g[1], e1 + pd), o1 = fma(h, g[5], bx);
    const double p2 = fma(h, g[2], e1 - pd), o2 = fma(h, g[6], by);
    const double p5 = fma(h, g[3], e5 + pxy), o5 = fma(h, g[7], 0.25 * (bx + by));
    const double p6 = fma(h, g[4], e5 - pxy), o6 = fma(h, g[8], 0.25 * (by - bx));
    fc[1] = p1 + o1;
    fc[3] = p1 - o1;
    fc[2] = p2 + o2;
    fc[4] = p2 - o2;
    fc[5] = p5 + o5;
    fc[7] = p5 - o5;
    fc[6] = p6 + o6;
    fc[8] = p6 - o6;
}

// Lattice-unit equilibrium over w_i, even part (r, Pf): used by the
// anti-bounce-back rule.
template <class T>
__device__ __forceinline__ T eq_even(int i, T r, T pxx, T pxy, T pyy) {
    const int e2 = ex(i) * ex(i) + ey(i) * ey(i);
    const T epe = T(ex(i) * ex(i)) * pxx + T(ey(i) * ey(i)) * pyy + T(2 * ex(i) * ey(i)) * pxy;
    const T rterm = (e2 == 0) ? T(2) * r : (e2 == 1 ? T(0.5) * r : -r);
    return rterm + T(1.5) * (T(3) * epe - (pxx + pyy));
}
template <class T>
__device__ __forceinline__ T eq_odd(int i, T a0, T a1) {
    return T(3) * (T(ex(i)) * a0 + T(ey(i)) * a1);
}

// Geometry of the extended state arrays.
struct Geo {
    int nx, ny;
    int64_t pitch, plane;
    bool perx, pery;
    __device__ __forceinline__ int64_t at(int x, int y) const { return int64_t(y + kPadRows) * pitch + x + kPadCols; }
};

// Stores v at (x, y) and at its periodic images (x +/- nx, y +/- ny) inside
// the 3-wide image band.  x in [-1, nx], y in [-1, ny].
template <class T>
__device__ __forceinline__ void store_img(T* base, const Geo& g, int x, int y, T v) {
    base[g.at(x, y)] = v;
    int ix = 0, iy = 0;
    if (g.perx) ix = (x < 3) ? g.nx : (x >= g.nx - 3 ? -g.nx : 0);
    if (g.pery) iy = (y < 3) ? g.ny : (y >= g.ny - 3 ? -g.ny : 0);
    if (ix) base[g.at(x + ix, y)] = v;
    if (iy) base[g.at(x, y + iy)] = v;
    if (ix && iy) base[g.at(x + ix, y + iy)] = v;
    // a periodic axis shorter than 6 nodes has a node in both bands
    if (g.perx && x < 3 && x >= g.nx - 3) {
        base[g.at(x - g.nx, y)] = v;
        if (iy) base[g.at(x - g.nx, y + iy)] = v;
    }
    if (g.pery && y < 3 && y >= g.ny - 3) {
        base[g.at(x, y - g.ny)] = v;
        if (ix) base[g.at(x + ix, y - g.ny)] = v;
        if (g.perx && x < 3 && x >= g.nx - 3) base[g.at(x - g.nx, y - g.ny)] = v;
    }
}

}  // namespace

}  // namespace lbm
