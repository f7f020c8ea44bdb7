// lbm_edge_tile.cuh -- one tile of the fused step on the edge bands of a
// body or of a batch's members (or of the initialisation), the body of the
// edge kernel (lbm_edge.cu).
//
// Nodes within 2 of a bounded edge (3 of a periodic seam) need the boundary
// machinery of Sec. 6: ghost values in Grad u and Div Q, bounced populations
// and periodic images.  A tile owns (tw - 4) x (th - 4) output nodes and has
// one thread per node of the tile and its 2-node halo:
//   stage A (every thread)      : pull-stream, first moment, predicted u*
//   stage B (1-node inner ring) : H = Grad u* with the ghost rules,
//                                 Q = P(F) + Pbar(H)
//   stage C (output nodes)      : 1S = rho0 b + Div Q, moments, corrected j
//                                 and u, equilibrium, BGK collision with He
//                                 forcing, stores, boundary rules of Sec. 6
// with a barrier between stages.  Every global load is issued in stage A, so
// a tile costs one memory latency plus its arithmetic.  The arithmetic is
// that of the interior kernel (lattice units, Q expanded without
// cancellation, collision by opposite pairs).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_kernels.h"
#include "lbm_pipeline.cuh"

namespace lbm {

namespace {

// Rare paths, kept out of line so the kernel's code stays small: stores of a
// node on a periodic axis shorter than 6 nodes, and the boundary rules of a
// node on a bounded edge.
template <class T>
__device__ __noinline__ void store_img_slow(T* base, Geo g, int x, int y, T v) {
    store_img(base, g, x, y, v);
}

__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return fma(a, b, c); }
// -fci + w x, w twice a lattice weight: wmul's product for FP32 storage, else
// one FMA.
template <class TS, class TC>
__device__ __forceinline__ TC back_value(TC fci, TC w, TC x) {
    if constexpr (std::is_same<TS, float>::value)
        return -fci + wmul<TS>(w, x);
    else
        return fma_rn(w, x, -fci);
}

// Eq. (abbcon) for link i with the node's post-collision population fci
// across a wall of outward normal (sx, sy) inv_len (inv_len = 1/sqrt(2) at a
// corner) carrying the traction (T0, T1) inv_len; Pbar* of Sec. 6 in the
// wall's frame from the quasi-traction g = -T* + Q N and the tangential
// entry of the populations' second moment.
template <class TS, class TC>
__device__ __forceinline__ TC abb_value(int i, TC fci, int sx, int sy, TC inv_len, TC T0, TC T1, TC r, TC pxx,
                                        TC pxy, TC pyy, TC q11, TC q12, TC q21, TC q22, TC inv_c2) {
    const TC N0 = TC(sx) * inv_len, N1 = TC(sy) * inv_len;
    const TC g0 = -T0 * inv_len + q11 * N0 + q12 * N1;
    const TC g1 = -T1 * inv_len + q21 * N0 + q22 * N1;
    const TC t0 = -N1, t1 = N0;
    const TC pnn = (N0 * g0 + N1 * g1) * inv_c2;
    const TC pnt = (t0 * g0 + t1 * g1) * inv_c2;
    const TC ptt = t0 * t0 * pxx + TC(2) * t0 * t1 * pxy + t1 * t1 * pyy;
    const TC sxx = pnn * N0 * N0 + TC(2) * pnt * N0 * t0 + ptt * t0 * t0;
    const TC syy = pnn * N1 * N1 + TC(2) * pnt * N1 * t1 + ptt * t1 * t1;
    const TC sxy = pnn * N0 * N1 + pnt * (N0 * t1 + t0 * N1) + ptt * t0 * t1;
    return back_value<TS>(fci, TC(2) * wgt<TC>(i), eq_even<TC>(i, r, sxx, sxy, syy));
}

// Stores a population that the boundary rules send back into the ghost cell
// (x, y), and into its images on a body with a periodic axis.
template <class T>
__device__ __forceinline__ void store_back(T* base, const Geo& g, int x, int y, T v) {
    if (g.perx || g.pery)
        store_img_slow(base, g, x, y, v);
    else
        base[g.at(x, y)] = v;
}

// The links of node (gx, gy) through one wall of outward normal (SX, SY), an
// edge of the body or a face of a hole: Eq. (bbcon) for a Dirichlet wall
// (dirichlet; wall momentum jh* = rho0 v* / c), else Eq. (abbcon) with the
// wall's traction.  fc: the node's post-collision populations; r, pxx, pyy:
// its moments; q: its Q (11, 12, 21, 22).  lo, hi: whether the diagonal link
// towards lower / higher coordinates along the wall leaves through this wall
// alone.  Along an axis the wall's frame is the lattice's, so the Poisson
// stress Pbar* of Sec. 6 is the quasi-traction and the tangential moment
// themselves, formed once for the wall's three links: about 35 operations,
// where the general form (abb_value) took 60 for each of them in a loop over
// all eight directions.  The operations that remain are abb_value's, in its
// order (what it adds and multiplies besides is exactly 0 and 1).
template <int SX, int SY, class TS, class TC>
__device__ __forceinline__ void wall_links(TS* fdst, const Geo& g, const StepParams& p, int gx, int gy, const TC* fc,
                                           TC r, TC pxx, TC pyy, const TC* q, bool dirichlet, TC jh0, TC jh1, TC T0,
                                           TC T1, TC inv_c2, bool lo, bool hi) {
    constexpr int S = SX + SY;  // +-1
    // the axis link and the diagonals towards lower and higher coordinates along the wall
    constexpr int ia = SX > 0 ? 1 : (SX < 0 ? 3 : (SY > 0 ? 2 : 4));
    constexpr int il = SX > 0 ? 8 : (SX < 0 ? 7 : (SY > 0 ? 6 : 7));
    constexpr int ih = SX > 0 ? 5 : (SX < 0 ? 6 : (SY > 0 ? 5 : 8));
    TC sxx, sxy, syy;
    if (SX != 0) {
        sxx = (TC(S) * (TC(S) * q[0] - T0)) * inv_c2;
        sxy = (TC(S) * (TC(S) * q[2] - T1)) * inv_c2;
        syy = pyy;
    } else {
        sxx = pxx;
        sxy = (TC(S) * (TC(S) * q[1] - T0)) * inv_c2;
        syy = (TC(S) * (TC(S) * q[3] - T1)) * inv_c2;
    }
    const TC tr = sxx + syy;
    auto link = [&](auto I) {
        constexpr int i = decltype(I)::value, oi = opp(i);
        constexpr bool diag = i > 4;
        TC val;
        if (dirichlet) {
            const TC e = TC(3) * (diag ? (TC(ex(i)) * jh0 + TC(ey(i)) * jh1) : TC(ex(i) + ey(i)) * (ex(i) != 0 ? jh0 : jh1));
            val = back_value<TS>(-fc[i], -(TC(2) * wgt<TC>(i)), e);
        } else {
            const TC epe = diag ? tr + TC(2 * ex(i) * ey(i)) * sxy : (ex(i) != 0 ? sxx : syy);
            const TC rterm = diag ? -r : TC(0.5) * r;
            val = back_value<TS>(fc[i], TC(2) * wgt<TC>(i), fma_rn(TC(1.5), fma_rn(TC(3), epe, -tr), rterm));
        }
        store_back(fdst + oi * g.plane, g, gx + ex(i), gy + ey(i), Codec<TS, TC>::st(val, oi, p));
    };
    link(std::integral_constant<int, ia>());
    if (lo) link(std::integral_constant<int, il>());
    if (hi) link(std::integral_constant<int, ih>());
}

// The link i of node (gx, gy) through a corner: of two bounded edges of the
// body, ea and eb (Eq. (bbcon) if either is Dirichlet, with the mean of their
// wall momenta if both are, else Eq. (abbcon) with N = (N1 + N2)/sqrt(2), T* =
// (T1 + T2)/sqrt(2)), or of the hole (two Neumann faces).
template <class TS, class TC, class UT>
__device__ __noinline__ void corner_link(TS* fdst, Geo g, const StepParams& p, const EdgeNow<TC, UT>* ea,
                                         const EdgeNow<TC, UT>* eb, int i, int gx, int gy, TC fci, TC r, TC pxx, TC pxy,
                                         TC pyy, TC q11, TC q12, TC q21, TC q22, TC T0, TC T1, TC inv_c2) {
    const bool da = ea && ea->kind == kDirichlet, db = eb && eb->kind == kDirichlet;
    TC val;
    if (da || db) {
        TC a0c, a1c;
        if (da && db) {
            a0c = TC(0.5) * (ea->jh[0] + eb->jh[0]);
            a1c = TC(0.5) * (ea->jh[1] + eb->jh[1]);
        } else {
            const EdgeNow<TC, UT>* e = da ? ea : eb;
            a0c = e->jh[0];
            a1c = e->jh[1];
        }
        val = back_value<TS>(-fci, -(TC(2) * wgt<TC>(i)), eq_odd<TC>(i, a0c, a1c));
    } else {
        val = abb_value<TS, TC>(i, fci, ex(i), ey(i), TC(0.70710678118654752440), T0, T1, r, pxx, pxy, pyy, q11, q12,
                                q21, q22, inv_c2);
    }
    const int oi = opp(i);
    store_img(fdst + oi * g.plane, g, gx + ex(i), gy + ey(i), Codec<TS, TC>::st(val, oi, p));
}

// A node's post-collision populations, moments and Q.
template <class TC>
struct BackNode {
    TC fc[9], r, pxx, pxy, pyy, q[4];
};

// Every link of node (gx, gy) into the hole: Eq. (abbcon) across the face it
// crosses, or both faces at a corner.  In FP32 a tile waits for instructions
// more than for arithmetic, and one small loop for all directions is faster
// than code for each face (wall_links, which saves operations and is kept for
// FP64): a 128 x 128 plate with a hole 7.9 us a step with that, 7.7 so.
template <class TS, class TC>
__device__ __forceinline__ void hole_links(TS* fdst, const Geo& g, const StepParams& p, int gx, int gy,
                                           const BackNode<TC>& n, TC inv_c2) {
#pragma unroll 1
    for (int i = 1; i < 9; ++i) {
        const int dx = gx + ex(i), dy = gy + ey(i);
        if (!in_hole(p.hole, dx, dy)) continue;
        const bool cx = ex(i) != 0 && in_hole(p.hole, dx, gy);
        const bool cy = ey(i) != 0 && in_hole(p.hole, gx, dy);
        const int sx = (cx || !cy) ? ex(i) : 0, sy = (cy || !cx) ? ey(i) : 0;
        TC T0 = TC(0), T1 = TC(0);
        if (sx != 0) {  // the face at x0 (entered along +x) or at x1
            const int fa = sx > 0 ? 0 : 1;
            T0 += TC(p.hole_T[2 * fa]);
            T1 += TC(p.hole_T[2 * fa + 1]);
        }
        if (sy != 0) {  // the face at y0 or at y1
            const int fa = sy > 0 ? 2 : 3;
            T0 += TC(p.hole_T[2 * fa]);
            T1 += TC(p.hole_T[2 * fa + 1]);
        }
        const TC inv_len = (sx != 0 && sy != 0) ? TC(0.70710678118654752440) : TC(1);
        const TC val = abb_value<TS, TC>(i, n.fc[i], sx, sy, inv_len, T0, T1, n.r, n.pxx, n.pxy, n.pyy, n.q[0], n.q[1],
                                         n.q[2], n.q[3], inv_c2);
        const int oi = opp(i);
        store_back(fdst + oi * g.plane, g, dx, dy, Codec<TS, TC>::st(val, oi, p));
    }
}

// The boundary rules of Sec. 6 for a node on a bounded edge or next to the
// hole, written into the ghost cells the links lead to.  edges: bits 0..3,
// the node lies on x-, x+, y-, y+; faces: bits 0..3, next to the hole's face
// at x0, x1, y0, y1; near_hole: within one node of the hole (then on no edge).
// Out of line: few nodes take it, and the tile's registers are spoken for.
template <class TS, class TC, class UT, bool HOLE>
__device__ __noinline__ void boundary_links(TS* fdst, Geo g, const StepParams& p, const EdgeNow<TC, UT>* s_edge,
                                            int gx, int gy, unsigned edges, unsigned faces, bool near_hole,
                                            BackNode<TC> n, TC inv_c2) {
    const bool exl = edges & 1, exh = edges & 2, eyl = edges & 4, eyh = edges & 8;
    auto edge = [&](auto SX, auto SY, int e, bool lo, bool hi) {
        const EdgeNow<TC, UT>& w = s_edge[e];
        wall_links<decltype(SX)::value, decltype(SY)::value, TS, TC>(fdst, g, p, gx, gy, n.fc, n.r, n.pxx, n.pyy, n.q,
                                                                     w.kind == kDirichlet, w.jh[0], w.jh[1], w.T[0],
                                                                     w.T[1], inv_c2, lo, hi);
    };
    using M1 = std::integral_constant<int, -1>;
    using Z0 = std::integral_constant<int, 0>;
    using P1 = std::integral_constant<int, 1>;
    if (exl) edge(M1(), Z0(), 0, !eyl, !eyh);
    if (exh) edge(P1(), Z0(), 1, !eyl, !eyh);
    if (eyl) edge(Z0(), M1(), 2, !exl, !exh);
    if (eyh) edge(Z0(), P1(), 3, !exl, !exh);
    if (HOLE && sizeof(TC) == 4 && near_hole) {
        hole_links<TS, TC>(fdst, g, p, gx, gy, n, inv_c2);
        return;
    }
    if (HOLE && near_hole) {
        auto face = [&](auto SX, auto SY, int fa) {
            constexpr int sx = decltype(SX)::value, sy = decltype(SY)::value;
            const bool lo = in_hole(p.hole, gx + (sx != 0 ? sx : -1), gy + (sx != 0 ? -1 : sy));
            const bool hi = in_hole(p.hole, gx + (sx != 0 ? sx : 1), gy + (sx != 0 ? 1 : sy));
            wall_links<sx, sy, TS, TC>(fdst, g, p, gx, gy, n.fc, n.r, n.pxx, n.pyy, n.q, false, TC(0), TC(0),
                                       TC(p.hole_T[2 * fa]), TC(p.hole_T[2 * fa + 1]), inv_c2, lo, hi);
        };
        if (faces & 1) face(P1(), Z0(), 0);  // entered along +x
        if (faces & 2) face(M1(), Z0(), 1);
        if (faces & 4) face(Z0(), P1(), 2);
        if (faces & 8) face(Z0(), M1(), 3);
    }
    if (!((exl || exh) && (eyl || eyh)) && !(HOLE && near_hole)) return;
    // the diagonal link through a corner of the body, or of the hole
#pragma unroll 1
    for (int i = 5; i < 9; ++i) {
        const EdgeNow<TC, UT>*ea = nullptr, *eb = nullptr;
        TC T0, T1;
        if (HOLE && near_hole) {  // into the hole through neither of its faces alone
            const int dx = gx + ex(i), dy = gy + ey(i);
            if (!in_hole(p.hole, dx, dy) || in_hole(p.hole, dx, gy) || in_hole(p.hole, gx, dy)) continue;
            const int fx = ex(i) > 0 ? 0 : 1, fy = ey(i) > 0 ? 2 : 3;
            T0 = TC(p.hole_T[2 * fx]) + TC(p.hole_T[2 * fy]);
            T1 = TC(p.hole_T[2 * fx + 1]) + TC(p.hole_T[2 * fy + 1]);
        } else {
            if (!((ex(i) < 0 ? exl : exh) && (ey(i) < 0 ? eyl : eyh))) continue;
            ea = &s_edge[ex(i) < 0 ? 0 : 1];
            eb = &s_edge[ey(i) < 0 ? 2 : 3];
            T0 = ea->T[0] + eb->T[0];
            T1 = ea->T[1] + eb->T[1];
        }
        corner_link<TS, TC, UT>(fdst, g, p, ea, eb, i, gx, gy, n.fc[i], n.r, n.pxx, n.pxy, n.pyy, n.q[0], n.q[1],
                                n.q[2], n.q[3], T0, T1, inv_c2);
    }
}

// |a| + |b| + |c| + |d| < 1e30.  FP64: on the exponents (each below 2^97 is
// enough), the sum itself only where those do not settle it.
__device__ __forceinline__ bool moderate(float a, float b, float c, float d) {
    return fabsf(a) + fabsf(b) + fabsf(c) + fabsf(d) < 1e30f;
}
__device__ __forceinline__ bool moderate(double a, double b, double c, double d) {
    auto mag = [](double x) { return __double2hiint(x) & 0x7fffffff; };
    if (max(max(mag(a), mag(b)), max(mag(c), mag(d))) < 0x46000000) return true;
    return fabs(a) + fabs(b) + fabs(c) + fabs(d) < 1e30;
}

// The tile `tile` of the body whose parameters are p (mode 0: one time step;
// mode 1: the initialisation).  Every thread of the CTA calls it (threads
// beyond tw x th idle through the barriers; t / tw by tile.inv_tw = ceil(2^16
// / tw), exact for t tw < 2^16).  Shared memory: su holds 2 x
// tw x th u-carry values, sq 4 x tw x th arithmetic values, sinit (mode 1)
// 4 x tw x th, s_edge the boundary data of the 4 edges and of a hole's faces
// (5 entries).  want_fields: also write u, v, r to p.fields.  HOLE: the
// body may have a hole (false: p.hole is not read, and the tile's code
// carries none of the hole's tests).  XJ (mode 0): the extrapolated scheme,
// whose carries are E = u(t) + F (the u* of stage A), D = ku jh(t) and
// F = ku (3 jh(t) - jh(t - dt)) (the initialisation reads p.scheme instead).
template <class TS, class TC, class UT, int MODE, bool HOLE, bool XJ>
__device__ __forceinline__ void edge_tile_body(const EdgeTile& tile, const StepParams& p, bool want_fields, UT* su,
                                               TC* sq, TC* sinit, EdgeNow<TC, UT>* s_edge) {
    const int t = threadIdx.x;

    // boundary data that do not depend on the time, while the previous launch
    // still runs (their FP64 operations take longer than a memory round trip)
    if (t < 4 && p.bc[t].steady) edge_now<TC, UT>(s_edge[t], p.bc[t], 0.0, p.lat_d[kLatRho0OverC]);

    // the collision of this launch is at t_now = n_now dt; the step counter
    // is read here and used once stage A has issued its loads, so that the
    // two memory round trips overlap
    grid_wait();  // before the first read of what the previous step wrote
    // the next launch may start now: not before this wait, which would let the
    // one after it start too, and tiles of three steps then crowd some SMs while
    // others run empty (an FP32 plate of 301 x 203 with a hole 10.3 us a step,
    // 8.3 so; of 150 x 150 9.0 and 7.3; 256 x 256 8.2 either way)
    if (sizeof(TC) == 4) grid_launch_dependents();
    int64_t n_now = 0;
    if (MODE == 0 && t < 4) n_now = p.counter[p.parity] + 1;

    LatConsts<TC> k;
    k.load(p);
    Geo g;
    g.nx = p.nx;
    g.ny = p.ny;
    g.pitch = p.pitch;
    g.plane = p.plane;
    g.perx = p.periodic_x != 0;
    g.pery = p.periodic_y != 0;
    const int nx = g.nx, ny = g.ny;
    const int64_t pitch = g.pitch, plane = g.plane;
    const TS* __restrict__ fsrc = static_cast<const TS*>(p.f_src);
    TS* __restrict__ fdst = static_cast<TS*>(p.f_dst);
    const void* __restrict__ a_src = p.a_src;
    void* __restrict__ a_dst = p.a_dst;
    const typename UT::CView as0 = UT::cview(a_src, 0, plane), as1 = UT::cview(a_src, 1, plane);
    const typename UT::View ad0 = UT::view(a_dst, 0, plane), ad1 = UT::view(a_dst, 1, plane);
    const TC* __restrict__ s_src = static_cast<const TC*>(p.s_src);
    TC* __restrict__ s_dst = static_cast<TC*>(p.s_dst);

    // ---- this thread's node: raw coordinates (an image beyond a periodic
    // seam) and node coordinates
    const int tw = tile.tw, th = tile.th;
    const int ty = (t * int(tile.inv_tw)) >> 16, tx = t - ty * tw;  // ty >= th: an idle thread
    const int nxo = tile.x1 - tile.x0, nyo = tile.y1 - tile.y0;  // output extent
    const int hx = tile.hx, hy = tile.hy;  // halo before the output nodes
    const int gxr = tile.x0 - hx + tx, gyr = tile.y0 - hy + ty;
    const bool okx = g.perx ? (gxr >= -2 && gxr < nx + 2) : (gxr >= 0 && gxr < nx);
    const bool oky = g.pery ? (gyr >= -2 && gyr < ny + 2) : (gyr >= 0 && gyr < ny);
    // (an image is at most 2 beyond the seam, and an axis has 3 nodes or more)
    const int gx = !g.perx ? gxr : (gxr < 0 ? gxr + nx : (gxr >= nx ? gxr - nx : gxr));
    const int gy = !g.pery ? gyr : (gyr < 0 ? gyr + ny : (gyr >= ny ? gyr - ny : gyr));
    // a node of the hole is not part of the body: it holds nothing, and the
    // cells of the hole next to its faces receive the populations the
    // anti-bounce-back rule sends back
    const bool holed = HOLE && p.hole[0] < p.hole[1];  // the body has a hole (uniform)
    const bool removed = holed && in_hole(p.hole, gx, gy);
    const bool inA = okx && oky && ty < th && !removed;
    const bool inB = inA && tx >= hx - 1 && tx <= hx + nxo && ty >= hy - 1 && ty <= hy + nyo;
    const bool inC = tx >= hx && tx < hx + nxo && ty >= hy && ty < hy + nyo && !removed;
    // a removed neighbour along an axis is a face of the hole: a bounded edge
    // for the ghost rules
    const bool hxl = holed && in_hole(p.hole, gx - 1, gy), hxh = holed && in_hole(p.hole, gx + 1, gy);
    const bool hyl = holed && in_hole(p.hole, gx, gy - 1), hyh = holed && in_hole(p.hole, gx, gy + 1);
    const bool gxl = (!g.perx && gx == 0) || hxl, gxh = (!g.perx && gx == nx - 1) || hxh;
    const bool gyl = (!g.pery && gy == 0) || hyl, gyh = (!g.pery && gy == ny - 1) || hyh;
    // within one node of the hole (a link may enter it)
    const bool near_hole =
        holed && gx >= p.hole[0] - 1 && gx <= p.hole[1] && gy >= p.hole[2] - 1 && gy <= p.hole[3];
    // first and second inward neighbours (used only by a ghost rule)
    const int tx1 = gxl ? min(tx + 1, tw - 1) : max(tx - 1, 0);
    const int tx2 = gxl ? min(tx + 2, tw - 1) : max(tx - 2, 0);
    const int ty1 = gyl ? min(ty + 1, th - 1) : max(ty - 1, 0);
    const int ty2 = gyl ? min(ty + 2, th - 1) : max(ty - 2, 0);
    const int txm = max(tx - 1, 0), txp = min(tx + 1, tw - 1);
    const int tym = max(ty - 1, 0), typ = min(ty + 1, th - 1);
    const int64_t o = g.at(gxr, gyr);  // raw position in the planes

    // ---------------- stage A: pull-stream, first moment, predicted u*
    TC f[9];
    TC so0 = TC(0), so1 = TC(0);  // source carry (XJ: D) of the node (stage C)
    TC fo0 = TC(0), fo1 = TC(0);  // XJ: F of the node
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = TC(0);
    if (MODE == 0 && inA) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
            f[i] = Codec<TS, TC>::ld(fsrc[int64_t(i) * plane + o - ex(i) - int64_t(ey(i)) * pitch], i, p);
        const UT A0 = UT::load(as0, o, p);
        const UT A1 = UT::load(as1, o, p);
        if constexpr (sizeof(TC) == 8) {  // FP64 goes on with sums and differences of opposite populations
            double h[9];
            pairs64(f, h);
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = h[i];
        }
        if (inC) {
            so0 = s_src[o];
            so1 = s_src[o + plane];
        }
        if (XJ) {  // u* = E
            if (inC) {
                fo0 = s_src[o + 2 * plane];
                fo1 = s_src[o + 3 * plane];
            }
            su[(ty * 2) * tw + tx] = A0;
            su[(ty * 2 + 1) * tw + tx] = A1;
        } else {
            TC m0, m1;
            if constexpr (sizeof(TC) == 8) {
                momentum64(f, m0, m1);
            } else {
                m0 = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
                m1 = (f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7]);
            }
            su[(ty * 2) * tw + tx] = A0.add(k.ku * m0);
            su[(ty * 2 + 1) * tw + tx] = A1.add(k.ku * m1);
        }
    } else if (MODE == 1 && inA) {
        const int64_t hh = (int64_t(gy) * nx + gx) * 2;
        su[(ty * 2) * tw + tx] = UT::from_double(p.u0 ? p.u0[hh] : 0.0);
        su[(ty * 2 + 1) * tw + tx] = UT::from_double(p.u0 ? p.u0[hh + 1] : 0.0);
    }
    if (tile.lead && t == 0) p.counter[p.parity ^ 1] = n_now;
    if (t < 4 && !p.bc[t].steady)
        edge_now<TC, UT>(s_edge[t], p.bc[t], double(n_now) * p.dt, p.lat_d[kLatRho0OverC]);
    if (HOLE && t == 4) s_edge[4].kind = kNeumann;  // the faces of a hole (only the kind is read)
    __syncthreads();

    // ---------------- stage B: H = Grad u*, Q = P(F) + Pbar(H)
    bool bad = false;
    if (inB) {
        const EdgeNow<TC, UT>& ebx = s_edge[(hxl || hxh) ? 4 : (gxl ? 0 : 1)];
        const EdgeNow<TC, UT>& eby = s_edge[(hyl || hyh) ? 4 : (gyl ? 2 : 3)];
        TC hh[2][2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const UT* r0 = su + (ty * 2 + c) * tw;
            const UT u0 = r0[tx];
            hh[c][0] = du_axis<TC, UT>(r0[txm], u0, r0[txp], r0[tx1], r0[tx2], gxl, gxh, ebx, c) * k.inv_2dx;
            hh[c][1] = du_axis<TC, UT>(su[(tym * 2 + c) * tw + tx], u0, su[(typ * 2 + c) * tw + tx],
                                       su[(ty1 * 2 + c) * tw + tx], su[(ty2 * 2 + c) * tw + tx], gyl, gyh, eby,
                                       c) *
                       k.inv_2dx;
        }
        TC q11, q12, q21, q22;
        const TC J =
            stress_remainder<TC>(hh[0][0], hh[0][1], hh[1][0], hh[1][1], k.lam, k.mu, q11, q12, q21, q22);
        bad |= not_positive(J) || !moderate(q11, q12, q21, q22);
        TC* qr = sq + (ty * 4) * tw + tx;
        qr[0] = q11;
        qr[tw] = q12;
        qr[2 * tw] = q21;
        qr[3 * tw] = q22;
        if (MODE == 1) {
            const TC tr = hh[0][0] + hh[1][1];
            TC* ir = sinit + (ty * 4) * tw + tx;
            ir[0] = -k.rho0 * tr;
            ir[tw] = -k.mu * (TC(2) * hh[0][0] + tr) * k.inv_c2;
            ir[2 * tw] = -k.mu * (hh[0][1] + hh[1][0]) * k.inv_c2;
            ir[3 * tw] = -k.mu * (TC(2) * hh[1][1] + tr) * k.inv_c2;
        }
    }
    __syncthreads();

    // ---------------- stage C: source, moments, collision, stores
    if (inC) {
        // s = (dt / c) 1S, 1S = rho0 b + Div(P + Pbar)   (Eq. source1)
        TC dQ[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const TC* r0 = sq + (ty * 4 + c) * tw;
            if ((c & 1) == 0)  // Q_a1: derivative along x
                dQ[c] = dq_axis<TC>(r0[txm], r0[tx], r0[txp], r0[tx1], r0[tx2], gxl, gxh);
            else  // Q_a2: derivative along y
                dQ[c] = dq_axis<TC>(sq[(tym * 4 + c) * tw + tx], r0[tx], sq[(typ * 4 + c) * tw + tx],
                                    sq[(ty1 * 4 + c) * tw + tx], sq[(ty2 * 4 + c) * tw + tx], gyl, gyh);
        }
        const TC sn0 = k.sb0 + k.sq_scale * (dQ[0] + dQ[1]);
        const TC sn1 = k.sb1 + k.sq_scale * (dQ[2] + dQ[3]);

        const UT ux = su[(ty * 2) * tw + tx], uy = su[(ty * 2 + 1) * tw + tx];
        TC r, j0, j1, pxx, pxy, pyy;
        TC du0 = TC(0), du1 = TC(0);  // predictor correction of u*
        constexpr bool PAIRS = MODE == 0 && sizeof(TC) == 8;
        if (MODE == 0) {
            TC m0, m1;
            if constexpr (PAIRS) {
                momentum64(f, m0, m1);
            } else {
                r = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
                m0 = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
                m1 = (f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7]);
                const TC dg = (f[5] + f[6]) + (f[7] + f[8]);
                pxx = (f[1] + f[3]) + dg;
                pyy = (f[2] + f[4]) + dg;
                pxy = (f[5] - f[6]) + (f[7] - f[8]);
            }
            if (XJ) {  // u(t + dt) = u(t) + ku (jh(t) + jh) = E - (F - D) + ku jh
                j0 = m0 + TC(0.5) * sn0;
                j1 = m1 + TC(0.5) * sn1;
                du0 = k.ku * j0 - (fo0 - so0);
                du1 = k.ku * j1 - (fo1 - so1);
            } else if (p.scheme == 1) {
                j0 = m0 + TC(0.5) * sn0;
                j1 = m1 + TC(0.5) * sn1;
                du0 = k.ku * (TC(0.5) * (sn0 - so0));
                du1 = k.ku * (TC(0.5) * (sn1 - so1));
            } else {
                j0 = m0 + TC(0.5) * so0;
                j1 = m1 + TC(0.5) * so1;
            }
        } else {
            // initialisation of Algorithm 1: r = -rho0 Div u0, j = rho0 v0,
            // Pbar = Pbar(Grad u0) (from stage B), f = f^eq
            const TC* ir = sinit + (ty * 4) * tw + tx;
            r = ir[0];
            pxx = ir[tw];
            pxy = ir[2 * tw];
            pyy = ir[3 * tw];
            const int64_t hh = (int64_t(gy) * nx + gx) * 2;
            j0 = k.rho0_over_c * TC(p.v0 ? p.v0[hh] : 0.0);
            j1 = k.rho0_over_c * TC(p.v0 ? p.v0[hh + 1] : 0.0);
        }

        TC fc[9];
        if constexpr (PAIRS) {
            TC dg;
            collide64(f, j0, j1, sn0, sn1, k, fc, dg, r);
            pxx = f[1] + dg;
            pyy = f[2] + dg;
            pxy = f[3] - f[4];
        } else {
            // equilibrium (Sec. 5), He forcing (Eq. source), BGK collision
            // (Eq. col), by opposite pairs: f^col_i = (1 - omega) f_i
            //   + w_i (omega E_i + 3 e_i.(omega jh + (1 - omega/2) s)),
            // E_i the even part of f^eq_i / w_i (equal for i and its opposite)
            const TC tr15 = TC(1.5) * (pxx + pyy);
            const TC E0 = TC(2) * r - tr15;
            const TC Ex = TC(0.5) * r + TC(4.5) * pxx - tr15;
            const TC Ey = TC(0.5) * r + TC(4.5) * pyy - tr15;
            const TC Ed = -r + TC(4.5) * (pxx + pyy) - tr15;
            const TC Ep = Ed + TC(9) * pxy, Em = Ed - TC(9) * pxy;
            const TC w0 = wgt<TC>(0), w1 = wgt<TC>(1), w5 = wgt<TC>(5);
            if (MODE == 1) {
                const TC o0 = TC(3) * j0, o1 = TC(3) * j1;
                f[0] = w0 * E0;
                f[1] = w1 * (Ex + o0);
                f[3] = w1 * (Ex - o0);
                f[2] = w1 * (Ey + o1);
                f[4] = w1 * (Ey - o1);
                f[5] = w5 * (Ep + o0 + o1);
                f[7] = w5 * (Ep - o0 - o1);
                f[6] = w5 * (Em - o0 + o1);
                f[8] = w5 * (Em + o0 - o1);
            }
            const TC b0 = TC(3) * (k.omega * j0 + k.force_pref * sn0);
            const TC b1 = TC(3) * (k.omega * j1 + k.force_pref * sn1);
            const TC ax = wmul<TS>(w1, k.omega * Ex), ay = wmul<TS>(w1, k.omega * Ey);
            const TC ap = wmul<TS>(w5, k.omega * Ep), am = wmul<TS>(w5, k.omega * Em);
            const TC bx = wmul<TS>(w1, b0), by = wmul<TS>(w1, b1);
            const TC bp = wmul<TS>(w5, b0 + b1), bm = wmul<TS>(w5, b1 - b0);
            fc[0] = k.one_m_omega * f[0] + wmul<TS>(w0, k.omega * E0);
            fc[1] = k.one_m_omega * f[1] + (ax + bx);
            fc[3] = k.one_m_omega * f[3] + (ax - bx);
            fc[2] = k.one_m_omega * f[2] + (ay + by);
            fc[4] = k.one_m_omega * f[4] + (ay - by);
            fc[5] = k.one_m_omega * f[5] + (ap + bp);
            fc[7] = k.one_m_omega * f[7] + (ap - bp);
            fc[6] = k.one_m_omega * f[6] + (am + bm);
            fc[8] = k.one_m_omega * f[8] + (am - bm);
        }

        // stores, with the periodic images of nodes near a seam
        const bool short_x = g.perx && nx < 6, short_y = g.pery && ny < 6;
        const int64_t img_x = (!g.perx || short_x) ? 0 : (gx < 3 ? nx : (gx >= nx - 3 ? -nx : 0));
        const int64_t img_y =
            (!g.pery || short_y) ? 0 : (gy < 3 ? int64_t(ny) * pitch : (gy >= ny - 3 ? -int64_t(ny) * pitch : 0));
        const bool slow = short_x || short_y;
        auto put = [&](auto* base, auto v) {
            if (slow) {
                store_img_slow(base, g, gx, gy, v);
                return;
            }
            base[o] = v;
            if (img_x) base[o + img_x] = v;
            if (img_y) base[o + img_y] = v;
            if (img_x && img_y) base[o + img_y + img_x] = v;
        };
#pragma unroll
        for (int i = 0; i < 9; ++i) put(fdst + i * plane, Codec<TS, TC>::st(fc[i], i, p));

        // links that leave the body through a bounded edge or enter the hole
        if (gxl || gxh || gyl || gyh || near_hole) {
            const TC* qr = sq + (ty * 4) * tw + tx;
            BackNode<TC> n;
#pragma unroll
            for (int i = 0; i < 9; ++i) n.fc[i] = fc[i];
            n.r = r;
            n.pxx = pxx;
            n.pxy = pxy;
            n.pyy = pyy;
#pragma unroll
            for (int c = 0; c < 4; ++c) n.q[c] = qr[c * tw];
            // the body's edges (a node next to the hole is next to none), the hole's faces
            const unsigned edges = unsigned(gxl && !hxl) | unsigned(gxh && !hxh) << 1 | unsigned(gyl && !hyl) << 2 |
                                   unsigned(gyh && !hyh) << 3;
            const unsigned faces = unsigned(hxh) | unsigned(hxl) << 1 | unsigned(hyh) << 2 | unsigned(hyl) << 3;
            boundary_links<TS, TC, UT, HOLE>(fdst, g, p, s_edge, gx, gy, edges, faces, HOLE && near_hole, n, k.inv_c2);
        }

        // carries for the next step: A' = u + ku (jh + s/2), u = u* + du;
        // the extrapolated scheme: E' = E - F + 4 D', D' = ku jh,
        // F' = 3 D' - D (before the first step jh(-dt) = jh(0): D = D',
        // F = 2 D', and E' = u0 + 2 D')
        const bool xj = XJ || (MODE == 1 && p.scheme == 2);
        const TC ka0 = xj ? k.ku * j0 : k.ku * (j0 + TC(0.5) * sn0);
        const TC ka1 = xj ? k.ku * j1 : k.ku * (j1 + TC(0.5) * sn1);
        const TC f0 = MODE == 1 ? TC(2) * ka0 : fo0, f1 = MODE == 1 ? TC(2) * ka1 : fo1;
        const UT A0 = xj ? ux.add(TC(4) * ka0 - f0).renorm() : ux.add(du0 + ka0).renorm();
        const UT A1 = xj ? uy.add(TC(4) * ka1 - f1).renorm() : uy.add(du1 + ka1).renorm();
        UT::store(A0, A1, ad0, ad1, p, put);
        if (xj) {
            const TC d0 = MODE == 1 ? ka0 : so0, d1 = MODE == 1 ? ka1 : so1;
            put(s_dst, ka0);
            put(s_dst + plane, ka1);
            put(s_dst + 2 * plane, TC(3) * ka0 - d0);
            put(s_dst + 3 * plane, TC(3) * ka1 - d1);
        } else {
            put(s_dst, sn0);
            put(s_dst + plane, sn1);
        }
        if (want_fields && p.fields != nullptr) {
            const int64_t fo = int64_t(gy) * nx + gx;
            const int64_t np = int64_t(nx) * ny;
            p.fields[fo] = ux.add(du0).to_double();
            p.fields[np + fo] = uy.add(du1).to_double();
            p.fields[2 * np + fo] = double(j0 * k.c_over_rho0);
            p.fields[3 * np + fo] = double(j1 * k.c_over_rho0);
            p.fields[4 * np + fo] = double(r);
            if (!(isfinite(j0) && isfinite(j1))) bad = true;  // in the arithmetic type: no FP64 work
        }
    }
    if (bad) atomicOr(p.flag, 1);
}

}  // namespace

}  // namespace lbm
