// lbm_interior.cu -- the fused step for the interior of the body.
//
// One launch advances the body from t_n to t_n+1 (Algorithm 1 of arXiv
// 2208.13769, with the paper's footnote predictor for u).  1S at a node needs
// P + Pbar on its 4 neighbours, which need u on a 2-node halo, which needs the
// streamed populations there.
//
// Every node at least 2 nodes from a bounded edge (3 from a periodic seam)
// needs none of the boundary machinery: no ghost rule in Grad u or Div Q, no
// bounced population, no periodic image.  This kernel advances exactly those
// nodes; the edge kernel of lbm_edge.cu advances the thin bands along the
// edges in the same step (both read the same source buffers and write
// disjoint nodes).
//
// Each CTA owns a strip of W <= 124 columns (strips never overlap; the first
// and last strip of a body may be narrower) and a chunk of rows, one thread
// per column plus a 2-column halo on each side, and walks the rows as a
// three-stage pipeline with a lag of one row per stage (written here for a
// walk down the chunk; chunks of odd index walk up it, the same with the
// row order mirrored):
//   stage A, row a     : pull-stream, first moment, predicted u*   (W + 4 cols)
//   stage B, row a - 1 : H = Grad u*, Q = P(F) + Pbar(H)           (W + 2 cols)
//   stage C, row a - 2 : 1S = rho0 b + Div Q, corrected j and u, equilibrium,
//                        BGK collision with He forcing, store       (W cols)
// The 9 population segments of each row arrive in a ring of shared-memory
// slots by tiled asynchronous copies (cp.async.bulk.tensor, one mbarrier per
// slot), the two carries with them.  u* and Q live in rolling buffers.
//
// Lattice units inside the kernels: m = sum_i e_i f_i, Pf = sum_i e_i e_i f_i,
// s = (dt / c) 1S, jh = j / c, so that the equilibrium (Sec. 5) reads
//   f_i^eq = w_i [ r (2 - 3/2 |e_i|^2) + 3 e_i.jh + 3/2 (3 e_i.Pf.e_i - tr Pf) ]
// and no rounded physical constant enters the lattice dynamics.
//
// State per node (two ping-pong copies):
//   f^col_i                                    (9 planes, storage type)
//   A = u_n + dX/(2 rho0) (jh_n + s_n / 2)     (u-carry, 2 comps)
//   s_n                                        (source carry, 2 comps)
// so that u*_n+1 = A + dX/(2 rho0) m  and  jh_n+1 = m + s_(n+1 or n) / 2.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_kernels.h"
#include "lbm_pipeline.cuh"

namespace lbm {

namespace {

// Shared memory of the interior tile: a 128-byte header (the ring's
// mbarriers, at most 8, and the abort word), the u* rows [3][2][NT] and the
// rows of (Q11, Q21) [2][2][NT], then the ring.
constexpr int kSmemHeader = 128;
constexpr int kSmemAbort = 64;
template <class UT, class TC, int NT>
__host__ __device__ constexpr size_t interior_smem_fixed() {
    return (kSmemHeader + sizeof(UT) * 6 * NT + sizeof(TC) * 4 * NT + 127) / 128 * 128;
}

// One slot of the ring: everything an iteration of the row loop reads from
// global memory, as boxes of tensor maps (InteriorMaps) that each start on a
// 128-byte boundary.
//  - The populations of stage A's row a.  A pulled row takes plane i from
//    row a - ey(i): planes {0, 1}, {5, 6} and {7, 8} come in pairs from one
//    row each, and {2, 3, 4} from rows a - 1, a, a + 1 as one box, by a map
//    whose plane stride is one plane plus one row.  The issuing thread runs
//    7 copies with constant coordinates instead of 9 and 6 loads whose 64-bit
//    addresses it and the others compute each row (483 warp instructions per
//    32 nodes against 545 at 4096 x 2048 in FP32).
//  - The u-carry of row a, and the source carry of the row that stage C of
//    the iteration before works on (three rows behind a).  Loaded into
//    registers one row ahead they arrived late (issuing the source's half a
//    row later still cost 10 us of 173); here every slot is in flight.
// A segment of the populations spans columns x0 - 3 .. x0 + W + 2 of a strip
// of W <= NT - 4 output columns from a 16-byte aligned start (up to 16 /
// sizeof(TS) - 1 columns before x0 - 3), one of a carry columns x0 - 2 ..
// x0 + W + 1.
template <class TS, class TC, class UT, int NT, bool XJ>
struct RingSlot {
    static constexpr int up(int bytes) { return (bytes + 127) / 128 * 128; }
    static constexpr int ES = int(sizeof(TS)), CS = int(sizeof(TC));
    static constexpr int SEG = sizeof(TS) == 2 ? NT + 16 : NT + 8;  // elements of a population segment
    static constexpr int SEGC = NT + 16 / CS;                       // words of a carry segment
    static constexpr int SEGL = NT + 8;                             // 16-bit low words of the u-carry
    static constexpr int NA = UT::layout == kCarryPair ? 4 : 2;     // u-carry planes in words of TC
    static constexpr int NL = UT::layout == kCarryPair16 ? 2 : 0;   // and in 16-bit words
    static constexpr int NS = XJ ? 4 : 2;                           // source-carry planes
    static constexpr int F2 = up(2 * SEG * ES), F3 = up(3 * SEG * ES);
    static constexpr int A = 3 * F2 + F3, L = A + up(NA * SEGC * CS), S = L + up(NL * SEGL * 2);
    static constexpr int BYTES = S + up(NS * SEGC * CS);
    static constexpr int TX_S = NS * SEGC * CS;  // bytes copied: the source carry, and all
    static constexpr int TX = 9 * SEG * ES + NA * SEGC * CS + NL * SEGL * 2 + TX_S;
    // byte offset of plane i's segment
    __host__ __device__ static constexpr int plane(int i) {
        return i < 2 ? i * SEG * ES
                     : (i < 5 ? 3 * F2 + (i - 2) * SEG * ES
                              : (i < 7 ? F2 + (i - 5) * SEG * ES : 2 * F2 + (i - 7) * SEG * ES));
    }
    // the population of direction i pulled by the column whose element of
    // plane 0 is at f
    __device__ __forceinline__ static TS pop(const unsigned char* f, int i) {
        return *reinterpret_cast<const TS*>(f + plane(i) - ex(i) * ES);
    }
    // the stored u-carry of component c: ec, el the column's words in a carry
    // segment and in a segment of low words
    __device__ __forceinline__ static typename UT::Raw carry(const unsigned char* slot, int c, int ec, int el) {
        const TC* a = reinterpret_cast<const TC*>(slot + A) + ec;
        if constexpr (UT::layout == kCarryOne)
            return typename UT::Raw{a[c * SEGC]};
        else if constexpr (UT::layout == kCarryPair)
            return typename UT::Raw{a[2 * c * SEGC], a[(2 * c + 1) * SEGC]};
        else
            return typename UT::Raw{a[c * SEGC], reinterpret_cast<const __half*>(slot + L)[c * SEGL + el]};
    }
    // plane c of the source carry
    __device__ __forceinline__ static TC source(const unsigned char* slot, int c, int ec) {
        return reinterpret_cast<const TC*>(slot + S)[c * SEGC + ec];
    }
};

// Slots of the ring for lbm_tuning.ring_slots rows in flight or in work (the
// row in work sits in registers).
__host__ __device__ constexpr int ring_depth(int ring_slots) { return ring_slots - 1; }

}  // namespace

// One tile (column strip bx, row chunk by of the rectangle tg) of one body,
// the only tile of its CTA.  Returns false if a wait gave up or a copy was
// refused (reported in p.flag).  Stage C takes the populations of its row
// from registers that stage A filled two rows earlier, and Q12, Q22 of the
// rows above and below from registers of stage B.  UNROLL3: the row loop
// unrolled by 3 (the row buffers' indices fixed at compile time, the kept
// values changing roles instead of moving: fewer instructions, more
// registers; faster for the formats whose registers allow it).  XJ: the
// extrapolated scheme, whose carries are E = u(t) + F (the u* of stage A, in
// the u-carry planes), D = ku jh(t) and F = ku (3 jh(t) - jh(t - dt)) (in
// the source planes); else u* is A + ku m and the source planes hold the
// last source.  PAIRS: FP32 operations by pairs in one instruction, where both
// components of the displacement are FP32 pairs.
template <class TS, class TC, class UT, int NT, bool XJ, bool UNROLL3, bool REV, bool PAIRS>
__device__ __forceinline__ bool interior_tile(const StepParams& p, const InteriorMaps* maps, const TileGeom& tg,
                                              int bx, int y_begin, int y_end, double* fields) {
    using Slot = RingSlot<TS, TC, UT, NT, XJ>;
    const int W = tg.strip_w;
    constexpr int ALIGN_COLS = 16 / int(sizeof(TS));

    extern __shared__ __align__(128) unsigned char smem[];
    const int R = ring_depth(p.ring_slots);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem);
    // a wait gave up: read after the row's first barrier, so every thread
    // takes the same decision
    volatile int* s_abort = reinterpret_cast<volatile int*>(smem + kSmemAbort);
    UT* su = reinterpret_cast<UT*>(smem + kSmemHeader);                        // u*: [3][2][NT]
    TC* sq = reinterpret_cast<TC*>(smem + kSmemHeader + sizeof(UT) * 6 * NT);  // Q11, Q21: [2][2][NT]
    unsigned char* ring = smem + interior_smem_fixed<UT, TC, NT>();

    LatConsts<TC> k;
    k.load(p);
    // u* then lies by words: the high words of both components, the low ones
    constexpr bool PK = PAIRS && sizeof(TC) == 4 && UT::layout != kCarryOne && !XJ;
    float2* su2 = reinterpret_cast<float2*>(su);
    const int64_t pitch = p.pitch, plane = p.plane;
    const int t = threadIdx.x;
    const int rx0 = tg.rect[0], rx1 = tg.rect[1];
    // strip bx of the strip grid, clipped to the rectangle
    const int x0 = tg.strip_x0 + bx * W;
    const int x_lo = max(rx0, x0), x_hi = min(rx1, x0 + W);
    if (x_lo >= x_hi || y_begin >= y_end) return true;
    // first column of the row segments: 16-byte aligned, inside the plane
    int seg0 = x0 - 3;
    seg0 = (seg0 >= 0 ? seg0 : seg0 - (ALIGN_COLS - 1)) / ALIGN_COLS * ALIGN_COLS;
    if (seg0 < -kPadCols) seg0 = -kPadCols;

    const int gx = x0 - 2 + t;  // this thread's column
    const bool colA = gx >= x_lo - 2 && gx < x_hi + 2;
    const bool colB = gx >= x_lo - 1 && gx < x_hi + 1;
    const bool colC = gx >= x_lo && gx < x_hi;
    const int tm = t > 0 ? t - 1 : t, tp = t < NT - 1 ? t + 1 : t;
    // where the segments start in a plane's row, and this column in them
    const int xf = seg0 + kPadCols, xc = (x0 - 2 + kPadCols) & ~(16 / int(sizeof(TC)) - 1),
              xl = (x0 - 2 + kPadCols) & ~7;
    const int e_own = (gx - seg0) * int(sizeof(TS)), ec = gx + kPadCols - xc, el = gx + kPadCols - xl;

    // the row walk: down the chunk, or up it (REV), so that two chunks
    // sharing a boundary read its halo rows at the same time (both at their
    // start or both at their end) and the second read hits L2; stage A's row
    // a = a0 + sg q, stage B at a - sg, stage C at a - 2 sg
    constexpr bool rev = REV;
    constexpr int sg = REV ? -1 : 1;
    const int a0 = rev ? y_end + 1 : y_begin - 2;
    const int niter = (y_end - y_begin) + 4;

    // the copies of iteration j into ring slot s (thread 0): iteration niter
    // holds only the source carry of the last one's stage C.  A copy's first
    // column must start on a 16-byte boundary: a tile whose does not (none
    // does, by seg0) is refused before anything is issued, in p.flag (bit 8)
    const uint32_t ring_at = smem_addr(ring), bars_at = smem_addr(bars);
    auto issue_row = [&](int j, int s) {
        const uint32_t dst = ring_at + uint32_t(s * Slot::BYTES), bar = bars_at + uint32_t(s * 8);
        const int r = a0 + sg * j + kPadRows;
        const bool all = j < niter;
        mbar_expect_tx(&bars[s], uint32_t(all ? Slot::TX : Slot::TX_S));
        tensor_load(dst + Slot::S, &maps->s, xc, r - 3 * sg, 0, bar);
        if (!all) return;
        tensor_load(dst, &maps->f, xf, r, 0, bar);                      // planes 0, 1 of row a
        tensor_load(dst + Slot::F2, &maps->f, xf, r - 1, 5, bar);       // 5, 6 of row a - 1
        tensor_load(dst + 2 * Slot::F2, &maps->f, xf, r + 1, 7, bar);   // 7, 8 of row a + 1
        tensor_load(dst + 3 * Slot::F2, &maps->f3, xf, r - 1, 0, bar);  // 2, 3, 4 of rows a - 1, a, a + 1
        tensor_load(dst + Slot::A, &maps->a, xc, r, 0, bar);
        if (Slot::NL > 0) tensor_load(dst + Slot::L, &maps->lo, xl, r, 0, bar);
    };
    if (xf < 0 || xf % ALIGN_COLS != 0) {  // uniform over the CTA
        if (t == 0) atomicOr(p.flag, 8);
        return false;
    }

    uint32_t phase = 0, issued = 0;
    if (t == 0) {
        *s_abort = 0;
        for (int s = 0; s < R; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (t == 0) {
        fence_proxy_async();  // the CTA's earlier shared-memory accesses precede the copies into the ring
        for (int j = 0; j < R && j <= niter; ++j) {
            issue_row(j, j);
            issued |= 1u << j;
        }
    }

    // Addresses: a base per plane, the same for every thread of the CTA
    // (column gx of thread 0 in the tile's lowest row), and a 32-bit offset
    // from it, which advances by a row (the host keeps a tile's rows few
    // enough for its byte offsets to fit, interior_max_rows).
    const uint32_t pitch32 = uint32_t(pitch);
    uint32_t off_a = uint32_t(t) + (rev ? uint32_t(niter - 1) * pitch32 : 0u);  // row a of stage A, this column
    const uint32_t dpitch = rev ? 0u - pitch32 : pitch32;                       // to the walk's next row
    const int64_t base = int64_t(y_begin - 2 + kPadRows) * pitch + (x0 - 2) + kPadCols;
    TS* fd[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) fd[i] = static_cast<TS*>(p.f_dst) + int64_t(i) * plane + base;
    const typename UT::View ad0 = UT::view(p.a_dst, 0, plane).shifted(base);
    const typename UT::View ad1 = UT::view(p.a_dst, 1, plane).shifted(base);
    TC* sd[Slot::NS];
#pragma unroll
    for (int i = 0; i < Slot::NS; ++i) sd[i] = static_cast<TC*>(p.s_dst) + int64_t(i) * plane + base;
    bool bad = false;
    // waits for slot s's copies
    auto wait_slot = [&](int s) {
        if (!mbar_wait(&bars[s], (phase >> s) & 1u)) *s_abort = 1;
        phase ^= 1u << s;
        issued &= ~(1u << s);
    };
    wait_slot(0);
    int ra = 0;
    // rows kept in registers for stage C two iterations later: the
    // populations of this column as stage A pulled them, Q12 and Q22 of stage B
    TC F0[9], F1[9], F2[9], V0[2], V1[2], V2[2];
#pragma unroll
    for (int i = 0; i < 9; ++i) F0[i] = F1[i] = F2[i] = TC(0);
#pragma unroll
    for (int i = 0; i < 2; ++i) V0[i] = V1[i] = V2[i] = TC(0);
    // One row of the pipeline.  sa = q mod 3 selects the u* row buffer (a
    // compile-time constant when the loop is unrolled by 3); gcur receives
    // stage A's populations of row a and vcur stage B's Q12, Q22 of row
    // a - sg, fp2 and vp2 hold those of two iterations ago.  Returns false
    // when the tile gives up.
    auto row = [&](int q, auto sa, TC* gcur, const TC* fp2, TC* vcur, const TC* vp2) -> bool {
        const int sA = sa;                    // slot of row a
        const int sB = sA == 0 ? 2 : sA - 1;  // slot of row a - 1
        const int sC = sA == 2 ? 0 : sA + 1;  // slot of row a - 2
        const int rn = ra + 1 == R ? 0 : ra + 1;  // ring slot of the next iteration

        // ---------------- stage A: row a
        if (colA) {
            const unsigned char* slot = ring + ra * Slot::BYTES;
            const unsigned char* pf = slot + e_own;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                if constexpr (PK && sizeof(TS) == 2)
                    gcur[i] = float(Slot::pop(pf, i));
                else
                    gcur[i] = Codec<TS, TC>::ld(Slot::pop(pf, i), i, p);
            }
            if constexpr (PK && sizeof(TS) == 2) scale9(gcur, p.dec_scale);
            if constexpr (sizeof(TC) == 8) {  // FP64 keeps them as sums and differences of opposite ones
                double f[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) f[i] = gcur[i];
                pairs64(f, gcur);
            }
            const UT A0 = UT::decode(Slot::carry(slot, 0, ec, el), p), A1 = UT::decode(Slot::carry(slot, 1, ec, el), p);
            if (XJ) {  // u* = u(t) + ku (3 jh(t) - jh(t - dt)) = E
                su[(sA * 2) * NT + t] = A0;
                su[(sA * 2 + 1) * NT + t] = A1;
            } else {
                const TC* g = gcur;
                if constexpr (PK) {
                    const float2 D = sub2(f2(g[1], g[2]), f2(g[3], g[4]));
                    const float2 m = add2(add2(D, f2(g[5] - g[6], g[5] - g[8])), f2(g[8] - g[7], g[6] - g[7]));
                    su2[(sA * 2) * NT + t] = f2(A0.hi, A1.hi);
                    su2[(sA * 2 + 1) * NT + t] = add2(f2(A0.lo, A1.lo), product2(f2(k.ku), m));
                } else {
                    TC m0, m1;
                    if constexpr (sizeof(TC) == 8) {
                        momentum64(g, m0, m1);
                    } else {
                        m0 = (g[1] - g[3]) + (g[5] - g[6]) + (g[8] - g[7]);
                        m1 = (g[2] - g[4]) + (g[5] - g[8]) + (g[6] - g[7]);
                    }
                    su[(sA * 2) * NT + t] = A0.add(k.ku * m0);
                    su[(sA * 2 + 1) * NT + t] = A1.add(k.ku * m1);
                }
            }
        }
        __syncthreads();
        if (*s_abort) return false;
        if (t == 0 && q + R <= niter) {  // into the slot that stage A has just read
            fence_proxy_async();
            issue_row(q + R, ra);
            issued |= 1u << ra;
        }
        // ---------------- stage B: row a - sg
        if (colB && q >= 2) {
            const UT* r0 = su + (sB * 2) * NT;
            // the rows below and above (a - 2 sg and a in the walk)
            const UT* rm = su + ((rev ? sA : sC) * 2) * NT;
            const UT* rp = su + ((rev ? sC : sA) * 2) * NT;
            TC h11, h12, h21, h22;
            if constexpr (PK) {
                const float2* q0 = reinterpret_cast<const float2*>(r0);
                const float2* qm = reinterpret_cast<const float2*>(rm);
                const float2* qp = reinterpret_cast<const float2*>(rp);
                const float2 dx = add2(sub2(q0[tp], q0[tm]), sub2(q0[NT + tp], q0[NT + tm]));
                const float2 dy = add2(sub2(qp[t], qm[t]), sub2(qp[NT + t], qm[NT + t]));
                h11 = dx.x * k.inv_2dx;
                h21 = dx.y * k.inv_2dx;
                h12 = dy.x * k.inv_2dx;
                h22 = dy.y * k.inv_2dx;
            } else {
                h11 = r0[tp].minus(r0[tm]) * k.inv_2dx;
                h21 = r0[NT + tp].minus(r0[NT + tm]) * k.inv_2dx;
                h12 = rp[t].minus(rm[t]) * k.inv_2dx;
                h22 = rp[NT + t].minus(rm[NT + t]) * k.inv_2dx;
            }
            TC q11, q12, q21, q22;
            const TC J = stress_remainder<TC>(h11, h12, h21, h22, k.lam, k.mu, q11, q12, q21, q22);
            bad |= not_positive(J);  // also catches a non-finite displacement gradient
            TC* qr = sq + (q & 1) * 2 * NT;
            qr[t] = q11;
            qr[NT + t] = q21;
            vcur[0] = q12;
            vcur[1] = q22;
        }
        wait_slot(rn);
        __syncthreads();

        // ---------------- stage C: row a - 2 sg
        if (colC && q >= 4) {
            const int gy = a0 + sg * (q - 2);
            const unsigned char* next = ring + rn * Slot::BYTES;
            const TC so0 = Slot::source(next, 0, ec), so1 = Slot::source(next, 1, ec);  // source carry (XJ: D)
            TC fo0 = TC(0), fo1 = TC(0);                                                // XJ: F
            if (XJ) {
                fo0 = Slot::source(next, Slot::NS - 2, ec);
                fo1 = Slot::source(next, Slot::NS - 1, ec);
            }
            const TC* qc = sq + ((q & 1) ^ 1) * 2 * NT;                      // Q11, Q21 of row a - 2 sg
            const TC* qm = rev ? vcur : vp2;                                 // Q12, Q22 of the row below it
            const TC* qp = rev ? vp2 : vcur;                                 // and of the row above it
            // s = (dt / c) 1S, 1S = rho0 b + Div(P + Pbar)   (Eq. source1)
            const TC sn0 = k.sb0 + k.sq_scale * ((qc[tp] - qc[tm]) + (qp[0] - qm[0]));
            const TC sn1 = k.sb1 + k.sq_scale * ((qc[NT + tp] - qc[NT + tm]) + (qp[1] - qm[1]));

            const TC* f = fp2;
            TC r, m0, m1, pxx, pyy, pxy;
            if constexpr (sizeof(TC) == 8) {
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
            TC j0, j1, du0 = TC(0), du1 = TC(0);
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

            TC fc[9];
            if constexpr (sizeof(TC) == 8) {
                TC dg;
                collide64(f, j0, j1, sn0, sn1, k, fc, dg, r);
            } else {
                if constexpr (PK) {
                    collide2<TS>(f, r, pxx, pyy, pxy, f2(j0, j1), f2(sn0, sn1), k, fc);
                } else {
                    // equilibrium, He forcing and BGK collision by opposite pairs
                    const TC tr15 = TC(1.5) * (pxx + pyy);
                    const TC E0 = TC(2) * r - tr15;
                    const TC Ex = TC(0.5) * r + TC(4.5) * pxx - tr15;
                    const TC Ey = TC(0.5) * r + TC(4.5) * pyy - tr15;
                    const TC Ed = -r + TC(4.5) * (pxx + pyy) - tr15;
                    const TC Ep = Ed + TC(9) * pxy, Em = Ed - TC(9) * pxy;
                    const TC w0 = wgt<TC>(0), w1 = wgt<TC>(1), w5 = wgt<TC>(5);
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
            }
            if constexpr (PK && sizeof(TS) == 2) scale9(fc, p.enc_scale);
            const uint32_t o = off_a - 2 * dpitch;  // row a - 2 sg = gy
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                if constexpr (PK && sizeof(TS) == 2)
                    *elem(fd[i], o) = TS(fc[i]);  // scaled above
                else
                    *elem(fd[i], o) = Codec<TS, TC>::st(fc[i], i, p);
            }

            // carries: A' = u + ku (jh + s/2), u = u* + du;  s' = s
            // (XJ: E' = u + ku (3 jh - jh(t)) = E - F + 4 D', D' = ku jh,
            // F' = 3 D' - D)
            UT ux, uy;
            if constexpr (PK) {
                const float2 uh = su2[(sC * 2) * NT + t], ul = su2[(sC * 2 + 1) * NT + t];
                ux = UT{uh.x, ul.x};
                uy = UT{uh.y, ul.y};
            } else {
                ux = su[(sC * 2) * NT + t];
                uy = su[(sC * 2 + 1) * NT + t];
            }
            UT A0, A1;
            const TC ka0 = XJ ? k.ku * j0 : k.ku * (j0 + TC(0.5) * sn0);
            const TC ka1 = XJ ? k.ku * j1 : k.ku * (j1 + TC(0.5) * sn1);
            if constexpr (PK) {
                float2 hi = f2(ux.hi, uy.hi), lo = add2(f2(ux.lo, uy.lo), f2(du0 + ka0, du1 + ka1));
                renorm2(hi, lo);
                A0 = UT{hi.x, lo.x};
                A1 = UT{hi.y, lo.y};
            } else {
                A0 = XJ ? ux.add(TC(4) * ka0 - fo0).renorm() : ux.add(du0 + ka0).renorm();
                A1 = XJ ? uy.add(TC(4) * ka1 - fo1).renorm() : uy.add(du1 + ka1).renorm();
            }
            auto put = [o](auto* at, auto v) { *elem(at, o) = v; };
            UT::store(A0, A1, ad0, ad1, p, put);
            *elem(sd[0], o) = XJ ? ka0 : sn0;
            *elem(sd[1], o) = XJ ? ka1 : sn1;
            if (XJ) {
                *elem(sd[Slot::NS - 2], o) = TC(3) * ka0 - so0;
                *elem(sd[Slot::NS - 1], o) = TC(3) * ka1 - so1;
            }
            if (fields != nullptr) {
                const int64_t fo = int64_t(gy) * p.nx + gx;
                const int64_t np = int64_t(p.nx) * p.ny;
                fields[fo] = ux.add(du0).to_double();
                fields[np + fo] = uy.add(du1).to_double();
                fields[2 * np + fo] = double(j0 * k.c_over_rho0);
                fields[3 * np + fo] = double(j1 * k.c_over_rho0);
                fields[4 * np + fo] = double(r);
                if (!(isfinite(j0) && isfinite(j1))) bad = true;  // in the arithmetic type: no FP64 work
            }
        }
        ra = rn;
        off_a += dpitch;
        return true;
    };
    if (UNROLL3) {
        // the kept values change roles instead of moving: iteration q's in
        // F[q mod 3], those of q - 2 in F[(q + 1) mod 3]
        for (int q = 0; q < niter;) {
            if (!row(q, std::integral_constant<int, 0>(), F0, F1, V0, V1) || ++q >= niter) break;
            if (!row(q, std::integral_constant<int, 1>(), F1, F2, V1, V2) || ++q >= niter) break;
            if (!row(q, std::integral_constant<int, 2>(), F2, F0, V2, V0) || ++q >= niter) break;
        }
    } else {
        // F1 and F2 keep the values of the last two iterations, moved after each
        int sa = 0;
        for (int q = 0; q < niter; ++q) {
            TC gcur[9], vcur[2];
            if (!row(q, sa, gcur, F2, vcur, V2)) break;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                F2[i] = F1[i];
                F1[i] = gcur[i];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                V2[i] = V1[i];
                V1[i] = vcur[i];
            }
            sa = sa == 2 ? 0 : sa + 1;
        }
    }
    if (bad) atomicOr(p.flag, 1);
    if (*s_abort) {
        if (t == 0) {
            atomicOr(p.flag, 4);
            for (int s = 0; s < R; ++s)
                if (issued & (1u << s)) (void)mbar_wait(&bars[s], (phase >> s) & 1u);
        }
        return false;
    }
    return true;
}

// One CTA per tile over the launch's rectangles (one 1-D grid; a body
// without a hole has one rectangle).
// Whether the chunks of a single body alternate their row walk (the two
// directions as two compiled paths of the tile).  In one wave the chunks
// above and below a boundary then read its halo rows together: FP32 with
// the compensated carry reads 61.0 DRAM bytes per node instead of 63.9 and
// runs 2.4 % faster.  Not for the unrolled row loop, whose two copies made
// the plain-carry FP32 and 16-bit kernels 9 to 10 % slower.
template <bool UNROLL3>
__host__ __device__ constexpr bool alternate_walk() {
    return !UNROLL3;
}

template <class TS, class TC, class UT, int NT, int MINB, bool XJ, bool UNROLL3>
__global__ void __launch_bounds__(NT, MINB)
    interior_step_kernel(const __grid_constant__ StepParams p, const __grid_constant__ InteriorRects R,
                         const __grid_constant__ InteriorMaps maps) {
    const InteriorItem it = R.items[blockIdx.x];
    // the rectangle by constant indices (no indexed reads of the parameters)
    const TileGeom tg = it.inst == 0 ? R.g[0] : (it.inst == 1 ? R.g[1] : (it.inst == 2 ? R.g[2] : R.g[3]));
    const bool up = it.rows < 0;
    const int y1 = it.y0 + (up ? -it.rows : it.rows);
    if (alternate_walk<UNROLL3>() && up)
        interior_tile<TS, TC, UT, NT, XJ, UNROLL3, true, true>(p, &maps, tg, it.strip, it.y0, y1, p.fields);
    else
        interior_tile<TS, TC, UT, NT, XJ, UNROLL3, false, true>(p, &maps, tg, it.strip, it.y0, y1, p.fields);
}

// The interiors of a batch of bodies for one time step: one CTA per interior
// tile (member rectangle, strip, chunk) of a list ordered longest first, the
// tile's parameters (the member's, with the rectangle and its strip grid)
// read from the device table into shared memory.  The tile is the
// single-body kernel's, so every node of a member takes the same arithmetic
// as when the member is stepped alone.
template <class TS, class TC, class UT, int NT, int MINB, bool UNROLL3>
__global__ void __launch_bounds__(NT, MINB) batch_interior_kernel(const __grid_constant__ BatchInteriorLaunch L) {
    __shared__ __align__(16) StepParams sp;
    const InteriorItem it = L.items[blockIdx.x];
    {
        const int4* src = reinterpret_cast<const int4*>(L.params + it.inst);
        int4* dst = reinterpret_cast<int4*>(&sp);
        for (int q = int(threadIdx.x); q < int(sizeof(StepParams) / 16); q += NT) dst[q] = src[q];
    }
    const InteriorMaps* maps = L.maps + it.inst;
    if (threadIdx.x == 0) {  // the thread that issues the copies
        acquire_tensor_map(&maps->f);
        acquire_tensor_map(&maps->f3);
        acquire_tensor_map(&maps->a);
        if (UT::layout == kCarryPair16) acquire_tensor_map(&maps->lo);
        acquire_tensor_map(&maps->s);
    }
    __syncthreads();
    const TileGeom tg = {{sp.rect[0], sp.rect[1], sp.rect[2], sp.rect[3]}, sp.strip_x0, sp.strip_w};
    const bool up = it.rows < 0;
    const int y1 = it.y0 + (up ? -it.rows : it.rows);
    double* fields = L.fields ? sp.fields : nullptr;
    // with 16-bit storage pairs let a 7th CTA on the SM, which costs the long
    // tiles more than they save (128 bodies of 64 to 512 nodes a side: 281 us a
    // step, 270 without); FP32 32 bodies of 64 to 1024 244 and 246
    constexpr bool kPairs = sizeof(TS) == 4;
    if (alternate_walk<UNROLL3>() && up)
        interior_tile<TS, TC, UT, NT, false, UNROLL3, true, kPairs>(sp, maps, tg, it.strip, it.y0, y1, fields);
    else
        interior_tile<TS, TC, UT, NT, false, UNROLL3, false, kPairs>(sp, maps, tg, it.strip, it.y0, y1, fields);
}

template <class TS, class TC, class UT, int NT, bool XJ>
size_t interior_smem_bytes(int ring_slots) {
    return interior_smem_fixed<UT, TC, NT>() +
           size_t(RingSlot<TS, TC, UT, NT, XJ>::BYTES) * size_t(ring_depth(ring_slots));
}

// The kernel's limit of dynamic shared memory, on the current device, that of
// the deepest ring: the same whatever ring a body or a batch runs with, so that
// planning one never lowers it under another's launches, on any device and from
// any thread.  (A launch takes what its own ring needs.)
template <class TS, class TC, class UT, int NT, bool XJ, class Kernel>
cudaError_t allow_any_ring(Kernel kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(interior_smem_bytes<TS, TC, UT, NT, XJ>(kMaxRing)));
}

template <class TS, class TC, class UT, int NT, int MINB, bool UNROLL3, bool XJ>
cudaError_t launch_interior_x(const StepParams& p, const InteriorRects& R, const InteriorMaps& maps, cudaStream_t s) {
    auto kern = interior_step_kernel<TS, TC, UT, NT, MINB, XJ, UNROLL3>;
    const size_t sm = interior_smem_bytes<TS, TC, UT, NT, XJ>(p.ring_slots);
    if (R.total <= 0) return cudaSuccess;
    kern<<<R.total, NT, sm, s>>>(p, R, maps);
    return cudaGetLastError();
}

// (the extrapolated scheme's variant keeps the rotating loop: its extra
// carries leave no registers for the unrolled one)
template <class TS, class TC, class UT, int NT, int MINB, bool UNROLL3>
cudaError_t launch_interior_t(const StepParams& p, const InteriorRects& R, const InteriorMaps& maps, cudaStream_t s) {
    return p.scheme == 2 ? launch_interior_x<TS, TC, UT, NT, MINB, false, true>(p, R, maps, s)
                         : launch_interior_x<TS, TC, UT, NT, MINB, UNROLL3, false>(p, R, maps, s);
}

template <class TS, class TC, class UT, int NT, int MINB, bool UNROLL3>
cudaError_t launch_batch_interior_t(const BatchInteriorLaunch& L, int ring_slots, cudaStream_t s, int* resident) {
    auto kern = batch_interior_kernel<TS, TC, UT, NT, MINB, UNROLL3>;
    const size_t sm = interior_smem_bytes<TS, TC, UT, NT, false>(ring_slots);
    if (resident) {  // CTAs per SM of this kernel with this ring
        *resident = 0;
        cudaError_t e = allow_any_ring<TS, TC, UT, NT, false>(kern);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(resident, kern, NT, sm);
        if (e != cudaSuccess) return e;
    }
    if (L.nitems <= 0) return cudaSuccess;
    kern<<<L.nitems, NT, sm, s>>>(L);
    return cudaGetLastError();
}

// The row loops of the single-body interior kernel (launch_interior); the
// register caps hold six CTAs per SM (the parameters come from shared
// memory here, not the launch's constant bank, which takes more registers
// unless capped: 96 to 104).
cudaError_t launch_batch_interior(int fmt, const BatchInteriorLaunch& L, int ring_slots, cudaStream_t s,
                                  int* resident) {
    constexpr int NT = kInteriorThreads;
    switch (fmt) {
        case kFmtF64:
            return launch_batch_interior_t<double, double, UPlain<double>, NT, 3, false>(L, ring_slots, s, resident);
        case kFmtF32:
            return launch_batch_interior_t<float, float, UPlain<float>, NT, 6, true>(L, ring_slots, s, resident);
        case kFmtF32C:
            return launch_batch_interior_t<float, float, UComp, NT, 6, false>(L, ring_slots, s, resident);
        case kFmtF32H:
            return launch_batch_interior_t<float, float, UCompH, NT, 6, false>(L, ring_slots, s, resident);
        case kFmtF16:
            return launch_batch_interior_t<__half, float, UComp, NT, 6, true>(L, ring_slots, s, resident);
        case kFmtBF16:
            return launch_batch_interior_t<__nv_bfloat16, float, UComp, NT, 6, true>(L, ring_slots, s, resident);
    }
    return cudaErrorInvalidValue;
}

void interior_strips(int fmt, int rx0, int rx1, int aligned, int* strip_x0, int* strip_w, int* nstrips) {
    int W = 124, xg = rx0;  // 128 threads: the strip and its 2-column halo on each side
    if (aligned == 1 || aligned == 2) {
        // the fewest strips of equal width on a grid of 32-byte sectors
        // (aligned 1: 8 columns of a 4- or 8-byte plane, 16 of a 2-byte
        // plane), so that no two CTAs store into one sector even when they
        // run far apart in time, or of 16-byte units (aligned 2: 2, 4 or 8
        // columns, wider strips of 16-bit storage at the price of a shared
        // sector at each strip boundary); column x sits at x + kPadCols of a
        // plane row and rows start 256-byte aligned
        const bool half = fmt == kFmtF16 || fmt == kFmtBF16;
        const int es = fmt == kFmtF64 ? 8 : (half ? 2 : 4);
        const int sec = aligned == 1 ? (half ? 16 : 8) : 16 / es;
        const int wmax = 124 / sec * sec;
        const int g0 = ((-kPadCols) % sec + sec) % sec - sec;  // g0 + kPadCols is a multiple of sec
        auto fdiv = [](int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); };
        xg = g0 + fdiv(rx0 - g0, sec) * sec;
        const int span = rx1 - xg, n = (span + wmax - 1) / wmax;
        W = ((span + n - 1) / n + sec - 1) / sec * sec;
    }
    *strip_x0 = xg;
    *strip_w = W;
    *nstrips = (rx1 - xg + W - 1) / W;  // the first and last strips may be partial
}

template <class TS, class TC, class UT, int NT, bool XJ, class Kernel>
int interior_occupancy_k(Kernel kern, int ring_slots) {
    int n = 0;
    cudaError_t e = allow_any_ring<TS, TC, UT, NT, XJ>(kern);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, NT,
                                                          interior_smem_bytes<TS, TC, UT, NT, XJ>(ring_slots));
    return e == cudaSuccess ? n : 0;
}
template <class TS, class TC, class UT, int NT, int MINB, bool UNROLL3>
int interior_occupancy_t(bool xj, int ring_slots) {
    return xj ? interior_occupancy_k<TS, TC, UT, NT, true>(interior_step_kernel<TS, TC, UT, NT, MINB, true, false>,
                                                           ring_slots)
              : interior_occupancy_k<TS, TC, UT, NT, false>(interior_step_kernel<TS, TC, UT, NT, MINB, false, UNROLL3>,
                                                            ring_slots);
}

// Per format: the minimum CTAs per SM (the register cap) and the row loop's
// form: FP16 / BF16 run the unrolled loop (72 registers, so 7 CTAs of one body
// fit an SM; held to 6 by their shared memory, 1000 x 1000 with a hole took
// 23.5 us a step instead of 22.4 and 2200 x 1800 69.7 instead of 72.8), plain-
// carry FP32 too at 72 registers (3 % at 4096 x 2048); the compensated carry
// has no registers to spare and runs the rotating loop (the unrolled one gained
// nothing for one body and made batches slower).
int interior_occupancy(int fmt, bool xj, int ring_slots) {
    switch (fmt) {
        case kFmtF64: return interior_occupancy_t<double, double, UPlain<double>, 128, 3, false>(xj, ring_slots);
        case kFmtF32: return interior_occupancy_t<float, float, UPlain<float>, 128, 7, true>(xj, ring_slots);
        case kFmtF32C: return interior_occupancy_t<float, float, UComp, 128, 6, false>(xj, ring_slots);
        case kFmtF32H: return interior_occupancy_t<float, float, UCompH, 128, 6, false>(xj, ring_slots);
        case kFmtF16: return interior_occupancy_t<__half, float, UComp, 128, 6, true>(xj, ring_slots);
        default: return interior_occupancy_t<__nv_bfloat16, float, UComp, 128, 6, true>(xj, ring_slots);
    }
}

int64_t interior_items(const int rect[4], int inst, int strips, const ChunkLevels& L, InteriorItem* out, int64_t cap) {
    int64_t n = 0;
    int y = rect[2], by = 0;
    for (int k = 0; k < 4; ++k)
        for (int c = 0; c < L.count[k] && y < rect[3]; ++c, ++by) {
            const int rows = std::min(L.rows[k], rect[3] - y);
            for (int bx = 0; bx < strips; ++bx, ++n)
                if (out && n < cap) out[n] = InteriorItem{inst, bx, y, (by & 1) ? -rows : rows};
            y += rows;
        }
    return n;
}

namespace {

using EncodeTiled = decltype(&cuTensorMapEncodeTiled);

// The driver's encoder (the library does not link against libcuda).
EncodeTiled encode_tiled() {
    static const EncodeTiled fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<EncodeTiled>(f);
    }();
    return fn;
}

// The maps of one state with the boxes of RingSlot.
template <class TS, class TC, class UT, bool XJ>
bool encode_maps(const void* f, const void* a, const void* src, int64_t pitch, int64_t plane, int ny,
                 InteriorMaps* out) {
    using Slot = RingSlot<TS, TC, UT, kInteriorThreads, XJ>;
    const EncodeTiled enc = encode_tiled();
    if (!enc) return false;
    const int64_t rows = int64_t(ny) + 2 * kPadRows;
    // words of `es` bytes from `at` on; planes `step` bytes apart, of `nrows` rows; boxes of w columns of np planes
    auto make = [&](CUtensorMap* m, const void* at, int es, int64_t nrows, int nplanes, int64_t step, int w, int np) {
        const CUtensorMapDataType type = es == 8   ? CU_TENSOR_MAP_DATA_TYPE_UINT64
                                         : es == 4 ? CU_TENSOR_MAP_DATA_TYPE_UINT32
                                                   : CU_TENSOR_MAP_DATA_TYPE_UINT16;
        const cuuint64_t dim[3] = {cuuint64_t(pitch), cuuint64_t(nrows), cuuint64_t(nplanes)};
        const cuuint64_t stride[2] = {cuuint64_t(pitch * es), cuuint64_t(step)};
        const cuuint32_t box[3] = {cuuint32_t(w), 1, cuuint32_t(np)}, unit[3] = {1, 1, 1};
        return enc(m, type, 3, const_cast<void*>(at), dim, stride, box, unit, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    const char* f0 = static_cast<const char*>(f);
    const char* a0 = static_cast<const char*>(a);
    constexpr int ES = Slot::ES, CS = Slot::CS;
    constexpr bool half_lo = UT::layout == kCarryPair16;  // components 1.5 planes apart, low words after the high ones
    return make(&out->f, f0, ES, rows, 9, plane * ES, Slot::SEG, 2) &&
           make(&out->f3, f0 + 2 * plane * ES, ES, rows - 2, 3, (plane + pitch) * ES, Slot::SEG, 3) &&
           make(&out->a, a0, CS, rows, Slot::NA, half_lo ? plane * 6 : plane * CS, Slot::SEGC, Slot::NA) &&
           (!half_lo || make(&out->lo, a0 + plane * 4, 2, rows, 2, plane * 6, Slot::SEGL, 2)) &&
           make(&out->s, src, CS, rows, Slot::NS, plane * CS, Slot::SEGC, Slot::NS);
}

}  // namespace

cudaError_t interior_maps(int fmt, bool xj, const void* f, const void* a, const void* s, int64_t pitch, int64_t plane,
                          int ny, InteriorMaps* out) {
    memset(out, 0, sizeof(*out));
    auto enc = [&](auto ts, auto tc, auto ut) {
        using TS = decltype(ts);
        using TC = decltype(tc);
        using UT = decltype(ut);
        return xj ? encode_maps<TS, TC, UT, true>(f, a, s, pitch, plane, ny, out)
                  : encode_maps<TS, TC, UT, false>(f, a, s, pitch, plane, ny, out);
    };
    bool ok = false;
    switch (fmt) {
        case kFmtF64: ok = enc(double(), double(), UPlain<double>()); break;
        case kFmtF32: ok = enc(float(), float(), UPlain<float>()); break;
        case kFmtF32C: ok = enc(float(), float(), UComp()); break;
        case kFmtF32H: ok = enc(float(), float(), UCompH()); break;
        case kFmtF16: ok = enc(__half(), float(), UComp()); break;
        case kFmtBF16: ok = enc(__nv_bfloat16(), float(), UComp()); break;
    }
    return ok ? cudaSuccess : cudaErrorNotSupported;
}

namespace {

constexpr int kMapWords = int(sizeof(InteriorMaps) / sizeof(int4));

__global__ void gather_maps(const InteriorMaps* const* from, InteriorMaps* to) {
    reinterpret_cast<int4*>(to + blockIdx.x)[threadIdx.x] =
        reinterpret_cast<const int4*>(from[blockIdx.x])[threadIdx.x];
    release_tensor_maps();
}

}  // namespace

// (Encoded and uploaded by the host for each batch, the maps of 256 members took
// 140 us of the 454 in which it was made; read where the members hold them, by a
// list, small batches' steps took up to 4 % longer.)
cudaError_t gather_interior_maps(const InteriorMaps* const* from, InteriorMaps* to, int n, cudaStream_t s) {
    gather_maps<<<unsigned(n), kMapWords, 0, s>>>(from, to);
    return cudaGetLastError();
}

cudaError_t launch_interior(int fmt, const StepParams& p0, const InteriorRects& R, const InteriorMaps& maps, cudaStream_t s,
                            bool fields) {
    StepParams p = p0;
    if (!fields) p.fields = nullptr;
    switch (fmt) {
        case kFmtF64: return launch_interior_t<double, double, UPlain<double>, 128, 3, false>(p, R, maps, s);
        case kFmtF32: return launch_interior_t<float, float, UPlain<float>, 128, 7, true>(p, R, maps, s);
        case kFmtF32C: return launch_interior_t<float, float, UComp, 128, 6, false>(p, R, maps, s);
        case kFmtF32H: return launch_interior_t<float, float, UCompH, 128, 6, false>(p, R, maps, s);
        case kFmtF16: return launch_interior_t<__half, float, UComp, 128, 6, true>(p, R, maps, s);
        case kFmtBF16: return launch_interior_t<__nv_bfloat16, float, UComp, 128, 6, true>(p, R, maps, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lbm
