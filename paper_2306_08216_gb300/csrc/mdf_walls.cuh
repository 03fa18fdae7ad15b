// mdf_walls.cuh -- fused MDF-FDLBM step with non-equilibrium
// extrapolation walls and/or a power-law fluid, on uniform or separable
// grids, marched by rows like the periodic fast path.
//
// The time step is that of mdf_step.cu (Sec. 2.2 Steps (1)-(4) of
// arXiv:2306.08216 with Eqs. 2.3.24-2.3.25, f32x2 pairs for alpha = u, v)
// with the same row march as mdf_step_fast.cu: populations 2 and 4 keep
// what their y stencils need of fbar^+ and f(t+h) in registers (five-row windows
// in march_window, for a single problem; carried sums in march_walls, for
// batches), populations 1
// and 3 run their x stencils through double-buffered exchange rows, fhat^+
// waits in a shared ring, and one barrier orders each row.  On top of that:
//  * walls (Secs. 4.3-4.4): wall nodes take the non-equilibrium
//    extrapolation of their wall-normal interior neighbour (the diagonal one
//    at corners) for f(t+h) and for fhat(t+dt), written by the neighbour's
//    thread; next to a wall the second-order upwind point beyond it is
//    replaced by its linear extrapolation (stream2 with the wall flag);
//    rows beyond a y wall are not wrapped (TMA fills them with zeros, and
//    nothing reads them);
//  * power law: the relaxation rates of every node follow from its
//    non-equilibrium first moment in Step 1 and wait two rows in a register
//    window for the recovery of Step 3.
// f(t+h) of a wall node is needed only by the stencils of interior nodes:
// pops 1 and 3 of a wall column go to the exchange row (written by the
// thread of the adjacent interior column), pops 2 and 4 of a wall row to the
// registers of the same column (south: when row 1 is formed; north:
// from row ny-2 through a one-row shared buffer, one iteration later).
//
// This header holds the march and its kernel templates; mdf_step_walls.cu
// instantiates the FP32 kernels and the entry points, mdf_step_walls16.cu
// the batched kernels with 16-bit storage (FP32 u, v, P plus FP16/BF16
// non-equilibrium pairs, as on the periodic fast path).
#pragma once

#include <algorithm>
#include <type_traits>

#include "mdf_device.cuh"

namespace mdf {

namespace {

using namespace dev;

__device__ __forceinline__ F2 pair_of(unsigned long long bits) {
    F2 a;
    a.r = bits;
    return a;
}

struct W3 {
    F2 w1, w0, w2;
};

__device__ __forceinline__ W3 weights(float k, float step, const StepArgs &a) {
    W3 w;
    w.w1 = splat(-step * k * a.a1);
    w.w0 = splat(-step * k * a.a0);
    w.w2 = splat(-step * k * a.am2);
    return w;
}

// One TMA row: 10 FP32 planes, or u, v, P and 4 planes of 16-bit pairs.
template <int ST>
constexpr int walls_row_planes() {
    return ST == STORAGE_FP32 ? NPLANES : DEV_PLANES;
}

// Rows of fhat in flight, and the force rows (p-4 .. p+2) every thread keeps of
// its own column, copied two rows ahead (see mdf_step_fast.cu); with 256
// threads one TMA slot makes room for them.
constexpr int WALL_FORCE_ROWS = 8;
template <int NT, bool FORCED>
__host__ __device__ constexpr int walls_slots() {
    return FORCED && NT == 256 ? 2 : TMA_SLOTS;
}

template <int NT, bool FORCED, int ST = STORAGE_FP32>
constexpr int walls_smem() {
    return walls_slots<NT, FORCED>() * walls_row_planes<ST>() * NT * 4 + RING * 5 * NT * 8 + 4 * (2 * NT * 8) +
           2 * NT * 8 + walls_slots<NT, FORCED>() * 8 + (FORCED ? WALL_FORCE_ROWS * 2 * NT * 4 : 0);
}

// Store one node in the layout of the storage mode (with the periodic
// images of a periodic x axis when XPER).
template <int ST, bool XPER>
__device__ __forceinline__ void store_node_st(const StepArgs &a, int row, int X, const F2 v[5]) {
    if (ST == STORAGE_FP32) store_node<XPER>(a, row, X, v);
    else store_node_dev<ST, XPER>(a, row, X, v);
}

// One block's march over strip bx, band by.  FORCED: body force, force rate
// or source present (read at run time); otherwise those terms are compiled out.
// ROLL: the march loop is not unrolled; otherwise it is unrolled by two.  The
// two compute the same values, in nearly the same time (power-law cavities of
// 65^2 to 513^2, us a step, unrolled / rolled: 16 of them 75.0 / 75.3, 512
// 1425 / 1429; Newtonian ones 53.8 / 53.1 and 1175 / 1159).  The y stencils carry seven values per stage
// from row to row (YCarry): with five-row register windows the loop was either
// five bodies long, which missed the instruction cache, or rotated a hundred
// registers a row, and took 168 registers (four blocks of 96 threads per SM;
// now at most 128 and five).
// ST: the storage mode of the state (16-bit: fhat is rebuilt from the
// stored u, v, P and non-equilibrium pairs on load, and stored back in that
// form, as on the periodic fast path).
template <int NT, int MK, bool PL, bool FORCED, bool ROLL, int ST>
__device__ __forceinline__ void march_walls(const CUtensorMap *tmap, const StepArgs &a, int bx, int by,
                                            unsigned char *smem, volatile int *s_abort) {
    constexpr int SLOTS = walls_slots<NT, FORCED>();
    constexpr int TROW = walls_row_planes<ST>() * NT * 4;  // one TMA row
    constexpr int PROW = 5 * NT * 8;        // one fhat^+ ring row
    constexpr int XROW = 2 * NT * 8;        // one exchange row: pops 1, 3
    unsigned char *tma = smem;
    unsigned char *ringP = tma + SLOTS * TROW;
    unsigned char *xB0 = ringP + RING * PROW;  // fbar^+ of pops 1, 3 of row p (two buffers)
    unsigned char *xF0 = xB0 + 2 * XROW;       // f(t+h) of pops 1, 3 of row q (two buffers)
    unsigned char *nrow = xF0 + 2 * XROW;      // f(t+h) of pops 2, 4 of the north wall row
    uint64_t *mbar = reinterpret_cast<uint64_t *>(nrow + 2 * NT * 8);
    unsigned char *ringF = reinterpret_cast<unsigned char *>(mbar + SLOTS);  // force field rows (FORCED)

    const int t = threadIdx.x;
    const int x0 = bx * a.W;
    const int X = x0 - 4 + t;
    const int y0 = by * a.H;
    const int y1 = min(y0 + a.H, a.ny);
    const int nIt = (y1 - y0) + 8;
    const int rowBase = y0 - 4;
    const float c = a.c, inv2c = a.inv2c;
    const int ny = a.ny;
    const bool xwall = a.xwall, ywall = a.ywall;
    const bool colx_wall = xwall && (X == 0 || X == a.nx - 1);
    const bool colx_out = xwall && (X < 0 || X >= a.nx);
    const bool xadj_p = xwall && X == 1, xadj_m = xwall && X == a.nx - 2;
    const bool col_in = X >= -GHOST && X < a.nx + GHOST;  // has a padded-field entry

    // abort flags, one per row parity: a flag is read after the barrier of its
    // row, and a thread can set it again only two barriers later
    if (t == 0) {
        s_abort[0] = s_abort[1] = 0;
        for (int i = 0; i < SLOTS; ++i) mbar_init(&mbar[i], 1);
        fence_mbar_init();
    }
    __syncthreads();
    // row p of the domain (beyond a y wall: as it is), and the next one to load
    int rp = ywall ? rowBase : wrap(rowBase, ny), lrow = rp;
    auto after = [&](int r) { return !ywall && r + 1 == ny ? 0 : r + 1; };
    auto before = [&](int r, int k) { return !ywall && r < k ? r - k + ny : r - k; };
    auto load_row = [&](int slot) {
        mbar_expect_tx(&mbar[slot], TROW);
        tma_load_row(tmap, &mbar[slot], tma + slot * TROW, x0, lrow);
        lrow = after(lrow);
    };
    int issued = min(SLOTS, nIt);
    if (t == 0)
        for (int i = 0; i < issued; ++i) load_row(i);

    // body force (fields): F of this column two rows ahead of every row; the dt
    // step reads the same rows unless a force rate gave it planes of its own
    const bool ffield = FORCED && a.force_mode == 2;
    const bool fd_same = ffield && a.force_mode_d == 2 && a.Fxdp == a.Fxp && a.Fydp == a.Fyp;
    int frow = rp;
    auto force_slot = [&](int it) { return ringF + ((it & (WALL_FORCE_ROWS - 1)) * 2 * NT + t) * 4; };
    auto copy_force = [&](int it) {
        if (ffield && it < nIt) {
            if (col_in && frow >= 0 && frow < ny) {
                const long long e = (long long)frow * a.pitch + GHOST + X;
                if (index_ok(a, e, a.plane)) {
                    cp_async4(force_slot(it), a.Fxp + e);
                    cp_async4(force_slot(it) + NT * 4, a.Fyp + e);
                }
            }
            frow = after(frow);
        }
        cp_async_commit();
    };
    auto force_ring = [&](int it) {
        const unsigned char *q = force_slot(it);
        return mk2(lds1(q, 0), lds1(q, NT * 4));
    };
    auto force_h = [&](int it, F2 factor) {
        if (a.force_mode == 0) return splat(0.0f);
        return factor * (ffield ? force_ring(it) : mk2(a.Fx, a.Fy));
    };
    auto force_dt = [&](int it, int row, F2 factor) {
        if (a.force_mode_d == 0) return splat(0.0f);
        if (fd_same) return factor * force_ring(it);
        if (a.force_mode_d == 1) return factor * mk2(a.Fxd, a.Fyd);
        if (!col_in) return splat(0.0f);
        return factor * field_pair(a, a.Fxdp, a.Fydp, (long long)row * a.pitch + GHOST + X);
    };
    if (FORCED) {
        copy_force(0);
        copy_force(1);
    }

    W3 wxh, wxd;
    if (MK == METRIC_UNIFORM) {
        wxh = {pair_of(a.pwxh[0]), pair_of(a.pwxh[1]), pair_of(a.pwxh[2])};
        wxd = {pair_of(a.pwxd[0]), pair_of(a.pwxd[1]), pair_of(a.pwxd[2])};
    } else {
        const float kx = a.kxv[min(GHOST + X, a.pitch - 1)];
        wxh = weights(kx, a.h, a);
        wxd = weights(kx, a.dt, a);
    }
    auto wyh = [&](float k) {
        return MK == METRIC_UNIFORM ? W3{pair_of(a.pwyh[0]), pair_of(a.pwyh[1]), pair_of(a.pwyh[2])}
                                    : weights(k, a.h, a);
    };
    auto wyd = [&](float k) {
        return MK == METRIC_UNIFORM ? W3{pair_of(a.pwyd[0]), pair_of(a.pwyd[1]), pair_of(a.pwyd[2])}
                                    : weights(k, a.dt, a);
    };
    const F2 zero = splat(0.0f);
    const bool calc = t >= 2 && t < NT - 2 && !colx_out && !colx_wall;          // forms fbar and f
    const bool outc = t >= 4 && t < NT - 4 && X >= 0 && X < a.nx && !colx_wall;  // forms outputs

    // carried from row to row
    YCarry<F2> cb, cf;    // fbar^+ (pass 1) and f(t+h) (pass 2) of pops 2, 4
    F2 D1[3], D2[3];      // fbar of pops 0, 1, 3 of rows p-1, p-2 (x part done)
    F2 XI[2];             // pass-2 x increments of pops 1, 3 of row r
    float R1[2], R2[2];   // power law: recovery rates (rkp, rk) of rows p-1, p-2
    cb.clear(zero);
    cf.clear(zero);
    D1[0] = D1[1] = D1[2] = D2[0] = D2[1] = D2[2] = XI[0] = XI[1] = zero;
    R1[0] = R1[1] = R2[0] = R2[1] = 0.0f;
    float k0 = 0.0f, k1 = 0.0f, k2 = 0.0f, k3 = 0.0f, k4 = 0.0f;  // stretched: c eta_y of rows p .. p-4

    int tslot = 0, phase = 0;  // TMA ring
    int pring = 0;             // ring row of row p
    bool aborted = false;
    constexpr int UNROLL = ROLL ? 1 : 2;
#pragma unroll UNROLL
    for (int it = 0; it < nIt; ++it) {
        const int par = it & 1;
        if (FORCED) {
            copy_force(it + 2);
            cp_async_wait<2>();  // the copies of row p have landed
        }
        unsigned char *xB = xB0 + par * XROW;
        unsigned char *xF = xF0 + par * XROW;
        const unsigned char *xFp = xF0 + (par ^ 1) * XROW;
        // ring rows of q = p - 2 and r = p - 4
        const int qring = pring >= 2 ? pring - 2 : pring + 3, rring = pring == 4 ? 0 : pring + 1;
        // ---------------------------------------------- S2: row p
        const bool p_in = !ywall || (rp >= 0 && rp < ny);
        F2 own1, own3, b0, b2, b4;
        float rk0 = 0.0f, rk1 = 0.0f;
        {
            if (!mbar_wait_bounded(&mbar[tslot], (uint32_t)phase)) s_abort[par] = 1;
            const float *src = reinterpret_cast<const float *>(tma + tslot * TROW);
            F2 g[5], n[5], o[5];
            if (ST == STORAGE_FP32) {
#pragma unroll
                for (int j = 0; j < 5; ++j) g[j] = mk2(src[j * NT + t], src[(5 + j) * NT + t]);
                const Mom2 m = (FORCED && a.r_mode && p_in && col_in)
                                   ? moments2r(g, c, a.rk_hat * source_at(a, rp, X))
                                   : moments2(g, c);
                noneq2(g, m, inv2c, n);
            } else {
                // fhat = feq(u, v, P) + n from the stored fields (16-bit
                // modes carry no source term)
                const unsigned *w = reinterpret_cast<const unsigned *>(src + DEV_FPLANES * NT);
                const F2 inv = splat(a.ninv);
                F2 nn[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) nn[j] = unpack16<ST>(w[j * NT + t]) * inv;
                dev_build(src[t], src[NT + t], src[2 * NT + t], nn, inv2c, g, n);
            }
            const F2 n13 = n[1] - n[3], n24 = n[2] - n[4];
            F2 mKp = pair_of(a.pmKp), Dp = pair_of(a.pDp), mKb = pair_of(a.pmKb), Db = pair_of(a.pDb);
            if (PL) {
                float gx1, gx2, gy1, gy2;
                split2(splat(c) * n13, gx1, gx2);
                split2(splat(c) * n24, gy1, gy2);
                const float sxy = 0.5f * (gy1 + gx2);
                const float gg = sqrtf(2.0f * (gx1 * gx1 + gy2 * gy2 + 2.0f * sxy * sxy));
                const Rates Rr = rates_nu(power_law_nu(gg, a), a.s_ratio, a.a_pl);
                mKp = splat(-(1.0f - Rr.rpp));
                Dp = splat(0.5f * (Rr.rp - Rr.rpp));
                mKb = splat(-(1.0f - Rr.rbp));
                Db = splat(0.5f * (Rr.rb - Rr.rbp));
                rk0 = Rr.rkp;
                rk1 = Rr.rk;
            }
            relax2(g, n, n13, n24, mKp, Dp, o);
            unsigned char *dP = ringP + pring * PROW;
#pragma unroll
            for (int j = 0; j < 5; ++j) sts2(dP, (j * NT + t) * 8, o[j]);
            relax2(g, n, n13, n24, mKb, Db, o);
            sts2(xB, t * 8, o[1]);
            sts2(xB, (NT + t) * 8, o[3]);
            own1 = o[1];
            own3 = o[3];
            b0 = o[0];
            b2 = o[2];
            b4 = o[4];
        }
        // one barrier per row (exchange rows double-buffered by row parity)
        __syncthreads();
        if (s_abort[par]) {
            aborted = true;
            break;
        }
        if (t == 0 && issued < nIt) {
            fence_proxy_async();
            load_row(tslot);
            ++issued;
        }
        if (++tslot == SLOTS) {
            tslot = 0;
            phase ^= 1;
        }
        if (MK != METRIC_UNIFORM) {
            k4 = k3;
            k3 = k2;
            k2 = k1;
            k1 = k0;
            k0 = p_in ? a.kyv[rp] : 0.0f;
        }
        // ---------------------------------------------- S1: pass-2 x increments of row q - 1
        F2 XN[2] = {zero, zero};
        if (outc) {
            const F2 f1p1 = lds2(xFp, (t + 1) * 8), f1 = lds2(xFp, t * 8);
            const F2 f1m1 = lds2(xFp, (t - 1) * 8), f1m2 = lds2(xFp, (t - 2) * 8);
            const F2 f3m1 = lds2(xFp, (NT + t - 1) * 8), f3 = lds2(xFp, (NT + t) * 8);
            const F2 f3p1 = lds2(xFp, (NT + t + 1) * 8), f3p2 = lds2(xFp, (NT + t + 2) * 8);
            XN[0] = stream2<true>(zero, f1p1, f1, f1m1, f1m2, xadj_p, wxd.w1, wxd.w0, wxd.w2);
            XN[1] = stream2<true>(zero, f3m1, f3, f3p1, f3p2, xadj_m, wxd.w1, wxd.w0, wxd.w2);
        }
        // ---------------------------------------------- S3: row q = p - 2, then S0: row r = p - 4
        if (calc) {
            const int q = before(rp, 2), r = rowBase + it - 4;
            const W3 wh0 = wyh(k0), wh1 = wyh(k1), wh2 = wyh(k2);  // rows p, p-1, q
            F2 hF = zero, hFq = zero;
            if (FORCED) {
                if (p_in) hF = force_h(it, pair_of(a.phw));
                if (!ywall || (q >= 0 && q < ny)) hFq = force_h(it - 2, pair_of(a.phw));
            }
            // fbar of row q: pops 0, 1, 3 from two rows ago, 2 and 4 completed by row p
            F2 fb[5];
            fb[0] = D2[0];
            fb[1] = D2[1];
            fb[3] = D2[2];
            fb[2] = cb.two();
            fb[4] = cb.template four<true>(FORCED ? cb.b4 + hFq : cb.b4, b4, ywall && q == ny - 2, wh2);
            // row p: pass 1, x part; its y part begins
#pragma unroll
            for (int k = 0; k < 3; ++k) D2[k] = D1[k];
            D1[0] = FORCED ? b0 + hF : b0;
            D1[1] = stream2<true>(FORCED ? own1 + hF : own1, lds2(xB, (t + 1) * 8), own1, lds2(xB, (t - 1) * 8),
                                  lds2(xB, (t - 2) * 8), xadj_p, wxh.w1, wxh.w0, wxh.w2);
            D1[2] = stream2<true>(FORCED ? own3 + hF : own3, lds2(xB, (NT + t - 1) * 8), own3,
                                  lds2(xB, (NT + t + 1) * 8), lds2(xB, (NT + t + 2) * 8), xadj_m, wxh.w1, wxh.w0,
                                  wxh.w2);
            cb.template push<true>(b2, b4, FORCED ? b2 + hF : b2, ywall && rp == 1, wh0, wh1);
            // Step 3: f = feq + (I + h/2 Lt)^-1 (fbar - feq); f of pops 2, 4 of row q
            F2 f2 = zero, f4 = zero;
            if (!ywall || (q > 0 && q < ny - 1)) {
                F2 mKk = pair_of(a.pmKk), Dk = pair_of(a.pDk);
                if (PL) {
                    mKk = splat(-(1.0f - R2[0]));
                    Dk = splat(0.5f * (R2[1] - R2[0]));
                }
                const Mom2 m = (FORCED && a.r_mode && col_in) ? moments2r(fb, c, a.rk_bar * source_at(a, q, X))
                                                              : moments2(fb, c);
                F2 n[5], f[5];
                noneq2(fb, m, inv2c, n);
                relax2(fb, n, n[1] - n[3], n[2] - n[4], mKk, Dk, f);
                sts2(xF, t * 8, f[1]);
                sts2(xF, (NT + t) * 8, f[3]);
                f2 = f[2];
                f4 = f[4];
                F2 w[5];
                if (xadj_p) {  // west wall column of this row: pops 1, 3 for the x stencils
                    nee2(f, a.uw[0], a.vw[0], inv2c, w);
                    sts2(xF, (t - 1) * 8, w[1]);
                    sts2(xF, (NT + t - 1) * 8, w[3]);
                }
                if (xadj_m) {
                    nee2(f, a.uw[1], a.vw[1], inv2c, w);
                    sts2(xF, (t + 1) * 8, w[1]);
                    sts2(xF, (NT + t + 1) * 8, w[3]);
                }
                if (ywall && q == 1) {  // south wall row (q - 1): pops 2, 4 for the y stencils
                    nee2(f, a.uw[2], a.vw[2], inv2c, w);
                    cf.a2 = w[2];
                    cf.a4 = w[4];
                }
                if (ywall && q == ny - 2) {  // north wall row, taken up next iteration
                    nee2(f, a.uw[3], a.vw[3], inv2c, w);
                    sts2(nrow, t * 8, w[2]);
                    sts2(nrow, (NT + t) * 8, w[4]);
                }
            } else if (q == ny - 1) {
                // north wall row: pops 2, 4 of its NEE value were formed with row ny-2
                f2 = lds2(nrow, t * 8);
                f4 = lds2(nrow, (NT + t) * 8);
            }
            // Step 4: row r is complete, the y part of row q begins
            const W3 wd2 = wyd(k2), wd3 = wyd(k3), wd4 = wyd(k4);  // rows q, q-1, r
            const bool r_out = it >= 8 && !(ywall && (r == 0 || r == ny - 1));
            const unsigned char *Pr = ringP + rring * PROW, *Pq = ringP + qring * PROW;
            F2 out[5];
            out[0] = lds2(Pr, t * 8);
            out[1] = lds2(Pr, (NT + t) * 8);
            out[3] = lds2(Pr, (3 * NT + t) * 8);
            out[4] = lds2(Pr, (4 * NT + t) * 8);
            F2 base2 = lds2(Pq, (2 * NT + t) * 8);
            if (FORCED) {
                if (r_out) {
                    const F2 fr = force_dt(it - 4, r, pair_of(a.pdw));
                    out[0] = out[0] + fr;
                    out[1] = out[1] + fr;
                    out[3] = out[3] + fr;
                    out[4] = out[4] + fr;
                }
                if (!ywall || (q >= 0 && q < ny)) base2 = base2 + force_dt(it - 2, q, pair_of(a.pdw));
            }
            out[1] = out[1] + XI[0];
            out[3] = out[3] + XI[1];
            out[2] = cf.two();
            out[4] = cf.template four<true>(out[4], f4, ywall && r == ny - 2, wd4);
            cf.template push<true>(f2, f4, base2, ywall && q == 1, wd2, wd3);
            XI[0] = XN[0];
            XI[1] = XN[1];
            if (r_out && outc) {
                const bool yadj_p = ywall && r == 1, yadj_m = ywall && r == ny - 2;
                if (xwall) store_node_st<ST, false>(a, r, X, out);
                else store_node_st<ST, true>(a, r, X, out);
                F2 w[5];
                if (xadj_p) { nee2(out, a.uw[0], a.vw[0], inv2c, w); store_node_st<ST, false>(a, r, 0, w); }
                if (xadj_m) { nee2(out, a.uw[1], a.vw[1], inv2c, w); store_node_st<ST, false>(a, r, a.nx - 1, w); }
                if (yadj_p || yadj_m) {
                    const int rr = yadj_p ? 0 : ny - 1;
                    const int side = yadj_p ? 2 : 3;
                    nee2(out, a.uw[side], a.vw[side], inv2c, w);
                    if (xwall) store_node_st<ST, false>(a, rr, X, w);
                    else store_node_st<ST, true>(a, rr, X, w);
                    if (xadj_p) { nee2(out, a.uw[0], a.vw[0], inv2c, w); store_node_st<ST, false>(a, rr, 0, w); }
                    if (xadj_m) { nee2(out, a.uw[1], a.vw[1], inv2c, w); store_node_st<ST, false>(a, rr, a.nx - 1, w); }
                }
            }
        }
        if (PL) {
            R2[0] = R1[0];
            R2[1] = R1[1];
            R1[0] = rk0;
            R1[1] = rk1;
        }
        pring = pring == RING - 1 ? 0 : pring + 1;
        rp = after(rp);
    }
    if (FORCED) cp_async_wait<0>();
    if (aborted && t == 0) {
        for (int it = issued - SLOTS; it < issued; ++it) {
            if (it < 0) continue;
            mbar_wait_bounded(&mbar[it % SLOTS], (uint32_t)((it / SLOTS) & 1));
        }
        atomicCAS(a.err, DEVERR_NONE, DEVERR_TMA_TIMEOUT);
    }
    // every copy was consumed: the barriers may be invalidated for reuse
    __syncthreads();
    if (t == 0)
        for (int i = 0; i < SLOTS; ++i) mbar_inval(&mbar[i]);
    __syncthreads();
}

// The same march for a single problem, with its y stencils in five-row register
// windows and the loop unrolled by five, so that every window slot is a
// compile-time index: no register moves and the output row first in the
// iteration make the shorter row latency, which decides where a problem's short
// bands leave a block few rows (700 x 600 nodes: 18.5 us a step against 19.9 of
// march_walls; stretched 1200 x 700 channel 35 against 38).  On a full GPU, in
// the batches, march_walls is the faster (512 power-law cavities 1.81 -> 1.57 ms a
// step).
template <int NT, int MK, bool PL, int FORCE>
__device__ __forceinline__ void march_window(const CUtensorMap *tmap, const StepArgs &a, int bx, int by,
                                             unsigned char *smem, volatile int *s_abort) {
    constexpr int SLOTS = walls_slots<NT, FORCE == FORCE_ANY>();
    constexpr int TROW = NPLANES * NT * 4;  // one TMA row
    constexpr int PROW = 5 * NT * 8;        // one fhat^+ ring row
    constexpr int XROW = 2 * NT * 8;        // one exchange row: pops 1, 3
    unsigned char *tma = smem;
    unsigned char *ringP = tma + SLOTS * TROW;
    unsigned char *xB0 = ringP + RING * PROW;  // fbar^+ of pops 1, 3 of row p (two buffers)
    unsigned char *xF0 = xB0 + 2 * XROW;       // f(t+h) of pops 1, 3 of row q (two buffers)
    unsigned char *nrow = xF0 + 2 * XROW;      // f(t+h) of pops 2, 4 of the north wall row
    uint64_t *mbar = reinterpret_cast<uint64_t *>(nrow + 2 * NT * 8);
    unsigned char *ringF = reinterpret_cast<unsigned char *>(mbar + SLOTS);  // force field rows (FORCE_ANY)

    const int t = threadIdx.x;
    const int x0 = bx * a.W;
    const int X = x0 - 4 + t;
    const int y0 = by * a.H;
    const int y1 = min(y0 + a.H, a.ny);
    const int nIt = (y1 - y0) + 9;
    const int rowBase = y0 - 4;
    const float c = a.c, inv2c = a.inv2c;
    const int ny = a.ny;
    const bool xwall = a.xwall, ywall = a.ywall;
    const bool colx_wall = xwall && (X == 0 || X == a.nx - 1);
    const bool colx_out = xwall && (X < 0 || X >= a.nx);
    const bool xadj_p = xwall && X == 1, xadj_m = xwall && X == a.nx - 2;
    const bool col_in = X >= -GHOST && X < a.nx + GHOST;  // has a padded-field entry

    // abort flags, one per row parity: a flag is read after the barrier of its
    // row, and a thread can set it again only two barriers later
    if (t == 0) {
        s_abort[0] = s_abort[1] = 0;
        for (int i = 0; i < SLOTS; ++i) mbar_init(&mbar[i], 1);
        fence_mbar_init();
    }
    __syncthreads();
    // row p of the domain (beyond a y wall: as it is), and the next one to load
    int rp = ywall ? rowBase : wrap(rowBase, ny), lrow = rp;
    auto after = [&](int r) { return !ywall && r + 1 == ny ? 0 : r + 1; };
    auto before = [&](int r, int k) { return !ywall && r < k ? r - k + ny : r - k; };
    auto load_row = [&](int slot) {
        mbar_expect_tx(&mbar[slot], TROW);
        tma_load_row(tmap, &mbar[slot], tma + slot * TROW, x0, lrow);
        lrow = after(lrow);
    };
    int issued = min(SLOTS, nIt);
    if (t == 0)
        for (int i = 0; i < issued; ++i) load_row(i);

    // body force (fields): F of this column two rows ahead of every row; the dt
    // step reads the same rows unless a force rate gave it planes of its own
    const bool ffield = FORCE == FORCE_ANY && a.force_mode == 2;
    const bool fd_same = ffield && a.force_mode_d == 2 && a.Fxdp == a.Fxp && a.Fydp == a.Fyp;
    int frow = rp;
    auto force_slot = [&](int it) { return ringF + ((it & (WALL_FORCE_ROWS - 1)) * 2 * NT + t) * 4; };
    auto copy_force = [&](int it) {
        if (ffield && it < nIt) {
            if (col_in && frow >= 0 && frow < ny) {
                const long long e = (long long)frow * a.pitch + GHOST + X;
                if (index_ok(a, e, a.plane)) {
                    cp_async4(force_slot(it), a.Fxp + e);
                    cp_async4(force_slot(it) + NT * 4, a.Fyp + e);
                }
            }
            frow = after(frow);
        }
        cp_async_commit();
    };
    auto force_ring = [&](int it) {
        const unsigned char *q = force_slot(it);
        return mk2(lds1(q, 0), lds1(q, NT * 4));
    };
    auto force_h = [&](int it, F2 factor) {
        if (a.force_mode == 0) return splat(0.0f);
        return factor * (ffield ? force_ring(it) : mk2(a.Fx, a.Fy));
    };
    auto force_dt = [&](int it, int row, F2 factor) {
        if (a.force_mode_d == 0) return splat(0.0f);
        if (fd_same) return factor * force_ring(it);
        if (FORCE == FORCE_CONST || a.force_mode_d == 1) return factor * mk2(a.Fxd, a.Fyd);
        if (!col_in) return splat(0.0f);
        return factor * field_pair(a, a.Fxdp, a.Fydp, (long long)row * a.pitch + GHOST + X);
    };
    if (FORCE == FORCE_ANY) {
        copy_force(0);
        copy_force(1);
    }

    W3 wxh, wxd;
    if (MK == METRIC_UNIFORM) {
        wxh = {pair_of(a.pwxh[0]), pair_of(a.pwxh[1]), pair_of(a.pwxh[2])};
        wxd = {pair_of(a.pwxd[0]), pair_of(a.pwxd[1]), pair_of(a.pwxd[2])};
    } else {
        const float kx = a.kxv[min(GHOST + X, a.pitch - 1)];
        wxh = weights(kx, a.h, a);
        wxd = weights(kx, a.dt, a);
    }
    const F2 zero = splat(0.0f);
    const bool calc = t >= 2 && t < NT - 2 && !colx_out && !colx_wall;          // forms fbar and f
    const bool outc = t >= 4 && t < NT - 4 && X >= 0 && X < a.nx && !colx_wall;  // forms outputs

    F2 BY[5][2];    // fbar^+ of pops 2, 4
    F2 D013[5][3];  // fbar of pops 0, 1, 3 (x part done)
    F2 FY[5][2];    // f(t+h) of pops 2, 4
    F2 XF[5][2];    // pass-2 x increments of pops 1, 3
    float RK[5][2]; // power law: recovery rates (rkp, rk) of the row
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        BY[s][0] = BY[s][1] = FY[s][0] = FY[s][1] = XF[s][0] = XF[s][1] = zero;
        D013[s][0] = D013[s][1] = D013[s][2] = zero;
        RK[s][0] = RK[s][1] = 0.0f;
    }

    int tslot = 0;
    bool aborted = false;
    // One row iteration: window slot K of row p (and of row p - 5 before its
    // write), slots s1..s4 of rows p-1..p-4, row ps of the fhat^+ ring.
    // Returns false when the block aborts.
    auto row = [&](const int it, auto kc, const int ps) -> bool {
        constexpr int k = decltype(kc)::value;
        constexpr int s1 = (k + 4) % 5, s2 = (k + 3) % 5, s3 = (k + 2) % 5, s4 = (k + 1) % 5;
        {
            if (FORCE == FORCE_ANY) {
                copy_force(it + 2);
                cp_async_wait<2>();  // the copies of row p have landed
            }
            unsigned char *xB = xB0 + (it & 1) * XROW;
            const unsigned char *xFp = xF0 + ((it & 1) ^ 1) * XROW;
            unsigned char *xF = xF0 + (it & 1) * XROW;
            // ---------------------------------------------- S0: output row r = p - 5
            if (it >= 9 && outc) {
                const int r = rowBase + it - 5;  // in [y0, y1): a row of the domain
                if (!(ywall && (r == 0 || r == a.ny - 1))) {
                    const unsigned char *Pr = ringP + ps * PROW;
                    F2 out[5];
#pragma unroll
                    for (int j = 0; j < 5; ++j) out[j] = lds2(Pr, (j * NT + t) * 8);
                    if (FORCE != FORCE_NONE) {
                        const F2 fF = force_dt(it - 5, r, pair_of(a.pdw));
#pragma unroll
                        for (int j = 0; j < 5; ++j) out[j] = out[j] + fF;
                    }
                    out[1] = out[1] + XF[k][0];
                    out[3] = out[3] + XF[k][1];
                    W3 wy;
                    if (MK == METRIC_UNIFORM) wy = {pair_of(a.pwyd[0]), pair_of(a.pwyd[1]), pair_of(a.pwyd[2])};
                    else wy = weights(a.kyv[r], a.dt, a);
                    const bool yadj_p = ywall && r == 1, yadj_m = ywall && r == a.ny - 2;
                    out[2] = stream2<true>(out[2], FY[s4][0], FY[k][0], FY[s1][0], FY[s2][0], yadj_p, wy.w1, wy.w0,
                                           wy.w2);
                    out[4] = stream2<true>(out[4], FY[s1][1], FY[k][1], FY[s4][1], FY[s3][1], yadj_m, wy.w1, wy.w0,
                                           wy.w2);
                    if (xwall) store_node<false>(a, r, X, out);
                    else store_node<true>(a, r, X, out);
                    F2 w[5];
                    if (xadj_p) { nee2(out, a.uw[0], a.vw[0], inv2c, w); store_node<false>(a, r, 0, w); }
                    if (xadj_m) { nee2(out, a.uw[1], a.vw[1], inv2c, w); store_node<false>(a, r, a.nx - 1, w); }
                    if (yadj_p || yadj_m) {
                        const int rr = yadj_p ? 0 : a.ny - 1;
                        const int side = yadj_p ? 2 : 3;
                        nee2(out, a.uw[side], a.vw[side], inv2c, w);
                        if (xwall) store_node<false>(a, rr, X, w);
                        else store_node<true>(a, rr, X, w);
                        if (xadj_p) { nee2(out, a.uw[0], a.vw[0], inv2c, w); store_node<false>(a, rr, 0, w); }
                        if (xadj_m) { nee2(out, a.uw[1], a.vw[1], inv2c, w); store_node<false>(a, rr, a.nx - 1, w); }
                    }
                }
            }
            // ---------------------------------------------- S2: row p
            const bool p_in = !ywall || (rp >= 0 && rp < a.ny);
            F2 own1, own3;
            {
                if (!mbar_wait_bounded(&mbar[tslot], (uint32_t)((it / SLOTS) & 1))) s_abort[it & 1] = 1;
                const float *src = reinterpret_cast<const float *>(tma + tslot * TROW);
                F2 g[5], n[5], o[5];
#pragma unroll
                for (int j = 0; j < 5; ++j) g[j] = mk2(src[j * NT + t], src[(5 + j) * NT + t]);
                const Mom2 m = (FORCE == FORCE_ANY && a.r_mode && p_in && col_in)
                                   ? moments2r(g, c, a.rk_hat * source_at(a, rp, X))
                                   : moments2(g, c);
                noneq2(g, m, inv2c, n);
                const F2 n13 = n[1] - n[3], n24 = n[2] - n[4];
                F2 mKp = pair_of(a.pmKp), Dp = pair_of(a.pDp), mKb = pair_of(a.pmKb), Db = pair_of(a.pDb);
                if (PL) {
                    float gx1, gx2, gy1, gy2;
                    split2(splat(c) * n13, gx1, gx2);
                    split2(splat(c) * n24, gy1, gy2);
                    const float sxy = 0.5f * (gy1 + gx2);
                    const float gg = sqrtf(2.0f * (gx1 * gx1 + gy2 * gy2 + 2.0f * sxy * sxy));
                    const Rates Rr = rates_nu(power_law_nu(gg, a), a.s_ratio, a.a_pl);
                    mKp = splat(-(1.0f - Rr.rpp));
                    Dp = splat(0.5f * (Rr.rp - Rr.rpp));
                    mKb = splat(-(1.0f - Rr.rbp));
                    Db = splat(0.5f * (Rr.rb - Rr.rbp));
                    RK[k][0] = Rr.rkp;
                    RK[k][1] = Rr.rk;
                }
                relax2(g, n, n13, n24, mKp, Dp, o);
                unsigned char *dP = ringP + ps * PROW;
#pragma unroll
                for (int j = 0; j < 5; ++j) sts2(dP, (j * NT + t) * 8, o[j]);
                relax2(g, n, n13, n24, mKb, Db, o);
                sts2(xB, t * 8, o[1]);
                sts2(xB, (NT + t) * 8, o[3]);
                own1 = o[1];
                own3 = o[3];
                BY[k][0] = o[2];
                BY[k][1] = o[4];
                D013[k][0] = o[0];
            }
            // one barrier per row (exchange rows double-buffered by row parity)
            __syncthreads();
            if (s_abort[it & 1]) return false;
            if (t == 0 && issued < nIt) {
                fence_proxy_async();
                load_row(tslot);
                ++issued;
            }
            tslot = (tslot == SLOTS - 1) ? 0 : tslot + 1;
            // ---------------------------------------------- S1: pass-2 x increments of row p-3
            if (it >= 5 && outc) {
                const F2 f1p1 = lds2(xFp, (t + 1) * 8), f1 = lds2(xFp, t * 8);
                const F2 f1m1 = lds2(xFp, (t - 1) * 8), f1m2 = lds2(xFp, (t - 2) * 8);
                const F2 f3m1 = lds2(xFp, (NT + t - 1) * 8), f3 = lds2(xFp, (NT + t) * 8);
                const F2 f3p1 = lds2(xFp, (NT + t + 1) * 8), f3p2 = lds2(xFp, (NT + t + 2) * 8);
                XF[s3][0] = stream2<true>(zero, f1p1, f1, f1m1, f1m2, xadj_p, wxd.w1, wxd.w0, wxd.w2);
                XF[s3][1] = stream2<true>(zero, f3m1, f3, f3p1, f3p2, xadj_m, wxd.w1, wxd.w0, wxd.w2);
            }
            // ---------------------------------------------- S3
            if (calc) {
                // pass 1, x part of row p
                F2 hF = zero;
                if (FORCE != FORCE_NONE && p_in) hF = force_h(it, pair_of(a.phw));
                D013[k][0] = D013[k][0] + hF;
                D013[k][1] = stream2<true>(own1 + hF, lds2(xB, (t + 1) * 8), own1, lds2(xB, (t - 1) * 8),
                                           lds2(xB, (t - 2) * 8), xadj_p, wxh.w1, wxh.w0, wxh.w2);
                D013[k][2] = stream2<true>(own3 + hF, lds2(xB, (NT + t - 1) * 8), own3, lds2(xB, (NT + t + 1) * 8),
                                           lds2(xB, (NT + t + 2) * 8), xadj_m, wxh.w1, wxh.w0, wxh.w2);
                const int q = before(rp, 2);
                if (it >= 4 && (!ywall || (q >= 0 && q < a.ny))) {
                    if (ywall && q == a.ny - 1) {
                        // north wall row: pops 2, 4 of its NEE value were formed with row ny-2
                        FY[s2][0] = lds2(nrow, t * 8);
                        FY[s2][1] = lds2(nrow, (NT + t) * 8);
                    } else if (!(ywall && q == 0)) {
                        F2 hFq = zero;
                        if (FORCE != FORCE_NONE) hFq = force_h(it - 2, pair_of(a.phw));
                        W3 wy;
                        if (MK == METRIC_UNIFORM) wy = {pair_of(a.pwyh[0]), pair_of(a.pwyh[1]), pair_of(a.pwyh[2])};
                        else wy = weights(a.kyv[q], a.h, a);
                        const bool yadj_p = ywall && q == 1, yadj_m = ywall && q == a.ny - 2;
                        F2 fb[5];
                        fb[0] = D013[s2][0];
                        fb[1] = D013[s2][1];
                        fb[3] = D013[s2][2];
                        fb[2] = stream2<true>(BY[s2][0] + hFq, BY[s1][0], BY[s2][0], BY[s3][0], BY[s4][0], yadj_p,
                                              wy.w1, wy.w0, wy.w2);
                        fb[4] = stream2<true>(BY[s2][1] + hFq, BY[s3][1], BY[s2][1], BY[s1][1], BY[k][1], yadj_m,
                                              wy.w1, wy.w0, wy.w2);
                        // Step 3: f = feq + (I + h/2 Lt)^-1 (fbar - feq)
                        F2 mKk = pair_of(a.pmKk), Dk = pair_of(a.pDk);
                        if (PL) {
                            mKk = splat(-(1.0f - RK[s2][0]));
                            Dk = splat(0.5f * (RK[s2][1] - RK[s2][0]));
                        }
                        const Mom2 m = (FORCE == FORCE_ANY && a.r_mode && col_in) ? moments2r(fb, c, a.rk_bar * source_at(a, q, X))
                                                            : moments2(fb, c);
                        F2 n[5], f[5];
                        noneq2(fb, m, inv2c, n);
                        relax2(fb, n, n[1] - n[3], n[2] - n[4], mKk, Dk, f);
                        sts2(xF, t * 8, f[1]);
                        sts2(xF, (NT + t) * 8, f[3]);
                        FY[s2][0] = f[2];
                        FY[s2][1] = f[4];
                        F2 w[5];
                        if (xadj_p) {  // west wall column of this row: pops 1, 3 for the x stencils
                            nee2(f, a.uw[0], a.vw[0], inv2c, w);
                            sts2(xF, (t - 1) * 8, w[1]);
                            sts2(xF, (NT + t - 1) * 8, w[3]);
                        }
                        if (xadj_m) {
                            nee2(f, a.uw[1], a.vw[1], inv2c, w);
                            sts2(xF, (t + 1) * 8, w[1]);
                            sts2(xF, (NT + t + 1) * 8, w[3]);
                        }
                        if (yadj_p) {  // south wall row (slot of row q - 1): pops 2, 4 for the y stencils
                            nee2(f, a.uw[2], a.vw[2], inv2c, w);
                            FY[s3][0] = w[2];
                            FY[s3][1] = w[4];
                        }
                        if (yadj_m) {  // north wall row, taken up next iteration
                            nee2(f, a.uw[3], a.vw[3], inv2c, w);
                            sts2(nrow, t * 8, w[2]);
                            sts2(nrow, (NT + t) * 8, w[4]);
                        }
                    }
                }
            }
        }
        rp = after(rp);
        return true;
    };
    using std::integral_constant;
    for (int it0 = 0; it0 < nIt && !aborted; it0 += 5) {
        if (!row(it0, integral_constant<int, 0>{}, 0)) { aborted = true; break; }
        if (it0 + 1 >= nIt) break;
        if (!row(it0 + 1, integral_constant<int, 1>{}, 1)) { aborted = true; break; }
        if (it0 + 2 >= nIt) break;
        if (!row(it0 + 2, integral_constant<int, 2>{}, 2)) { aborted = true; break; }
        if (it0 + 3 >= nIt) break;
        if (!row(it0 + 3, integral_constant<int, 3>{}, 3)) { aborted = true; break; }
        if (it0 + 4 >= nIt) break;
        if (!row(it0 + 4, integral_constant<int, 4>{}, 4)) { aborted = true; break; }
    }
    if (FORCE == FORCE_ANY) cp_async_wait<0>();
    if (aborted && t == 0) {
        for (int it = issued - SLOTS; it < issued; ++it) {
            if (it < 0) continue;
            mbar_wait_bounded(&mbar[it % SLOTS], (uint32_t)((it / SLOTS) & 1));
        }
        atomicCAS(a.err, DEVERR_NONE, DEVERR_TMA_TIMEOUT);
    }
}

// Resident blocks the register budget is sized for: march_walls 5 x 96 threads
// (it takes up to 128 registers; power law on stretched grids spills 8 to 36
// bytes), march_window 3 x 128 (up to 166) or 2 x 256 (128, spilling 16 to 112
// bytes except in the plainest forms, and still the faster of the two where its
// bands fit the grid better: 1200 x 700 power-law cavity 41.8 us a step against 46.8).
constexpr int kWallsBatchBlocks = 5;
template <int NT>
constexpr int walls_min_blocks() {
    return NT <= 128 ? 3 : 2;
}

template <int NT, int MK, bool PL, int FORCE>
__global__ void __launch_bounds__(NT, walls_min_blocks<NT>())
    walls_kernel(const __grid_constant__ CUtensorMap tmap, const StepArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ volatile int s_abort[2];
    march_window<NT, MK, PL, FORCE>(&tmap, a, blockIdx.x, blockIdx.y, smem, s_abort);
}

// Persistent batch form (each_item).
// FORCED if any problem of the batch has a force, force rate or source;
// ROLL selects the rolled march, ST the storage mode (see march_walls).
template <int NT, int MK, bool PL, bool FORCED, bool ROLL, int ST>
__global__ void __launch_bounds__(NT, kWallsBatchBlocks)
    walls_batch_kernel(const BatchItem *__restrict__ items, int nitems, int *queue, const StepArgs *__restrict__ args,
                       const CUtensorMap *__restrict__ maps) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ volatile int s_abort[2];
    each_item(items, nitems, queue, [&](const BatchItem &item) {
        march_walls<NT, MK, PL, FORCED, ROLL, ST>(&maps[item.problem], args[item.problem], item.bx, item.by, smem,
                                                  s_abort);
        return !(s_abort[0] || s_abort[1]);
    });
}

template <int NT, int MK, bool PL, int FORCE>
cudaError_t launch_t(const CUtensorMap *tmap, const StepArgs &args, const StepPlan &plan, cudaStream_t stream) {
    auto k = walls_kernel<NT, MK, PL, FORCE>;
    constexpr int smem = walls_smem<NT, FORCE == FORCE_ANY>();
    static std::atomic<unsigned long long> configured{0};  // devices set up
    if (needs_device_setup(configured)) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        mark_device_setup(configured);
    }
    k<<<dim3(plan.gx, plan.gy), NT, smem, stream>>>(*tmap, args);
    return cudaGetLastError();
}

template <int NT, int MK, bool PL>
cudaError_t occupancy_t(int *occ, int *smem) {
    // the variant with force fields holds force rows as well: report the largest
    // shared memory and the smallest occupancy of the three
    *occ = 1 << 30;
    *smem = 0;
    const auto variant = [&](auto k, int bytes) {
        int o = 0;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k, NT, bytes);
        *occ = std::min(*occ, o);
        *smem = std::max(*smem, bytes);
        return e;
    };
    cudaError_t e = variant(walls_kernel<NT, MK, PL, FORCE_NONE>, walls_smem<NT, false>());
    if (e == cudaSuccess) e = variant(walls_kernel<NT, MK, PL, FORCE_CONST>, walls_smem<NT, false>());
    if (e == cudaSuccess) e = variant(walls_kernel<NT, MK, PL, FORCE_ANY>, walls_smem<NT, true>());
    return e;
}

template <int NT, int MK, bool PL, bool FORCED, bool ROLL, int ST>
cudaError_t batch_launch_ft(const BatchItem *items, int nitems, int *queue, const StepArgs *args, const CUtensorMap *maps,
                            int grid, cudaStream_t stream) {
    auto k = walls_batch_kernel<NT, MK, PL, FORCED, ROLL, ST>;
    constexpr int smem = walls_smem<NT, FORCED, ST>();
    static std::atomic<unsigned long long> configured{0};  // devices set up
    if (needs_device_setup(configured)) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        mark_device_setup(configured);
    }
    k<<<grid, NT, smem, stream>>>(items, nitems, queue, args, maps);
    return cudaGetLastError();
}

// The batch kernels of one storage mode: both march forms with FP32
// storage, the rolled form only with 16-bit storage (the form a full GPU
// keeps; small 16-bit batches have the tile kernel beside it).
template <int ST>
constexpr bool walls_unrolled_batch() {
    return ST == STORAGE_FP32;
}

template <int NT, int MK, bool PL, int ST>
cudaError_t batch_launch_t(const BatchItem *items, int nitems, int *queue, const StepArgs *args, const CUtensorMap *maps, int grid,
                           int forced, int roll, cudaStream_t stream) {
    if constexpr (walls_unrolled_batch<ST>()) {
        if (!roll) {
            if (forced) return batch_launch_ft<NT, MK, PL, true, false, ST>(items, nitems, queue, args, maps, grid, stream);
            return batch_launch_ft<NT, MK, PL, false, false, ST>(items, nitems, queue, args, maps, grid, stream);
        }
    } else {
        if (!roll) return cudaErrorInvalidConfiguration;
    }
    if (forced) return batch_launch_ft<NT, MK, PL, true, true, ST>(items, nitems, queue, args, maps, grid, stream);
    return batch_launch_ft<NT, MK, PL, false, true, ST>(items, nitems, queue, args, maps, grid, stream);
}

// Occupancy of one batch kernel variant.
template <int NT, int MK, bool PL, bool FORCED, bool ROLL, int ST>
cudaError_t batch_occupancy_v(int *occ) {
    auto k = walls_batch_kernel<NT, MK, PL, FORCED, ROLL, ST>;
    constexpr int smem = walls_smem<NT, FORCED, ST>();
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, NT, smem);
    return e;
}

template <int NT, int MK, bool PL, int ST>
cudaError_t batch_occupancy_t(int *occ, int *smem) {
    // take the smallest occupancy of the variants, and the shared memory of
    // those with a force
    int o[4] = {1 << 30, 1 << 30, 1 << 30, 1 << 30};
    *smem = walls_smem<NT, true, ST>();
    cudaError_t e = batch_occupancy_v<NT, MK, PL, false, true, ST>(&o[0]);
    if (e == cudaSuccess) e = batch_occupancy_v<NT, MK, PL, true, true, ST>(&o[1]);
    if constexpr (walls_unrolled_batch<ST>()) {
        if (e == cudaSuccess) e = batch_occupancy_v<NT, MK, PL, false, false, ST>(&o[2]);
        if (e == cudaSuccess) e = batch_occupancy_v<NT, MK, PL, true, false, ST>(&o[3]);
    }
    *occ = std::min(std::min(o[0], o[1]), std::min(o[2], o[3]));
    return e;
}

#define MDF_WALLS_DISPATCH(NTV, FN, ...)                                             \
    switch ((metric == METRIC_SEPARABLE ? 2 : 0) + (power_law ? 1 : 0)) {            \
        case 0: return FN<NTV, METRIC_UNIFORM, false>(__VA_ARGS__);                   \
        case 1: return FN<NTV, METRIC_UNIFORM, true>(__VA_ARGS__);                    \
        case 2: return FN<NTV, METRIC_SEPARABLE, false>(__VA_ARGS__);                 \
        default: return FN<NTV, METRIC_SEPARABLE, true>(__VA_ARGS__);                 \
    }

#define MDF_WALLS_DISPATCH_ST(NTV, STV, FN, ...)                                     \
    switch ((metric == METRIC_SEPARABLE ? 2 : 0) + (power_law ? 1 : 0)) {            \
        case 0: return FN<NTV, METRIC_UNIFORM, false, STV>(__VA_ARGS__);              \
        case 1: return FN<NTV, METRIC_UNIFORM, true, STV>(__VA_ARGS__);               \
        case 2: return FN<NTV, METRIC_SEPARABLE, false, STV>(__VA_ARGS__);            \
        default: return FN<NTV, METRIC_SEPARABLE, true, STV>(__VA_ARGS__);            \
    }

template <int NT, int MK, bool PL>
cudaError_t launch_f(const CUtensorMap *tmap, const StepArgs &args, const StepPlan &plan, cudaStream_t stream) {
    switch (force_kind(args)) {
        case FORCE_NONE: return launch_t<NT, MK, PL, FORCE_NONE>(tmap, args, plan, stream);
        case FORCE_CONST: return launch_t<NT, MK, PL, FORCE_CONST>(tmap, args, plan, stream);
        default: return launch_t<NT, MK, PL, FORCE_ANY>(tmap, args, plan, stream);
    }
}

template <int NT>
cudaError_t launch_nt(const CUtensorMap *tmap, const StepArgs &args, int metric, const StepPlan &plan,
                      cudaStream_t stream) {
    const int power_law = args.power_law;
    MDF_WALLS_DISPATCH(NT, launch_f, tmap, args, plan, stream)
}

}  // namespace

// Batches use 96-thread blocks (strips of 88 columns): the 2^k + 1 node
// sides of a cavity sweep waste fewer thread columns than with 120-column
// strips (513 nodes: 6 x 96 = 576 threads against 5 x 128 = 640).
constexpr int kWallsBatchNT = 96;

}  // namespace mdf
