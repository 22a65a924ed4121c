// The FP64 EPR (Eq. IID7-IID11) and moment streaming (Eq. IIE3) in lattice form, for 1D and 2D
// cells with a row table.  GB300 issues one FP64 warp instruction per SM every 16 cycles, in which
// its four schedulers issue up to 64 FP32 or integer ones: the number of FP64 operations per cell
// is the time of the FP64 path, and everything else here is arranged around that count.
//   - The velocity set is swept from the lattice point nearest to u outwards, row by row, and
//     along a row outwards from its centre.  On the lattice the exponent is a polynomial in
//     integer offsets (k, j), so populations follow from multiplicative forward differences in
//     both directions: a row costs about a dozen products where seven exponentials stood, and the
//     error growth (~n^3/6 ulp over n steps) starts at the centre.
//   - The children of split points are a lattice of spacing 1/2 of their own, swept the same way.
//   - Hot cells (R_ac above kSweepR) start every row from its own exponentials instead, seven to ten
//     of them to 25 points and more, since ratios compounded over so many rows lose too much.
//   - A Newton pass sums only the residual's moments (degree <= 3 and <= 2) in FP64, as power sums
//     of the integer offsets (exact weights, made by integer operations) moved to thermal units
//     once per pass.  The Jacobian and the solve of an update are FP32, from the same populations:
//     an update only steers the iteration, whose FP64 residual is judged against the tolerance as
//     before, and an update with a Jacobian to 2^-24 leaves about 1e-5 of the residual, far below
//     what the quadratic step itself leaves until the residual is at rounding.
//   - The membership decisions come from the row table, taken once per cell.
// A solve that breaks down here is redone by the all-FP64 Newton (solve_fg), so what converges and
// what falls back is decided there.
// Against one exponential per row start and third ratio, FP64 moments to degree 6 and single shares of
// every child, a step of a 731 x 523 four-quadrant flow (RT 0.25-1.5) went from 30.3 to 8.3 ms, and its
// error against 64-bit arithmetic from 5.1e-16 to 4.1e-16.
#pragma once

#include <cstdint>

#include "lelbm_df.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// exp(x) in FP64 with integer instructions: Tang's table-driven method (ACM TOMS 15, 1989) in 64-bit
// fixed point.  x log2(e) = n + j / 512 + rho, 2^(j/512) from a table, 2^rho from five Taylor terms.
// Every step carries at least 59 bits, so the result is rounded once (0.62 ulp at most).  About 70
// integer instructions, some 20 issue cycles of an SM, where the library's exp takes about 17 FP64
// instructions, 16 cycles each.
// ---------------------------------------------------------------------------
// 2^(w 2^-55) = P 2^(n - 62), P in [2^62, 2^63].
__device__ __forceinline__ unsigned long long exp2_q62(long long w, int& n) {
    const int hi = (int)(w >> 32);
    n = hi >> 23;
    const unsigned long long T = __ldg(&c_exp2.t[(hi >> 14) & 511]);
    const unsigned long long L = __umul64hi((unsigned long long)w << 18, 0xB17217F7D1CF79ACull);  // 512 rho ln 2
    const unsigned l = (unsigned)(L >> 32);
    const unsigned long long q2 = __umul64hi(L, L);
    const unsigned q3 = __umulhi((unsigned)(q2 >> 32), l), q4 = __umulhi(q3, l), q5 = __umulhi(q4, l);
    // rho ln 2 = L / 512: the terms L/2^9, L^2/2^19, L^3/(6 2^27), L^4/(24 2^36) and (to a few per cent)
    // L^5/(120 2^45), with 64 fractional bits
    const unsigned long long e = (L >> 9) + (q2 >> 19) + ((unsigned long long)__umulhi(q3, 0xAAAAAAABu) << 3) +
                                 (__umulhi(q4, 0xAAAAAAABu) >> 8) + (q5 >> 20);
    return T + __umul64hi(T, e);
}

__device__ __forceinline__ double exp_int(double x) {
    const int xh = __double2hiint(x);
    const int ex = (xh >> 20) & 0x7ff;
    if (ex >= 1023 + 7) return exp(x);  // |x| >= 128, infinite or NaN
    // |x| log2(e) with 55 fractional bits
    const unsigned long long m =
        ((unsigned long long)((xh & 0xfffff) | (ex ? 0x100000 : 0)) << 43) | ((unsigned long long)(unsigned)__double2loint(x) << 11);
    const unsigned long long p = __umul64hi(m, 0xB8AA3B295C17F0BCull);  // mantissa x log2(e) / 2, 63 bits below the point
    const int sh = 1023 + 7 - ex;                                       // >= 1: p holds |x| log2(e) 2^(62 - (ex - 1023))
    unsigned long long w = sh < 64 ? (((p >> (sh - 1)) + 1) >> 1) : 0ull;
    const long long ws = xh < 0 ? -(long long)w : (long long)w;
    int n;
    const unsigned long long P = exp2_q62(ws, n) + 512;  // round to 53 bits
    // P = 2^62 + ...: adding it above the exponent field carries its leading one into the exponent
    return __longlong_as_double((long long)(P >> 10) + ((long long)(n + 1022) << 52));
}

// Coefficients d[ix(a, b)] of k^a j^b in the exponent 1 + sum_j lam_j T_j at the thermal points
// (x0 + k h, y0 + j h).
template <int D, bool FLUON>
__device__ __forceinline__ void lattice_poly(const double* lam, double x0, double y0, double h, double* d) {
    using Q = DFPop<D, FLUON>;
    constexpr int P = Q::P;
#pragma unroll
    for (int j = 0; j < Q::N; j++) d[Q::ix(bx<D, FLUON>(j), by<D, FLUON>(j))] = lam[j];
    d[0] += 1.0;
#pragma unroll
    for (int b = 0; b <= (D == 2 ? P : 0); b++) {
        const int n = P - b;
#pragma unroll
        for (int k = 0; k < P; k++)
#pragma unroll
            for (int i = P - 1; i >= 0; i--)
                if (k < n && i >= k && i < n) d[Q::ix(i, b)] = fma(x0, d[Q::ix(i + 1, b)], d[Q::ix(i, b)]);
    }
    if constexpr (D == 2) {
#pragma unroll
        for (int a = 0; a <= P; a++) {
            const int n = P - a;
#pragma unroll
            for (int k = 0; k < P; k++)
#pragma unroll
                for (int i = P - 1; i >= 0; i--)
                    if (k < n && i >= k && i < n) d[Q::ix(a, i)] = fma(y0, d[Q::ix(a, i + 1)], d[Q::ix(a, i)]);
        }
    }
    double hp[P + 1];
    hp[0] = 1.0;
#pragma unroll
    for (int k = 1; k <= P; k++) hp[k] = hp[k - 1] * h;
#pragma unroll
    for (int b = 0; b <= (D == 2 ? P : 0); b++)
#pragma unroll
        for (int a = 0; a + b <= P; a++)
            if (a + b > 0) d[Q::ix(a, b)] *= hp[a + b];
}

// Ratios of neighbouring populations at an anchor, from the exponent polynomial p (lattice_poly).
// Second and third ratios compound over a sweep, so they are exponentials of their own where a long
// row needs it (along x) and products of at most two factors elsewhere.
template <int D, bool FLUON>
struct SweepFactors {
    double e0, r, l, r2, r3, l3;            // population, ratios to k = +1 and -1, second and third ratios
    double el, l2;                          // 1D, apart: population at k = -1 and second ratio there (l from there)
    double u, ud, u2, u2d, u3, u3d;         // ratios of e0 to the rows j = +1 and -1, second, third
    double m11, i11, m12, i12, m21, i21;    // exp(-+p_11), exp(-+p_12), exp(-+p_21)

    // apart (1D): the left side starts from exponentials of its own, at k = -1
    __device__ __forceinline__ void init(const double* p, double wgt, bool apart) {
        using Q = DFPop<D, FLUON>;
        constexpr int NE = FLUON ? (D == 1 ? 6 : 17) : (D == 1 ? 4 : 9);
        double a[NE];
        const double p10 = p[Q::ix(1, 0)], p20 = p[Q::ix(2, 0)];
        const double p30 = FLUON ? p[FLUON ? Q::ix(3, 0) : 0] : 0.0;
        a[0] = p[0];
        a[1] = p10 + p20 + p30;
        a[2] = D == 1 && apart ? 3.0 * p20 - p10 - 7.0 * p30 : p20 - p10 - p30;
        a[3] = 2.0 * p20 + 6.0 * p30;
        if constexpr (FLUON) {
            a[4] = 6.0 * p30;
            a[5] = -a[4];
        }
        if constexpr (D == 2) {
            constexpr int o = FLUON ? 6 : 4;
            const double p01 = p[Q::ix(0, 1)], p02 = p[Q::ix(0, 2)];
            const double p03 = FLUON ? p[FLUON ? Q::ix(0, 3) : 0] : 0.0;
            a[o] = p01 + p02 + p03;
            a[o + 1] = p02 - p01 - p03;
            a[o + 2] = 2.0 * p02 + 6.0 * p03;
            a[o + 3] = p[Q::ix(1, 1)];
            a[o + 4] = -a[o + 3];
            if constexpr (FLUON) {
                a[11] = 6.0 * p03;
                a[12] = -a[11];
                a[13] = p[Q::ix(1, 2)];
                a[14] = -a[13];
                a[15] = p[Q::ix(2, 1)];
                a[16] = -a[15];
            }
        }
        // one code site in 2D (inlined copies would crowd the instruction caches); side by side in 1D, where a
        // small batch waits for this chain
#pragma unroll(D == 1 ? NE : 1)
        for (int k = 0; k < NE; k++) a[k] = exp_int(-a[k]);
        e0 = wgt * a[0];
        r = a[1];
        l = a[2];
        r2 = a[3];
        if constexpr (FLUON) {
            r3 = a[4];
            l3 = a[5];
        }
        if (D == 1 && apart) {
            el = wgt * exp_int(p10 - p20 + p30 - p[0]);
            if constexpr (FLUON) l2 = exp_int(12.0 * p30 - 2.0 * p20);
        }
        if constexpr (D == 2) {
            constexpr int o = FLUON ? 6 : 4;
            u = a[o];
            ud = a[o + 1];
            u2 = a[o + 2];
            m11 = a[o + 3];
            i11 = a[o + 4];
            if constexpr (FLUON) {
                u3 = a[11];
                u3d = a[12];
                u2d = u2 * (u3d * u3d);
                m12 = a[13];
                i12 = a[14];
                m21 = a[15];
                i21 = a[16];
            }
        }
    }
};

// The row state of one population and its advance to the next row (up or down).
template <int D, bool FLUON>
struct SweepRows {
    double E, R, L, R2;            // at k = 0 of the row: population, ratios to the right and left, second ratio
    double U, U2, U3, V, VL, W, V2, V2L;

    __device__ __forceinline__ void start(const SweepFactors<D, FLUON>& f, bool down) {
        E = f.e0;
        R = f.r;
        L = f.l;
        R2 = f.r2;
        if constexpr (D == 2) {
            U = down ? f.ud : f.u;
            U2 = FLUON && down ? f.u2d : f.u2;
            V = down ? f.i11 : f.m11;
            VL = down ? f.m11 : f.i11;
            if constexpr (FLUON) {
                const double a21 = down ? f.i21 : f.m21;
                U3 = down ? f.u3d : f.u3;
                V *= f.m12 * a21;
                VL *= f.i12 * a21;
                V2 = f.m12 * f.m12;
                V2L = f.i12 * f.i12;
                W = a21 * a21;
            }
        }
    }
    __device__ __forceinline__ void advance() {
        if constexpr (D == 2) {
            E *= U;
            U *= U2;
            R *= V;
            L *= VL;
            if constexpr (FLUON) {
                U2 *= U3;
                V *= V2;
                VL *= V2L;
                R2 *= W;
            }
        }
    }
};

// Rows that one anchor serves on each side: a new anchor every 2 kAnchorRows + 1 rows bounds the
// compounded rounding of tall sets; up to R_ac = 7 (RT = 3.5 at n = 4) one anchor serves all.
constexpr int kAnchorRows = 8;

// Acoustic radius up to which 2D sweeps compound along y too.  The mean error of a population (weighted by
// it, against 64 bits; the general stencil, whose rows each start afresh, in brackets): RT 0.6 1.6e-16
// (1.3e-15), RT 9.4 1.3e-15 (1.5e-15), but with sweeps RT 10 1.3e-15 (1.0e-15), RT 16 2.2e-15 (6.6e-16)
// and RT 32 5.0e-15 (1.0e-15).  Beyond, rows that start afresh in the lattice form: RT 10 4.9e-16, RT 16
// 6.2e-16, RT 32 1.0e-15.  Time of a step: 128^2 at RT 16 4.8 -> 5.5 ms (13.1 on the general stencil),
// 64^2 at RT 32 8.2 -> 7.7 ms (17.6).
constexpr int kSweepR = 12;

// In 1D the left side of a row longer than this starts from exponentials of its own: RT 16 4.4e-16 (4.8e-16),
// RT 150 9.4e-15 (9.4e-15), where from the centre's it lost a third more.  On every row they would cost
// a 400-cell tube 6 % (the chain of a cell is what its step waits for).
constexpr int kSweepLeft = 11;

// The populations of one side of a row, from its point at thermal x outwards in steps of h (signed): with its
// own exponentials, but for the last ratio, which is the same on every row.
struct SideF {
    double e, r, r2;
    __device__ __forceinline__ void start(const double* c, double x, double h, double w) {
        const double h2 = h * h, c3 = 3.0 * c[3] * x;
        e = w * exp_int(-(((c[3] * x + c[2]) * x + c[1]) * x + c[0]));
        r = exp_int(-(h * fma(x, fma(2.0, c[2], c3), c[1]) + h2 * (c[2] + c3 + c[3] * h)));
        r2 = exp_int(-2.0 * h2 * (c[2] + c3 + 3.0 * c[3] * h));
    }
};
struct SideG {
    double e, r;
    __device__ __forceinline__ void start(const double* c, double x, double h, double w) {
        e = w * exp_int(-((c[2] * x + c[1]) * x + c[0]));
        r = exp_int(-h * (c[1] + c[2] * (2.0 * x + h)));
    }
};

// Visits the lattice points (x0 + k h, y0 + j h) of rows jlo..jhi: ext(j, i0, i1, h0, h1) gives a
// row's points i0..i1 without the hole h0..h1 (empty: h0 = 1, h1 = 0); point(k, j, f, g) gets every
// point with its populations (weights wf, wg included), row_end(j) follows a row that is not empty.
// FRESH: every row starts from exponentials of its own, on both sides of its centre.
template <int D, bool FRESH, class Ext, class Pt, class RowEnd>
__device__ __forceinline__ void lattice_sweep(const double* lf, const double* lg, bool doF, bool doG, double x0,
                                              double y0, double h, double wf, double wg, int jlo, int jhi,
                                              const Ext& ext, Pt& point, RowEnd& row_end) {
    if constexpr (FRESH) {
        const double h3 = 6.0 * (h * h) * h;
        const double r3 = doF ? exp_int(-h3 * lf[D == 1 ? 3 : 6]) : 0.0, l3 = doF ? exp_int(h3 * lf[D == 1 ? 3 : 6]) : 0.0;
        const double r2g = doG ? exp_int(-2.0 * (h * h) * lg[D == 1 ? 2 : 3]) : 0.0;
#pragma unroll 1
        for (int j = jlo; j <= jhi; j++) {
            int i0, i1, h0, h1;
            ext(j, i0, i1, h0, h1);
            if (i0 > i1) continue;
            double cf[4], cg[3];
            row_coeffs<D>(lf, lg, fma(widen((float)j), h, y0), cf, cg);
#pragma unroll 1
            for (int left = 0; left < 2; left++) {
                const int n = left ? -i0 : i1;
                if (n < left) continue;
                const double x = left ? x0 - h : x0, hs = left ? -h : h, t3 = left ? l3 : r3;
                SideF f{0.0, 0.0, 0.0};
                SideG g{0.0, 0.0};
                if (doF) f.start(cf, x, hs, wf);
                if (doG) g.start(cg, x, hs, wg);
#pragma unroll 1
                for (int i = left; i <= n; i++) {
                    const int k = left ? -i : i;
                    if (k >= i0 && k <= i1 && (k < h0 || k > h1)) point(k, j, f.e, g.e);
                    f.e *= f.r;
                    f.r *= f.r2;
                    f.r2 *= t3;
                    g.e *= g.r;
                    g.r *= r2g;
                }
            }
            row_end(j);
        }
        return;
    }
    bool apart = false;
    if constexpr (D == 1) {
        int i0, i1, h0, h1;
        ext(0, i0, i1, h0, h1);
        apart = i0 < -kSweepLeft;
    }
    int ja = 0;
    while (ja - kAnchorRows > jlo) ja -= 2 * kAnchorRows + 1;
#pragma unroll 1
    for (; ja - kAnchorRows <= jhi; ja += 2 * kAnchorRows + 1) {
        SweepFactors<D, true> ff;
        SweepFactors<D, false> fg;
        if (doF) {
            double p[DFPop<D, true>::NB];
            lattice_poly<D, true>(lf, x0, fma(widen((float)ja), h, y0), h, p);
            ff.init(p, wf, apart);
        }
        if (doG) {
            double p[DFPop<D, false>::NB];
            lattice_poly<D, false>(lg, x0, fma(widen((float)ja), h, y0), h, p);
            fg.init(p, wg, apart);
        }
        const double l3sq = doF ? ff.l3 * ff.l3 : 0.0;
#pragma unroll 1
        for (int down = 0; down < (D == 2 ? 2 : 1); down++) {
            SweepRows<D, true> sf;
            SweepRows<D, false> sg;
            if (doF) sf.start(ff, down);
            if (doG) sg.start(fg, down);
            const int step = down ? -1 : 1;
            const int j_end = down ? max(jlo, ja - kAnchorRows) : min(jhi, ja + kAnchorRows);
#pragma unroll 1
            for (int j = ja; step * (j_end - j) >= 0; j += step) {
                int i0 = 0, i1 = -1, h0, h1;
                if (j >= jlo && j <= jhi && !(down && j == ja)) ext(j, i0, i1, h0, h1);
                if (i0 <= i1) {
#pragma unroll 1
                    for (int left = 0; left < 2; left++) {
                        double e = 0.0, r = 0.0, r2 = 0.0, r3 = 0.0, eg = 0.0, rg = 0.0;
                        if (doF) {
                            e = apart && left ? ff.el : sf.E;
                            r = left ? sf.L : sf.R;
                            r2 = !left ? sf.R2 : (apart ? ff.l2 : sf.R2 * l3sq);
                            r3 = left ? ff.l3 : ff.r3;
                        }
                        if (doG) {
                            eg = apart && left ? fg.el : sg.E;
                            rg = left ? sg.L : sg.R;
                        }
                        const int n = left ? -i0 : i1;
#pragma unroll 1
                        for (int i = apart ? left : 0; i <= n; i++) {
                            const int k = left ? -i : i;
                            if (!(left && i == 0) && k >= i0 && k <= i1 && (k < h0 || k > h1)) point(k, j, e, eg);
                            if (doF) {
                                e *= r;
                                r *= r2;
                                r2 *= r3;
                            }
                            if (doG) {
                                eg *= rg;
                                rg *= fg.r2;
                            }
                        }
                    }
                    row_end(j);
                }
                if (doF) sf.advance();
                if (doG) sg.advance();
            }
        }
    }
}

// The one or two lattices of a cell's velocity set: lattice 0 holds the level-0 points (spacing 1,
// anchored at the integer velocity nearest to u), lattice 1 the children of split points (spacing
// 1/2, anchored a quarter cell below it).
template <int D>
struct CellLattice {
    int xn, yn;      // anchor of lattice 0
    int n;           // lattices in use
    double fx, fy;   // u - (xn, yn)

    __device__ __forceinline__ void init(const CellState<D>& c, const RowTable<D>& tab) {
        fx = c.u[0] - (double)tab.xc;
        xn = tab.xc + (fx > 0.5 ? 1 : 0);
        fx = c.u[0] - (double)xn;
        fy = 0.0;
        yn = 0;
        if constexpr (D == 2) {
            fy = c.u[1] - (double)tab.yc;
            yn = tab.yc + (fy > 0.5 ? 1 : 0);
            fy = c.u[1] - (double)yn;
        }
        n = (D == 2 ? tab.band_n > 0 : tab.a <= tab.b) ? 2 : 1;
    }
    // rows of lattice `child`
    __device__ __forceinline__ void rows(const RowTable<D>& tab, bool child, int& jlo, int& jhi) const {
        jlo = jhi = 0;
        if constexpr (D == 2) {
            jlo = tab.y_first - yn;
            jhi = jlo + tab.nrows - 1;
            if (child) {
                jlo = 2 * (jlo + tab.band_first);
                jhi = jlo + 2 * tab.band_n - 1;
            }
        }
    }
    __device__ __forceinline__ void ext(const RowTable<D>& tab, bool child, int j, int& i0, int& i1, int& h0,
                                        int& h1) const {
        int x0, x1, a, b;
        if constexpr (D == 2) {
            tab.row_ext(yn + (child ? j >> 1 : j) - tab.y_first, x0, x1, a, b);
        } else {
            x0 = tab.x0;
            x1 = tab.x1;
            a = tab.a;
            b = tab.b;
        }
        if (child) {
            i0 = 2 * (a - xn);
            i1 = 2 * (b - xn) + 1;
            h0 = 1;
            h1 = 0;
            if (a > b) i1 = i0 - 1;
        } else {
            i0 = x0 - xn;
            i1 = x1 - xn;
            h0 = a - xn;
            h1 = b - xn;
            if (a > b) {
                h0 = 1;
                h1 = 0;
            }
        }
    }
};

// Power sums L[ix(a, b)] = sum k^a j^b f of a lattice (spacing hs in thermal units, u at (fx, fy) in
// its units) -> the moments sum x^a y^b f in thermal units about u, added to T.
template <int D, bool FLUON>
__device__ __forceinline__ void add_thermal(const double* Ls, double fx, double fy, double hs, double* T) {
    using Q = DFPop<D, FLUON>;
    constexpr int P = Q::P;
    double sp[P + 1];
    sp[0] = 1.0;
#pragma unroll
    for (int k = 1; k <= P; k++) sp[k] = sp[k - 1] * hs;
    double K[Q::NB];
#pragma unroll
    for (int k = 0; k < Q::NB; k++) K[k] = Ls[k];
    moments_about<D, P>(K, fx, fy);
#pragma unroll
    for (int b = 0; b <= (D == 2 ? P : 0); b++)
#pragma unroll
        for (int a = 0; a + b <= P; a++)
            T[Q::ix(a, b)] = a + b > 0 ? fma(K[Q::ix(a, b)], sp[a + b], T[Q::ix(a, b)]) : T[Q::ix(a, b)] + K[Q::ix(a, b)];
}

// One pass over the velocity set: the thermal moments of degree <= 3 of f (if doF) and <= 2 of g
// (if doG) in FP64 (TF, TG) and the Jacobian's moments in FP32 (MF, MG).  Returns the point count.
template <int D, bool FRESH>
__device__ __forceinline__ unsigned int moment_pass64(const CellState<D>& c, const RowTable<D>& tab,
                                                      const CellLattice<D>& lat, const double* lf, const double* lg,
                                                      bool doF, bool doG, double* TF, double* TG, float* MF,
                                                      float* MG) {
    using MS = MomentSet<D>;
    using QF = DFPop<D, true>;
    using QG = DFPop<D, false>;
#pragma unroll
    for (int i = 0; i < QF::NB; i++) TF[i] = 0.0;
#pragma unroll
    for (int i = 0; i < QG::NB; i++) TG[i] = 0.0;
#pragma unroll
    for (int i = 0; i < MS::NF; i++) MF[i] = 0.f;
#pragma unroll
    for (int i = 0; i < MS::NG; i++) MG[i] = 0.f;
    unsigned int q = 0;
#pragma unroll 1
    for (int l = 0; l < lat.n; l++) {
        const bool child = l == 1;
        const double hs = child ? 0.5 * c.inv_sig : c.inv_sig;
        const double ox = child ? 2.0 * lat.fx + 0.5 : lat.fx;  // u from the anchor, in spacings
        const double oy = child ? 2.0 * lat.fy + 0.5 : lat.fy;
        const float h32 = (float)hs, x32 = (float)(-ox * hs), y32 = (float)(-oy * hs);
        const double w = child ? (D == 2 ? 0.25 : 0.5) : 1.0;
        double LF[QF::NB], LG[QG::NB], S[4], G[3];
        float SF[MS::PF + 1], SG[MS::PG + 1];
#pragma unroll
        for (int i = 0; i < QF::NB; i++) LF[i] = 0.0;
#pragma unroll
        for (int i = 0; i < QG::NB; i++) LG[i] = 0.0;
        auto clear = [&]() {
#pragma unroll
            for (int a = 0; a < 4; a++) S[a] = 0.0;
#pragma unroll
            for (int a = 0; a < 3; a++) G[a] = 0.0;
#pragma unroll
            for (int a = 0; a <= MS::PF; a++) SF[a] = 0.f;
#pragma unroll
            for (int a = 0; a <= MS::PG; a++) SG[a] = 0.f;
        };
        clear();
        auto point = [&](int k, int, double f, double g) {
            q++;
            const float kf = (float)k;  // k^2 and k^3 exact in FP32 up to |k| = 256
            const double k1 = widen(kf), k2 = widen(kf * kf);
            const float x = fmaf(kf, h32, x32);
            const float x2 = x * x, x3 = x2 * x, x4 = x2 * x2;
            const float pw[7] = {1.f, x, x2, x3, x4, x4 * x, x3 * x3};
            if (doF) {
                const double k3 = widen(kf * kf * kf);
                S[0] += f;
                S[1] = fma(k1, f, S[1]);
                S[2] = fma(k2, f, S[2]);
                S[3] = fma(k3, f, S[3]);
                const float ff = narrow(f);
#pragma unroll
                for (int a = 0; a <= MS::PF; a++) SF[a] = fmaf(pw[a], ff, SF[a]);
            }
            if (doG) {
                G[0] += g;
                G[1] = fma(k1, g, G[1]);
                G[2] = fma(k2, g, G[2]);
                const float gf = narrow(g);
#pragma unroll
                for (int a = 0; a <= MS::PG; a++) SG[a] = fmaf(pw[a], gf, SG[a]);
            }
        };
        auto row_end = [&](int j) {
            if constexpr (D == 1) {
#pragma unroll
                for (int a = 0; a < 4; a++) LF[a] = S[a];
#pragma unroll
                for (int a = 0; a < 3; a++) LG[a] = G[a];
#pragma unroll
                for (int a = 0; a <= MS::PF; a++) MF[a] += SF[a];
#pragma unroll
                for (int a = 0; a <= MS::PG; a++) MG[a] += SG[a];
            } else {
                const float jf = (float)j, y = fmaf(jf, h32, y32);
                const double jp[4] = {1.0, widen(jf), widen(jf * jf), widen(jf * jf * jf)};
                float yp[MS::PF + 1];
                yp[0] = 1.f;
#pragma unroll
                for (int k = 1; k <= MS::PF; k++) yp[k] = yp[k - 1] * y;
                if (doF) {
#pragma unroll
                    for (int b = 0; b <= 3; b++)
#pragma unroll
                        for (int a = 0; a + b <= 3; a++)
                            LF[QF::ix(a, b)] = b ? fma(jp[b], S[a], LF[QF::ix(a, b)]) : LF[QF::ix(a, b)] + S[a];
#pragma unroll
                    for (int b = 0; b <= MS::PF; b++)
#pragma unroll
                        for (int a = 0; a + b <= MS::PF; a++)
                            MF[tix(a, b, MS::PF)] = fmaf(SF[a], yp[b], MF[tix(a, b, MS::PF)]);
                }
                if (doG) {
#pragma unroll
                    for (int b = 0; b <= 2; b++)
#pragma unroll
                        for (int a = 0; a + b <= 2; a++)
                            LG[QG::ix(a, b)] = b ? fma(jp[b], G[a], LG[QG::ix(a, b)]) : LG[QG::ix(a, b)] + G[a];
#pragma unroll
                    for (int b = 0; b <= MS::PG; b++)
#pragma unroll
                        for (int a = 0; a + b <= MS::PG; a++)
                            MG[tix(a, b, MS::PG)] = fmaf(SG[a], yp[b], MG[tix(a, b, MS::PG)]);
                }
                clear();
            }
        };
        int jlo, jhi;
        lat.rows(tab, child, jlo, jhi);
        auto ext = [&](int j, int& i0, int& i1, int& h0, int& h1) { lat.ext(tab, child, j, i0, i1, h0, h1); };
        lattice_sweep<D, FRESH>(lf, lg, doF, doG, -ox * hs, -oy * hs, hs, w, w, jlo, jhi, ext, point, row_end);
        if (doF) add_thermal<D, true>(LF, ox, oy, hs, TF);
        if (doG) add_thermal<D, false>(LG, ox, oy, hs, TG);
    }
    return q;
}

// Newton update from the FP64 residual and the FP32 Jacobian of one pass (Eq. IID8-IID11).
// Returns as newton_step_tol.
template <int D, bool FLUON>
__device__ __forceinline__ int newton_step64(const double* T, const float* Mom, const double* con, double* lam,
                                             double tol, int max_iter, int it) {
    using Q = DFPop<D, FLUON>;
    constexpr int N = Q::N, PJ = Q::PJ;
    float x[N];
    long long worst = 0;
#pragma unroll
    for (int j = 0; j < N; j++) {
        const double r = T[Q::ix(bx<D, FLUON>(j), by<D, FLUON>(j))] - con[j];
        worst = max_abs_bits(r, worst);
        x[j] = narrow_signed(r);
    }
    if (worst >= kInfBits) return -1;
    const bool conv = worst <= __double_as_longlong(tol);
    if (!conv && it >= max_iter) return -2;
    float A[N * (N + 1) / 2];
#pragma unroll
    for (int i = 0; i < N; i++)
#pragma unroll
        for (int j = 0; j <= i; j++)
            A[tri(i, j)] = Mom[D == 1 ? bx<D, FLUON>(i) + bx<D, FLUON>(j)
                                      : tix(bx<D, FLUON>(i) + bx<D, FLUON>(j), by<D, FLUON>(i) + by<D, FLUON>(j), PJ)];
    if (!ldlt_solve<float, N>(A, x)) return -1;
    bool fin = true;
#pragma unroll
    for (int j = 0; j < N; j++) {
        fin = fin && isfinite(x[j]);
        lam[j] += widen(x[j]);
    }
    if (!fin) return -1;
    return conv ? 1 : 0;
}

// Joint Newton iterations of both populations as solve_fg, with lattice-form passes.
template <int D, bool FRESH = false>
__device__ __forceinline__ void solve_fg64(const CellState<D>& c, const RowTable<D>& tab, const CellLattice<D>& lat,
                                           const double* conF, const double* conG, bool has_g, double* lf, double* lg,
                                           const Model& m, int& sf, int& sg, unsigned int& npf, unsigned int& npg) {
    bool fa = true, ga = has_g;
    sf = 0;
    sg = 0;
#pragma unroll 1
    for (int it = 0; fa || ga; it++) {
        double TF[DFPop<D, true>::NB], TG[DFPop<D, false>::NB];
        float MF[MomentSet<D>::NF], MG[MomentSet<D>::NG];
        const unsigned int q = moment_pass64<D, FRESH>(c, tab, lat, lf, lg, fa, ga, TF, TG, MF, MG);
        if (ga) {
            npg += q;
            const int r = newton_step64<D, false>(TG, MG, conG, lg, m.tol, m.max_iter, it);
            sg = r < 0 ? r : sg + 1;
            ga = r == 0;
        }
        if (fa) {
            npf += q;
            const int r = newton_step64<D, true>(TF, MF, conF, lf, m.tol, m.max_iter, it);
            sf = r < 0 ? r : sf + 1;
            fa = r == 0;
        }
    }
}

}  // namespace lbm
