// Checks of the device headers' per-cell functions on the CPU (see cuda_host.h), for
// test_device_code.py.
#include "cuda_host.h"

#include <random>
#include <vector>

#include "lelbm_step.cuh"

using namespace lbm;
typedef long double real;

namespace {

constexpr int kGrid = 64;  // cells a side of the periodic grid that takes the deposits

struct Cell {
    Model m{};
    Geometry g{};
    CellState<2> c{};
    Stencil<2> st{};
    RowTable<2> tab{};
    CellLattice<2> lat{};
    char2 rows[kRowsMax];
    double conF[10], conG[6], lf[10], lg[6];  // constraints and the FP64 solution
    std::vector<uint8_t> type;
    std::vector<double> M;
    std::vector<float2> pop;
    std::vector<float2> etab;
    long long beta[10];

    Cell() : type(kGrid * kGrid, CELL_FLUID), M(11 * kGrid * kGrid), pop(kDfPopCap), etab(kExpTab) {
        m.K = 2.0;
        m.n_conf = 4.0;
        m.r_min = 2.0;
        m.refine_div = m.refine_rad = 3.0;
        m.max_refine = 4;
        m.Pr = 1.0;
        m.tol = 1e-12;
        m.max_iter = 60;
        set_derived_params(m, 2);
        g.D = 2;
        g.NX = g.NY = g.nx = g.ny = kGrid;
        g.ncell = kGrid * kGrid;
        g.periodic[0] = g.periodic[1] = 1;
        exp2_table_init(etab.data());
    }
    // a cell at temperature RT (about), with constraints off equilibrium by up to noneq; false
    // where the FP64 path has no lattice-form solution
    template <class Rng>
    bool draw(Rng& rng, double RT, double noneq, double umag) {
        std::uniform_real_distribution<double> U(-1.0, 1.0);
        c.rho = 1.0;
        c.RT = RT * (1.0 + 0.03 * U(rng));
        c.sig = std::sqrt(c.RT);
        c.inv_sig = 1.0 / c.sig;
        c.u[0] = umag * U(rng);
        c.u[1] = umag * U(rng);
        st.init(c, m);
        tab.build(c, st, rows);
        for (int j = 0; j < 10; j++) conF[j] = (j == 0 || j == 3 || j == 5) + (j > 2 ? noneq * U(rng) : 0.0);
        for (int j = 0; j < 6; j++) conG[j] = (j == 0 || j == 3 || j == 5) + (j > 0 ? noneq * U(rng) : 0.0);
        if (!tab.ok) return false;
        lat.init(c, tab);
        maxwell_start_fg<2, 10, 6>(c.RT, lf, lg);
        int sf, sg;
        unsigned pf = 0, pg = 0;
        solve_fg64<2>(c, tab, lat, conF, conG, true, lf, lg, m, sf, sg, pf, pg);
        return sf >= 0 && sg >= 0;
    }
    // puts the drawn cell into Min as moments, with the drawn non-equilibrium phonon constraints, and takes it
    // through the collision; false as draw
    bool collide_at(std::vector<double>& Min, long long cell) {
        double Me[11];
        eq_moments<2>(m.K, c.rho, c.u, c.RT, Me);
        Me[9] += c.rho * m.K * c.RT * c.sig * conG[1];
        Me[10] += c.rho * m.K * c.RT * c.sig * conG[2];
        for (int i = 0; i < 11; i++) Min[(size_t)i * kGrid * kGrid + cell] = Me[i];
        collide<2>(Me, m, c);
        if (!c.ok) return false;
        st.init(c, m);
        tab.build(c, st, rows);
        if (!tab.ok) return false;
        lat.init(c, tab);
        for (int j = 0; j < 10; j++) conF[j] = c.cf[j];
        for (int j = 0; j < 6; j++) conG[j] = c.cg[j];
        maxwell_start_fg<2, 10, 6>(c.RT, lf, lg);
        int sf, sg;
        unsigned pf = 0, pg = 0;
        solve_fg64<2>(c, tab, lat, conF, conG, true, lf, lg, m, sf, sg, pf, pg);
        return sf >= 0 && sg >= 0;
    }
    DFStream stream(double mass, int pop_cap) {
        DFStream ds{};
        ds.g = &g;
        ds.type = type.data();
        ds.Mout = M.data();
        ds.at = cell_place<2>(g, (kGrid / 2) * kGrid + kGrid / 2);
        ds.beta = beta;
        ds.pop = pop.data();
        ds.pop_stride = 1;
        ds.pop_cap = pop_cap;
        df_split(mass, ds.mh, ds.ml);
        return ds;
    }
    // Largest residual (thermal units) of what lies in M, deposited with mass 1, against the
    // constraints of the fluons or the phonons.  The stored heat flux is the sum of two constraints.
    double residual(bool fluon) const {
        real T[11] = {};
        for (int k = 0; k < 11; k++)
            for (int i = 0; i < kGrid * kGrid; i++) T[k] += M[(size_t)k * kGrid * kGrid + i];
        const real ux = c.u[0], uy = c.u[1], s = c.inv_sig, uu = ux * ux + uy * uy;
        real worst = 0;
        auto take = [&](real v) { worst = std::max(worst, fabsl(v)); };
        if (!fluon) {
            take(T[8] - conG[0]);
            take((T[9] - ux * T[8]) * s - conG[1]);
            take((T[10] - uy * T[8]) * s - conG[2]);
            return (double)worst;
        }
        const real n = T[0], x = T[1], y = T[2], xx = T[3], xy = T[4], yy = T[5];
        take(n - conF[0]);
        take((x - ux * n) * s - conF[1]);
        take((y - uy * n) * s - conF[2]);
        take((xx - 2 * ux * x + ux * ux * n) * s * s - conF[3]);
        take((xy - ux * y - uy * x + ux * uy * n) * s * s - conF[4]);
        take((yy - 2 * uy * y + uy * uy * n) * s * s - conF[5]);
        const real ud = ux * x + uy * y;
        const real qx = T[6] - ux * (xx + yy) - 2 * (ux * xx + uy * xy) + 2 * ux * ud + uu * x - uu * ux * n;
        const real qy = T[7] - uy * (xx + yy) - 2 * (ux * xy + uy * yy) + 2 * uy * ud + uu * y - uu * uy * n;
        take((qx * s * s * s - conF[6] - conF[7]) / 2);
        take((qy * s * s * s - conF[8] - conF[9]) / 2);
        return (double)worst;
    }
};

template <bool FLUON>
int population(Cell& k, const double* start, double mass, int pop_cap, ThreadCounters& tc, double xm = 0.0,
               double* solution = nullptr) {
    double lam[10];
    for (int j = 0; j < DFPop<2, FLUON>::N; j++) lam[j] = start[j];
    DFStream ds = k.stream(mass, pop_cap);
    const int u = df_population<2, FLUON>(k.m, k.c, k.tab, lam, FLUON ? k.conF : k.conG, k.etab.data(),
                                   xm > 0.0 ? xm : k.st.R + 2.0, ds, tc);
    for (int j = 0; solution && j < DFPop<2, FLUON>::N; j++) solution[j] = lam[j];
    return u;
}

template <bool FLUON>
void judged(double RT, double noise, double tol, int trials, unsigned seed, double* out) {
    std::mt19937_64 rng(seed);
    std::normal_distribution<double> N01;
    Cell k;
    k.m.tol = tol;
    for (int i = 0; i < 4; i++) out[i] = 0.0;
    for (int t = 0; t < trials; t++) {
        if (!k.draw(rng, RT, 0.1, 1.0)) continue;
        double start[10];
        for (int j = 0; j < DFPop<2, FLUON>::N; j++)
            start[j] = (double)(float)((FLUON ? k.lf[j] : k.lg[j]) + noise * N01(rng));
        ThreadCounters tc{}, full{};
        std::fill(k.M.begin(), k.M.end(), 0.0);
        const bool ok = population<FLUON>(k, start, 1.0, kDfPopCap, tc) >= 0;
        out[0] += 1.0;
        out[3] += tc.redo;
        if (!ok) continue;
        out[1] = std::max(out[1], k.residual(FLUON));
        const std::vector<double> kept = k.M;
        std::fill(k.M.begin(), k.M.end(), 0.0);
        population<FLUON>(k, start, 1.0, 0, full);  // every population evaluated twice
        out[2] += kept != k.M;
    }
}

// |X| up to which the fixed-point exponents of the phonons' multipliers lam stay in range.
float reach(const Cell& k, const double* lam) {
    long long beta[10];
    float lo = 0.f, hi = 1000.f;
    while (std::nextafterf(lo, hi) < hi) {
        const float mid = lo + 0.5f * (hi - lo);
        const bool in = fix_poly<2, false>(lam, k.c.inv_sig, k.c.u[0] - (double)k.tab.xc, k.c.u[1] - (double)k.tab.yc,
                                           (double)mid, beta);
        (in ? lo : hi) = mid;
    }
    return lo;
}

// Errors of the lattice-form populations (out[0]: mean, weighted by the population; out[1]: largest relative
// one) and of the general stencil's (out[2], out[3]) against extended precision, f and g.
template <int D>
void populations(double RT, int trials, unsigned seed, double* out) {
    constexpr int NF = Dim<D>::NF, NG = Dim<D>::NG;
    std::mt19937_64 rng(seed);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    Model m{};
    m.K = 2.0;
    m.n_conf = 4.0;
    m.r_min = 2.0;
    m.refine_div = m.refine_rad = 3.0;
    m.max_refine = 4;
    set_derived_params(m, D);
    real err[2] = {}, sum = 0;
    double worst[2] = {};
    for (int t = 0; t < trials; t++) {
        CellState<D> c{};
        c.rho = 1.0;
        c.RT = RT * (1.0 + 0.02 * U(rng));
        c.sig = std::sqrt(c.RT);
        c.inv_sig = 1.0 / c.sig;
        for (int a = 0; a < D; a++) c.u[a] = 2.0 * U(rng);
        Stencil<D> st;
        st.init(c, m);
        char2 rows[kRowsMax];
        RowTable<D> tab;
        tab.build(c, st, rows);
        if (!tab.ok) continue;
        CellLattice<D> lat;
        lat.init(c, tab);
        double lf[NF], lg[NG];
        maxwell_start_fg<D, NF, NG>(c.RT, lf, lg);
        for (double& v : lf) v += 0.01 * U(rng);
        for (double& v : lg) v += 0.01 * U(rng);
        auto take = [&](int who, const real* v, double f, double g) {
            const real x = (v[0] - c.u[0]) * c.inv_sig, y = D == 2 ? (v[D - 1] - c.u[D - 1]) * c.inv_sig : 0;
            for (int p = 0; p < 2; p++) {
                real e = 1;
                for (int j = 0; j < (p ? NG : NF); j++)
                    e += (real)(p ? lg[j] : lf[j]) * powl(x, p ? bx<D, false>(j) : bx<D, true>(j)) *
                         powl(y, p ? by<D, false>(j) : by<D, true>(j));
                const real exact = expl(-e), d = fabsl((p ? g : f) - exact);
                err[who] += d;
                worst[who] = std::max(worst[who], (double)(d / exact));
                if (who == 0) sum += exact;
            }
        };
        for (int l = 0; l < lat.n; l++) {
            const bool child = l == 1;
            const double hs = child ? 0.5 * c.inv_sig : c.inv_sig;
            const double ox = child ? 2.0 * lat.fx + 0.5 : lat.fx, oy = child ? 2.0 * lat.fy + 0.5 : lat.fy;
            auto point = [&](int k, int j, double f, double g) {
                const real v[2] = {child ? lat.xn - 0.25L + 0.5L * k : (real)(lat.xn + k),
                                   child ? lat.yn - 0.25L + 0.5L * j : (real)(lat.yn + j)};
                take(0, v, f, g);
            };
            auto row_end = [](int) {};
            auto ext = [&](int j, int& i0, int& i1, int& h0, int& h1) { lat.ext(tab, child, j, i0, i1, h0, h1); };
            int jlo, jhi;
            lat.rows(tab, child, jlo, jhi);
            if (D == 1 || st.R <= kSweepR)
                lattice_sweep<D, false>(lf, lg, true, true, -ox * hs, -oy * hs, hs, 1.0, 1.0, jlo, jhi, ext, point,
                                        row_end);
            else
                lattice_sweep<D, true>(lf, lg, true, true, -ox * hs, -oy * hs, hs, 1.0, 1.0, jlo, jhi, ext, point,
                                       row_end);
        }
        auto row = [&](int cy, int xa, int xb) {
            double cf[4], cg[3];
            row_coeffs<D>(lf, lg, D == 2 ? ((double)cy - c.u[D - 1]) * c.inv_sig : 0.0, cf, cg);
            auto point = [&](int k, double, double f, double g) {
                const real v[2] = {(real)(xa + k), (real)cy};
                take(1, v, f, g);
            };
            row_eval(cf, cg, true, true, ((double)xa - c.u[0]) * c.inv_sig, c.inv_sig, xb - xa + 1, point);
        };
        auto leaf = [&](const double* cp, double) {
            const double x = (cp[0] - c.u[0]) * c.inv_sig, y = D == 2 ? (cp[D - 1] - c.u[D - 1]) * c.inv_sig : 0.0;
            double cf[4], cg[3];
            row_coeffs<D>(lf, lg, y, cf, cg);
            const real v[2] = {cp[0], D == 2 ? cp[D - 1] : 0.0};
            take(1, v, std::exp(-(((cf[3] * x + cf[2]) * x + cf[1]) * x + cf[0])),
                 std::exp(-((cg[2] * x + cg[1]) * x + cg[0])));
        };
        st.for_each_row(row, leaf);
    }
    for (int k = 0; k < 2; k++) {
        out[2 * k] = (double)(err[k] / sum);
        out[2 * k + 1] = worst[k];
    }
}

}  // namespace

extern "C" {

// The mixed path's finish of one population from multipliers that are off by `noise`: out = cells drawn,
// the largest true residual of a deposit that passed the check, cells streamed from kept
// populations, deposits taken back.
void check_judged(int fluon, double RT, double noise, double tol, int trials, unsigned seed, double* out) {
    if (fluon)
        judged<true>(RT, noise, tol, trials, seed, out);
    else
        judged<false>(RT, noise, tol, trials, seed, out);
}

// A phonon deposit taken back: out = cells drawn, the largest of what stays of a moment against its
// largest value, cells streamed from kept populations, cells whose updated multipliers alone are out of the
// fixed-point range (edge = 1: the range is set between the start's reach and the update's).
void check_take_back(double RT, double noise, int edge, int trials, unsigned seed, double* out) {
    std::mt19937_64 rng(seed);
    std::normal_distribution<double> N01;
    Cell k;
    const long long cell = (kGrid / 2) * kGrid + kGrid / 2;
    std::vector<double> Min(11 * kGrid * kGrid);  // the moments that the collision takes the cell from
    for (int i = 0; i < 4; i++) out[i] = 0.0;
    for (int t = 0; t < trials; t++) {
        if (!k.draw(rng, RT, 0.1, 1.0) || !k.collide_at(Min, cell)) continue;
        double start[6], lam[6];
        for (int j = 0; j < 6; j++) start[j] = lam[j] = (double)(float)(k.lg[j] + noise * N01(rng));
        double xm = k.st.R + 2.0;
        ThreadCounters tc{};
        if (edge) {
            DFStream ds = k.stream(1.0, 0);
            double r[6], rmax;
            float MJ[DFPop<2, false>::NJ], dl[6];
            if (!df_pass<2, false, DF_CORR>(k.c.u[0], k.c.u[1], k.c.inv_sig, k.tab, lam, k.conG, k.etab.data(), xm, r,
                                            rmax, MJ, ds, tc.ls, tc.pdfc, k.beta) ||
                !df_update<2, false>(MJ, r, lam, dl))
                continue;
            const float a = reach(k, start), b = reach(k, lam);
            if (!(b < a)) continue;
            xm = a;
            out[3] += 1.0;
        }
        const double mass = k.c.rho * k.m.K * k.c.RT;
        std::fill(k.M.begin(), k.M.end(), 0.0);
        const int u = population<false>(k, start, mass, kDfPopCap, tc, xm, lam);
        if (u < 0) continue;
        out[0] += 1.0;
        const std::vector<double> made = k.M;
        DFStream ds = k.stream(1.0, kDfPopCap);
        if (u & kFromKept) {
            df_take_back<2>(k.m, k.g, Min.data(), cell, k.tab, start, u & (kFromKept - 1), k.etab.data(), xm, ds, tc);
        } else {  // as mixed_block
            double r[6], rmax;
            df_split(-mass, ds.mh, ds.ml);
            df_pass<2, false, DF_STREAM>(k.c.u[0], k.c.u[1], k.c.inv_sig, k.tab, lam, k.conG, k.etab.data(), xm, r, rmax,
                                         nullptr, ds, tc.ls, tc.pdf, k.beta);
        }
        for (int i = 8; i < 11; i++) {
            double top = 0.0, left = 0.0;
            for (int j = 0; j < kGrid * kGrid; j++) {
                top = std::max(top, std::fabs(made[(size_t)i * kGrid * kGrid + j]));
                left = std::max(left, std::fabs(k.M[(size_t)i * kGrid * kGrid + j]));
            }
            out[1] = std::max(out[1], left / top);
        }
        std::fill(k.M.begin(), k.M.end(), 0.0);
        population<false>(k, start, mass, 0, tc, xm);
        out[2] += made != k.M;
    }
}

void check_populations(int D, double RT, int trials, unsigned seed, double* out) {
    if (D == 1)
        populations<1>(RT, trials, seed, out);
    else
        populations<2>(RT, trials, seed, out);
}

long long check_pop_threads(int D, long long ncell, int n_inst, int sms) { return df_pop_threads(D, ncell, n_inst, sms); }

// The FP64 arithmetic in integer instructions and short forms, on n random arguments: out = largest error of
// exp_int in ulps over |x| < 128, of recip64 and of quotient in ulps, then how many of the other results were wrong:
// narrow (truncation; zero below 2^-126, infinity from 2^128), widen (exact), quarter (exact).
void check_arithmetic(int n, unsigned seed, double* out) {
    std::mt19937_64 rng(seed);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    for (int i = 0; i < 6; i++) out[i] = 0.0;
    auto ulps = [](double got, real exact) {
        int e;
        std::frexp((double)exact, &e);
        return (double)(fabsl(got - exact) / ldexpl(1.0L, e - 53));
    };
    const double edge[] = {0.0, -0.0, 1e-300, -1e-300, 1e-17, 0.6931471805599453, -0.6931471805599453, 127.999, -127.999,
                           0x1p-60, -0x1p-52, 64.0, -64.0};
    const int n_edge = (int)(sizeof edge / sizeof edge[0]);
    for (int i = 0; i < n; i++) {
        const double x = i < n_edge ? edge[i] : (i % 3 ? 128.0 * U(rng) : std::ldexp(U(rng), i % 60 - 56));
        out[0] = std::max(out[0], ulps(exp_int(x), expl((real)x)));
        const double b = std::ldexp(1.0 + std::fabs(U(rng)), (int)(rng() % 190) - 95);
        const double a = std::ldexp(U(rng), (int)(rng() % 40) - 20);
        const double y = recip64(b);
        out[1] = std::max(out[1], ulps(y, 1.0L / (real)b));
        out[2] = std::max(out[2], ulps(quotient(a, b, y), (real)a / (real)b));
        const double v = std::ldexp(1.0 + std::fabs(U(rng)), (int)(rng() % 300) - 150);
        const float f = narrow(v);
        const float want = v < 0x1p-126 ? 0.f : (v >= 0x1p128 ? INFINITY : std::nextafterf((float)v, 0.f));
        out[3] += v >= 0x1p-126 && v < 0x1p128 ? !((double)f <= v && (f == (float)v || f == want)) : f != want;
        out[4] += std::isfinite(f) && (widen(f) != (double)f || widen(-f) != -(double)f);
        const double w = i % 2 ? -v : v;
        out[5] += quarter(w) != 0.25 * w || quarter(std::ldexp(w, -900)) != 0.25 * std::ldexp(w, -900);
    }
    out[4] += widen(0x1p-130f) != 0.0;
    out[5] += quarter(0.0) != 0.0 || !std::isinf(quarter(INFINITY));
}

}
