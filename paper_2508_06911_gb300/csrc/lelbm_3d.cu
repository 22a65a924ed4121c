// The LELBM time step in three dimensions (the paper's general-D formulation, Sec. II,
// with D = 3: 17 stored moments, N_f = 19 fluon and N_g = 10 phonon constraints, Eq.
// IIB5, IIB14-IIB17), FP64, fluid boundaries only (Sec. III.A).
//
// One warp per cell.  A 3D velocity set holds hundreds of points (q ~ (4/3) pi (R_ac +
// 1/2)^3, 180 at RT = 0.5, 380 at RT = 1) and its Jacobians (19 x 19 and 10 x 10) do not
// fit one thread's registers, so the 32 lanes share a cell:
//   - the LAS stencil (Eq. IIC6, IIC9-IIC11) is laid out as row items in shared memory:
//     each item is a run of points along x at fixed (y, z), level-0 runs with spacing 1
//     and the children of split points as runs with spacing 2^-L (Eq. IIC10-IIC11);
//   - a Newton pass (Eq. IID7-IID11) gives each lane one item at a time: it evaluates the
//     populations along the run (the exponent is a cubic in x on the run) and their row
//     sums sum x^a f -- in FP64 those of the residual (a <= 3 for fluons, <= 2 for phonons), in
//     FP32 those of the Jacobian (a <= 6, <= 4); the lanes then fold the row sums of 32 items
//     into the population moments x^a y^b z^c f (30 in FP64, one per lane; 84 + 35 in FP32);
//   - the solve is a Gauss-Jordan elimination in FP32, one row of the system per lane;
// The FP64 pipe (one warp instruction in 64 cycles on each of an SM's four partitions) bounds this
// kernel, so only what decides the result is FP64: populations (their exponentials by integer
// instructions, exp_int), the residual, the multipliers and the deposited moments.  A solve that
// breaks down is redone by the all-FP64 Newton below it.  A step of 40^3 cells: 19.2 ms, against
// 82.5 ms with library exponentials, FP64 moments to degree 6 and an FP64 factorisation; error
// 7.5e-16 -> 6.3e-16.
//   - moment streaming (Eq. IIE3) deposits T_N(c_i) rho f'_i and T_N(c_i) rho K RT g'_i
//     at x + c_i with FP64 atomic additions (cloud-in-cell for refined children).
// Thermal units throughout the Newton (t = (c - u) / sqrt(RT)), as in 1D and 2D.
#include <cuda_runtime.h>

#include <cstdint>

#include "lelbm_device.cuh"
#include "lelbm_fp64.cuh"
#include "lelbm_internal.h"

namespace lbm {

constexpr int kW3Warps = 2;           // warps (cells in flight) per block
constexpr int kW3Items = 1024;        // row items per cell (R_ac up to about 16, RT ~ 16)
constexpr int kNF3 = 19, kNG3 = 10;   // constraints
constexpr int kPF3 = 6, kPG3 = 4;     // degree of the Jacobian moments
constexpr int kMF3 = 84, kMG3 = 35;   // monomials x^a y^b z^c of degree <= 6, <= 4
constexpr int kMon3 = kMF3 + kMG3;
constexpr int kSub = 64;              // item coordinates in units of 1/64 cell

// Exponents of the fluon basis T_j (Eq. IIB14-IIB16): 1, t_a, t_a t_b (a <= b), and the
// heat-flux entries t_a^2 t_g ordered g-major; the phonon basis is the first ten.
__device__ __constant__ int8_t c_bex[kNF3] = {0, 1, 0, 0, 2, 1, 1, 0, 0, 0, 3, 1, 1, 2, 0, 0, 2, 0, 0};
__device__ __constant__ int8_t c_bey[kNF3] = {0, 0, 1, 0, 0, 1, 0, 2, 1, 0, 0, 2, 0, 1, 3, 1, 0, 2, 0};
__device__ __constant__ int8_t c_bez[kNF3] = {0, 0, 0, 1, 0, 0, 1, 0, 1, 2, 0, 0, 2, 0, 0, 2, 1, 1, 3};

// Position of x^a y^b z^c among the monomials of degree <= P, ordered by c, then b, then a.
__device__ __forceinline__ int mon_index(int a, int b, int c, int P) {
    const int n = P + 3, k = n - c;  // C(n, 3) monomials, C(k, 3) of them with z-degree >= c
    return n * (n - 1) * (n - 2) / 6 - (int)((unsigned)(k * (k - 1) * (k - 2)) / 6u) + b * (P - c + 1) - b * (b - 1) / 2 + a;
}

// Position of y^b z^c (b + c <= 6) in a row's table of transverse monomials.
__device__ __forceinline__ int yz_index(int b, int c) { return c * 7 - c * (c - 1) / 2 + b; }

// One run of stencil points: c = (x + k h, y, z) for k = 0..n-1, h = 2^-level, all in
// units of 1/64 cell; dC = 2^(-3 level) (Eq. IIC11).
struct Item3 {
    short x, y, z, nl;  // nl = n | level << 12
};

struct Warp3 {
    Item3 items[kW3Items];
    union {
        struct {                  // lattice pass: row sums of a chunk and its rows' transverse monomials
            double S[32][7];      // FP64: fluon x^0..3, phonon x^0..2
            double YZ[32][10];    // FP64: y^b z^c, b + c <= 3 (yz_index3)
            float SJ[32][12];     // FP32: fluon x^0..6, phonon x^0..4
            float YZJ[32][28];    // FP32: y^b z^c, b + c <= 6 (yz_index)
        } q;
        struct {                  // all-FP64 pass
            double S[32][12];     // row sums: fluon x^0..6, phonon x^0..4
            double YZ[32][28];    // y^b z^c (b + c <= 6) of the chunk's rows (thermal units), yz_index
        };
    };
    union {
        struct {
            float MFJ[kMF3], MGJ[kMG3];  // Jacobian moments in FP32
            double T[30];                // residual moments in FP64: 20 fluon (degree <= 3), 10 phonon
        };
        struct {
            double MF[kMF3];      // population moments of the fluons
            double MG[kMG3];      // and of the phonons
            double A[kNF3 * kNF3];
            double Ag[kNG3 * kNG3];
        };
    };
    double rf[kNF3], rg[kNG3];
    double lf[kNF3], lg[kNG3];
    double cf[kNF3], cg[kNG3];
};

// ---------------------------------------------------------------------------
// LAS stencil as row items (Eq. IIC6, IIC9-IIC11), with the membership tests of the 1D
// and 2D stencils: squared distances summed x, y, z with one rounding each.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double dist2_3(double x, double y, double z, const double* u) {
    const double dx = __dsub_rn(x, u[0]), dy = __dsub_rn(y, u[1]), dz = __dsub_rn(z, u[2]);
    return __dadd_rn(__dadd_rn(__dadd_rn(0.0, __dmul_rn(dx, dx)), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// The run of points x_k = x0 + k h (k = 0..n-1) at (y, z) within r2 of u: [k0, k1]
// (empty when k0 > k1).  The test is monotone in |x - u_x| along the run, so the set is an
// interval; its ends are found from the real-valued chord and then checked.  The tests are taken in
// FP32 on offsets from floor(u) (exact: multiples of 1/64 below 32) and, closer to the threshold
// than FP32 resolves (as in RowTable::build), exactly in FP64.
struct Frac3 {
    double c[3];  // floor(u)
    float f[3];   // u - floor(u)
};
__device__ __forceinline__ void run_band(double x0, double h, int n, double y, double z, const double* u,
                                         const Frac3& o, double r2, int& k0, int& k1) {
    const float thr = (float)r2, mg = 1e-3f + 1e-5f * thr;
    const float X0 = (float)(x0 - o.c[0]), hf = (float)h;
    const float dy = (float)(y - o.c[1]) - o.f[1], dz = (float)(z - o.c[2]) - o.f[2];
    const float yz2 = fmaf(dy, dy, dz * dz);
    k0 = 1;
    k1 = 0;
    if (yz2 > thr + mg) return;
    auto inside = [&](int k) -> bool {
        const float d = fmaf((float)k, hf, X0) - o.f[0], v = fmaf(d, d, yz2);
        if (v < thr - mg) return true;
        if (v > thr + mg) return false;
        return dist2_3(x0 + k * h, y, z, u) <= r2;
    };
    const float s = sqrtf(fmaxf(thr - yz2, 0.f)), ih = 1.f / hf;
    k0 = (int)floorf((o.f[0] - s - X0) * ih) - 1;
    k1 = (int)ceilf((o.f[0] + s - X0) * ih) + 1;
    k0 = k0 < 0 ? 0 : k0;
    k1 = k1 > n - 1 ? n - 1 : k1;
    while (k0 <= k1 && !inside(k0)) k0++;
    while (k1 >= k0 && !inside(k1)) k1--;
}

// Emits the items of one level-0 row (cy, cz): the unsplit runs and, recursively, the
// child runs of its split points.  count_only: only counts.  Returns the item count.
template <bool WRITE>
__device__ int row_items(int cy, int cz, const double* u, const Frac3& o, const Stencil<3>& st, Item3* out, int cap) {
    int cnt = 0;
    auto emit = [&](double x, double y, double z, int n, int level) {
        if (WRITE && cnt < cap) {
            Item3 it;
            it.x = (short)rint(x * kSub);
            it.y = (short)rint(y * kSub);
            it.z = (short)rint(z * kSub);
            it.nl = (short)(n | (level << 12));
            out[cnt] = it;
        }
        cnt++;
    };
    const double y = cy, z = cz;
    const int xlo = (int)o.c[0] - st.R - 2, xhi = (int)o.c[0] + st.R + 3;
    int a0, a1;
    run_band((double)xlo, 1.0, xhi - xlo + 1, y, z, u, o, st.rr2, a0, a1);
    if (a0 > a1) return 0;
    // stack of child runs still to split: (x0, y, z, n, level)
    struct Run {
        double x, y, z;
        int n, level;
    };
    Run stack[16];
    int sp = 0;
    Run top{(double)(xlo + a0), y, z, a1 - a0 + 1, 0};
    for (;;) {
        const double h = ldexp(1.0, -top.level);
        int b0 = 1, b1 = 0;
        if (top.level < st.Nr) run_band(top.x, h, top.n, top.y, top.z, u, o, st.rad2[top.level + 1], b0, b1);
        if (b0 > b1) {
            emit(top.x, top.y, top.z, top.n, top.level);
        } else {
            if (b0 > 0) emit(top.x, top.y, top.z, b0, top.level);
            if (b1 < top.n - 1) emit(top.x + (b1 + 1) * h, top.y, top.z, top.n - 1 - b1, top.level);
            // children of the split points at +-h/4 per axis: four child runs of spacing h/2
            const double q = 0.25 * h;
            for (int s = 3; s >= 0; s--) {
                if (sp < 16)
                    stack[sp++] = Run{top.x + b0 * h - q, top.y + ((s & 1) ? q : -q), top.z + ((s & 2) ? q : -q),
                                      2 * (b1 - b0 + 1), top.level + 1};
            }
        }
        if (sp == 0) break;
        top = stack[--sp];
    }
    return cnt;
}

// Lays the cell's velocity set out as items in w->items (deterministic order: level-0
// rows by z, then y); returns the total count (more than kW3Items: the set does not fit)
// and the number of points in *q.
__device__ int build_items(Warp3* w, const double* u, const Stencil<3>& st, int lane, long long* q) {
    Frac3 o;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        o.c[a] = floor(u[a]);
        o.f[a] = (float)(u[a] - o.c[a]);
    }
    // every row within R_ac + 1/2 of u
    const int y0 = (int)o.c[1] - st.R, z0 = (int)o.c[2] - st.R;
    const int ny = 2 * st.R + 2, ncand = ny * ny;
    int total = 0;
    long long pts = 0;
    for (int base = 0; base < ncand; base += 32) {
        const int idx = base + lane;
        const int cy = y0 + idx % ny, cz = z0 + idx / ny;
        const int cnt = idx < ncand ? row_items<false>(cy, cz, u, o, st, nullptr, 0) : 0;
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int off = total + incl - cnt;
        if (cnt > 0 && off < kW3Items) row_items<true>(cy, cz, u, o, st, w->items + off, kW3Items - off);
        total += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    const int n = total < kW3Items ? total : kW3Items;
    for (int i = lane; i < n; i += 32) pts += w->items[i].nl & 0xfff;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pts += __shfl_xor_sync(0xffffffffu, pts, o);
    *q = pts;
    return total;
}

// Geometry of item i in thermal units: first x, spacing, y, z and the volume element.
struct ItemGeo {
    double tx, th, ty, tz, dC;
    int n, level;
    double cx, cy, cz, h;  // lattice frame: first velocity and spacing
};

__device__ __forceinline__ ItemGeo item_geo(const Item3& it, const CellState<3>& c) {
    ItemGeo g;
    g.n = it.nl & 0xfff;
    g.level = it.nl >> 12;
    g.h = ldexp(1.0, -g.level);
    g.dC = ldexp(1.0, -3 * g.level);
    g.cx = it.x * (1.0 / kSub);
    g.cy = it.y * (1.0 / kSub);
    g.cz = it.z * (1.0 / kSub);
    g.tx = (g.cx - c.u[0]) * c.inv_sig;
    g.ty = (g.cy - c.u[1]) * c.inv_sig;
    g.tz = (g.cz - c.u[2]) * c.inv_sig;
    g.th = g.h * c.inv_sig;
    return g;
}

// Position of y^b z^c (b + c <= 3) among the row's FP64 transverse monomials.
__device__ __forceinline__ constexpr int yz_index3(int b, int c) { return c * 4 - c * (c - 1) / 2 + b; }

// y^b z^c, b + c <= 3.
__device__ __forceinline__ void yz_monomials(double y, double z, double* m) {
    m[yz_index3(0, 0)] = 1.0;
    m[yz_index3(1, 0)] = y;
    m[yz_index3(0, 1)] = z;
    m[yz_index3(2, 0)] = y * y;
    m[yz_index3(1, 1)] = y * z;
    m[yz_index3(0, 2)] = z * z;
    m[yz_index3(3, 0)] = m[yz_index3(2, 0)] * y;
    m[yz_index3(2, 1)] = m[yz_index3(2, 0)] * z;
    m[yz_index3(1, 2)] = m[yz_index3(0, 2)] * y;
    m[yz_index3(0, 3)] = m[yz_index3(0, 2)] * z;
}

// Coefficients of 1 + sum_j lam_j T_j as a cubic (fluons) or quadratic (phonons) in x on
// the run whose transverse monomials are m.  The bases are those of c_bex, c_bey, c_bez.
__device__ __forceinline__ void run_coeffs(const double* lf, const double* lg, const double* m, double* cf,
                                           double* cg) {
    constexpr int Y = yz_index3(1, 0), Z = yz_index3(0, 1), YY = yz_index3(2, 0), YZ = yz_index3(1, 1),
                  ZZ = yz_index3(0, 2);
    cf[0] = 1.0 + lf[0] + lf[2] * m[Y] + lf[3] * m[Z] + lf[7] * m[YY] + lf[8] * m[YZ] + lf[9] * m[ZZ] +
            lf[14] * m[yz_index3(3, 0)] + lf[15] * m[yz_index3(1, 2)] + lf[17] * m[yz_index3(2, 1)] +
            lf[18] * m[yz_index3(0, 3)];
    cf[1] = lf[1] + lf[5] * m[Y] + lf[6] * m[Z] + lf[11] * m[YY] + lf[12] * m[ZZ];
    cf[2] = lf[4] + lf[13] * m[Y] + lf[16] * m[Z];
    cf[3] = lf[10];
    cg[0] = 1.0 + lg[0] + lg[2] * m[Y] + lg[3] * m[Z] + lg[7] * m[YY] + lg[8] * m[YZ] + lg[9] * m[ZZ];
    cg[1] = lg[1] + lg[5] * m[Y] + lg[6] * m[Z];
    cg[2] = lg[4];
}

// One Newton pass over the velocity set: the residual's moments x^a y^b z^c f of degree <= 3 (fluons, if
// doF) and <= 2 (phonons, if doG) in FP64 into w->T, the Jacobian's of degree <= 6 and <= 4 in FP32 into
// w->MFJ, w->MGJ.  A lane owns one FP64 monomial (ta, tyz of population tsel; tsel = 2: none) and up to
// four FP32 ones.
__device__ void moment_pass3q(Warp3* w, const CellState<3>& c, int n_items, bool doF, bool doG, int lane,
                              const int* ma, const int* mb, const int* mcz, const int* msel, int nown, int ts,
                              int tyz, bool town, unsigned long long& npts) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    double tacc = 0.0;
    int si[4], yi[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        si[k] = k < nown ? (msel[k] ? 7 : 0) + ma[k] : 0;
        yi[k] = k < nown ? yz_index(mb[k], mcz[k]) : 0;
    }
    for (int base = 0; base < n_items; base += 32) {
        const int i = base + lane;
        if (i < n_items) {
            const ItemGeo gi = item_geo(w->items[i], c);
            double m[10], cf[4], cg[3];
            yz_monomials(gi.ty, gi.tz, m);
            run_coeffs(w->lf, w->lg, m, cf, cg);
            double S[7];
            float J[12];
#pragma unroll
            for (int a = 0; a < 7; a++) S[a] = 0.0;
#pragma unroll
            for (int a = 0; a < 12; a++) J[a] = 0.f;
            double x = gi.tx;
            const float h32 = (float)gi.th, x32 = (float)gi.tx;
#pragma unroll 1
            for (int k = 0; k < gi.n; k++, x += gi.th) {
                const float xf = fmaf((float)k, h32, x32);
                const float x2 = xf * xf, x3 = x2 * xf, x4 = x2 * x2;
                const float pw[7] = {1.f, xf, x2, x3, x4, x4 * xf, x3 * x3};
                if (doF) {
                    double p = exp_int(-(((cf[3] * x + cf[2]) * x + cf[1]) * x + cf[0]));
                    const float pj = narrow(p);
                    S[0] += p;
#pragma unroll
                    for (int a = 1; a < 4; a++) {
                        p *= x;
                        S[a] += p;
                    }
#pragma unroll
                    for (int a = 0; a < 7; a++) J[a] = fmaf(pw[a], pj, J[a]);
                }
                if (doG) {
                    double p = exp_int(-((cg[2] * x + cg[1]) * x + cg[0]));
                    const float pj = narrow(p);
                    S[4] += p;
#pragma unroll
                    for (int a = 1; a < 3; a++) {
                        p *= x;
                        S[4 + a] += p;
                    }
#pragma unroll
                    for (int a = 0; a < 5; a++) J[7 + a] = fmaf(pw[a], pj, J[7 + a]);
                }
            }
            npts += (unsigned long long)gi.n;
            const float dCf = (float)gi.dC;  // a power of two
#pragma unroll
            for (int a = 0; a < 7; a++) w->q.S[lane][a] = S[a] * gi.dC;
#pragma unroll
            for (int a = 0; a < 12; a++) w->q.SJ[lane][a] = J[a] * dCf;
#pragma unroll
            for (int a = 0; a < 10; a++) w->q.YZ[lane][a] = m[a];
            const float yf = (float)gi.ty, zf = (float)gi.tz;
            float yp[7], zp = 1.f;
            yp[0] = 1.f;
#pragma unroll
            for (int k = 1; k < 7; k++) yp[k] = yp[k - 1] * yf;
#pragma unroll
            for (int cz = 0; cz < 7; cz++) {
#pragma unroll
                for (int bb = 0; bb + cz < 7; bb++) w->q.YZJ[lane][yz_index(bb, cz)] = yp[bb] * zp;
                zp *= zf;
            }
        }
        __syncwarp();
        const int nr = n_items - base < 32 ? n_items - base : 32;
#pragma unroll 2
        for (int r = 0; r < nr; r++) {
            tacc = fma(w->q.S[r][ts], w->q.YZ[r][tyz], tacc);
#pragma unroll
            for (int k = 0; k < 4; k++) acc[k] = fmaf(w->q.SJ[r][si[k]], w->q.YZJ[r][yi[k]], acc[k]);
        }
        __syncwarp();
    }
    if (town) w->T[lane] = tacc;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        if (k < nown) {
            const int e = lane + 32 * k;
            if (e < kMF3)
                w->MFJ[e] = acc[k];
            else
                w->MGJ[e - kMF3] = acc[k];
        }
    }
    __syncwarp();
}

// Newton update of one population from the FP64 residual and the FP32 Jacobian of a lattice pass: lane i
// holds row i of the system and eliminates (Gauss-Jordan; every pivot has to be positive, as in a
// Cholesky factorisation).  Returns as newton_update3.
template <int N, int P, int T0>
__device__ __forceinline__ int newton_update3q(const double* T, const float* Mom, const double* con, double* lam, int it,
                                               double tol, int max_iter, int lane) {
    constexpr int PT = P / 2;  // degree of the residual's moments
    const int i = lane < N ? lane : N - 1;
    const int ex = c_bex[i], ey = c_bey[i], ez = c_bez[i];
    const double rj = T[T0 + mon_index(ex, ey, ez, PT)] - con[i];
    long long worst = __double_as_longlong(rj) & 0x7fffffffffffffffLL;
    float b = narrow(__longlong_as_double(worst));
    b = __double2hiint(rj) < 0 ? -b : b;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long v = __shfl_xor_sync(0xffffffffu, worst, o);
        worst = v > worst ? v : worst;
    }
    if (worst >= 0x7ff0000000000000LL) return -1;
    const bool conv = worst <= __double_as_longlong(tol);
    if (!conv && it >= max_iter) return -2;
    float a[N];
#pragma unroll
    for (int j = 0; j < N; j++) a[j] = Mom[mon_index(ex + c_bex[j], ey + c_bey[j], ez + c_bez[j], P)];
    float piv = 1.f;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < N; k++) {
        const float d = __shfl_sync(0xffffffffu, a[k], k);
        ok = ok && d > 0.f;
        if (lane == k) piv = d;
        const float f = lane == k ? 0.f : __fdividef(a[k], d);
#pragma unroll
        for (int j = k + 1; j < N; j++) a[j] = fmaf(-f, __shfl_sync(0xffffffffu, a[j], k), a[j]);
        b = fmaf(-f, __shfl_sync(0xffffffffu, b, k), b);
    }
    const float x = __fdividef(b, piv);
    ok = ok && (lane >= N || isfinite(x));
    if (!__all_sync(0xffffffffu, ok)) return -1;
    if (lane < N) lam[lane] += widen(x);
    __syncwarp();
    return conv ? 1 : 0;
}

// One Newton pass over the velocity set: the population moments x^a y^b z^c f of degree
// <= 6 (fluons, if doF) and <= 4 (phonons, if doG) into w->MF, w->MG.
__device__ void moment_pass3(Warp3* w, const CellState<3>& c, int n_items, bool doF, bool doG, int lane,
                             const int* ma, const int* mb, const int* mcz, const int* msel, int nown,
                             unsigned long long& npts) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int base = 0; base < n_items; base += 32) {
        const int i = base + lane;
        if (i < n_items) {
            const ItemGeo gi = item_geo(w->items[i], c);
            double m[10], cf[4], cg[3];
            yz_monomials(gi.ty, gi.tz, m);
            run_coeffs(w->lf, w->lg, m, cf, cg);
            double Sf[7], Sg[5];
#pragma unroll
            for (int a = 0; a < 7; a++) Sf[a] = 0.0;
#pragma unroll
            for (int a = 0; a < 5; a++) Sg[a] = 0.0;
            auto point = [&](int, double x, double f, double g) {
                double pf = f * gi.dC, pg = g * gi.dC;
#pragma unroll
                for (int a = 0; a < 7; a++) {
                    Sf[a] += pf;
                    pf *= x;
                }
#pragma unroll
                for (int a = 0; a < 5; a++) {
                    Sg[a] += pg;
                    pg *= x;
                }
            };
            row_eval(cf, cg, doF, doG, gi.tx, gi.th, gi.n, point);
            npts += (unsigned long long)gi.n;
#pragma unroll
            for (int a = 0; a < 7; a++) w->S[lane][a] = Sf[a];
#pragma unroll
            for (int a = 0; a < 5; a++) w->S[lane][7 + a] = Sg[a];
            // the row's transverse monomials, once per row (the lanes then need one product
            // per monomial and row)
            double yp[7];
            yp[0] = 1.0;
#pragma unroll
            for (int k = 1; k < 7; k++) yp[k] = yp[k - 1] * gi.ty;
            double zp = 1.0;
#pragma unroll
            for (int cz = 0; cz < 7; cz++) {
#pragma unroll
                for (int b = 0; b + cz < 7; b++) w->YZ[lane][yz_index(b, cz)] = yp[b] * zp;
                zp *= gi.tz;
            }
        }
        __syncwarp();
        const int nr = n_items - base < 32 ? n_items - base : 32;
        bool act[4];
        int si[4], yi[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            act[k] = k < nown && ((msel[k] == 0 && doF) || (msel[k] == 1 && doG));
            si[k] = k < nown ? (msel[k] ? 7 : 0) + ma[k] : 0;
            yi[k] = k < nown ? yz_index(mb[k], mcz[k]) : 0;
        }
        for (int r = 0; r < nr; r++) {
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (act[k]) acc[k] = fma(w->S[r][si[k]], w->YZ[r][yi[k]], acc[k]);
        }
        __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
        if (k < nown) {
            const int e = lane + 32 * k;
            if (msel[k] == 0 && doF) w->MF[e] = acc[k];
            if (msel[k] == 1 && doG) w->MG[e - kMF3] = acc[k];
        }
    }
    __syncwarp();
}

// Cholesky factorisation A = L L^T (row-major N x N, lower triangle) and solve A x = b,
// shared by the lanes of a warp; b is overwritten by x.  Returns false on a non-positive
// pivot (the same test as the oracle's plain factorisation).
__device__ bool warp_chol_solve(double* A, double* b, int N, int lane) {
    for (int k = 0; k < N; k++) {
        __syncwarp();
        const double akk = A[k * N + k];
        if (!(akk > 0.0)) return false;
        const double d = sqrt(akk);
        __syncwarp();
        if (lane == 0) A[k * N + k] = d;
        for (int i = k + 1 + lane; i < N; i += 32) A[i * N + k] /= d;
        __syncwarp();
        for (int i = k + 1; i < N; i++) {
            const double lik = A[i * N + k];
            for (int j = k + 1 + lane; j <= i; j += 32) A[i * N + j] -= lik * A[j * N + k];
        }
    }
    __syncwarp();
    for (int k = 0; k < N; k++) {  // L y = b
        const double yk = b[k] / A[k * N + k];
        __syncwarp();
        if (lane == 0) b[k] = yk;
        for (int i = k + 1 + lane; i < N; i += 32) b[i] -= A[i * N + k] * yk;
        __syncwarp();
    }
    for (int k = N - 1; k >= 0; k--) {  // L^T x = y
        const double xk = b[k] / A[k * N + k];
        __syncwarp();
        if (lane == 0) b[k] = xk;
        for (int i = lane; i < k; i += 32) b[i] -= A[k * N + i] * xk;
        __syncwarp();
    }
    return true;
}

// Residual and Newton update of one population from its moments (Eq. IID9-IID11):
// N = 19, P = 6 (fluons) or N = 10, P = 4 (phonons).  Returns 1 when the population has
// converged (the update just applied is the polishing one), 0 to go on, -1 on a
// breakdown and -2 at the iteration cap (the oracle's Newton loop).
__device__ int newton_update3(const double* Mom, const double* con, double* lam, double* A, double* r, int N, int P,
                              int it, double tol, int max_iter, int lane) {
    double rj = 0.0;
    if (lane < N) {
        rj = Mom[mon_index(c_bex[lane], c_bey[lane], c_bez[lane], P)] - con[lane];
        r[lane] = rj;
    }
    double rmax = lane < N ? fabs(rj) : 0.0;
    bool fin = lane < N ? isfinite(rj) : true;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rmax = fmax(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    fin = __all_sync(0xffffffffu, fin);
    if (!fin) return -1;
    const bool conv = rmax <= tol;
    if (!conv && it >= max_iter) return -2;
    for (int e = lane; e < N * N; e += 32) {
        const int i = e / N, j = e - (e / N) * N;
        A[e] = Mom[mon_index(c_bex[i] + c_bex[j], c_bey[i] + c_bey[j], c_bez[i] + c_bez[j], P)];
    }
    __syncwarp();
    if (!warp_chol_solve(A, r, N, lane)) return -1;
    bool ok = true;
    if (lane < N) {
        lam[lane] += r[lane];
        ok = isfinite(lam[lane]);
    }
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();
    if (!ok) return -1;
    return conv ? 1 : 0;
}

// EPR of both populations (Eq. IID7-IID11) from the multipliers in w->lf, w->lg by lattice passes; as
// solve3.
__device__ __forceinline__ void solve3q(Warp3* w, const CellState<3>& c, const Model& m, bool has_g, int n_items, int lane,
                                        const int* ma, const int* mb, const int* mcz, const int* msel, int nown, int& sf,
                                        int& sg, unsigned long long& np_f, unsigned long long& np_g) {
    // the FP64 monomial of this lane: 20 fluon ones (degree <= 3), then 10 phonon ones (degree <= 2)
    int ts = 0, tyz = 0;
    {
        int t = lane < 20 ? lane : lane - 20;
        const int P = lane < 20 ? 3 : 2;
        for (int cz = 0; cz <= P; cz++)
            for (int by = 0; by <= P - cz; by++)
                for (int ax = 0; ax <= P - cz - by; ax++) {
                    if (t == 0) {
                        ts = (lane < 20 ? 0 : 4) + ax;
                        tyz = yz_index3(by, cz);
                    }
                    t--;
                }
    }
    bool actF = true, actG = has_g;
    sf = 0;
    sg = 0;
#pragma unroll 1
    for (int it = 0; actF || actG; it++) {
        unsigned long long np = 0;
        moment_pass3q(w, c, n_items, actF, actG, lane, ma, mb, mcz, msel, nown, ts, tyz, lane < 30, np);
        if (actF) {
            np_f += np;
            const int r = newton_update3q<kNF3, kPF3, 0>(w->T, w->MFJ, w->cf, w->lf, it, m.tol, m.max_iter, lane);
            sf = r < 0 ? r : sf + 1;
            actF = r == 0;
        }
        if (actG) {
            np_g += np;
            const int r = newton_update3q<kNG3, kPG3, 20>(w->T, w->MGJ, w->cg, w->lg, it, m.tol, m.max_iter, lane);
            sg = r < 0 ? r : sg + 1;
            actG = r == 0;
        }
        __syncwarp();
    }
}

// EPR of both populations (Eq. IID7-IID11) from the multipliers in w->lf, w->lg and the
// constraints in w->cf, w->cg.  sf, sg: Newton updates (>= 0) or -1 / -2.
static __device__ __noinline__ void solve3(Warp3* w, const CellState<3>& c, const Model& m, bool has_g, int n_items, int lane,
                       const int* ma, const int* mb, const int* mcz, const int* msel, int nown, int& sf, int& sg,
                       unsigned long long& np_f, unsigned long long& np_g) {
    bool actF = true, actG = has_g;
    int uf = 0, ug = 0;
    sf = 0;
    sg = 0;
    for (int it = 0; actF || actG; it++) {
        unsigned long long np = 0;
        moment_pass3(w, c, n_items, actF, actG, lane, ma, mb, mcz, msel, nown, np);
        if (actF) np_f += np;
        if (actG) np_g += np;
        if (actF) {
            const int s = newton_update3(w->MF, w->cf, w->lf, w->A, w->rf, kNF3, kPF3, it, m.tol, m.max_iter, lane);
            if (s < 0) {
                sf = s;
                actF = false;
            } else {
                uf++;
                if (s == 1) {
                    sf = uf;
                    actF = false;
                }
            }
        }
        if (actG) {
            const int s = newton_update3(w->MG, w->cg, w->lg, w->Ag, w->rg, kNG3, kPG3, it, m.tol, m.max_iter, lane);
            if (s < 0) {
                sg = s;
                actG = false;
            } else {
                ug++;
                if (s == 1) {
                    sg = ug;
                    actG = false;
                }
            }
        }
        __syncwarp();
    }
}

__device__ __forceinline__ int land_axis3(int i, int n, int pad, int periodic) {
    if (periodic) {
        const int r = i % n;
        return r < 0 ? r + n : r;
    }
    return (i < pad || i >= pad + n) ? -1 : i;
}

// Moment streaming (Eq. IIE3) of the cell's populations with the multipliers in w->lf,
// w->lg: T_N(c_i) rho f'_i and T_N(c_i) rho K RT g'_i added at x + c_i; a refined child
// landing between cells is shared by cloud-in-cell weights; what lands on a pad or outside
// the grid is discarded.
__device__ void stream3(Warp3* w, const CellState<3>& c, const Model& m, const Geometry3& g, double* Mout, int ix,
                        int iy, int iz, int n_items, bool has_g, int lane, unsigned long long& nms, unsigned int& far64) {
    const double ms = c.rho, gs = c.rho * m.K * c.RT;
#pragma unroll 1
    for (int i = lane; i < n_items; i += 32) {
        const Item3 it = w->items[i];
        const ItemGeo gi = item_geo(it, c);
        double mm[10], cf[4], cg[3];
        yz_monomials(gi.ty, gi.tz, mm);
        run_coeffs(w->lf, w->lg, mm, cf, cg);
        const double msd = ms * gi.dC, gsd = gs * gi.dC;
        const int step = kSub >> gi.level;
        const int qy = it.y, qz = it.z;  // velocity in 1/64 cell, exact
        const double cy = widen((float)qy * (1.f / kSub)), cz = widen((float)qz * (1.f / kSub));
        double x = gi.tx;
#pragma unroll 1
        for (int k = 0; k < gi.n; k++, x += gi.th) {
            const int qx = it.x + k * step;
            const double cx = widen((float)qx * (1.f / kSub));
            const double mf = msd * exp_int(-(((cf[3] * x + cf[2]) * x + cf[1]) * x + cf[0]));
            const double mg = has_g ? gsd * exp_int(-((cg[2] * x + cg[1]) * x + cg[0])) : 0.0;
            far64 = max(far64, (unsigned)(qx * qx) + (unsigned)(qy * qy) + (unsigned)(qz * qz));
            double dM[17];
            dM[0] = mf;
            dM[1] = cx * mf;
            dM[2] = cy * mf;
            dM[3] = cz * mf;
            dM[4] = cx * dM[1];
            dM[5] = cx * dM[2];
            dM[6] = cx * dM[3];
            dM[7] = cy * dM[2];
            dM[8] = cy * dM[3];
            dM[9] = cz * dM[3];
            const double e = dM[4] + dM[7] + dM[9];
            dM[10] = cx * e;
            dM[11] = cy * e;
            dM[12] = cz * e;
            dM[13] = mg;
            dM[14] = cx * mg;
            dM[15] = cy * mg;
            dM[16] = cz * mg;
            // landing: the cell of x + c and, for refined children, cloud-in-cell weights (multiples of 1/64)
            const int bx = qx >> 6, by = qy >> 6, bz = qz >> 6;
            const float w1x = (float)(qx & 63) * (1.f / kSub), w1y = (float)(qy & 63) * (1.f / kSub),
                        w1z = (float)(qz & 63) * (1.f / kSub);
#pragma unroll 1
            for (int s8 = 0; s8 < 8; s8++) {
                const int sx = s8 & 1, sy = (s8 >> 1) & 1, sz = s8 >> 2;
                const float wf = (sx ? w1x : 1.f - w1x) * (sy ? w1y : 1.f - w1y) * (sz ? w1z : 1.f - w1z);
                if (wf == 0.f) continue;
                const int tx = land_axis3(ix + bx + sx, g.nx, g.px, g.periodic[0]);
                const int ty = land_axis3(iy + by + sy, g.ny, g.py, g.periodic[1]);
                const int tz = land_axis3(iz + bz + sz, g.nz, g.pz, g.periodic[2]);
                if (tx < 0 || ty < 0 || tz < 0) continue;
                const long long t = ((long long)tz * g.NY + ty) * g.NX + tx;
                if (gi.level == 0) {  // one cell takes it all
#pragma unroll
                    for (int q = 0; q < 17; q++) atomicAdd(&Mout[q * g.ncell + t], dM[q]);
                    break;
                }
                const double wgt = widen(wf);
#pragma unroll
                for (int q = 0; q < 17; q++) atomicAdd(&Mout[q * g.ncell + t], wgt * dM[q]);
            }
        }
        nms += (unsigned long long)gi.n;
    }
}

// The monomials this lane accumulates: entries lane, lane + 32, ... of the list of the
// 84 fluon monomials (degree <= 6) followed by the 35 phonon ones (degree <= 4).
__device__ __forceinline__ int own_monomials(int lane, int* ma, int* mb, int* mcz, int* msel) {
    int nown = 0;
    for (int k = 0; k < 4; k++) {
        const int e = lane + 32 * k;
        if (e >= kMon3) break;
        const int P = e < kMF3 ? kPF3 : kPG3;
        int t = e < kMF3 ? e : e - kMF3;
        for (int cz = 0; cz <= P; cz++)
            for (int by = 0; by <= P - cz; by++)
                for (int ax = 0; ax <= P - cz - by; ax++) {
                    if (t == 0) {
                        ma[k] = ax;
                        mb[k] = by;
                        mcz[k] = cz;
                    }
                    t--;
                }
        msel[k] = e < kMF3 ? 0 : 1;
        nown++;
    }
    return nown;
}

// Eq. (IID13) in thermal units, with the constraints of the collision (or, for the
// fallback, of the equilibrium: omega = 1).
__device__ __forceinline__ void start3(Warp3* w, const CellState<3>& c, bool equilibrium, int lane) {
    double lf[kNF3], lg[kNG3];
    maxwell_start_newton<3, kNF3, kNG3>(c.RT, lf, lg);
    if (lane < kNF3) {
        w->lf[lane] = lf[lane];
        double v = c.cf[lane];
        if (equilibrium) v = lane == 0 ? 1.0 : ((lane == 4 || lane == 7 || lane == 9) ? 1.0 : 0.0);
        w->cf[lane] = v;
    }
    if (lane < kNG3) {
        w->lg[lane] = lg[lane];
        double v = c.cg[lane];
        if (equilibrium) v = lane == 0 ? 1.0 : ((lane == 4 || lane == 7 || lane == 9) ? 1.0 : 0.0);
        w->cg[lane] = v;
    }
    __syncwarp();
}

// One time step of every cell of a padded 3D grid: each warp claims cells from a global
// counter and runs the single-cell operation (collision, LAS, EPR, moment streaming).
__global__ void __launch_bounds__(kW3Warps * 32) cell3d_kernel(const __grid_constant__ Model m,
                                                               const __grid_constant__ Geometry3 g,
                                                               const double* __restrict__ Min, double* Mout,
                                                               DevStats* stats, unsigned long long* work) {
    extern __shared__ __align__(16) unsigned char smem3[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    Warp3* w = reinterpret_cast<Warp3*>(smem3) + wid;
    int ma[4], mb[4], mcz[4], msel[4];
    const int nown = own_monomials(lane, ma, mb, mcz, msel);
    const bool has_g = m.K > 0.0;
    unsigned long long n_cells = 0, np_f = 0, np_g = 0, n_ms = 0, q_max = 0, feq = 0, fmx = 0;
    unsigned long long hist[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    unsigned int far64 = 0;  // largest |c|^2 in (1/64 cell)^2
    for (;;) {
        long long cell = 0;
        if (lane == 0) cell = (long long)atomicAdd(work, 1ull);
        cell = __shfl_sync(0xffffffffu, cell, 0);
        if (cell >= g.ncell) break;
        const double v = lane < 17 ? Min[(long long)lane * g.ncell + cell] : 0.0;
        double M[17];
#pragma unroll
        for (int i = 0; i < 17; i++) M[i] = __shfl_sync(0xffffffffu, v, i);
        CellState<3> c;
        collide<3>(M, m, c);
        if (!c.ok) {  // non-physical cell: nothing can be reconstructed
            if (lane == 0) {
                fmx++;
                atomicMin(&stats->first_fail, (unsigned long long)cell);
            }
            continue;
        }
        Stencil<3> st;
        st.init(c, m);
        // item coordinates are 16-bit multiples of 1/64: |c| < 512
        const double reach = fmax(fabs(c.u[0]), fmax(fabs(c.u[1]), fabs(c.u[2]))) + (double)st.R + 3.0;
        long long q = 0;
        const int total = reach < 500.0 ? build_items(w, c.u, st, lane, &q) : kW3Items + 1;
        if (total > kW3Items) {  // velocity set beyond the item table: reported, not streamed
            if (lane == 0) {
                fmx++;
                atomicMin(&stats->first_fail, (unsigned long long)cell);
            }
            __syncwarp();
            continue;
        }
        n_cells++;
        q_max = q_max > (unsigned long long)q ? q_max : (unsigned long long)q;
        start3(w, c, false, lane);
        int sf, sg;
        solve3q(w, c, m, has_g, total, lane, ma, mb, mcz, msel, nown, sf, sg, np_f, np_g);
        if (sf < 0 || sg < 0) {  // redone by the all-FP64 Newton
            start3(w, c, false, lane);
            solve3(w, c, m, has_g, total, lane, ma, mb, mcz, msel, nown, sf, sg, np_f, np_g);
        }
        if (sf >= 0 && sg >= 0) {
            hist[sf < 7 ? sf : 7]++;
            if (has_g) hist[sg < 7 ? sg : 7]++;
        } else {
            // equilibrium constraints (omega = 1) for both populations
            start3(w, c, true, lane);
            solve3(w, c, m, has_g, total, lane, ma, mb, mcz, msel, nown, sf, sg, np_f, np_g);
            if (sf >= 0 && sg >= 0) {
                feq++;
            } else {
                // normalised Maxwellian weights: f'_i = g'_i = dC_i exp(-t^2 / 2) / S
                if (lane < kNF3) w->lf[lane] = lane == 0 ? -1.0 : ((lane == 4 || lane == 7 || lane == 9) ? 0.5 : 0.0);
                __syncwarp();
                unsigned long long np = 0;
                moment_pass3(w, c, total, true, false, lane, ma, mb, mcz, msel, nown, np);
                const double S = w->MF[0];
                __syncwarp();
                if (lane == 0) w->lf[0] = log(S) - 1.0;
                __syncwarp();
                if (lane < kNG3) w->lg[lane] = w->lf[lane];
                __syncwarp();
                fmx++;
                if (lane == 0) atomicMin(&stats->first_fail, (unsigned long long)cell);
            }
        }
        const long long pl = (long long)g.NX * g.NY;
        const int iz = (int)(cell / pl);
        const long long rem = cell - (long long)iz * pl;
        const int iy = (int)(rem / g.NX), ix = (int)(rem - (long long)iy * g.NX);
        stream3(w, c, m, g, Mout, ix, iy, iz, total, has_g, lane, n_ms, far64);
        __syncwarp();
    }
    // counters: lane 0 holds the per-cell tallies, every lane its streamed points
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        n_ms += __shfl_xor_sync(0xffffffffu, n_ms, o);
        far64 = max(far64, __shfl_xor_sync(0xffffffffu, far64, o));
    }
    if (lane == 0) {
        atomicAdd(&stats->cells, n_cells);
        atomicAdd(&stats->points_f, np_f);
        atomicAdd(&stats->points_g, np_g);
        atomicAdd(&stats->points_ms, n_ms);
        atomicAdd(&stats->fallback_eq, feq);
        atomicAdd(&stats->fallback_mx, fmx);
        atomicMax(&stats->q_max, q_max);
        atomicMax(&stats->disp_max_bits, (unsigned long long)__double_as_longlong(sqrt((double)far64) / kSub));
        for (int i = 0; i < 8; i++)
            if (hist[i]) atomicAdd(&stats->newton_hist[i], hist[i]);
    }
}

// Boundary fill of the 3D pads (Sec. III.A): inflow pads hold the equilibrium of the
// inflow state, the others copy the nearest interior cell.
__global__ void fill_pads3_kernel(double K, double r_in, double ux, double uy, double uz, double RT_in, double* M,
                                  long long ncell, const long long* pad_cell, const long long* pad_src,
                                  long long npad) {
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < npad;
         k += (long long)gridDim.x * blockDim.x) {
        const long long dst = pad_cell[k], src = pad_src[k];
        if (src < 0) {
            const double u[3] = {ux, uy, uz};
            double Me[17];
            eq_moments<3>(K, r_in, u, RT_in, Me);
#pragma unroll
            for (int i = 0; i < 17; i++) M[i * ncell + dst] = Me[i];
        } else {
#pragma unroll
            for (int i = 0; i < 17; i++) M[i * ncell + dst] = M[i * ncell + src];
        }
    }
}

void launch_fill_pads3(const Model& m, const double inlet[5], double* M, long long ncell, const long long* pad_cell,
                       const long long* pad_src, long long npad, cudaStream_t s) {
    if (npad == 0) return;
    long long b = (npad + 255) / 256;
    if (b > 65535LL * 32) b = 65535LL * 32;
    fill_pads3_kernel<<<(int)b, 256, 0, s>>>(m.K, inlet[0], inlet[1], inlet[2], inlet[3], inlet[4], M, ncell, pad_cell,
                                            pad_src, npad);
}

int cell3d_blocks(int device) {
    static bool attr_set = false;
    if (!attr_set) {
        cudaFuncSetAttribute(cell3d_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(Warp3) * kW3Warps));
        attr_set = true;
    }
    int sms = 0, per_sm = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cell3d_kernel, kW3Warps * 32, sizeof(Warp3) * kW3Warps);
    return sms * (per_sm < 1 ? 1 : per_sm);
}

void launch_cell3d(const Model& m, const Geometry3& g, const double* Min, double* Mout, DevStats* st,
                   unsigned long long* work, int blocks, cudaStream_t s) {
    cell3d_kernel<<<blocks, kW3Warps * 32, sizeof(Warp3) * kW3Warps, s>>>(m, g, Min, Mout, st, work);
}

}  // namespace lbm
