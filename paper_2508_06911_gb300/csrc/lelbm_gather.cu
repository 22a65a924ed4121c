// Deterministic moment streaming (Eq. IIE3) for the FP64 2D path: a gather instead of a
// scatter.  The cell kernel leaves every cell's converged multipliers (after the polishing
// update, or of the fallback it took) in Model::det_lam; this kernel then computes, for
// each target cell, the sum of T_N(c_i) rho f'_i and T_N(c_i) rho K RT g'_i over every source
// cell whose stencil point c_i lands on the target -- a level-0 point exactly at x + c_i, a
// refined child by its cloud-in-cell share -- in a fixed order of sources and points.  No
// atomics: the result does not depend on the order in which blocks run, so two runs give
// the same bits.
//
// A block owns a 32 x 8 tile of targets.  Source cells within the reach H of the tile (H =
// the largest |u_a| + R_ac + 1/2 of the step, plus one cell for cloud-in-cell shares) are
// staged through shared memory two rows by 64 columns at a time: their macroscopic variables
// (Eq. IIB6), stencil parameters (Eq. IIC6, IIC9) and multipliers; each thread then walks
// the staged sources inside its own window.  Periodic axes wrap the source coordinate, so a
// source that reaches a target through several images contributes once per image, as in
// the scatter.
//
// FP64 instructions bound the kernel.  Most pairs in the window (2 H + 1)^2 are no points of the
// source's set, so membership is decided in FP32 on offsets from floor(u) (as in RowTable::build: only
// a test closer to its threshold than FP32 resolves goes to FP64); a pair that is a point takes 45
// FP64 operations, its exponentials being integer code (exp_int).  384 x 320 step, cell kernel
// included: 7.1 ms with FP64 tests and library exponentials here, 3.5 ms so.
#include <cuda_runtime.h>

#include <cstdint>

#include "lelbm_device.cuh"
#include "lelbm_fp64.cuh"
#include "lelbm_internal.h"

namespace lbm {

constexpr int kGTX = 32, kGTY = 8;  // target tile
constexpr int kGRB = 2, kGCW = 64;  // staged chunk: source rows x columns

struct GSrc {
    double ux, uy, inv_sig, rr2, mf, mg;  // mf = rho, mg = rho K RT (Eq. IIE3)
    double lf[10], lg[6];
    float fx, fy;  // u - floor(u)
    int bx, by;    // floor(u)
    int R, Nr, ok;
};

// Adds the moment fractions of one population point c (lattice frame, relative to its
// source) of weight w (volume dC times cloud-in-cell share), to acc (Eq. IIE3).
__device__ __forceinline__ void gather_point(const GSrc& s, bool has_g, double cx, double cy, double w, double* acc) {
    const double x = (cx - s.ux) * s.inv_sig, y = (cy - s.uy) * s.inv_sig;
    double cf[4], cg[3];
    row_coeffs<2>(s.lf, s.lg, y, cf, cg);
    const double mf = w * s.mf * exp_int(-(((cf[3] * x + cf[2]) * x + cf[1]) * x + cf[0]));
    const double mg = has_g ? w * s.mg * exp_int(-((cg[2] * x + cg[1]) * x + cg[0])) : 0.0;
    double v[11];
    stored_moments<2, true, true>(cx, cy, mf, mg, v);
#pragma unroll
    for (int k = 0; k < 11; k++) acc[k] += v[k];
}

// Is the lattice point at (dx, dy) within distance^2 thr of the source's u (inclusive)?
__device__ __forceinline__ bool gather_inside(const GSrc& s, int dx, int dy, double thr, float thr32) {
    const float ex = (float)(dx - s.bx) - s.fx, ey = (float)(dy - s.by) - s.fy;
    const float v = fmaf(ex, ex, ey * ey), mg = 1e-3f + 1e-5f * thr32;
    if (v < thr32 - mg) return true;
    if (v > thr32 + mg) return false;
    const double a = __dsub_rn((double)dx, s.ux), b = __dsub_rn((double)dy, s.uy);  // as Stencil::dist2
    return __dadd_rn(__dadd_rn(0.0, __dmul_rn(a, a)), __dmul_rn(b, b)) <= thr;
}

__global__ void __launch_bounds__(kGTX * kGTY) gather2d_kernel(const __grid_constant__ Model m,
                                                               const __grid_constant__ Geometry g,
                                                               const double* __restrict__ Min, double* __restrict__ Mout,
                                                               DevStats* stats) {
    __shared__ GSrc src[kGRB][kGCW];
    const int H = *m.det_halo;
    const bool has_g = m.K > 0.0;
    const int lx = threadIdx.x % kGTX, ly = threadIdx.x / kGTX;
    const int tx0 = blockIdx.x * kGTX, ty0 = blockIdx.y * kGTY;
    const int tx = tx0 + lx, ty = ty0 + ly;
    // interior targets receive; pads and cells off the array do not (Sec. III)
    const int px = g.periodic[0] ? 0 : g.pad, py = g.periodic[1] ? 0 : g.pad;
    const bool recv = tx >= px && tx < px + g.nx && ty >= py && ty < py + g.ny;
    double acc[11];
#pragma unroll
    for (int k = 0; k < 11; k++) acc[k] = 0.0;
    unsigned long long n_dep = 0;
    double rad2[5];
#pragma unroll
    for (int L = 0; L < 5; L++) {
        rad2[L] = m.rad2[L];
    }
    const int sx_lo = tx0 - H, sx_hi = tx0 + kGTX - 1 + H;
    const int sy_lo = ty0 - H, sy_hi = ty0 + kGTY - 1 + H;
    for (int sy0 = sy_lo; sy0 <= sy_hi; sy0 += kGRB) {
        for (int sx0 = sx_lo; sx0 <= sx_hi; sx0 += kGCW) {
            __syncthreads();
            for (int e = threadIdx.x; e < kGRB * kGCW; e += blockDim.x) {
                const int r = e / kGCW, k = e - r * kGCW;
                int sx = sx0 + k, sy = sy0 + r;
                GSrc& s = src[r][k];
                s.ok = 0;
                if (sx > sx_hi || sy > sy_hi) continue;
                if (g.periodic[0]) {
                    sx %= g.NX;
                    if (sx < 0) sx += g.NX;
                } else if (sx < 0 || sx >= g.NX) {
                    continue;
                }
                if (g.periodic[1]) {
                    sy %= g.NY;
                    if (sy < 0) sy += g.NY;
                } else if (sy < 0 || sy >= g.NY) {
                    continue;
                }
                const long long cell = (long long)sy * g.NX + sx;
                double M[11];
#pragma unroll
                for (int i = 0; i < 11; i++) M[i] = Min[i * g.ncell + cell];
                CellState<2> c;
                double RT, usq;
                if (!cell_macros<2>(M, m, c.rho, c.u, RT, usq)) continue;
                c.RT = RT;
                c.sig = sqrt(RT);
                c.inv_sig = recip64(c.sig);
                Stencil<2> st;
                st.init(c, m);
                s.ux = c.u[0];
                s.uy = c.u[1];
                s.bx = (int)floor(c.u[0]);
                s.by = (int)floor(c.u[1]);
                s.fx = (float)(c.u[0] - (double)s.bx);
                s.fy = (float)(c.u[1] - (double)s.by);
                s.inv_sig = c.inv_sig;
                s.rr2 = st.rr2;
                s.mf = c.rho;
                s.mg = c.rho * m.K * c.RT;
                s.R = st.R;
                s.Nr = st.Nr;
#pragma unroll
                for (int j = 0; j < 10; j++) s.lf[j] = m.det_lam[(long long)j * g.ncell + cell];
#pragma unroll
                for (int j = 0; j < 6; j++) s.lg[j] = m.det_lam[(long long)(10 + j) * g.ncell + cell];
                s.ok = 1;
            }
            __syncthreads();
            if (!recv) continue;
            // the staged sources inside this target's window |t - s| <= H, in order
            for (int r = 0; r < kGRB; r++) {
                const int dy = ty - (sy0 + r);
                if (dy < -H || dy > H || sy0 + r > sy_hi) continue;
                const int k0 = max(0, tx - H - sx0), k1 = min(kGCW - 1, tx + H - sx0);
                for (int k = k0; k <= k1; k++) {
                    const GSrc& s = src[r][k];
                    if (!s.ok) continue;
                    const int dx = tx - (sx0 + k);  // the point c = (dx, dy) of the source
                    const float ex = (float)(dx - s.bx) - s.fx, ey = (float)(dy - s.by) - s.fy;
                    const float reach = (float)s.R + 2.6f;
                    if (ex * ex + ey * ey > reach * reach) continue;
                    const float rr = (float)s.R + 0.5f, rr32 = rr * rr, split32 = (float)rad2[1];
                    // a level-0 point that is not split lands exactly on the target
                    if (gather_inside(s, dx, dy, s.rr2, rr32) &&
                        (s.Nr == 0 || !gather_inside(s, dx, dy, rad2[1], split32))) {
                        gather_point(s, has_g, widen((float)dx), widen((float)dy), 1.0, acc);
                        n_dep++;
                    }
                    // children of split points whose cloud-in-cell share reaches the target
                    const float near = sqrtf(split32) + 1.6f;
                    if (s.Nr == 0 || fabsf(ex) > near || fabsf(ey) > near) continue;
#pragma unroll 1
                    for (int py0 = dy - 1; py0 <= dy + 1; py0++) {
#pragma unroll 1
                        for (int px0 = dx - 1; px0 <= dx + 1; px0++) {
                            if (!gather_inside(s, px0, py0, s.rr2, rr32) ||
                                !gather_inside(s, px0, py0, rad2[1], split32))
                                continue;
                            if (s.Nr == 1) {  // four children at +-1/4
#pragma unroll 1
                                for (int k = 0; k < 4; k++) {
                                    const float cx = (float)px0 + ((k & 1) ? 0.25f : -0.25f);
                                    const float cy = (float)py0 + ((k & 2) ? 0.25f : -0.25f);
                                    const float wx = 1.f - fabsf(cx - (float)dx), wy = 1.f - fabsf(cy - (float)dy);
                                    if (wx > 0.f && wy > 0.f) {
                                        gather_point(s, has_g, widen(cx), widen(cy), widen(0.25f * wx * wy), acc);
                                        n_dep++;
                                    }
                                }
                                continue;
                            }
                            Stencil<2> st;
                            st.u[0] = s.ux;
                            st.u[1] = s.uy;
                            st.rr2 = s.rr2;
                            st.R = s.R;
                            st.Nr = s.Nr;
#pragma unroll
                            for (int L = 0; L < 5; L++) st.rad2[L] = rad2[L];
                            const double c0[2] = {(double)px0, (double)py0};
                            auto leaf = [&](const double* cl, double dC) {
                                const double wx = 1.0 - fabs(cl[0] - (double)dx), wy = 1.0 - fabs(cl[1] - (double)dy);
                                if (wx > 0.0 && wy > 0.0) {
                                    gather_point(s, has_g, cl[0], cl[1], dC * (wx * wy), acc);
                                    n_dep++;
                                }
                            };
                            st.visit0(c0, leaf);
                        }
                    }
                }
            }
        }
    }
    if (tx < g.NX && ty < g.NY) {
        const long long t = (long long)ty * g.NX + tx;
#pragma unroll
        for (int k = 0; k < 11; k++) Mout[k * g.ncell + t] = recv ? acc[k] : 0.0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n_dep += __shfl_xor_sync(0xffffffffu, n_dep, o);
    if ((threadIdx.x & 31) == 0 && n_dep) atomicAdd(&stats->points_ms, n_dep);
}

void launch_gather2d(const Model& m, const Geometry& g, const double* Min, double* Mout, DevStats* st,
                     cudaStream_t s) {
    const dim3 grid((g.NX + kGTX - 1) / kGTX, (g.NY + kGTY - 1) / kGTY);
    gather2d_kernel<<<grid, kGTX * kGTY, 0, s>>>(m, g, Min, Mout, st);
}

}  // namespace lbm
