// Allocation-free time step (lelbm_step_noalloc in include/lelbm.h).
//
// Who needs it: callers that must not allocate device memory.  Examples:
//   - an application that owns all device memory through its own pool or a
//     fixed memory budget;
//   - code on a latency-critical path, where cudaFree synchronises the whole
//     device and cudaMalloc can fail or fragment mid-run.
// Such a caller passes the input and output moment buffers it already owns.
// Everything else the step needs (counters, the 1D instance table) lives in
// the file-scope array g_noalloc_scratch below.
//
// The array is a static __device__ variable.  Every GPU on which the library
// is loaded holds its 512 KiB until the process exits.  All calls share it
// and it keeps the last call's contents, so every call clears what must start
// at zero.  Calls whose work overlaps on the GPU (for example on two streams)
// race on it.
//
// In host code the name g_noalloc_scratch is only a host-side stand-in, not a
// device address.  The device address comes from cudaGetSymbolAddress, taken
// once per device with that device current (on the first call there).
// Device code uses the array directly.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>

#include "../../include/lelbm.h"
#include "lelbm_step.cuh"

namespace lbm {
namespace {

constexpr int kMaxInst = LELBM_NOALLOC_MAX_INSTANCES;
// byte layout of the scratch array
constexpr size_t kStatsOff = 0;
constexpr size_t kLenOff = 1024;                                  // int[kMaxInst]
constexpr size_t kPadOff = kLenOff + sizeof(int) * kMaxInst;      // int[kMaxInst]
constexpr size_t kBlkOff = kPadOff + sizeof(int) * kMaxInst;      // long long[kMaxInst + 1]
constexpr size_t kScratchBytes = kBlkOff + sizeof(long long) * (kMaxInst + 1);
static_assert(sizeof(DevStats) <= kLenOff, "counters overflow their slot");
static_assert(kScratchBytes <= 512 * 1024, "scratch larger than stated");

static __device__ __align__(256) unsigned char g_noalloc_scratch[512 * 1024];

__device__ __forceinline__ DevStats* scratch_stats() {
    return reinterpret_cast<DevStats*>(g_noalloc_scratch + kStatsOff);
}
__device__ __forceinline__ const int* scratch_len() {
    return reinterpret_cast<const int*>(g_noalloc_scratch + kLenOff);
}
__device__ __forceinline__ const int* scratch_pad() {
    return reinterpret_cast<const int*>(g_noalloc_scratch + kPadOff);
}
__device__ __forceinline__ long long* scratch_blk() {
    return reinterpret_cast<long long*>(g_noalloc_scratch + kBlkOff);
}

// Geometry of the step, passed by value.
struct Topo {
    int D;
    long long ncell;
    int NX, NY;          // 2D padded sizes
    int nx, ny, pad;     // 2D interior and pad
    int periodic[2];
    int bc[4];
    int n_inst;          // 1D instances
    int uniform_pad;     // 1D: pad of every instance, or -1 to read the per-instance table
    double inlet[4];
};

// Exclusive prefix sum of the 1D block sizes (pads + interior) into blk[0..n].
__global__ void instance_scan_kernel(int n, int periodic, int uniform_pad) {
    __shared__ long long part[1024];
    const int* len = scratch_len();
    const int* pad = scratch_pad();
    long long* blk = scratch_blk();
    const int per = (n + blockDim.x - 1) / blockDim.x;
    const int b0 = threadIdx.x * per;
    long long s = 0;
    for (int b = b0; b < n && b < b0 + per; b++)
        s += len[b] + (periodic ? 0 : 2LL * (uniform_pad >= 0 ? uniform_pad : pad[b]));
    part[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long acc = 0;
        for (int i = 0; i < (int)blockDim.x; i++) {
            const long long v = part[i];
            part[i] = acc;
            acc += v;
        }
    }
    __syncthreads();
    long long acc = part[threadIdx.x];
    for (int b = b0; b < n && b < b0 + per; b++) {
        blk[b] = acc;
        acc += len[b] + (periodic ? 0 : 2LL * (uniform_pad >= 0 ? uniform_pad : pad[b]));
    }
    if (b0 < n && b0 + per >= n) blk[n] = acc;
}

__device__ __forceinline__ int find_instance(const long long* blk, int n, long long cell) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (blk[mid] <= cell)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

template <int D>
__global__ void __launch_bounds__(128) noalloc_cell_kernel(Model m, Topo t, const double* __restrict__ Min,
                                                           double* Mout) {
    constexpr int NM = Dim<D>::NM, NF = Dim<D>::NF, NG = Dim<D>::NG;
    DevStats* stats = scratch_stats();
    const long long* blk = scratch_blk();
    const int* len = scratch_len();
    const int* pads = scratch_pad();
    __shared__ BlockCounters bc;
    __shared__ ThreadCounters s_tc[128];
    __shared__ double s_con[128][NF + NG];                                  // constraints of each thread's cell
    __shared__ char2 s_rows[D == 2 ? 128 : 1][D == 2 ? kRowsMax : 1];       // and its row table
    double* conF = s_con[threadIdx.x];
    double* conG = conF + NF;
    counters_init(bc);
    s_tc[threadIdx.x] = ThreadCounters{0, 0, 0, 0, 0, 0, {0, 0.0, 0, 0}, 0, 0, 0};
    ThreadCounters& tc = s_tc[threadIdx.x];
    __syncthreads();
    Geometry g{};  // what the landing rules read (no walls; the 1D instance comes with the cell)
    g.D = D;
    g.NX = t.NX;
    g.NY = t.NY;
    g.ncell = t.ncell;
    g.nx = t.nx;
    g.ny = t.ny;
    g.pad = t.pad;
    g.periodic[0] = t.periodic[0];
    g.periodic[1] = t.periodic[1];

    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x; cell < t.ncell; cell += stride) {
        // where this cell's moments come from (Sec. III.A fill, done on the fly); the same
        // rules as fill_pads_kernel and the pad-source lists the handle builds at create
        long long src = cell;
        bool inflow = false;
        long long lo = 0;
        int n = 0, ix = 0, iy = 0;
        if constexpr (D == 1) {
            const int b = find_instance(blk, t.n_inst, cell);
            const int p = t.periodic[0] ? 0 : (t.uniform_pad >= 0 ? t.uniform_pad : pads[b]);
            n = len[b];
            lo = blk[b] + p;
            if (cell < lo) {
                inflow = t.bc[0] == LELBM_BC_INFLOW;
                src = lo;
            } else if (cell >= lo + n) {
                inflow = t.bc[1] == LELBM_BC_INFLOW;
                src = lo + n - 1;
            }
        } else {
            iy = (int)(cell / t.NX);
            ix = (int)(cell - (long long)iy * t.NX);
            const int px = t.periodic[0] ? 0 : t.pad, py = t.periodic[1] ? 0 : t.pad;
            const bool inx = ix >= px && ix < px + t.nx, iny = iy >= py && iy < py + t.ny;
            if (!(inx && iny)) {
                inflow = (ix < px && t.bc[0] == LELBM_BC_INFLOW) || (ix >= px + t.nx && t.bc[1] == LELBM_BC_INFLOW) ||
                         (iy < py && t.bc[2] == LELBM_BC_INFLOW) || (iy >= py + t.ny && t.bc[3] == LELBM_BC_INFLOW);
                const int sx = ix < px ? px : (ix >= px + t.nx ? px + t.nx - 1 : ix);
                const int sy = iy < py ? py : (iy >= py + t.ny ? py + t.ny - 1 : iy);
                src = (long long)sy * t.NX + sx;
            }
        }
        double M[NM];
        if (inflow) {
            const double uin[2] = {t.inlet[1], t.inlet[2]};
            eq_moments<D>(m.K, t.inlet[0], uin, t.inlet[3], M);
        } else {
#pragma unroll
            for (int i = 0; i < NM; i++) M[i] = Min[i * t.ncell + src];
        }
        CellState<D> c;
        collide<D>(M, m, c);  // as prepare_cell (lelbm_step.cuh) on the FP64 path
        if (!c.ok) {
            atomicAdd(&bc.fmx, 1ull);
            atomicMin(&stats->first_fail, (unsigned long long)cell);
            continue;
        }
        tc.cells++;
        Stencil<D> st;
        st.init(c, m);
        double lf[NF], lg[NG];
        maxwell_start_newton<D, NF, NG>(c.RT, lf, lg);
#pragma unroll
        for (int j = 0; j < NF; j++) conF[j] = c.cf[j];
#pragma unroll
        for (int j = 0; j < NG; j++) conG[j] = c.cg[j];
        RowTable<D> tab;
        tab.build(c, st, s_rows[D == 2 ? threadIdx.x : 0]);
        Absorbed none;  // no walls here
        fp64_cell<D>(m, g, nullptr, Mout, stats, CellPlace{cell, lo, n, ix, iy}, bc, tc, conF, conG, c, st, tab, lf, lg,
                     false, none);
    }
    counters_flush(bc, tc, stats);
}

// Device address of g_noalloc_scratch, looked up once per device.
std::mutex g_addr_mutex;
unsigned char* g_addr[64] = {};

}  // namespace
}  // namespace lbm

using namespace lbm;

extern "C" int lelbm_step_noalloc(const lelbm_params* p, const double* m_in, double* m_out, lelbm_stats* stats) {
    if (!p || !m_in || !m_out) return LELBM_E_INVAL;
    if (p->dims != 1 && p->dims != 2) return LELBM_E_INVAL;
    if (p->solid || p->precision != LELBM_FP64 || p->deterministic) return LELBM_E_INVAL;
    if (p->nx < 1 || p->ny < 1 || (p->dims == 1 && p->ny != 1)) return LELBM_E_INVAL;
    if (!(p->K >= 0.0) || !(p->nu_shear >= 0.0) || !(p->prandtl > 0.0) || !(p->tol > 0.0)) return LELBM_E_INVAL;
    if (p->max_newton < 1 || p->max_newton > 60 || p->max_refine < 0 || p->max_refine > 4) return LELBM_E_INVAL;
    for (int a = 0; a < p->dims; a++) {
        const int l = p->bc[2 * a], r = p->bc[2 * a + 1];
        if (l < 0 || l > 2 || r < 0 || r > 2) return LELBM_E_INVAL;
        if ((l == LELBM_BC_PERIODIC) != (r == LELBM_BC_PERIODIC)) return LELBM_E_INVAL;
        if (l != LELBM_BC_PERIODIC && p->dims == 2 && p->pad < 1) return LELBM_E_INVAL;
    }
    const int nb = (p->dims == 1 && p->n_batch > 1) ? p->n_batch : 1;
    if (nb > kMaxInst) return LELBM_E_INVAL;  // beyond the scratch array's capacity
    const bool periodic_x = p->bc[0] == LELBM_BC_PERIODIC;
    if (p->dims == 1 && !periodic_x && !(nb > 1 && p->pads) && p->pad < 1) return LELBM_E_INVAL;
    if (nb > 1 && !p->lengths) return LELBM_E_INVAL;

    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LELBM_E_CUDA;
    unsigned char* base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_addr_mutex);
        if (!g_addr[dev]) {
            void* ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess) return LELBM_E_CUDA;
            g_addr[dev] = static_cast<unsigned char*>(ptr);
        }
        base = g_addr[dev];
    }
    cudaStream_t s = (cudaStream_t)p->stream;

    Model m{};
    m.K = p->K;
    m.nu_s = p->nu_shear;
    m.nu_b = p->nu_bulk;
    m.Pr = p->prandtl;
    m.limiter = p->limiter;
    m.n_conf = p->n_conform;
    m.r_min = p->r_min;
    m.refine_div = p->refine_div;
    m.refine_rad = p->refine_rad;
    m.max_refine = p->max_refine;
    m.tol = p->tol;
    m.max_iter = p->max_newton;
    set_derived_params(m, p->dims);

    Topo t{};
    t.D = p->dims;
    t.periodic[0] = periodic_x;
    t.periodic[1] = p->dims == 2 ? p->bc[2] == LELBM_BC_PERIODIC : 1;
    for (int i = 0; i < 4; i++) {
        t.bc[i] = p->bc[i];
        t.inlet[i] = p->inlet[i];
    }
    t.n_inst = nb;
    long long ncell = 0;
    if (p->dims == 1) {
        // instance lengths and pads go straight from the caller's host arrays into the scratch
        if (nb > 1) {
            if (cudaMemcpyAsync(base + kLenOff, p->lengths, sizeof(int) * nb, cudaMemcpyHostToDevice, s) != cudaSuccess)
                return LELBM_E_CUDA;
        } else {
            if (cudaMemcpyAsync(base + kLenOff, &p->nx, sizeof(int), cudaMemcpyHostToDevice, s) != cudaSuccess)
                return LELBM_E_CUDA;
        }
        const int* pads_src = (nb > 1 && p->pads) ? p->pads : nullptr;
        if (pads_src) {
            for (int b = 0; b < nb; b++)
                if (!periodic_x && pads_src[b] < 1) return LELBM_E_INVAL;
            if (cudaMemcpyAsync(base + kPadOff, pads_src, sizeof(int) * nb, cudaMemcpyHostToDevice, s) != cudaSuccess)
                return LELBM_E_CUDA;
        }
        t.uniform_pad = pads_src ? -1 : p->pad;
        for (int b = 0; b < nb; b++) {
            const int n = nb > 1 ? p->lengths[b] : p->nx;
            if (n < 1) return LELBM_E_INVAL;
            ncell += n + (periodic_x ? 0 : 2LL * (pads_src ? pads_src[b] : p->pad));
        }
        instance_scan_kernel<<<1, 1024, 0, s>>>(nb, periodic_x ? 1 : 0, t.uniform_pad);
    } else {
        const int px = t.periodic[0] ? 0 : p->pad, py = t.periodic[1] ? 0 : p->pad;
        t.NX = p->nx + 2 * px;
        t.NY = p->ny + 2 * py;
        t.nx = p->nx;
        t.ny = p->ny;
        t.pad = (t.periodic[0] && t.periodic[1]) ? 0 : p->pad;
        ncell = (long long)t.NX * t.NY;
    }
    t.ncell = ncell;

    // counters start at zero (first_fail at its "none" value); the output is accumulated into
    DevStats z;
    std::memset(&z, 0, sizeof z);
    z.first_fail = ~0ull;
    if (cudaMemcpyAsync(base + kStatsOff, &z, sizeof z, cudaMemcpyHostToDevice, s) != cudaSuccess) return LELBM_E_CUDA;
    const int nm = p->dims == 1 ? 6 : 11;
    if (cudaMemsetAsync(m_out, 0, sizeof(double) * nm * ncell, s) != cudaSuccess) return LELBM_E_CUDA;

    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long need = (ncell + 127) / 128;
    long long cap = 8LL * (sms > 0 ? sms : 1);
    const int blocks = (int)(need < cap ? need : cap);
    if (p->dims == 1)
        noalloc_cell_kernel<1><<<blocks, 128, 0, s>>>(m, t, m_in, m_out);
    else
        noalloc_cell_kernel<2><<<blocks, 128, 0, s>>>(m, t, m_in, m_out);
    if (cudaGetLastError() != cudaSuccess) return LELBM_E_CUDA;

    if (stats) {
        DevStats d;
        if (cudaMemcpyAsync(&d, base + kStatsOff, sizeof d, cudaMemcpyDeviceToHost, s) != cudaSuccess) return LELBM_E_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return LELBM_E_CUDA;
        std::memset(stats, 0, sizeof *stats);
        stats->steps = 1;
        stats->cells = (long long)d.cells;
        for (int i = 0; i < 64; i++) stats->newton_hist[i] = (long long)d.newton_hist[i];
        stats->fallback_eq = (long long)d.fallback_eq;
        stats->fallback_mx = (long long)d.fallback_mx;
        stats->q_max = (long long)d.q_max;
        double dm;
        std::memcpy(&dm, &d.disp_max_bits, sizeof dm);
        stats->disp_max = dm;
        stats->first_fail_cell = d.first_fail == ~0ull ? -1 : (long long)d.first_fail;
        stats->points_f = (long long)d.points_f;
        stats->points_g = (long long)d.points_g;
        stats->points_ms = (long long)d.points_ms;
        if (d.fallback_mx) return LELBM_E_EPR;
    }
    return LELBM_OK;
}
