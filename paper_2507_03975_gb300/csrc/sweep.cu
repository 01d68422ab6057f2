// Kinetic step of SI / GSIS: the first-order-upwind discrete-ordinate sweep
// (Sec. 4.1, Eqs. (RTE_d), (Iij) with psi = 0, Eq. (RTE_SI) steady) and its
// angular moments (Eqs. (def_rho), (def_F), (RTE_M0)), plus the per-problem
// set-up of the coefficients every iteration reuses.
//
// Sweep layout.  Work unit = (direction s, band of 32 rows).  A warp owns one
// unit: lane l owns row 32*band + l (counted from the upwind wall) and walks
// the row from the upwind wall, one cell per step, lane l lagging lane l-1 by
// one step, so the upwind south value is the value lane l-1 produced one step
// earlier (one warp shuffle) and the upwind west value is the lane's own
// previous result (a register).  Lane 0 takes its south value from the band
// below (its last-row results, handed over value by value through a global
// row whose slots read "unwritten" until stored) or from the inflow on the
// first band.  Each compute warp is paired with helper warps that stage the
// cell data of the coming steps in shared memory, fetch the south values and
// write the results out, so the compute warp touches global memory only to
// hand its last row on.
// Every wait is bounded and reports kErrTimeout instead of hanging.
//
// All intensities of the last sweep stay in HBM as I[s][cell] (needed by the
// moment reduction, the pseudo-time delta form of Sec. 4.3 and the final
// second moment).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cstring>
#include <map>
#include <mutex>
#include <type_traits>
#include <vector>

#include "divide.cuh"
#include "gsis_internal.cuh"
#include "moments_fixed.cuh"

namespace gsis {

namespace {

constexpr double kInvFourPi = 0.079577471545947667884441881686257;   // 1 / (4 pi)

// --------------------------------------------------------------- set-up
// |mu_s|/dx_i and |eta_s|/dy_j per sorted direction (both precisions).
__global__ void coef_kernel(int nx, int ny, int K, const double* __restrict__ dx,
                            const double* __restrict__ dy, const double* __restrict__ qmu,
                            const double* __restrict__ qeta, double* acoef, double* bcoef,
                            float* acoef_f, float* bcoef_f)
{
    const int tot_a = K * nx, tot = K * (nx + ny);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += gridDim.x * blockDim.x) {
        if (t < tot_a) {
            const int s = t / nx, i = t - s * nx;
            const double v = fabs(qmu[s]) / dx[i];
            acoef[t] = v;
            if (acoef_f) acoef_f[t] = (float)v;
        } else {
            const int u = t - tot_a;
            const int s = u / ny, j = u - s * ny;
            const double v = fabs(qeta[s]) / dy[j];
            bcoef[u] = v;
            if (bcoef_f) bcoef_f[u] = (float)v;
        }
    }
}

// Per cell: sigma_t, pseudo-time shift (Eqs. (cfl_pse), (tau_pse),
// dx_ref = min(dx_i, dy_j)), the finite-volume synthetic operator
// (Eqs. (elem_mtx_M), (Gamma_ij_com2) on the Cartesian mesh:
// Gamma = 2 / (3 (sigma_i h_i + sigma_j h_j)); boundary
// beta = 2/(3 sigma_i h_i) + 1/4 from Eq. (macro_bc_delta_flux)), input checks
// (opacities, sources and inflow finite; opacities non-negative).  Bound by
// the FP64 pipe: thirteen divisions a cell.  synth = 0 (a kinetic step alone,
// source iteration): no synthetic operator and no HoT weights, and with no
// pseudo-time and no intensity gradient no division is left (256x256:
// 26.7 -> 4.5 us).
__global__ void cell_setup_kernel(int nx, int ny, const double* __restrict__ dx,
                                  const double* __restrict__ dy, const double* __restrict__ sa,
                                  const double* __restrict__ ss, const double* __restrict__ q,
                                  const double* __restrict__ inflow, int n_inflow,
                                  double shift0, double cfl_p, double beta, double* sigt, float* sigt_f,
                                  double* shift, float* shift_f, int synth, double* diag, double* cx,
                                  double* cy, double* hw, double* bface, double* gw, float* gw_f,
                                  float* sigt_d, int* err)
{
    const int N = nx * ny;
    if (inflow)
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_inflow; t += gridDim.x * blockDim.x)
            if (!isfinite(inflow[t])) atomicOr(err, kErrBadInput);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const int j = c / nx, i = c - j * nx;
        const double a = sa[c], s = ss[c], st = a + s;
        if (!(a >= 0.0) || !(s >= 0.0) || !(st > 0.0) || !isfinite(st) || !isfinite(q[c]))
            atomicOr(err, kErrBadInput);
        sigt[c] = st;
        if (sigt_f) sigt_f[c] = (float)st;
        const double hx = dx[i], hy = dy[j];
        // neighbour optical distances |sigma_i r^L - sigma_j r^R|
        double th = 0.0;
        double gE = 0.0, gW = 0.0, gN = 0.0, gS = 0.0;
        const bool dist = synth || beta > 0.0;
        if (dist && i + 1 < nx) {
            const double o = 0.5 * (st * hx + (sa[c + 1] + ss[c + 1]) * dx[i + 1]);
            th = fmax(th, o);
            if (synth) gE = 1.0 / (3.0 * o);
        }
        if (dist && i > 0) {
            const double o = 0.5 * (st * hx + (sa[c - 1] + ss[c - 1]) * dx[i - 1]);
            th = fmax(th, o);
            if (synth) gW = 1.0 / (3.0 * o);
        }
        if (dist && j + 1 < ny) {
            const double o = 0.5 * (st * hy + (sa[c + nx] + ss[c + nx]) * dy[j + 1]);
            th = fmax(th, o);
            if (synth) gN = 1.0 / (3.0 * o);
        }
        if (dist && j > 0) {
            const double o = 0.5 * (st * hy + (sa[c - nx] + ss[c - nx]) * dy[j - 1]);
            th = fmax(th, o);
            if (synth) gS = 1.0 / (3.0 * o);
        }
        const double ref = fmin(hx, hy);
        double sh = shift0;   // 1/(c dt) of a time step (0 when steady)
        if (cfl_p > 0.0) sh += 1.0 / (cfl_p * ref);
        if (beta > 0.0) sh += th / (beta * ref);
        shift[c] = sh;
        if (shift_f) shift_f[c] = (float)sh;
        if (sigt_d) sigt_d[c] = (float)(st + sh);
        if (!synth && !gw) continue;
        // D = V sigma_a + sum_int A Gamma + sum_bnd A beta
        double d = hx * hy * a + hy * (gE + gW) + hx * (gN + gS);
        const double bx = 2.0 / (3.0 * st * hx) + 0.25, by = 2.0 / (3.0 * st * hy) + 0.25;
        if (i == 0) d += hy * bx;
        if (i == nx - 1) d += hy * bx;
        if (j == 0) d += hx * by;
        if (j == ny - 1) d += hx * by;
        diag[c] = d;
        cx[c] = hy * gE;
        cy[c] = hx * gN;
        // adaptive least-squares gradient on the Cartesian mesh (Eqs. (shifted_j),
        // (new_vector), (LSF_mdf)): G_x = sum_{E,W} d_j (rho_j - rho_i) / sum d_j^2
        // with d_E = +(hx/2 + (sigma_E/sigma_i) dx_E/2), d_W = -(...); the weights
        // d_j / sum d^2 carry the 1/(3 sigma_t) of the high-order terms (Eq. (GSIS_HoT))
        {
            double dE = 0.0, dW = 0.0, dN = 0.0, dS = 0.0;
            if (i + 1 < nx) dE = 0.5 * hx + ((sa[c + 1] + ss[c + 1]) / st) * 0.5 * dx[i + 1];
            if (i > 0) dW = -(0.5 * hx + ((sa[c - 1] + ss[c - 1]) / st) * 0.5 * dx[i - 1]);
            if (j + 1 < ny) dN = 0.5 * hy + ((sa[c + nx] + ss[c + nx]) / st) * 0.5 * dy[j + 1];
            if (j > 0) dS = -(0.5 * hy + ((sa[c - nx] + ss[c - nx]) / st) * 0.5 * dy[j - 1]);
            const double inv3s = 1.0 / (3.0 * st);
            const double sx = dE * dE + dW * dW, sy = dN * dN + dS * dS;
            const double fx = sx > 0.0 ? inv3s / sx : 0.0, fy = sy > 0.0 ? inv3s / sy : 0.0;
            hw[c] = dE * fx;
            hw[N + c] = dW * fx;
            hw[2 * N + c] = dN * fy;
            hw[3 * N + c] = dS * fy;
            if (gw) {   // the same least-squares gradient for the intensities (no 1/(3 sigma_t))
                const double gx = sx > 0.0 ? 1.0 / sx : 0.0, gy = sy > 0.0 ? 1.0 / sy : 0.0;
                const double g4[4] = {dE * gx, dW * gx, dN * gy, dS * gy};
                for (int t = 0; t < 4; ++t) {
                    gw[(size_t)t * N + c] = g4[t];
                    if (gw_f) gw_f[(size_t)t * N + c] = (float)g4[t];
                }
            }
        }
        // boundary faces: area * beta (Eq. (macro_bc_delta_flux)), faces W, E, S, N
        if (i == 0) bface[j] = hy * bx;
        if (i == nx - 1) bface[ny + j] = hy * bx;
        if (j == 0) bface[2 * ny + i] = hx * by;
        if (j == ny - 1) bface[2 * ny + nx + i] = hx * by;
    }
}

// 1 / (sigma_t + shift + |mu|/dx + |eta|/dy) in sweep order (FP64 sweep).
// Directions with the same |mu| and |eta| (the four reflections in every
// level-symmetric set) share the value at a cell: the division, which bounds
// this kernel, is done once, for the first of them (rrep), and stored in each
// one's own order along the list rnext.  A block forms one band's values on
// COLS columns in shared memory (columns -31 .. nx + 30: those outside the
// mesh are zero, as are rows beyond it) and writes each order's diagonals
// from there, a step's 32 lanes at a time: written straight from the cells,
// two of the four orders scattered each store over 32 rows of the table.  A
// pitch of COLS makes the diagonals conflict-free (stride COLS -+ 1, odd).
// 256^2 S12: 116 us before the shared division, 58 before the tiles, 44 now;
// 1024^2 S16: 2.87, 1.34, 0.84 ms (its divisions and sums take 0.55 ms of the
// FP64 pipe); 64^2 S8 7.4 us with 16 columns (64: 14, two blocks per three SMs).
template <int COLS>
__global__ void __launch_bounds__(256)
recip_kernel(int nx, int ny, int nb, const int* __restrict__ rrep, const int* __restrict__ rnext,
             const double* __restrict__ qmu, const double* __restrict__ qeta, const double* __restrict__ acoef,
             const double* __restrict__ bcoef, const double* __restrict__ sigt, const double* __restrict__ shift,
             double* rsw)
{
    __shared__ double v[32 * COLS];
    const int ns = nx + 31, band = blockIdx.y, s = rrep[blockIdx.z];
    const int c0 = (int)blockIdx.x * COLS - 31, c1 = min(c0 + COLS, nx + 31);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = 8;
    int mn = rnext[s];   // the next order of the list, its signs one turn ahead
    const bool xp = qmu[s] >= 0.0, yp = qeta[s] >= 0.0;
#pragma unroll
    for (int k = threadIdx.x; k < 32 * COLS; k += 256) {
        const int c = c0 + k % COLS, jl = band * 32 + k / COLS;
        double r = 0.0;
        if (c >= 0 && c < nx && jl < ny) {
            const int i = xp ? c : nx - 1 - c;
            const int j = yp ? jl : ny - 1 - jl;
            const int cell = i + nx * j;
            r = 1.0 / (sigt[cell] + shift[cell] + acoef[(size_t)s * nx + i] + bcoef[(size_t)s * ny + j]);
        }
        v[k] = r;
    }
    __syncthreads();
    const int jl = band * 32 + lane;
    bool sx = true, sy = true;
    for (int m = s; m >= 0;) {
        const int mnn = mn >= 0 ? rnext[mn] : -1;
        const double nmu = mn >= 0 ? qmu[mn] : 0.0, neta = mn >= 0 ? qeta[mn] : 0.0;
        const int mj = sy || jl >= ny ? jl : ny - 1 - jl, ml = mj & 31;   // this row in the order of m
        const int t0 = sx ? c0 : nx - c1;
        double* out = rsw + ((size_t)m * nb + (mj >> 5)) * ns * 32 + ml;
        for (int t = t0 + wid; t < t0 + (c1 - c0) + 31; t += nw) {
            const int c = sx ? t - ml : nx - 1 - (t - ml);
            if (t >= 0 && t < ns && c >= c0 && c < c1) out[(size_t)t * 32] = v[lane * COLS + c - c0];
        }
        sx = (nmu >= 0.0) == xp;
        sy = (neta >= 0.0) == yp;
        m = mn;
        mn = mnn;
    }
}

__global__ void fill_kernel(double* a, size_t n, double v)
{
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        a[t] = v;
}

__global__ void fillf_kernel(float* a, size_t n, float v)
{
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        a[t] = v;
}

// Angular source of the next sweep from rho (Eq. (RTE_SI)):
// src = (sigma_s rho + q)/4pi  (no pseudo-time correction; used by the
// stand-alone kinetic step and at start-up).
__global__ void source_kernel(int N, const double* __restrict__ ss, const double* __restrict__ q,
                              const double* __restrict__ rho, double* src, float* src_f)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const double v = (ss[c] * rho[c] + q[c]) * kInvFourPi;
        src[c] = v;
        if (src_f) src_f[c] = (float)v;
    }
}

// --------------------------------------------------------------- sweep
// Source of the sweep: isotropic (plain), isotropic plus the pseudo-time
// term shift * I^m (delta form), or the adjoint source
// w_s (a - mu_s bx - eta_s by) of the transposed kinetic step.
// kSrcDelta: the increment sweep of the second-order upwind delta form
// (Eqs. (RTE_d_increment), (delta_Iij), (RTE_d_mtx)): source = the residual
// R[s][cell], zero increment on inflow faces, stored result I + corr + dI.
constexpr int kSrcPlain = 0, kSrcPseudoTime = 1, kSrcAdjoint = 2, kSrcDelta = 3;
// Windows per chunk buffer beyond the source (and the FP32 sigma_t): the
// pseudo-time, adjoint and increment forms read two per-cell/per-ordinate
// arrays more, the plain form none.  (A time-step form that read I^n and
// the per-cell source, one window more, with 1/(c dt) as a constant, was
// measured when a pair had two warps, one for the copies: 1024^2 S16 sweep
// 1.09 -> 1.92 ms against the 0.40 ms of the per-ordinate source pass it saved.)
__host__ __device__ constexpr int sweep_xw(int mode) { return mode == kSrcPlain ? 0 : 2; }

template <typename T>
struct SweepArgs {
    int nx, ny, N, K, nb, nsteps;
    const T* acoef; const T* bcoef;
    const double* rsw;
    const T* sigt; const T* shift; const T* src;
    int src_stride;             // elements between ordinates' sources (0: one per-cell source for all)
    const T* iold;              // stored intensities of the delta form: I^m (pseudo-time) or I^n (time step)
    const T* ax; const T* ay;   // adjoint source: bx, by (src holds a)
    const double* qw;           // sorted weights (adjoint source)
    T* I; T* edge;
    const double* inflow;
    const int* perm; const double* qmu; const double* qeta;
    int* err; const int* done;
    unsigned int* tasks;     // unit counter (band-major order)
    unsigned int* exits;     // warps that have left
    unsigned int* arrived;   // CTAs that have started
    int* mode;               // 0 undecided, 1 static placement, 2 counter
    long long wait_cycles;
    int resident;            // the launch guarantees the whole grid resident: static placement, no counters
};

// Several independent problems in one launch: unit u of the launch lies in
// segment g (seg_start[g] <= u < seg_start[g + 1]); a segment is one band of
// one problem, all K_p of its directions.  Within a problem the bands appear
// in increasing order, so a unit's upstream unit has the smaller index.
template <typename T>
struct SweepBatch {
    const SweepArgs<T>* probs;   // [B]
    const int* seg_start;        // [nseg + 1]
    const int* seg_prob;         // [nseg]
    const int* seg_band;         // [nseg]
    int nseg, ntasks;
    int dynamic;                 // 1: counter order even when the grid is resident
    unsigned int* tasks; unsigned int* exits; unsigned int* arrived; int* mode;
    int* err;                    // the launch's own error bits (a wait outside any unit)
    long long wait_cycles;
};

template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(smem)), "l"(gmem), "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Band hand-off slots hold the bit pattern "all ones" (a NaN that no
// arithmetic produces) until the upstream band writes the value.
template <typename T> struct Bits;
template <> struct Bits<double> {
    using U = unsigned long long;
    static constexpr U empty = ~0ull;
    static __device__ __forceinline__ U load(const double* p)
    {
        U v;
        asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p));
        return v;
    }
    static __device__ __forceinline__ void store(double* p, double v)
    {
        asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v));
    }
    static __device__ __forceinline__ double value(U u) { return __longlong_as_double((long long)u); }
    static __device__ __forceinline__ void clear(double* p) { *reinterpret_cast<U*>(p) = empty; }
    // plain store of a result; no compiler memory clobber, so the shared-memory
    // loads of the next steps may be issued ahead of it
    static __device__ __forceinline__ void put(double* p, double v)
    {
        asm volatile("st.global.f64 [%0], %1;" ::"l"(p), "d"(v));
    }
};
template <> struct Bits<float> {
    using U = unsigned int;
    static constexpr U empty = ~0u;
    static __device__ __forceinline__ U load(const float* p)
    {
        U v;
        asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
        return v;
    }
    static __device__ __forceinline__ void store(float* p, float v)
    {
        asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(v));
    }
    static __device__ __forceinline__ float value(U u) { return __uint_as_float(u); }
    static __device__ __forceinline__ void clear(float* p) { *reinterpret_cast<U*>(p) = empty; }
    static __device__ __forceinline__ void put(float* p, float v)
    {
        asm volatile("st.global.f32 [%0], %1;" ::"l"(p), "f"(v));
    }
};

// What the load warp tells the other warps of its pair about a chunk (in the
// chunk's buffer): the unit, where its results and its hand-off row go, and
// the adjoint source's coefficients.
template <typename T>
struct alignas(16) SweepHdr {
    int task;                  // launch unit, -1: no more units
    int nchunks, nx, rows;     // rows of the band inside the mesh
    T* out;                    // I at (band row 0, sweep column 0)
    T* eo;                     // this band's hand-off row, by column
    int* err;
    int t0, dr, dc, put_edge;  // first step of the chunk; strides of `out`; a band above reads the last row
    T* ei;                     // the band below's hand-off row, or null (band 0)
    const double* in;          // band 0: inflow of sweep column c at in[c * in_step], or null (vacuum)
    long long in_step;
    T cw, cm, ce;              // adjoint source w (a - mu bx - eta by)
};

// Shared-memory plan of one pair's warps.  A chunk is SEG consecutive steps
// (64-byte row segments).  Each of the NBUF chunk buffers holds, for the
// lane's own row, the cell data of the SEG cells the lane updates in the
// chunk (padded rows: conflict-free column access), the column coefficients
// of the SEG + 31 columns the skewed lanes touch, the 1/d table rows of the
// chunk (FP64), the SEG south values of lane 0, the unit's row coefficients
// and wall values (first chunk) and the header.
template <typename T, int MODE>
struct SweepSmem {
    static constexpr bool PRE = sizeof(T) == 8;               // 1/d from the table
    static constexpr int XW = sweep_xw(MODE);
    // a preparation warp forms what the compute warp can take ready-made: 1/d
    // in FP32, the combined source of the pseudo-time and adjoint forms
    static constexpr bool PREP = !PRE || MODE == kSrcPseudoTime || MODE == kSrcAdjoint;
    static constexpr int WARPS = PREP ? 4 : 3;                // compute, load, south [, preparation]
    static constexpr int SEG = 64 / (int)sizeof(T);
    // Buffers per pair: deeper queues hide more of the copies' latency, but the
    // shared memory comes out of the L1 that the 64-byte windows, shifted by
    // one cell from row to row, find their shared sectors in (FP64 1024^2
    // S16: 3 buffers 0.89 ms, 4 1.04 ms; FP32 512^2 S12: 3, 4, 5 buffers 125,
    // 98, 109 us).
    static constexpr int NBUF = PRE ? 3 : 4;
    static constexpr int RS = SEG + 1;
    static constexpr int AW = SEG + 32;
    static constexpr int NW = (PRE ? 1 : 2) + XW;              // src, [sigt], [shift,] [I^m or I^n]
    static constexpr int W_SRC = 0;                           // window slots
    static constexpr int W_SIGT = 1;                          // FP32 only (no 1/d table)
    static constexpr int W_SHIFT = PRE ? 1 : 2;               // two extra windows only
    static constexpr int W_IOLD = PRE ? 2 : 3;
    static constexpr int WIN = 32 * RS;
    static constexpr size_t r16(size_t b) { return (b + 15) / 16 * 16; }
    static constexpr size_t off_r = r16(sizeof(T) * (size_t)NW * WIN);
    static constexpr size_t off_a = off_r + (PRE ? (size_t)SEG * 32 * sizeof(double) : 0);
    static constexpr size_t off_e = off_a + r16(sizeof(T) * (size_t)AW);
    static constexpr size_t off_c = off_e + r16(sizeof(T) * (size_t)SEG);
    static constexpr size_t off_h = off_c + 2 * 32 * sizeof(T);
    static constexpr size_t buf_bytes = off_h + r16(sizeof(SweepHdr<T>));
    static constexpr size_t bar_bytes = 4 * 8 * (size_t)NBUF;   // full, ready, done, empty
    static constexpr size_t off_buf = r16(bar_bytes);
    static constexpr size_t pair_bytes = off_buf + NBUF * buf_bytes;
    // pairs per CTA: 8 (two chains per SM sub-partition) where the shared
    // memory holds them (FP64 1024^2 S16: 6, 7, 8 pairs 0.985, 0.918, 0.887
    // ms; the FP64 pipe is saturated by six chains, 18.4 cycles an operation)
    static constexpr size_t kFit = kSweepSmemCap / pair_bytes;
    static constexpr size_t kWant = 8;
    static constexpr int PAIRS = (int)(kFit < kWant ? kFit : kWant);
    static constexpr int THREADS = PAIRS * WARPS * 32;
    static constexpr size_t bytes = PAIRS * pair_bytes;
    static_assert(PAIRS >= 4, "a sweep CTA needs at least one pair per sub-partition");
    static_assert(NBUF >= 3, "the preparation warp writes a chunk out two chunks behind");
};

// One persistent CTA per SM runs PAIRS "pairs" of a compute warp and its two
// or three helpers; a pair's load warp chooses the units (direction s, band),
// u = band * K + s, and hands each on in the headers of its chunk buffers.
// When the whole grid is resident (a cooperative launch, or every CTA checks in
// within a few microseconds) the units are placed statically: pair p of CTA c takes
// u = p G + c + i PAIRS G, so each SM's first units come from different
// bands and run at different times; every unit is owned by a running pair and
// waits only on u - K.  Otherwise (part of the grid held back by other work
// on the GPU) the pairs take units from a counter in increasing order, so a
// unit only waits on one that a running pair took earlier.  One atomic
// decision picks the mode for every CTA; the launch's last warp to leave
// re-arms the counters.
//
// The time of a sweep with few units is the wavefront's critical path:
// nx + ny steps plus, per band, a chunk and a hand-off.  So the compute warp
// does nothing but the steps; what it used to do beside them (waiting with 32
// arrivals per barrier, writing results out, FP32 reciprocals, the wall's
// conditionals) took as long again:
//
//   load warp     cp.async of the window data into a free buffer, header.
//                 Without a preparation warp it also writes finished chunks
//                 out before it refills their buffer.
//   south warp    lane 0's south values of a chunk: the inflow on band 0, else
//                 the upstream band's last-row results, polled until written
//                 (in a warp of its own: between the load warp's copies a
//                 poll came a round trip to L2 late at every chunk).
//   preparation   (PREP) per chunk, in place: FP32 1/d, the pseudo-time or
//   warp          adjoint source; then writes out the chunk two behind.
//   compute warp  SEG steps from shared memory, each result into the slot of
//                 the source it used, the last lane's also to the band's
//                 hand-off row.  Slots outside the mesh are computed like
//                 the others, from the nearest cell's data: no lane inside
//                 the mesh reads their results (lane l + 1 at step t reads
//                 lane l of step t - 1, the same column), the west value is
//                 set to the wall's at the lane's first column, and nothing
//                 of them is written out.
//
// Every wait is bounded; on time-out kErrTimeout is raised and the warp leaves
// after its copies in flight have landed.
//
// Before / after (one launch, us): FP64 64^2 S8 31 / 26, 256^2 S12 108 / 94
// (per-ordinate source; 88 with the south value from its slot) and 189 / 150
// (increment form), 200^2 S8 35 / 28 (24) and 51 / 40 (36, adjoint form),
// 1024^2 S16 919 / 887 (854); FP32 641x470 S6 254 / 96,
// 512^2 S12 190 / 98, batch of 24 problems 158 / 128.  Bounds now: FP64 with
// many units, the pipe (1024^2 S16: 14.2 M warp operations of 18.4 cycles on
// 152 SMs, 0.83 ms); with few, the chain of a step (253 cycles: three FP64
// operations and the store and load of a slot; 265 with a 64-bit shuffle);
// FP32, instruction issue of the four warps of a pair and the load warp's 34
// copy instructions a chunk.
template <typename T, int MODE, bool BATCH>
__global__ void __launch_bounds__(SweepSmem<T, MODE>::THREADS, 1)
sweep_kernel(const SweepArgs<T> a1, const SweepBatch<T> bt)
{
    constexpr bool PT = MODE == kSrcPseudoTime, ADJ = MODE == kSrcAdjoint, DELTA = MODE == kSrcDelta;
    using SM = SweepSmem<T, MODE>;
    using B = Bits<T>;
    using Hdr = SweepHdr<T>;
    constexpr bool PRE = SM::PRE, PREP = SM::PREP;
    constexpr int SEG = SM::SEG, NBUF = SM::NBUF, RS = SM::RS, NW = SM::NW;
    constexpr int RPI = 32 / SEG;   // rows per copy or write-out instruction
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int role = warp / SM::PAIRS, pair = warp - role * SM::PAIRS;   // 0 compute, 1 load, 2 south, 3 preparation
    unsigned char* pbase = smem_raw + (size_t)pair * SM::pair_bytes;
    unsigned long long* full = reinterpret_cast<unsigned long long*>(pbase);   // data and header
    unsigned long long* ready = full + NBUF;     // south values [, prepared]
    unsigned long long* done_b = ready + NBUF;   // steps finished
    unsigned long long* empty = done_b + NBUF;   // PREP: written out
    auto buf = [&](int b) { return pbase + SM::off_buf + (size_t)b * SM::buf_bytes; };

    if (threadIdx.x < SM::PAIRS) {
        unsigned long long* f = reinterpret_cast<unsigned long long*>(smem_raw + (size_t)threadIdx.x * SM::pair_bytes);
        for (int b = 0; b < NBUF; ++b) {
            mbar_init(f + b, 33);                        // 32 cp.async arrivals, the header
            mbar_init(f + NBUF + b, PREP ? 2 : 1);       // south values [, preparation]
            mbar_init(f + 2 * NBUF + b, 1);
            mbar_init(f + 3 * NBUF + b, 1);
        }
    }
    __syncthreads();

    const int G = gridDim.x;
    const int ntasks = BATCH ? bt.ntasks : a1.K * a1.nb;
    const long long budget = BATCH ? bt.wait_cycles : a1.wait_cycles;
    unsigned* const c_tasks = BATCH ? bt.tasks : a1.tasks;
    unsigned* const c_exits = BATCH ? bt.exits : a1.exits;
    unsigned* const c_arrived = BATCH ? bt.arrived : a1.arrived;
    int* const c_mode = BATCH ? bt.mode : a1.mode;
    int* const c_err = BATCH ? bt.err : a1.err;

    __shared__ int cta_mode, cta_stop;
    if (threadIdx.x == 0) {
        cta_stop = BATCH ? 0 : ld_volatile_int(a1.done) | ld_volatile_int(a1.err);
        int m = 1;
        const long long t0 = clock64();
        if (BATCH || !a1.resident) {
            atomicAdd(c_arrived, 1u);
            m = 0;
        }
        while (m == 0) {
            m = *reinterpret_cast<volatile int*>(c_mode);
            if (m != 0) break;
            if (*reinterpret_cast<volatile unsigned*>(c_arrived) >= (unsigned)G) atomicCAS(c_mode, 0, 1);
            else if (clock64() - t0 > 20000) atomicCAS(c_mode, 0, 2);
        }
        cta_mode = m;
    }
    __syncthreads();
    const bool placed = cta_mode == 1 && !(BATCH && bt.dynamic);

    // All lanes wait for the phase of chunk g; false (in all of them) on time-out.
    auto wait_all = [&](unsigned long long* bars, unsigned g, int* err) {
        const bool ok = __all_sync(kFull, mbar_wait(bars + g % NBUF, (g / NBUF) & 1, budget));
        if (!ok && lane == 0) atomicOr(err, kErrTimeout);
        return ok;
    };
    auto arrive_one = [&](unsigned long long* bar) {   // one arrival for the warp's accesses so far
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };
    // Results of a finished chunk: RPI rows of SEG consecutive cells per store.
    auto write_out = [&](unsigned g) {
        const unsigned char* bp = buf((int)(g % NBUF));
        const Hdr& h = *reinterpret_cast<const Hdr*>(bp + SM::off_h);
        const T* w = reinterpret_cast<const T*>(bp);
        const int kk = lane % SEG, r1 = lane / SEG, t0 = h.t0, nx = h.nx, rows = h.rows, dr = h.dr, dc = h.dc;
        T* out = h.out;
        constexpr int NI = SEG;   // 32 / RPI
        T v[NI];
#pragma unroll
        for (int u = 0; u < NI; ++u) {
            const int at = (r1 + u * RPI) * RS + kk;
            v[u] = w[SM::W_SRC * SM::WIN + at];
            if (DELTA) v[u] = (w[SM::W_IOLD * SM::WIN + at] + w[SM::W_SHIFT * SM::WIN + at]) + v[u];
        }
        if (rows == 32 && t0 >= 31 && t0 + SEG <= nx) {
            T* o = out + r1 * dr + (t0 + kk - r1) * dc;
            const int step = RPI * (dr - dc);
#pragma unroll
            for (int u = 0; u < NI; ++u) B::put(o + u * step, v[u]);
        } else {
#pragma unroll
            for (int u = 0; u < NI; ++u) {
                const int r = r1 + u * RPI, c = t0 + kk - r;
                if (r < rows && c >= 0 && c < nx) B::put(out + r * dr + c * dc, v[u]);
            }
        }
    };

    unsigned g = 0;   // chunks this warp has handled (buffer = g % NBUF)

    auto load_warp = [&]() {
        int next_static = pair * G + (int)blockIdx.x;
        bool first = true;
        // buffer of chunk g free: its previous chunk is written out
        auto acquire = [&](int* err) {
            if (g < NBUF) return true;
            if (PREP) return wait_all(empty, g - NBUF, err);
            if (!wait_all(done_b, g - NBUF, err)) return false;
            write_out(g - NBUF);
            __syncwarp();
            return true;
        };
        for (;;) {
            // next unit; -1: none left, or an error was raised.  In a batch the
            // units of a problem that has stopped (converged or failed) are skipped.
            int t = -1, pp = 0, lt = 0;
            if (lane == 0) {
                for (;;) {
                    if (placed) {
                        t = next_static;
                        next_static += SM::PAIRS * G;
                    } else {
                        if (first && pair >= SM::PAIRS / 2) {
                            // the second half of the pairs shares sub-partitions with the
                            // first half: let the first half take the first units, so that
                            // concurrently running units start on distinct sub-partitions
                            const unsigned want = min((unsigned)ntasks, (unsigned)(SM::PAIRS / 2) * (unsigned)G);
                            const long long t0 = clock64();
                            while (*reinterpret_cast<volatile unsigned*>(c_tasks) < want && clock64() - t0 < 20000)
                                __nanosleep(64);
                        }
                        first = false;
                        t = (int)atomicAdd(c_tasks, 1u);
                    }
                    if (t >= ntasks) { t = -1; break; }
                    if (!BATCH) {
                        if (ld_volatile_int(a1.err)) t = -1;
                        lt = t;
                        break;
                    }
                    const int sg = batch_find(bt.seg_start, bt.nseg, t);
                    pp = bt.seg_prob[sg];
                    const SweepArgs<T>& q = bt.probs[pp];
                    if (ld_volatile_int(q.done) | ld_volatile_int(q.err)) continue;
                    lt = bt.seg_band[sg] * q.K + (t - bt.seg_start[sg]);
                    break;
                }
            }
            const int task = __shfl_sync(kFull, t, 0), prob = __shfl_sync(kFull, pp, 0);
            const int ltask = __shfl_sync(kFull, lt, 0);
            first = false;
            if (task < 0) {   // end marker in the next buffer; without PREP the last chunks are still to be written
                if (!acquire(c_err)) return;
                const int b = (int)(g % NBUF);
                if (lane == 0) reinterpret_cast<Hdr*>(buf(b) + SM::off_h)->task = -1;
                cp_async_mbar_arrive(full + b);
                arrive_one(full + b);
                if (!PREP)
                    for (unsigned q = g >= NBUF ? g - NBUF + 1 : 0; q < g; ++q) {
                        if (!wait_all(done_b, q, c_err)) return;
                        write_out(q);
                    }
                return;
            }
            const SweepArgs<T>& a = BATCH ? bt.probs[prob] : a1;
            const int nx = a.nx, ny = a.ny, K = a.K, nb = a.nb, nsteps = a.nsteps;
            const int nchunks = (nsteps + SEG - 1) / SEG;
            const int band = ltask / K;
            const int s = ltask - band * K;
            const bool xpos = a.qmu[s] >= 0.0, ypos = a.qeta[s] >= 0.0;
            const int k = a.perm[s];
            const int rows = min(32, ny - band * 32);
            // cell of (band row r, sweep column c) = base0 + r * dr + c * dc
            const int dr = ypos ? nx : -nx, dc = xpos ? 1 : -1;
            const int base0 = (ypos ? band * 32 : ny - 1 - band * 32) * nx + (xpos ? 0 : nx - 1);
            const T* wsrc[NW];
            wsrc[SM::W_SRC] = a.src + (size_t)s * a.src_stride;
            if constexpr (!PRE) wsrc[SM::W_SIGT] = a.sigt;
            if constexpr (PT) {
                wsrc[SM::W_SHIFT] = a.shift;
                wsrc[SM::W_IOLD] = a.iold + (size_t)s * a.N;
            }
            if constexpr (ADJ) {
                wsrc[SM::W_SHIFT] = a.ax;
                wsrc[SM::W_IOLD] = a.ay;
            }
            if constexpr (DELTA) {   // residual and stored intensity of this ordinate, correction per cell
                wsrc[SM::W_SRC] = a.src + (size_t)s * a.N;
                wsrc[SM::W_SHIFT] = a.shift;
                wsrc[SM::W_IOLD] = a.iold + (size_t)s * a.N;
            }
            const T* arow = a.acoef + (size_t)s * nx;
            const double* rrow = PRE ? a.rsw + ((size_t)s * nb + band) * (size_t)nsteps * 32 : nullptr;
            T* edge_in = band > 0 ? a.edge + ((size_t)s * nb + band - 1) * nx : nullptr;
            T bj = T(0), wall = T(0);   // this lane's row: |eta|/dy, the intensity entering through the wall
            if (lane < rows) {
                const int j = ypos ? band * 32 + lane : ny - 1 - band * 32 - lane;
                bj = a.bcoef[(size_t)s * ny + j];
                if (a.inflow) wall = (T)a.inflow[(size_t)(xpos ? j : ny + j) * K + k];
            }
            const int kk = lane % SEG, r1 = lane / SEG;
            for (int m = 0; m < nchunks; ++m, ++g) {
                if (!acquire(a.err)) return;
                const int b = (int)(g % NBUF);
                unsigned char* bp = buf(b);
                T* wb = reinterpret_cast<T*>(bp);
                T* ab = reinterpret_cast<T*>(bp + SM::off_a);
                const int t0 = m * SEG;
                // row r of the band needs columns t0 - r .. t0 - r + SEG - 1
                if (rows == 32 && t0 >= 31 && t0 + SEG <= nx) {
                    // interior chunk: every row window lies inside the mesh
                    int cell = base0 + r1 * dr + (t0 + kk - r1) * dc;
                    const int dcell = RPI * (dr - dc);
                    T* dst = wb + r1 * RS + kk;
#pragma unroll
                    for (int r0 = 0; r0 < 32; r0 += RPI) {
#pragma unroll
                        for (int w = 0; w < NW; ++w) cp_async<sizeof(T)>(dst + w * SM::WIN, wsrc[w] + cell);
                        cell += dcell;
                        dst += RPI * RS;
                    }
                    const T* ap = arow + (xpos ? t0 - 31 : nx - 1 - (t0 - 31));
                    for (int u = lane; u < SEG + 31; u += 32) cp_async<sizeof(T)>(ab + u, ap + u * dc);
                } else {
                    // at the walls: the nearest cell's data where the window leaves the mesh
#pragma unroll
                    for (int r0 = 0; r0 < 32; r0 += RPI) {
                        const int r = r0 + r1;
                        const int c = min(max(t0 + kk - r, 0), nx - 1);
                        const int cell = base0 + min(r, rows - 1) * dr + c * dc;
#pragma unroll
                        for (int w = 0; w < NW; ++w) cp_async<sizeof(T)>(wb + w * SM::WIN + r * RS + kk, wsrc[w] + cell);
                    }
                    for (int u = lane; u < SEG + 31; u += 32) {
                        const int c = min(max(t0 - 31 + u, 0), nx - 1);
                        cp_async<sizeof(T)>(ab + u, arow + (xpos ? c : nx - 1 - c));
                    }
                }
                if constexpr (PRE) {
                    const int nv = min(SEG, nsteps - t0) * 32;   // doubles, multiple of 32
                    double* rb = reinterpret_cast<double*>(bp + SM::off_r);
                    const double* rp = rrow + (size_t)t0 * 32;
#pragma unroll
                    for (int v = 0; v < SEG * 32; v += 64)
                        if (v + 2 * lane < nv) cp_async<16>(rb + v + 2 * lane, rp + v + 2 * lane);
                }
                cp_async_mbar_arrive(full + b);
                if (m == 0) {
                    T* cx = reinterpret_cast<T*>(bp + SM::off_c);
                    cx[lane] = bj;
                    cx[32 + lane] = wall;
                }
                if (lane == 0) {
                    Hdr& h = *reinterpret_cast<Hdr*>(bp + SM::off_h);
                    h.task = task;
                    h.nchunks = nchunks;
                    h.nx = nx;
                    h.rows = rows;
                    h.out = a.I + (size_t)s * a.N + base0;
                    h.eo = a.edge + ((size_t)s * nb + band) * nx;
                    h.err = a.err;
                    h.t0 = t0;
                    h.dr = dr;
                    h.dc = dc;
                    h.put_edge = band < nb - 1;
                    h.ei = edge_in;
                    h.in = nullptr;
                    if (a.inflow) {   // sweep column 0's face of the wall below, then along the row
                        h.in = a.inflow + (size_t)((ypos ? 2 * ny : 2 * ny + nx) + (xpos ? 0 : nx - 1)) * K + k;
                        h.in_step = xpos ? K : -K;
                    }
                    if (ADJ && m == 0) {
                        const double ws = a.qw[s];
                        h.cw = (T)ws;
                        h.cm = (T)(-ws * a.qmu[s]);
                        h.ce = (T)(-ws * a.qeta[s]);
                    }
                }
                arrive_one(full + b);
            }
        }
    };

    // South values of lane 0: per chunk the inflow (band 0) or the band below's
    // last-row results, polled until they are written.
    auto south_warp = [&]() {
        using U = typename B::U;
        int* err = c_err;
        for (;;) {
            if (!wait_all(full, g, err)) return;
            const Hdr& h = *reinterpret_cast<const Hdr*>(buf((int)(g % NBUF)) + SM::off_h);
            if (h.task < 0) {
                arrive_one(ready + g % NBUF);
                return;
            }
            const int nchunks = h.nchunks, nx = h.nx;
            T* const ei = h.ei;
            const double* const in = h.in;
            const long long in_step = h.in_step;
            err = h.err;
            for (int m = 0; m < nchunks; ++m, ++g) {
                const int c = m * SEG + lane;
                const bool need = lane < SEG && c < nx;
                U u = B::empty;
                T ev = T(0);
                if (need) {   // in flight during the wait
                    if (ei) u = B::load(ei + c);
                    else if (in) ev = (T)in[c * in_step];
                }
                if (m > 0 && !wait_all(full, g, err)) return;
                if (ei) {
                    const long long start = clock64();
                    while (!__all_sync(kFull, !need || u != B::empty)) {
                        if (__any_sync(kFull, clock64() - start > budget)) {   // warp-uniform exit
                            if (lane == 0) atomicOr(err, kErrTimeout);
                            return;
                        }
                        if (need && u == B::empty) u = B::load(ei + c);
                    }
                    if (need) ev = B::value(u);
                }
                const int b = (int)(g % NBUF);
                if (lane < SEG) reinterpret_cast<T*>(buf(b) + SM::off_e)[lane] = ev;
                arrive_one(ready + b);
            }
            // every value of the upstream hand-off row has been taken:
            // mark it unwritten for the next sweep
            if (ei)
                for (int c = lane; c < nx; c += 32) B::clear(ei + c);
        }
    };

    auto prep_warp = [&]() {
        unsigned written = 0;   // chunks written out
        int* err = c_err;
        auto write_next = [&]() {
            if (!wait_all(done_b, written, err)) return false;
            write_out(written);
            arrive_one(empty + written % NBUF);
            ++written;
            return true;
        };
        for (;;) {
            if (!wait_all(full, g, err)) return;
            const Hdr& h0 = *reinterpret_cast<const Hdr*>(buf((int)(g % NBUF)) + SM::off_h);
            if (h0.task < 0) {
                arrive_one(ready + g % NBUF);
                while (written < g)
                    if (!write_next()) return;
                return;
            }
            const int nchunks = h0.nchunks;
            err = h0.err;
            const T cw = h0.cw, cm = h0.cm, ce = h0.ce;
            const T bj = reinterpret_cast<const T*>(buf((int)(g % NBUF)) + SM::off_c)[lane];
            for (int m = 0; m < nchunks; ++m, ++g) {
                if (m > 0 && !wait_all(full, g, err)) return;
                unsigned char* bp = buf((int)(g % NBUF));
                T* w = reinterpret_cast<T*>(bp) + lane * RS;
                const T* ab = reinterpret_cast<const T*>(bp + SM::off_a) + 31 - lane;
                float d[PRE ? 1 : SEG];
                unsigned dlo = ~0u, dhi = 0u;
#pragma unroll
                for (int tt = 0; tt < SEG; ++tt) {
                    T sv = w[SM::W_SRC * SM::WIN + tt];
                    if (ADJ) sv = fma(cm, w[SM::W_SHIFT * SM::WIN + tt], fma(ce, w[SM::W_IOLD * SM::WIN + tt], cw * sv));
                    T sh = T(0);
                    if (PT) {
                        sh = w[SM::W_SHIFT * SM::WIN + tt];
                        sv = fma(sh, w[SM::W_IOLD * SM::WIN + tt], sv);
                    }
                    if (ADJ || PT) w[SM::W_SRC * SM::WIN + tt] = sv;
                    if constexpr (!PRE) {
                        d[tt] = w[SM::W_SIGT * SM::WIN + tt] + ab[tt] + bj;
                        if (PT) d[tt] += sh;
                        dlo = min(dlo, __float_as_uint(d[tt]));
                        dhi = max(dhi, __float_as_uint(d[tt]));
                    }
                }
                if constexpr (!PRE) {
                    const bool plain = dlo >= kRcpLo && dhi <= kRcpHi;
#pragma unroll
                    for (int tt = 0; tt < SEG; ++tt)
                        w[SM::W_SIGT * SM::WIN + tt] = plain ? rcp_newton(d[tt]) : 0.f;
                    if (!plain) {
#pragma unroll
                        for (int tt = 0; tt < SEG; ++tt) w[SM::W_SIGT * SM::WIN + tt] = __frcp_rn(d[tt]);
                    }
                }
                arrive_one(ready + g % NBUF);
                if (g >= 2 && !write_next()) return;
            }
        }
    };

    auto compute_warp = [&]() {
        unsigned long long* in = ready;
        for (;;) {
            if (!wait_all(in, g, c_err)) return;
            const unsigned char* b0 = buf((int)(g % NBUF));
            const Hdr& h = *reinterpret_cast<const Hdr*>(b0 + SM::off_h);
            if (h.task < 0) return;
            const int nchunks = h.nchunks, nx = h.nx;
            const bool full_rows = h.rows == 32, put_edge = lane == 31 && h.put_edge;
            T* eo = h.eo;
            int* err = h.err;
            const T* cx = reinterpret_cast<const T*>(b0 + SM::off_c);
            const T bj = cx[lane], wall = cx[32 + lane];
            T IW = wall, Iprev = T(0);
            T sv_n = T(0), ai_n = T(0), r_n = T(0), e_n = T(0);   // next step's operands, read one step ahead
            bool ahead = false;                                   // ... of the next chunk already
            auto operands = [&](const unsigned char* bp, int tt) {
                const T* w = reinterpret_cast<const T*>(bp) + lane * RS + tt;
                sv_n = w[SM::W_SRC * SM::WIN];
                ai_n = (reinterpret_cast<const T*>(bp + SM::off_a) + 31 - lane)[tt];
                if constexpr (PRE) r_n = (reinterpret_cast<const T*>(bp + SM::off_r) + lane)[tt * 32];
                else r_n = w[SM::W_SIGT * SM::WIN];
                e_n = reinterpret_cast<const T*>(bp + SM::off_e)[tt];
            };
            for (int m = 0; m < nchunks; ++m, ++g) {
                if (!ahead) {
                    if (m > 0 && !wait_all(in, g, err)) return;
                    operands(buf((int)(g % NBUF)), 0);
                }
                ahead = false;
                unsigned char* bp = buf((int)(g % NBUF));
                T* res = reinterpret_cast<T*>(bp) + lane * RS;   // the source slots collect the results
                // FP64, south values of steps 1.. of the chunk: lane l - 1's previous
                // result from its slot, lane 0's from the south values
                const volatile T* south =
                    lane > 0 ? res - RS : reinterpret_cast<const T*>(bp + SM::off_e) + 1;
                const int t0 = m * SEG;
                auto steps = [&](auto wall_chunk) {
                    constexpr bool WALL = decltype(wall_chunk)::value;
#pragma unroll
                    for (int tt = 0; tt < SEG; ++tt) {
                        const T sv = sv_n, ai = ai_n, rinv = r_n, e = e_n;
                        if (tt + 1 < SEG) operands(bp, tt + 1);
                        else if (m + 1 < nchunks) {
                            // a look at the next chunk while this step's chain runs; not a wait:
                            // the band above may need this step first
                            const unsigned gn = g + 1;
                            ahead = __all_sync(kFull, mbar_test(in + gn % NBUF, (gn / NBUF) & 1));
                            if (ahead) operands(buf((int)(gn % NBUF)), 0);
                        }
                        if (WALL && t0 + tt == lane) IW = wall;   // the lane's first column
                        // lane l gets lane l-1's previous result; lane 0 the south value
                        T Isouth;
                        if (PRE && tt > 0) {
                            __syncwarp();
                            Isouth = south[tt - 1];
                        } else {
                            Isouth = __shfl_sync(kFull, lane == 31 ? e : Iprev, (lane + 31) & 31);
                        }
                        T acc = fma(ai, IW, sv);
                        acc = fma(bj, Isouth, acc);
                        const T Inew = acc * rinv;
                        IW = Inew;
                        Iprev = Inew;
                        res[SM::W_SRC * SM::WIN + tt] = Inew;
                        const int c = t0 + tt - 31;
                        if (put_edge && (!WALL || (c >= 0 && c < nx))) B::store(eo + c, Inew);
                    }
                };
                if (full_rows && t0 >= 31 && t0 + SEG <= nx) steps(std::false_type{});
                else steps(std::true_type{});
                arrive_one(done_b + g % NBUF);
            }
        }
    };

    if (!cta_stop) {
        if (role == 0) compute_warp();
        else if (role == 1) load_warp();
        else if (role == 2) south_warp();
        else prep_warp();
    }
    if (role == 1) cp_async_wait_all();
    // the launch's last warp to leave re-arms the counters for the next launch
    __syncwarp();
    if (lane == 0 && (BATCH || !a1.resident)) {
        __threadfence();
        if (atomicAdd(c_exits, 1u) == (unsigned)G * (unsigned)(SM::WARPS * SM::PAIRS) - 1u) {
            *c_tasks = 0u;
            *c_arrived = 0u;
            *c_mode = 0;
            *c_exits = 0u;
        }
    }
}

// --------------------------------------------------------------- moments
template <typename T>
struct MomArgs {
    int nx, ny, N, K;
    const T* I;
    const int* sidx;
    const double* mu; const double* eta; const double* w;   // original order
    double* rho; double* Fx; double* Fy;                    // may be null (F)
    double* Pxx; double* Pxy; double* Pyy;                  // may be null
    const double* rho_new;                                  // GSIS correction of P (or null)
    const int* done;
    const int* pairs;   // [K/2][2] x-reflection pairs (original k, the first with mu > 0), or null
    const MomQuad* quads;   // [K/4] reflection quads (FP64), or null
};

// FP64 moments of one cell by plain multiply-adds in the original direction
// order (cells that the fixed-point sums do not cover).
template <bool WITH_F, bool WITH_P>
__device__ __forceinline__ void moments_plain_cell(const MomArgs<double>& a, int c, double* out)
{
    double r = 0.0, fx = 0.0, fy = 0.0, pxx = 0.0, pxy = 0.0, pyy = 0.0;
#pragma unroll 1
    for (int k = 0; k < a.K; ++k) {
        const double v = a.I[(size_t)a.sidx[k] * a.N + c], w = a.w[k], m = a.mu[k], e = a.eta[k];
        r = fma(w, v, r);
        if (WITH_F) {
            fx = fma(w * m, v, fx);
            fy = fma(w * e, v, fy);
        }
        if (WITH_P) {
            pxx = fma(w * m * m, v, pxx);
            pxy = fma(w * m * e, v, pxy);
            pyy = fma(w * e * e, v, pyy);
        }
    }
    out[0] = r;
    if (WITH_F) { out[1] = fx; out[2] = fy; }
    if (WITH_P) { out[3] = pxx; out[4] = pxy; out[5] = pyy; }
}

// FP64 moments over reflection quads in fixed point (moments_fixed.cuh),
// one thread per cell.
template <bool WITH_F, bool WITH_P>
__device__ __forceinline__ void moments_quad_body(const MomArgs<double>& a, int bid, int nblk)
{
    constexpr int NM = WITH_P ? 6 : WITH_F ? 3 : 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    MomQuad* tab = reinterpret_cast<MomQuad*>(smem_raw);
    const int nq = a.K / 4;
    for (int t = threadIdx.x; t < nq * 16; t += blockDim.x) {
        unsigned v = reinterpret_cast<const unsigned*>(a.quads)[t];
        if ((t & 15) >= 4 && (t & 1)) v >>= 32 - FixedMoments<NM>::kFrac;
        reinterpret_cast<unsigned*>(tab)[t] = v;
    }
    __syncthreads();
    for (int c = bid * blockDim.x + threadIdx.x; c < a.N; c += nblk * blockDim.x) {
        FixedMoments<NM> f;
        double o[6];
        if (!f.run(tab, nq, a.I, (size_t)a.N, c, o)) moments_plain_cell<WITH_F, WITH_P>(a, c, o);
        if (a.rho) a.rho[c] = o[0];
        if (WITH_F) {
            a.Fx[c] = o[1];
            a.Fy[c] = o[2];
        }
        if (WITH_P) {
            double d = 0.0;   // moments of I + (rho_new - rho_half)/4pi: + drho/3 on the diagonal
            if (a.rho_new) d = (a.rho_new[c] - o[0]) / 3.0;
            a.Pxx[c] = o[3] + d;
            a.Pxy[c] = o[4];
            a.Pyy[c] = o[5] + d;
        }
    }
}

// Per cell, in original direction order k = 0..K-1:
// rho = sum w I, F = sum w Omega I, P = sum w Omega Omega I.
template <typename T, bool WITH_F, bool WITH_P>
__device__ __forceinline__ void moments_body(const MomArgs<T>& a, int bid, int nblk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* cf = reinterpret_cast<T*>(smem_raw);                     // [K][6]
    int* sk = reinterpret_cast<int*>(cf + 6 * a.K);             // [K]
    if (a.done && ld_volatile_int(a.done)) return;
    if constexpr (sizeof(T) == 8) {
        if (a.quads) {
            moments_quad_body<WITH_F, WITH_P>(a, bid, nblk);
            return;
        }
    }
    if (!WITH_P && a.pairs) {
        // Directions in x-reflection pairs k1 = (mu, eta), k2 = (-mu, eta)
        // with one weight: rho += w (I1 + I2), F_x += w mu (I1 - I2),
        // F_y += w eta (I1 + I2): five operations per pair instead of six
        // (FP32, and FP64 sets without reflection quads).
        const int np = a.K / 2;
        T* cp = cf;                                             // [np][3]: w, w mu, w eta of k1
        int* sp = reinterpret_cast<int*>(cf + 3 * np);          // [np][2]: sorted indices of k1, k2
        for (int p = threadIdx.x; p < np; p += blockDim.x) {
            const int k1 = a.pairs[2 * p], k2 = a.pairs[2 * p + 1];
            const double w = a.w[k1];
            cp[3 * p + 0] = (T)w;
            cp[3 * p + 1] = (T)(w * a.mu[k1]);
            cp[3 * p + 2] = (T)(w * a.eta[k1]);
            sp[2 * p] = a.sidx[k1];
            sp[2 * p + 1] = a.sidx[k2];
        }
        __syncthreads();
        for (int c = bid * blockDim.x + threadIdx.x; c < a.N; c += nblk * blockDim.x) {
            T r = T(0), fx = T(0), fy = T(0);
#pragma unroll 4
            for (int p = 0; p < np; ++p) {
                const T v1 = a.I[(size_t)sp[2 * p] * a.N + c];
                const T v2 = a.I[(size_t)sp[2 * p + 1] * a.N + c];
                const T sum = v1 + v2;
                r = fma(cp[3 * p + 0], sum, r);
                if (WITH_F) {
                    fx = fma(cp[3 * p + 1], v1 - v2, fx);
                    fy = fma(cp[3 * p + 2], sum, fy);
                }
            }
            if (a.rho) a.rho[c] = (double)r;
            if (WITH_F) {
                a.Fx[c] = (double)fx;
                a.Fy[c] = (double)fy;
            }
        }
        return;
    }
    for (int k = threadIdx.x; k < a.K; k += blockDim.x) {
        const double w = a.w[k], m = a.mu[k], e = a.eta[k];
        cf[6 * k + 0] = (T)w;
        cf[6 * k + 1] = (T)(w * m);
        cf[6 * k + 2] = (T)(w * e);
        cf[6 * k + 3] = (T)(w * m * m);
        cf[6 * k + 4] = (T)(w * m * e);
        cf[6 * k + 5] = (T)(w * e * e);
        sk[k] = a.sidx[k];
    }
    __syncthreads();
    for (int c = bid * blockDim.x + threadIdx.x; c < a.N; c += nblk * blockDim.x) {
        T r = T(0), fx = T(0), fy = T(0), pxx = T(0), pxy = T(0), pyy = T(0);
#pragma unroll 4
        for (int k = 0; k < a.K; ++k) {
            const T v = a.I[(size_t)sk[k] * a.N + c];
            r = fma(cf[6 * k + 0], v, r);
            if (WITH_F) {
                fx = fma(cf[6 * k + 1], v, fx);
                fy = fma(cf[6 * k + 2], v, fy);
            }
            if (WITH_P) {
                pxx = fma(cf[6 * k + 3], v, pxx);
                pxy = fma(cf[6 * k + 4], v, pxy);
                pyy = fma(cf[6 * k + 5], v, pyy);
            }
        }
        if (a.rho) a.rho[c] = (double)r;
        if (WITH_F) {
            a.Fx[c] = (double)fx;
            a.Fy[c] = (double)fy;
        }
        if (WITH_P) {
            double dxx = (double)pxx, dyy = (double)pyy;
            if (a.rho_new) {   // moments of I + (rho_new - rho_half)/4pi: + drho/3 on the diagonal
                const double d = (a.rho_new[c] - (double)r) / 3.0;
                dxx += d;
                dyy += d;
            }
            a.Pxx[c] = dxx;
            a.Pxy[c] = (double)pxy;
            a.Pyy[c] = dyy;
        }
    }
}

// Kinetic net flux through every boundary face, sum_k w_k (Omega_k . n) I_face,k
// (outgoing: boundary cell intensity, incoming: inflow).  One warp per face;
// lane l sums k = l, l+32, ... in order, then a fixed shuffle tree.
template <typename T>
struct BfArgs {
    int nx, ny, K;
    const T* I;
    const int* sidx;
    const double* mu; const double* eta; const double* w;   // original order
    const double* inflow;
    double* fb;
    const int* done;
};

template <typename T>
__device__ __forceinline__ void bflux_body(const BfArgs<T>& a, int bid, int nblk)
{
    if (a.done && ld_volatile_int(a.done)) return;
    const int nx = a.nx, ny = a.ny, K = a.K;
    const int nbf = 2 * (nx + ny), N = nx * ny;
    const int lane = threadIdx.x & 31;
    const int warps = (nblk * blockDim.x) >> 5;
    for (int f = (bid * blockDim.x + threadIdx.x) >> 5; f < nbf; f += warps) {
        int c, axis;
        double sgn;
        if (f < ny) { c = nx * f; axis = 0; sgn = -1.0; }
        else if (f < 2 * ny) { c = nx - 1 + nx * (f - ny); axis = 0; sgn = 1.0; }
        else if (f < 2 * ny + nx) { c = f - 2 * ny; axis = 1; sgn = -1.0; }
        else { c = (f - 2 * ny - nx) + nx * (ny - 1); axis = 1; sgn = 1.0; }
        T acc = T(0);
        for (int k = lane; k < K; k += 32) {
            const double on = sgn * (axis == 0 ? a.mu[k] : a.eta[k]);
            T Iface;
            if (on >= 0.0) Iface = a.I[(size_t)a.sidx[k] * N + c];
            else Iface = a.inflow ? (T)a.inflow[(size_t)f * K + k] : T(0);
            acc = fma((T)(a.w[k] * on), Iface, acc);
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if (lane == 0) a.fb[f] = (double)acc;
    }
}

template <typename T, bool WITH_F, bool WITH_P>
__global__ void __launch_bounds__(kRedBlock) moments_kernel(const MomArgs<T> a)
{
    moments_body<T, WITH_F, WITH_P>(a, blockIdx.x, gridDim.x);
}

template <typename T>
__global__ void __launch_bounds__(256) bflux_kernel(const BfArgs<T> a)
{
    bflux_body(a, blockIdx.x, gridDim.x);
}

// Moments and boundary fluxes of one problem in one launch: the first
// mblocks blocks take the cells, the rest the boundary faces.
template <typename T, bool WITH_F, bool WITH_P>
__global__ void __launch_bounds__(kRedBlock) moments_bflux_kernel(const MomArgs<T> m, const BfArgs<T> f, int mblocks)
{
    if ((int)blockIdx.x < mblocks) moments_body<T, WITH_F, WITH_P>(m, blockIdx.x, mblocks);
    else bflux_body(f, blockIdx.x - mblocks, gridDim.x - mblocks);
}

// Batched moments and boundary fluxes: problem p owns blocks
// [bstart[p], bstart[p + 1]); its first mblocks blocks take the cell moments,
// the rest the boundary faces.
template <typename T>
struct MomBatchRec {
    MomArgs<T> m;
    BfArgs<T> f;
    int mblocks;
};

template <typename T, bool WITH_F, bool WITH_P>
__global__ void __launch_bounds__(kRedBlock) moments_batch_kernel(const MomBatchRec<T>* __restrict__ tab,
                                                                  const int* __restrict__ bstart, int B)
{
    const int p = batch_find(bstart, B, blockIdx.x);
    const int b0 = __ldg(bstart + p), nblk = __ldg(bstart + p + 1) - b0, lb = blockIdx.x - b0;
    const int mb = tab[p].mblocks;
    if (lb < mb) {
        const MomArgs<T> a = tab[p].m;
        moments_body<T, WITH_F, WITH_P>(a, lb, mb);
    } else {
        const BfArgs<T> a = tab[p].f;
        bflux_body(a, lb - mb, nblk - mb);
    }
}

int grid_for(long long n, int block, int cap)
{
    long long g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

template <typename T, int MODE>
SweepArgs<T> sweep_args(const Plan& P)
{
    SweepArgs<T> a{};
    a.nx = P.nx; a.ny = P.ny; a.N = P.N; a.K = P.K; a.nb = P.nb; a.nsteps = P.nx + 31;
    if constexpr (sizeof(T) == 8) {
        a.acoef = P.acoef; a.bcoef = P.bcoef; a.sigt = P.sigt; a.shift = P.shift; a.src = P.src;
    } else {
        a.acoef = P.acoef_f; a.bcoef = P.bcoef_f; a.sigt = P.sigt_f; a.shift = P.shift_f; a.src = P.src_f;
    }
    a.rsw = P.rsw;
    a.I = static_cast<T*>(P.I);
    a.iold = P.In ? static_cast<const T*>(P.In) : a.I;
    a.edge = static_cast<T*>(P.edge);
    a.inflow = P.inflow;
    if (MODE == kSrcAdjoint) {   // transposed kinetic step: reflected direction, adjoint source
        if constexpr (sizeof(T) == 8) {
            a.src = P.adj_a; a.ax = P.adj_x; a.ay = P.adj_y;
        } else {
            a.src = P.adj_a_f; a.ax = P.adj_x_f; a.ay = P.adj_y_f;
            if (P.adj_sigt_f) a.sigt = P.adj_sigt_f;
        }
        a.I = static_cast<T*>(P.Iadj);
        a.inflow = P.adj_inflow;
    }
    if (MODE == kSrcDelta) {   // increment sweep: residual source, zero inflow increment, correction
        a.src = static_cast<const T*>(P.R);
        if constexpr (sizeof(T) == 8) a.shift = P.corr;
        else {
            a.shift = P.corr_f;
            a.sigt = P.sigt_d;
        }
        a.inflow = nullptr;
    }
    a.qw = P.qw;
    a.perm = P.perm; a.qmu = P.qmu; a.qeta = P.qeta;
    a.err = &P.status->error;
    a.done = &P.status->done;
    a.tasks = &P.status->sweep_tasks;
    a.exits = &P.status->sweep_exits;
    a.arrived = &P.status->sweep_arrived;
    a.mode = &P.status->sweep_mode;
    a.wait_cycles = P.wait_cycles;
    return a;
}

// One problem's sweep.  A cooperative launch guarantees the whole grid
// resident, so the units are placed without a check-in and the warps leave
// without counting: 2 us less, of 38 to 130 per iteration.  But it starts only
// when its whole grid fits, so that the sweeps of several streams take turns
// where plain launches share the SMs.  Source iteration on meshes 64 cells
// wide, us an iteration with 1 / 2 / 4 / 8 streams, cooperative | plain | the
// sweep before the roles of its warps were split (plain):
//   24 CTAs  44 / 46 /  52 /  63 | 46 / 48 /  53 /  65 |  59 /  63 /  78 / 118
//   60       65 / 67 /  75 / 137 | 66 / 69 /  77 / 113 |  86 /  91 / 110 / 168
//   72       71 / 73 /  95 / 187 | 73 / 75 /  90 / 133 |  95 /  99 / 125 / 185
//   84       77 / 79 / 120 / 238 | 79 / 82 / 100 / 145 | 103 / 108 / 136 / 205
//   96       85 / 88 / 156       | 86 / 89 / 112 / 163 | 113 / 120 / 150 / 222
// (152 CTAs, 128^2 S8: 69 / 100 / 196 | 71 / 90 / 116).  So cooperative where two
// such launches fit at once: there no number of streams is slower than with
// that form.  Beyond, and where the grid does not fit the SMs that the context
// may use, plain with its check-in.
template <typename T, int MODE>
cudaError_t launch_sweep_args(SweepArgs<T> a, int grid, int num_sms, cudaStream_t st)
{
    using SM = SweepSmem<T, MODE>;
    SweepBatch<T> none{};
    if (2 * grid <= num_sms) {
        a.resident = 1;
        void* args[] = {&a, &none};
        const cudaError_t e = cudaLaunchCooperativeKernel((const void*)sweep_kernel<T, MODE, false>, dim3(grid),
                                                          dim3(SM::THREADS), args, SM::bytes, st);
        if (e != cudaErrorCooperativeLaunchTooLarge) return e;
        cudaGetLastError();
    }
    a.resident = 0;
    sweep_kernel<T, MODE, false><<<grid, SM::THREADS, SM::bytes, st>>>(a, none);
    return cudaGetLastError();
}

template <typename T, int MODE>
cudaError_t launch_sweep_t(Plan& P, cudaStream_t st)
{
    const SweepArgs<T> a = sweep_args<T, MODE>(P);
    return launch_sweep_args<T, MODE>(a, P.sweep_grid, P.num_sms, st);
}

template <typename T, int MODE>
cudaError_t launch_sweep_batch_t(const BatchTables& bt, cudaStream_t st)
{
    SweepBatch<T> b{};
    b.probs = static_cast<const SweepArgs<T>*>(bt.sweep);
    b.seg_start = bt.seg_start;
    b.seg_prob = bt.seg_prob;
    b.seg_band = bt.seg_band;
    b.nseg = bt.nseg;
    b.ntasks = bt.ntasks;
    b.dynamic = bt.dynamic;
    b.tasks = &bt.status->sweep_tasks;
    b.exits = &bt.status->sweep_exits;
    b.arrived = &bt.status->sweep_arrived;
    b.mode = &bt.status->sweep_mode;
    b.err = &bt.status->error;
    b.wait_cycles = bt.wait_cycles;
    sweep_kernel<T, MODE, true><<<bt.sweep_grid, SweepSmem<T, MODE>::THREADS, SweepSmem<T, MODE>::bytes, st>>>(
        SweepArgs<T>{}, b);
    return cudaGetLastError();
}

// The fixed-point sums where the set allows them for the moments asked
// (mom_quads), except where the iteration amplifies the 1e-16 by
// which they differ from the loop's, so that there the sums keep their order
// and their bits.  Second order: the limiter makes it 3e-10 within 250
// iterations (256^2 S12 channel).  Steady pseudo-time (mquad_moments is then 0):
// its runs over media of several decades stop the FP32 synthetic solve after
// a few steps; 53x269 S14 over six decades ends 2e-9 apart, batches of such
// meshes, whose iteration counts then differ by one, up to 2e-6.  The loop
// takes 30.5 us there instead of 18.8 (256^2 S12), 5% of an iteration.
const MomQuad* moments_quads(const Plan& P, bool with_P)
{
    return P.mquad_moments >= (with_P ? 6 : 3) && P.order != 2 ? P.mquad : nullptr;
}

// Blocks of the cell moments: one cell per thread over reflection quads (no
// nearly empty last turn: 1024^2 would take 3.4 turns of 8 blocks per SM),
// else a grid-stride loop that re-uses the block's coefficient table.
template <typename T>
int moments_blocks(const Plan& P, bool with_P)
{
    return grid_for(P.N, kRedBlock, sizeof(T) == 8 && moments_quads(P, with_P) ? INT_MAX : P.num_sms * 8);
}

template <typename T>
size_t moments_smem(int K)
{
    return (size_t)K * (6 * sizeof(T) + sizeof(int)) + 16;
}

template <typename T>
BfArgs<T> bflux_args(const Plan& P, double* fb_out, const int* done)
{
    BfArgs<T> f{};
    f.nx = P.nx; f.ny = P.ny; f.K = P.K;
    f.I = static_cast<const T*>(P.I);
    f.sidx = P.sidx;
    f.mu = P.omu; f.eta = P.oeta; f.w = P.ow;
    f.inflow = P.inflow;
    f.fb = fb_out;
    f.done = done;
    return f;
}

template <typename T>
cudaError_t launch_moments_t(const Plan& P, bool with_F, bool with_P, double* rho_out, double* Fout,
                             double* Pout, bool gsis_correct, double* fb_out, bool force, cudaStream_t st)
{
    MomArgs<T> a{};
    a.nx = P.nx; a.ny = P.ny; a.N = P.N; a.K = P.K;
    a.I = static_cast<const T*>(P.I);
    a.sidx = P.sidx;
    a.pairs = P.has_mpair ? P.mpair : nullptr;
    a.quads = moments_quads(P, with_P);
    a.mu = P.omu;
    a.eta = P.oeta;
    a.w = P.ow;
    a.rho = rho_out;
    a.Fx = Fout ? Fout : P.Fx;
    a.Fy = Fout ? Fout + P.N : P.Fy;
    if (with_P) { a.Pxx = Pout; a.Pxy = Pout + P.N; a.Pyy = Pout + 2 * (size_t)P.N; }
    a.rho_new = gsis_correct ? P.rho_m : nullptr;
    a.done = force ? nullptr : &P.status->done;
    const size_t smem = moments_smem<T>(P.K);
    const int grid = moments_blocks<T>(P, with_P);
    if (P.order != 2) {   // cells and boundary faces in one launch
        static_assert(kRedBlock == 256, "the boundary-flux blocks take 256 threads");
        const BfArgs<T> f = bflux_args<T>(P, fb_out, a.done);
        const int fg = grid_for((long long)P.nbf * 32, 256, P.num_sms * 4);
        if (with_P) moments_bflux_kernel<T, true, true><<<grid + fg, kRedBlock, smem, st>>>(a, f, grid);
        else if (with_F) moments_bflux_kernel<T, true, false><<<grid + fg, kRedBlock, smem, st>>>(a, f, grid);
        else moments_bflux_kernel<T, false, false><<<grid + fg, kRedBlock, smem, st>>>(a, f, grid);
        return cudaGetLastError();
    }
    if (with_P) moments_kernel<T, true, true><<<grid, kRedBlock, smem, st>>>(a);
    else if (with_F) moments_kernel<T, true, false><<<grid, kRedBlock, smem, st>>>(a);
    else moments_kernel<T, false, false><<<grid, kRedBlock, smem, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (P.order == 2) return launch_uw2_bflux(P, fb_out, a.done, st);   // reconstructed outgoing faces
    bflux_kernel<T><<<grid_for((long long)P.nbf * 32, 256, P.num_sms * 4), 256, 0, st>>>(
        bflux_args<T>(P, fb_out, a.done));
    return cudaGetLastError();
}

template <typename T, int MODE, bool BATCH>
cudaError_t sweep_attr()
{
    return cudaFuncSetAttribute(sweep_kernel<T, MODE, BATCH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)SweepSmem<T, MODE>::bytes);
}

// Raises the dynamic shared-memory limit of fn to at least `bytes` (never
// lowers it: plans of different sizes may launch concurrently).
cudaError_t raise_smem_limit(const void* fn, size_t bytes)
{
    static std::mutex mu;
    static std::map<const void*, size_t> have;
    std::lock_guard<std::mutex> g(mu);
    size_t& h = have[fn];
    if (bytes <= h) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) h = bytes;
    return e;
}

template <typename T>
cudaError_t prepare_t(int K)
{
    static std::once_flag once;
    static cudaError_t first = cudaSuccess;
    std::call_once(once, [] {
        cudaError_t e;
        if ((e = sweep_attr<T, kSrcPlain, false>()) != cudaSuccess ||
            (e = sweep_attr<T, kSrcPseudoTime, false>()) != cudaSuccess ||
            (e = sweep_attr<T, kSrcAdjoint, false>()) != cudaSuccess ||
            (e = sweep_attr<T, kSrcDelta, false>()) != cudaSuccess ||
            (e = sweep_attr<T, kSrcPlain, true>()) != cudaSuccess ||
            (e = sweep_attr<T, kSrcPseudoTime, true>()) != cudaSuccess)
            first = e;
    });
    if (first != cudaSuccess) return first;
    const size_t ms = moments_smem<T>(K);
    cudaError_t e;
    if ((e = raise_smem_limit((const void*)moments_kernel<T, true, true>, ms)) != cudaSuccess) return e;
    if ((e = raise_smem_limit((const void*)moments_kernel<T, true, false>, ms)) != cudaSuccess) return e;
    if ((e = raise_smem_limit((const void*)moments_kernel<T, false, false>, ms)) != cudaSuccess) return e;
    if ((e = raise_smem_limit((const void*)moments_batch_kernel<T, true, false>, ms)) != cudaSuccess) return e;
    if ((e = raise_smem_limit((const void*)moments_bflux_kernel<T, true, true>, ms)) != cudaSuccess) return e;
    if ((e = raise_smem_limit((const void*)moments_bflux_kernel<T, true, false>, ms)) != cudaSuccess) return e;
    if ((e = raise_smem_limit((const void*)moments_bflux_kernel<T, false, false>, ms)) != cudaSuccess) return e;
    return raise_smem_limit((const void*)moments_batch_kernel<T, false, false>, ms);
}

template <typename T, int MODE, bool BATCH>
int sweep_occupancy()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sweep_kernel<T, MODE, BATCH>,
                                                      SweepSmem<T, MODE>::THREADS, SweepSmem<T, MODE>::bytes) != cudaSuccess)
        return 0;
    return n;
}

}  // namespace

// Asked of the driver once per device: both are constants of the device, and
// the clock rate costs 0.3-0.6 ms a query (64x64 S8 transport sweep: 684 us a
// call with two queries, 120-205 us without them and the set-up below).
DeviceInfo device_info()
{
    constexpr int kMaxDev = 64;
    static std::atomic<long long> known[kMaxDev];   // sms << 32 | clock_khz; 0: not asked yet
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return DeviceInfo{0, 0};
    long long v = dev < kMaxDev ? known[dev].load(std::memory_order_relaxed) : 0;
    if (v == 0) {
        int n = 0, khz = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev) != cudaSuccess)
            return DeviceInfo{0, 0};
        if (khz <= 0) khz = 2000000;
        v = ((long long)n << 32) | (long long)khz;
        if (dev < kMaxDev) known[dev].store(v, std::memory_order_relaxed);
    }
    return DeviceInfo{(int)(v >> 32), (int)(v & 0xffffffffll)};
}

cudaError_t launch_setup(const Plan& P, cudaStream_t st)
{
    const int tot = P.K * (P.nx + P.ny);
    coef_kernel<<<grid_for(tot, 256, 1024), 256, 0, st>>>(
        P.nx, P.ny, P.K, P.dx, P.dy, P.qmu, P.qeta, const_cast<double*>(P.acoef),
        const_cast<double*>(P.bcoef), P.fp32 ? const_cast<float*>(P.acoef_f) : nullptr,
        P.fp32 ? const_cast<float*>(P.bcoef_f) : nullptr);
    return cudaGetLastError();
}

// Per-cell set-up and the FP64 reciprocal table (pseudo-time controls given).
cudaError_t launch_cell_setup(const Plan& P, double cfl_p, double beta, cudaStream_t st)
{
    cell_setup_kernel<<<grid_for(P.N, 256, P.num_sms * 8), 256, 0, st>>>(
        P.nx, P.ny, P.dx, P.dy, P.sigma_a, P.sigma_s, P.q, P.inflow, P.nbf * P.K, P.shift0, cfl_p, beta, P.sigt,
        P.fp32 ? P.sigt_f : nullptr, P.shift, P.fp32 ? P.shift_f : nullptr,
        P.scheme == GSIS_SCHEME_GSIS || P.K == 0, P.diag, P.cx, P.cy, P.hw,
        P.bface, P.gw, P.gw_f, P.sigt_d, &P.status->error);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (!P.fp32 && P.nrep > 0) {
        // wide tiles (fewer steps that two blocks share) where they still give
        // every SM several blocks
        auto tiles = [&](int cols) { return (unsigned)((P.nx + 62 + cols - 1) / cols); };
        auto go = [&](auto kernel, int cols) {
            kernel<<<dim3(tiles(cols), P.nb, P.nrep), 256, 0, st>>>(P.nx, P.ny, P.nb, P.rrep, P.rnext, P.qmu, P.qeta,
                                                                    P.acoef, P.bcoef, P.sigt, P.shift,
                                                                    const_cast<double*>(P.rsw));
        };
        if ((long long)tiles(64) * P.nb * P.nrep >= 4ll * P.num_sms) go(recip_kernel<64>, 64);
        else go(recip_kernel<16>, 16);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_init_state(const Plan& P, cudaStream_t st)
{
    const int g = grid_for(P.N, 256, P.num_sms * 8);
    fill_kernel<<<g, 256, 0, st>>>(P.rho_m, P.N, 0.0);
    fill_kernel<<<g, 256, 0, st>>>(P.rho_h, P.N, 0.0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (P.order == 2) {   // no correction of the initial intensities
        fill_kernel<<<g, 256, 0, st>>>(P.corr, P.N, 0.0);
        if (P.fp32) fillf_kernel<<<g, 256, 0, st>>>(P.corr_f, P.N, 0.f);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (P.pt || P.order == 2) {   // I^0 = 0 (the delta form reads it)
        const size_t n = (size_t)P.K * P.N;
        if (P.fp32) fillf_kernel<<<grid_for((long long)n, 256, P.num_sms * 16), 256, 0, st>>>(static_cast<float*>(P.I), n, 0.f);
        else fill_kernel<<<grid_for((long long)n, 256, P.num_sms * 16), 256, 0, st>>>(static_cast<double*>(P.I), n, 0.0);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return launch_source_from(P, P.rho_m, st);
}

cudaError_t launch_source_from(const Plan& P, const double* rho_in, cudaStream_t st)
{
    source_kernel<<<grid_for(P.N, 256, P.num_sms * 8), 256, 0, st>>>(P.N, P.sigma_s, P.q, rho_in, P.src,
                                                                    P.fp32 ? P.src_f : nullptr);
    return cudaGetLastError();
}

cudaError_t launch_sweep(Plan& P, cudaStream_t st)
{
    if (P.pt && P.X && !P.fp32) {
        // FP64 pseudo-time form with its source already combined per ordinate
        // (X = src + shift I^m, formed by the update kernel): the plain sweep
        // over X takes one FP64 operation per update fewer, same bits
        SweepArgs<double> a = sweep_args<double, kSrcPlain>(P);
        a.src = P.X;
        a.src_stride = P.N;
        return launch_sweep_args<double, kSrcPlain>(a, P.sweep_grid, P.num_sms, st);
    }
    if (P.fp32 && P.pt && P.X_f) {
        // FP32 time step with its source combined per ordinate (X = src +
        // I^n/(c dt)) and its diagonal sigma_t + 1/(c dt): the plain sweep
        // over X reads two cell windows instead of four
        SweepArgs<float> a = sweep_args<float, kSrcPlain>(P);
        a.src = P.X_f;
        a.src_stride = P.N;
        a.sigt = P.sigt_d;
        return launch_sweep_args<float, kSrcPlain>(a, P.sweep_grid, P.num_sms, st);
    }
    if (P.fp32) {
        return P.pt ? launch_sweep_t<float, kSrcPseudoTime>(P, st)
                    : launch_sweep_t<float, kSrcPlain>(P, st);
    }
    return P.pt ? launch_sweep_t<double, kSrcPseudoTime>(P, st) : launch_sweep_t<double, kSrcPlain>(P, st);
}

cudaError_t launch_delta_sweep(Plan& P, cudaStream_t st)
{
    return P.fp32 ? launch_sweep_t<float, kSrcDelta>(P, st) : launch_sweep_t<double, kSrcDelta>(P, st);
}

cudaError_t launch_adjoint_sweep(Plan& P, cudaStream_t st)
{
    return P.fp32 ? launch_sweep_t<float, kSrcAdjoint>(P, st) : launch_sweep_t<double, kSrcAdjoint>(P, st);
}

template <typename T>
cudaError_t launch_sweep_pt_into_t(Plan& P, const void* src, const void* iold, void* out, cudaStream_t st)
{
    SweepArgs<T> a = sweep_args<T, kSrcPseudoTime>(P);
    a.src = static_cast<const T*>(src);
    a.iold = static_cast<const T*>(iold);
    a.I = static_cast<T*>(out);
    a.inflow = nullptr;
    return launch_sweep_args<T, kSrcPseudoTime>(a, P.sweep_grid, P.num_sms, st);
}

cudaError_t launch_sweep_pt_into(Plan& P, const void* src, const void* iold, void* out, cudaStream_t st)
{
    return P.fp32 ? launch_sweep_pt_into_t<float>(P, src, iold, out, st)
                  : launch_sweep_pt_into_t<double>(P, src, iold, out, st);
}

// Moments of the last sweep into the given outputs: rho always, F when
// with_F (Fout or the plan's F arrays), P when with_P (plus drho/3 on the
// diagonal when gsis_correct), boundary fluxes into fb_out.  force: run even
// after the device has stopped the iteration (final outputs).
cudaError_t launch_moments_to(const Plan& P, bool with_F, bool with_P, double* rho_out, double* Fout,
                              double* Pout, bool gsis_correct, double* fb_out, bool force, cudaStream_t st)
{
    if (P.fp32)
        return launch_moments_t<float>(P, with_F, with_P, rho_out, Fout, Pout, gsis_correct, fb_out, force, st);
    return launch_moments_t<double>(P, with_F, with_P, rho_out, Fout, Pout, gsis_correct, fb_out, force, st);
}

size_t sweep_batch_rec_bytes(int fp32)
{
    return fp32 ? sizeof(SweepArgs<float>) : sizeof(SweepArgs<double>);
}

void sweep_batch_rec(const Plan& P, void* out)
{
    if (P.fp32) {
        SweepArgs<float> a = P.pt ? sweep_args<float, kSrcPseudoTime>(P) : sweep_args<float, kSrcPlain>(P);
        if (P.pt && P.X_f) {   // the plain sweep over the per-ordinate source, as launch_sweep does
            a = sweep_args<float, kSrcPlain>(P);
            a.src = P.X_f;
            a.src_stride = P.N;
            a.sigt = P.sigt_d;
        }
        std::memcpy(out, &a, sizeof(a));
    } else {
        const SweepArgs<double> a = P.pt ? sweep_args<double, kSrcPseudoTime>(P) : sweep_args<double, kSrcPlain>(P);
        std::memcpy(out, &a, sizeof(a));
    }
}

cudaError_t launch_sweep_batch(const BatchTables& bt, cudaStream_t st)
{
    if (bt.fp32)   // with per-ordinate sources (ord_blocks > 0) the records describe plain sweeps
        return bt.pt && bt.ord_blocks == 0 ? launch_sweep_batch_t<float, kSrcPseudoTime>(bt, st)
                                           : launch_sweep_batch_t<float, kSrcPlain>(bt, st);
    return bt.pt ? launch_sweep_batch_t<double, kSrcPseudoTime>(bt, st) : launch_sweep_batch_t<double, kSrcPlain>(bt, st);
}

size_t mom_batch_rec_bytes(int fp32)
{
    return fp32 ? sizeof(MomBatchRec<float>) : sizeof(MomBatchRec<double>);
}

template <typename T>
int mom_batch_rec_t(const Plan& P, bool with_F, void* out)
{
    MomBatchRec<T> r{};
    r.m.nx = P.nx; r.m.ny = P.ny; r.m.N = P.N; r.m.K = P.K;
    r.m.I = static_cast<const T*>(P.I);
    r.m.sidx = P.sidx;
    r.m.pairs = P.has_mpair ? P.mpair : nullptr;
    r.m.quads = moments_quads(P, false);
    r.m.mu = P.omu; r.m.eta = P.oeta; r.m.w = P.ow;
    r.m.rho = P.rho_h;
    r.m.Fx = with_F ? P.Fx : nullptr;
    r.m.Fy = with_F ? P.Fy : nullptr;
    r.m.done = &P.status->done;
    r.f = bflux_args<T>(P, P.fb, &P.status->done);
    r.mblocks = moments_blocks<T>(P, false);
    std::memcpy(out, &r, sizeof(r));
    return r.mblocks + grid_for((long long)P.nbf * 32, kRedBlock, P.num_sms * 4);
}

// Batched record of the moments of one GSIS / SI iteration (rho^{m+1/2},
// F^{m+1/2} when with_F, boundary fluxes); returns the problem's blocks.
int mom_batch_rec(const Plan& P, bool with_F, void* out)
{
    return P.fp32 ? mom_batch_rec_t<float>(P, with_F, out) : mom_batch_rec_t<double>(P, with_F, out);
}

cudaError_t launch_moments_batch(const BatchTables& bt, cudaStream_t st)
{
    const int fp32 = bt.fp32;
    const size_t smem = fp32 ? moments_smem<float>(bt.maxK) : moments_smem<double>(bt.maxK);
    if (fp32) {
        const auto* tab = static_cast<const MomBatchRec<float>*>(bt.mom);
        if (bt.with_F) moments_batch_kernel<float, true, false><<<bt.mom_blocks, kRedBlock, smem, st>>>(tab, bt.mom_bstart, bt.B);
        else moments_batch_kernel<float, false, false><<<bt.mom_blocks, kRedBlock, smem, st>>>(tab, bt.mom_bstart, bt.B);
    } else {
        const auto* tab = static_cast<const MomBatchRec<double>*>(bt.mom);
        if (bt.with_F) moments_batch_kernel<double, true, false><<<bt.mom_blocks, kRedBlock, smem, st>>>(tab, bt.mom_bstart, bt.B);
        else moments_batch_kernel<double, false, false><<<bt.mom_blocks, kRedBlock, smem, st>>>(tab, bt.mom_bstart, bt.B);
    }
    return cudaGetLastError();
}

cudaError_t prepare_kernels(int K, int fp32, int pt)
{
    (void)pt;
    return fp32 ? prepare_t<float>(K) : prepare_t<double>(K);
}

int sweep_max_active_blocks(int fp32, int pt)
{
    // one grid for every variant a plan may launch (forward, pseudo-time,
    // adjoint): every warp pair must be resident, so take the smallest
    (void)pt;
    if (fp32)
        return std::min({sweep_occupancy<float, kSrcPlain, false>(), sweep_occupancy<float, kSrcPseudoTime, false>(),
                         sweep_occupancy<float, kSrcAdjoint, false>(), sweep_occupancy<float, kSrcDelta, false>(),
                         sweep_occupancy<float, kSrcPlain, true>(),
                         sweep_occupancy<float, kSrcPseudoTime, true>()});
    return std::min({sweep_occupancy<double, kSrcPlain, false>(), sweep_occupancy<double, kSrcPseudoTime, false>(),
                     sweep_occupancy<double, kSrcAdjoint, false>(), sweep_occupancy<double, kSrcDelta, false>(),
                     sweep_occupancy<double, kSrcPlain, true>(),
                     sweep_occupancy<double, kSrcPseudoTime, true>()});
}

}  // namespace gsis
