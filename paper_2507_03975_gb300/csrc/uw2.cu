// Second-order upwind (UW2) kinetic step in the paper's delta form (Sec. 4.1):
// the residual of the UW2 equations at the stored intensities, and the
// boundary kinetic flux with reconstructed outgoing face values.  The
// increment sweep itself is the sweep kernel's delta mode (csrc/sweep.cu).
//
// Per ordinate s and cell i (sorted direction index, I^m = I + corr):
//  * least-squares gradient with the adaptive shifted neighbour positions
//    (Sec. 5.2, Eqs. (shifted_j), (new_vector), (LSF_mdf)); on the Cartesian
//    mesh G_x = sum_{E,W} g_j (I_j - I_i) with the set-up weights g_j;
//  * Barth-Jespersen limiter psi (or none): the unlimited change to each face
//    Delta_f = G . (x_f - x_i) is scaled so that no face value leaves
//    [min, max] of the cell and its face neighbours;
//  * face values I_i + psi G . (x_f - x_i) (Eq. (Ii,k)) from the upwind side
//    (Eq. (Iij)), the inflow on incoming boundary faces;
//  * R = S - sigma_t I_i - mu (I_E - I_W)/dx - eta (I_N - I_S)/dy
//    (Eq. (RTE_d_res), steady, per unit volume).
// The residual kernel marches (a warp per ordinate and column strip, each
// limited gradient and face value formed once); the boundary flux reads
// global memory.
#include <cuda_runtime.h>

#include "divide.cuh"
#include "gsis_internal.cuh"

namespace gsis {

namespace {

template <typename T>
struct Uw2Args {
    int nx, ny, N, K;
    const T* I;                 // [K][N] stored intensities
    const T* corr;              // [N] isotropic correction (I^m = I + corr), or null
    const T* gw;                // [4][N] gradient weights E, W, N, S
    const double* dx; const double* dy;
    const T* src; const T* sigt;
    const double* qmu; const double* qeta; const int* perm;
    const double* inflow;       // [nbf][K] original direction index, or null
    T* R;                       // [K][N] out
    int limiter;                // 0 Barth-Jespersen, 1 none
    const int* done;
};

template <typename T>
__device__ __forceinline__ T value(const Uw2Args<T>& a, const T* Is, int c)
{
    return a.corr ? Is[c] + a.corr[c] : Is[c];
}

// Limited gradient from the cell value, the existing face neighbours' values
// and the least-squares weights.  The Barth-Jespersen factor uses that the
// four face changes are +-dfx, +-dfy: min over faces of the admissible ratio
// = min(hi - Ic, Ic - lo) / max(|dfx|, |dfy|) (one division, and none when no
// face needs limiting; correctly rounded division is monotone, so this is
// the per-face minimum exactly).
template <typename T>
__device__ __forceinline__ void limited_gradient_vals(T Ic, bool hE, T vE, bool hW, T vW, bool hN, T vN, bool hS,
                                                      T vS, T wE, T wW, T wN, T wS, T hx, T hy, int limiter, T& gx,
                                                      T& gy)
{
    T lo = Ic, hi = Ic;
    gx = T(0);
    gy = T(0);
    if (hE) { gx = fma(wE, vE - Ic, gx); lo = fmin(lo, vE); hi = fmax(hi, vE); }
    if (hW) { gx = fma(wW, vW - Ic, gx); lo = fmin(lo, vW); hi = fmax(hi, vW); }
    if (hN) { gy = fma(wN, vN - Ic, gy); lo = fmin(lo, vN); hi = fmax(hi, vN); }
    if (hS) { gy = fma(wS, vS - Ic, gy); lo = fmin(lo, vS); hi = fmax(hi, vS); }
    if (limiter != 0) return;
    const T dm = fmax(fabs(T(0.5) * hx * gx), fabs(T(0.5) * hy * gy));
    const T room = fmin(hi - Ic, Ic - lo);
    if (dm > T(0) && room < dm) {
        const T psi = room / dm;
        gx *= psi;
        gy *= psi;
    }
}

// Limited gradient of ordinate Is at cell (i, j), values from global memory.
template <typename T>
__device__ __forceinline__ void limited_gradient(const Uw2Args<T>& a, const T* Is, int i, int j, T& gx, T& gy)
{
    const int nx = a.nx, ny = a.ny, N = a.N;
    const int c = i + nx * j;
    const bool hE = i + 1 < nx, hW = i > 0, hN = j + 1 < ny, hS = j > 0;
    limited_gradient_vals(value(a, Is, c), hE, hE ? value(a, Is, c + 1) : T(0), hW, hW ? value(a, Is, c - 1) : T(0),
                          hN, hN ? value(a, Is, c + nx) : T(0), hS, hS ? value(a, Is, c - nx) : T(0), a.gw[c],
                          a.gw[N + c], a.gw[2 * (size_t)N + c], a.gw[3 * (size_t)N + c], (T)a.dx[i], (T)a.dy[j],
                          a.limiter, gx, gy);
}

// The Barth-Jespersen factor from the differences to the neighbours, east,
// west (negated), ahead, behind (negated; 0 where there is none) and the face
// changes hx/2 G_x, hy/2 G_y: false where the limiter does not act.  Rounding is
// monotone, so the largest difference is the difference to the largest value.
// In double on the bits: numbers of which one is >= 0 are ordered like their
// bits as signed integers; a comparison, a sign change or a magnitude would be
// an FP64 pipe instruction each (19 cycles per SM).
__device__ __forceinline__ bool limit(double dE, double dWn, double dA, double dBn, double cx, double cy, double& psi)
{
    constexpr long long S = 1ll << 63;
    const long long e = __double_as_longlong(dE), w = __double_as_longlong(dWn) ^ S, a = __double_as_longlong(dA),
                    b = __double_as_longlong(dBn) ^ S;
    const long long up = max(max(max(e, w), max(a, b)), 0ll), dn = max(max(max(e ^ S, w ^ S), max(a ^ S, b ^ S)), 0ll);
    const long long dm = max(__double_as_longlong(cx) & ~S, __double_as_longlong(cy) & ~S), room = min(up, dn);
    if (!(room < dm)) return false;
    psi = ratio(__longlong_as_double(room), __longlong_as_double(dm));
    return true;
}

__device__ __forceinline__ bool limit(float dE, float dWn, float dA, float dBn, float cx, float cy, float& psi)
{
    const float up = fmaxf(fmaxf(fmaxf(dE, -dWn), fmaxf(dA, -dBn)), 0.f);
    const float dn = fmaxf(fmaxf(fmaxf(-dE, dWn), fmaxf(-dA, dBn)), 0.f);
    const float dm = fmaxf(fabsf(cx), fabsf(cy)), room = fminf(up, dn);
    if (!(dm > 0.f) || !(room < dm)) return false;
    psi = room / dm;
    return true;
}

// Residual, one warp per ordinate, 29 columns and kUwRows rows.  The FP64
// pipe bounds it, so every quantity that two cells share is formed once:
// lanes are columns (the east difference is minus the right lane's west
// one, a face value goes to the downwind lane by shuffle) and the warp marches
// along y from the upwind side (the difference to the row behind and the
// face value on it are in registers).  Lanes at the ends and one row before
// the first only feed the others: 29 of 32 lanes, 16 of 17 rows count (32 rows,
// 8 warps per block: 582 us; 16 and 4: 565).  24 FP64 operations per cell and
// ordinate, 4 more with the limiter and six for its ratio where it acts; the cell-tile form before took FP64 comparisons, divisions
// by the spacings and each shared quantity twice.  The same bits: the
// limiter amplifies a rounding difference of 1e-16 to 3e-10 within 250
// iterations.  256^2 S12, FP64: 748 -> 482 us, without the limiter 362 us.
constexpr int kUwCols = 29, kUwRows = 16, kUwWarps = 4;
static_assert(kUwRows <= 32, "one lane holds 1/dy of one row");

template <typename T>
__global__ void __launch_bounds__(kUwWarps * 32) uw2_residual_kernel(const Uw2Args<T> a, int sx)
{
    if (a.done && ld_volatile_int(a.done)) return;
    const int lane = threadIdx.x & 31, s = blockIdx.y * kUwWarps + (threadIdx.x >> 5);
    if (s >= a.K) return;
    const int nx = a.nx, ny = a.ny, N = a.N, K = a.K;
    const int bx = blockIdx.x % sx, by = blockIdx.x / sx;
    const double mu = a.qmu[s], eta = a.qeta[s];
    const bool xp = mu >= 0.0, yp = eta >= 0.0;
    const int k = a.perm[s];
    const int i = bx * kUwCols + lane - (xp ? 2 : 1);
    const bool in = i >= 0 && i < nx;
    const bool hE = in && i + 1 < nx, hW = in && i > 0;
    const bool counts = in && (xp ? lane >= 2 && lane <= 30 : lane >= 1 && lane <= 29);
    const int ic = min(max(i, 0), nx - 1);
    const T hx = (T)a.dx[ic], hx2 = T(0.5) * hx, yx = T(1) / hx;
    const T sx2 = xp ? hx2 : -hx2, am = (T)fabs(mu), ae = (T)fabs(eta);
    const int ja = by * kUwRows, n = min(ny, ja + kUwRows) - ja;
    const int dj = yp ? 1 : -1;
    const int jf = yp ? ja : ja + n - 1;             // first row that counts
    const T* Is = a.I + (size_t)s * N;
    T* Rs = a.R + (size_t)s * N;
    auto row_in = [&](int j) { return j >= 0 && j < ny; };
    auto at = [&](int j) -> T {
        if (!in || !row_in(j)) return T(0);
        return value(a, Is, i + nx * j);
    };
    const int t0 = row_in(jf - dj) ? -1 : 0;
    int j = jf + t0 * dj;
    T Ic = at(j), vA = at(j + dj);
    T dBn = row_in(j - dj) ? Ic - at(j - dj) : T(0);  // from the row behind
    T fB = T(0);                                      // face value on its side
    if (t0 == 0 && a.inflow && in) fB = (T)a.inflow[(size_t)(yp ? 2 * ny + i : 2 * ny + nx + i) * K + k];
    // lane l: dy / 2 and 1/dy of row t = l
    const T hl = (T)a.dy[min(max(jf + lane * dj, 0), ny - 1)], hl2 = T(0.5) * hl, ry = T(1) / hl;
    const T hy2_up = t0 < 0 ? T(0.5) * (T)a.dy[jf - dj] : T(0);   // of the row before the first
    for (int t = t0; t < n; ++t, j += dj) {
        const int c = ic + nx * j;
        const T vAA = at(j + 2 * dj);   // used in the next turn
        const T wE = a.gw[c], wW = a.gw[N + c], wN = a.gw[2 * (size_t)N + c], wS = a.gw[3 * (size_t)N + c];
        const T sv = a.src[c], sg = a.sigt[c];
        T dE = __shfl_down_sync(kFull, Ic, 1) - Ic, dWn = __shfl_up_sync(kFull, dE, 1);
        if (!hE) dE = T(0);   // a missing neighbour has weight 0 and difference 0
        if (!hW) dWn = T(0);
        const T dA = row_in(j + dj) ? vA - Ic : T(0);
        T gx = fma(wW, -dWn, fma(wE, dE, T(0)));
        T gy;
        if (yp) gy = fma(wS, -dBn, fma(wN, dA, T(0)));
        else gy = fma(wS, dA, fma(wN, -dBn, T(0)));
        const T hs = __shfl_sync(kFull, hl2, t < 0 ? 0 : t), hy2 = t < 0 ? hy2_up : hs;
        T psi;
        if (a.limiter == 0 && limit(dE, dWn, dA, dBn, hx2 * gx, hy2 * gy, psi)) {
            gx *= psi;
            gy *= psi;
        }
        const T fx = fma(sx2, gx, Ic);   // downwind faces
        T fy;
        if (yp) fy = fma(hy2, gy, Ic);
        else fy = fma(-hy2, gy, Ic);
        T fu = xp ? __shfl_up_sync(kFull, fx, 1) : __shfl_down_sync(kFull, fx, 1);
        if (t >= 0) {
            if (in && (xp ? i == 0 : i == nx - 1))
                fu = a.inflow ? (T)a.inflow[(size_t)(xp ? j : ny + j) * K + k] : T(0);
            // mu (E - W) = |mu| (downwind - upwind), the same bits
            T r = fma(-sg, Ic, sv);
            r -= div_by(am * (fx - fu), hx, yx);
            r -= div_by(ae * (fy - fB), __shfl_sync(kFull, hl, t), __shfl_sync(kFull, ry, t));
            if (counts) Rs[c] = r;
        }
        fB = fy;
        dBn = dA;
        Ic = vA;
        vA = vAA;
    }
}

// Kinetic net flux through every boundary face with UW2 face values of the
// stored intensities (outgoing: reconstructed boundary cell, incoming: inflow);
// one warp per face, lanes over the original direction index.
template <typename T>
__global__ void __launch_bounds__(256) uw2_bflux_kernel(const Uw2Args<T> a, const int* __restrict__ sidx,
                                                        const double* __restrict__ mu, const double* __restrict__ eta,
                                                        const double* __restrict__ w, double* fb)
{
    if (a.done && ld_volatile_int(a.done)) return;
    const int nx = a.nx, ny = a.ny, K = a.K, N = a.N;
    const int nbf = 2 * (nx + ny);
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int f = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; f < nbf; f += warps) {
        int i, j, axis;
        double sgn;
        if (f < ny) { i = 0; j = f; axis = 0; sgn = -1.0; }
        else if (f < 2 * ny) { i = nx - 1; j = f - ny; axis = 0; sgn = 1.0; }
        else if (f < 2 * ny + nx) { i = f - 2 * ny; j = 0; axis = 1; sgn = -1.0; }
        else { i = f - 2 * ny - nx; j = ny - 1; axis = 1; sgn = 1.0; }
        const int c = i + nx * j;
        T acc = T(0);
        for (int k = lane; k < K; k += 32) {
            const double on = sgn * (axis == 0 ? mu[k] : eta[k]);
            T Iface;
            if (on >= 0.0) {
                const T* Is = a.I + (size_t)sidx[k] * N;
                T gx, gy;
                limited_gradient(a, Is, i, j, gx, gy);
                const T h = (T)(axis == 0 ? a.dx[i] : a.dy[j]);
                Iface = fma((T)sgn * T(0.5) * h, axis == 0 ? gx : gy, value(a, Is, c));
            } else {
                Iface = a.inflow ? (T)a.inflow[(size_t)f * K + k] : T(0);
            }
            acc = fma((T)(w[k] * on), Iface, acc);
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if (lane == 0) fb[f] = (double)acc;
    }
}

int grid_for(long long n, int block, int cap)
{
    long long g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

template <typename T>
Uw2Args<T> uw2_args(const Plan& P, bool with_corr, const int* done)
{
    Uw2Args<T> a{};
    a.nx = P.nx; a.ny = P.ny; a.N = P.N; a.K = P.K;
    a.I = static_cast<const T*>(P.I);
    a.dx = P.dx; a.dy = P.dy;
    a.qmu = P.qmu; a.qeta = P.qeta; a.perm = P.perm;
    a.inflow = P.inflow;
    a.R = static_cast<T*>(P.R);
    a.limiter = P.limiter;
    a.done = done;
    if constexpr (sizeof(T) == 8) {
        a.corr = with_corr ? P.corr : nullptr;
        a.gw = P.gw; a.src = P.src; a.sigt = P.sigt;
    } else {
        a.corr = with_corr ? P.corr_f : nullptr;
        a.gw = P.gw_f; a.src = P.src_f; a.sigt = P.sigt_f;
    }
    return a;
}

}  // namespace

cudaError_t launch_uw2_residual(const Plan& P, cudaStream_t st)
{
    const int sx = (P.nx + kUwCols - 1) / kUwCols, sy = (P.ny + kUwRows - 1) / kUwRows;
    const dim3 grid(sx * sy, (P.K + kUwWarps - 1) / kUwWarps);
    if (P.fp32) uw2_residual_kernel<float><<<grid, kUwWarps * 32, 0, st>>>(uw2_args<float>(P, true, &P.status->done), sx);
    else uw2_residual_kernel<double><<<grid, kUwWarps * 32, 0, st>>>(uw2_args<double>(P, true, &P.status->done), sx);
    return cudaGetLastError();
}

cudaError_t launch_uw2_bflux(const Plan& P, double* fb_out, const int* done, cudaStream_t st)
{
    const int g = grid_for((long long)P.nbf * 32, 256, P.num_sms * 4);
    if (P.fp32)
        uw2_bflux_kernel<float><<<g, 256, 0, st>>>(uw2_args<float>(P, false, done), P.sidx, P.omu, P.oeta, P.ow,
                                                   fb_out);
    else
        uw2_bflux_kernel<double><<<g, 256, 0, st>>>(uw2_args<double>(P, false, done), P.sidx, P.omu, P.oeta,
                                                    P.ow, fb_out);
    return cudaGetLastError();
}

}  // namespace gsis
