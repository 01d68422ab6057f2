// Angular moments of FP64 intensities in fixed point: per cell
//   rho = sum w I,  F = sum w Omega I,  P = sum w Omega Omega I
// over quadrature sets closed under both axis reflections with equal weights
// and without very small coefficients (mom_quads; every level-symmetric set).
//
// Why not FP64 FMAs: GB300 issues one FP64 instruction per SM every 16
// cycles, 64 issue slots of one sub-partition.  Five of them per pair of
// ordinates kept the FP64 pipe 91 % busy and the kernel at 0.58 ms on
// 1024^2 S16, where reading the intensities once takes 0.18 ms.  A 32 x 32 +
// 64 bit integer multiply-add takes 4 issue slots, so the sums run in
// integers: about 30 slots per ordinate and cell instead of 160.  1024^2
// S16: 0.584 -> 0.259 ms (4.7 TB/s); 256^2 S12: 30.5 -> 18.8 us, with P 66.6 ->
// 26.0 us.
//
// Form.  The four reflections of an ordinate, (mu, eta), (-mu, eta),
// (mu, -eta), (-mu, -eta), share one weight, so a quad adds
//   w (I1 + I2 + I3 + I4)        to rho   (w mu^2, w eta^2: P_xx, P_yy)
//   w mu (I1 - I2 + I3 - I4)     to F_x
//   w eta (I1 + I2 - I3 - I4)    to F_y
//   w mu eta (I1 - I2 - I3 + I4) to P_xy.
// A value's 53-bit mantissa goes into a 64-bit integer d with the cell's
// largest exponent at bit 60 (eight bits below the mantissa's own), its last
// bit set (inexact values then err by less than a unit either way, without a
// bias), so the four-term sums are exact integer additions.  Coefficients
// are 62-bit integers c = coefficient * 2^62 (those of a moment add up to at
// most pi), as c = 2^32 ch + 4 cl (with P, whose coefficients w mu^2 get small, all
// 32 low bits are kept: cl there is the low word itself).
//
// Error.  What is lost is below 2^-60 of the cell's largest intensity per
// ordinate, times its coefficient, and random; the FP64 loop loses up to 2^-53 of
// the partial sum per addition.  Where the largest intensity belongs to an
// ordinate of small coefficient c, the result can be as small as c times it,
// and the loss of the others is up to sqrt(sum c_q^2) / c times larger
// relative to it.  mom_quads keeps that ratio below 2^8 in every moment summed
// so: the random error is then below 1.2 2^-52, the loop's own in such a cell.
// S16: 2^5 in rho and F, 2^7.8 in P.  Product sets with more than a few
// polar levels, whose smallest w mu^2 are 2^-15 and less, exceed it: there the
// loss would be 1e-13 (16 x 16), and 4e-9 in rho for a weight of 1e-9.
// The order of the sum does not matter to integers, but
// the scale does: where a later chunk holds a larger exponent the sums are
// shifted down, the low bits of the high word into the next (a unit of the
// high word is 2^-57 of the largest intensity whatever the coefficient:
// dropped, it left P of an S16 beam with 5e-15; now 1e-15, the loop 2e-15).
//
// Values that the scheme does not cover (a cell with an infinity or a NaN,
// or whose largest value is below 2^-959) take the FP64 loop.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "reflections.h"

namespace gsis {

// One quad of the set: the four sorted directions and, per moment (rho, F_x,
// F_y, P_xx, P_xy, P_yy), the high and low 32 bits of its coefficient.
struct MomQuad {
    int s[4];
    unsigned c[6][2];
};

// Quads of the set (mu, eta, w) in `quads`, and the moments that may be summed
// over them: 6 (rho, F, P), 3 (rho, F) or 0.  Quads take distinct directions:
// a repeated direction is not a quad's.
inline int mom_quads(int K, const double* mu, const double* eta, const double* w, std::vector<MomQuad>& quads)
{
    constexpr double kSpread = 256.0;
    quads.clear();
    for (int s = 0; s < K; ++s)
        if (!(mu[s] != 0.0) || !(eta[s] != 0.0) || !(w[s] < 2.0)) return 0;
    if (K % 4 != 0) return 0;
    const std::vector<int> at = by_magnitude(K, mu, eta, w);
    double sum2[6] = {}, least[6] = {2.0, 2.0, 2.0, 2.0, 2.0, 2.0};
    for (int i = 0; i < K; i += 4) {
        MomQuad q{};
        unsigned signs = 0;
        const int a = at[i];
        auto alike = [&](int b) {
            return std::fabs(mu[b]) == std::fabs(mu[a]) && std::fabs(eta[b]) == std::fabs(eta[a]) && w[b] == w[a];
        };
        for (int r = 0; r < 4; ++r) {
            const int t = at[i + r], sign = (mu[t] < 0.0 ? 1 : 0) + (eta[t] < 0.0 ? 2 : 0);
            if (!alike(t)) return 0;
            signs |= 1u << sign;
            q.s[sign] = t;
        }
        if (signs != 15u || (i + 4 < K && alike(at[i + 4]))) return 0;
        const double m = std::fabs(mu[a]), e = std::fabs(eta[a]);
        const double cf[6] = {w[a], w[a] * m, w[a] * e, w[a] * m * m, w[a] * m * e, w[a] * e * e};
        for (int t = 0; t < 6; ++t) {
            const unsigned long long c = (unsigned long long)std::nearbyint(std::ldexp(cf[t], 62));
            q.c[t][0] = (unsigned)(c >> 32);
            q.c[t][1] = (unsigned)c;
            sum2[t] += cf[t] * cf[t];
            least[t] = std::min(least[t], cf[t]);
        }
        quads.push_back(q);
    }
    std::sort(quads.begin(), quads.end(), [](const MomQuad& a, const MomQuad& b) { return a.s[0] < b.s[0]; });
    int n = 0;
    while (n < 6 && std::sqrt(sum2[n]) <= kSpread * least[n]) ++n;
    return n < 3 ? 0 : n < 6 ? 3 : 6;
}

#ifdef __CUDACC__
template <int NM>
struct FixedMoments {
    static constexpr int kChunk = 4;   // quads whose 16 loads are in flight together
    static constexpr int kFrac = NM > 3 ? 32 : 30;   // bits of cl
    // |dh cl| < 2^(31 + kFrac) - 2^31, dl cl < 2^(32 + kFrac): with 30 bits a
    // chunk's four terms and the remainder fit 64 bits, with 32 one term does
    static constexpr bool kCarryEach = kFrac == 32;

    long long A[NM], B2[NM];           // sum dh ch, sum dh cl
    unsigned long long B[NM];          // sum dl ch
    unsigned long long C[NM];          // sum dl cl since the last carry
    int E;                             // the scale: biased exponent at d's bit 60

    __device__ __forceinline__ void carry(int m)
    {
        A[m] += B2[m] >> kFrac;
        B2[m] &= (1ll << kFrac) - 1;
        B[m] += C[m] >> kFrac;
        C[m] = 0;
    }

    __device__ __forceinline__ void add(int m, long long d, unsigned ch, unsigned cl)
    {
        const int dh = (int)(d >> 32);
        const unsigned dl = (unsigned)d;
        A[m] += (long long)dh * (int)ch;             // ch < 2^31
        B[m] += (unsigned long long)dl * ch;
        if constexpr (kFrac == 32) B2[m] += (long long)dh * (long long)(unsigned long long)cl;
        else B2[m] += (long long)dh * (int)cl;
        C[m] += (unsigned long long)dl * cl;
        if constexpr (kCarryEach) carry(m);
    }

    // A 2^64 + B 2^32 + B2 2^(64 - kFrac), in units of 2^(E - 1145): to FP64
    __device__ __forceinline__ double value(int m) const
    {
        const unsigned long long f = (B[m] & 0xffffffffull) + ((unsigned long long)B2[m] << (32 - kFrac));
        const long long a = A[m] + (long long)(B[m] >> 32) + (long long)(f >> 32);   // B2 < 2^kFrac: carried
        const double lo = fma((double)(unsigned)f, 0x1p-32, (double)(unsigned)a);
        const double v = fma((double)(int)(a >> 32), 0x1p32, lo);
        // E - 1081 lies in [-1017, 965]: both factors are normal numbers
        const int e = E - 1081, e1 = e / 2, e2 = e - e1;
        return v * __hiloint2double((e1 + 1023) << 20, 0) * __hiloint2double((e2 + 1023) << 20, 0);
    }

    // Moments of cell c over nq quads (tab: cl already of kFrac bits); false:
    // out is not written (see above).
    __device__ __forceinline__ bool run(const MomQuad* __restrict__ tab, int nq, const double* __restrict__ I,
                                        size_t N, int c, double* out)
    {
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            A[m] = B2[m] = 0;
            B[m] = C[m] = 0;
        }
        E = 0;
        bool ok = true, any = false;
        const unsigned long long* I64 = reinterpret_cast<const unsigned long long*>(I) + c;
        for (int q0 = 0; q0 < nq; q0 += kChunk) {
            unsigned long long v[4 * kChunk];
#pragma unroll
            for (int u = 0; u < kChunk; ++u)
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    v[4 * u + r] = q0 + u < nq ? __ldg(I64 + (size_t)tab[q0 + u].s[r] * N) : 0ull;
            unsigned mx = 0, sg = 0;
#pragma unroll
            for (int u = 0; u < 4 * kChunk; ++u) {
                const unsigned h = (unsigned)(v[u] >> 32);
                mx = max(mx, h & 0x7fffffffu);
                sg |= h;
            }
            const int En = max(E, (int)(mx >> 20));
            if (En < 64) {   // all zero: nothing to add; else too small for this scale
                unsigned long long o = 0;
#pragma unroll
                for (int u = 0; u < 4 * kChunk; ++u) o |= v[u] << 1;
                ok = ok && o == 0;
                continue;
            }
            if (mx >= 0x7ff00000u) ok = false;
            if (En > E) {
                const int sh = min(En - E, 63);
                if (any) {
#pragma unroll
                    for (int m = 0; m < NM; ++m) {   // what A loses goes to B
                        const unsigned long long ra = (unsigned long long)A[m] & ((1ull << sh) - 1);
                        A[m] >>= sh;
                        B[m] = (B[m] >> sh) + (sh <= 32 ? (ra << 32) >> sh : ra >> (sh - 32));
                        B2[m] >>= sh;
                    }
                }
                E = En;
            }
            any = true;
#pragma unroll
            for (int u = 0; u < 4 * kChunk; ++u) {
                const unsigned h = (unsigned)(v[u] >> 32), l = (unsigned)v[u];
                const unsigned n = (unsigned)(E - (int)((h >> 20) & 0x7ffu));   // a zero's is >= 64: shifted out
                const unsigned mh = (h & 0xfffffu) | 0x100000u;
                const unsigned long long m61 = ((unsigned long long)__funnelshift_l(l, mh, 8) << 32) | (l << 8);
                v[u] = n > 63u ? 0ull : (m61 >> n) | 1ull;
                if (sg >> 31) v[u] = h >> 31 ? 0ull - v[u] : v[u];
            }
#pragma unroll
            for (int u = 0; u < kChunk; ++u) {
                if (q0 + u >= nq) break;
                const MomQuad& q = tab[q0 + u];
                const long long i1 = (long long)v[4 * u], i2 = (long long)v[4 * u + 1], i3 = (long long)v[4 * u + 2],
                                i4 = (long long)v[4 * u + 3];
                const long long a = i1 + i2, b = i3 + i4;
                add(0, a + b, q.c[0][0], q.c[0][1]);
                if (NM >= 3) {
                    const long long p = i1 - i2, t = i3 - i4;
                    add(1, p + t, q.c[1][0], q.c[1][1]);
                    add(2, a - b, q.c[2][0], q.c[2][1]);
                    if (NM >= 6) {
                        add(3, a + b, q.c[3][0], q.c[3][1]);
                        add(4, p - t, q.c[4][0], q.c[4][1]);
                        add(5, a + b, q.c[5][0], q.c[5][1]);
                    }
                }
            }
            if constexpr (!kCarryEach) {
#pragma unroll
                for (int m = 0; m < NM; ++m) carry(m);
            }
        }
        if (!ok) return false;
        if (!any) E = 1081;
#pragma unroll
        for (int m = 0; m < NM; ++m) out[m] = value(m);
        return true;
    }
};
#endif

}  // namespace gsis
