// csrc/moments_fixed.cuh compiled for the host: the device functions it calls
// are restated, so that its arithmetic can be compared with exact sums without
// a GPU (test_moments_fixed_host.py).
#define __CUDACC__
#define __device__
#define __forceinline__ inline
#define __restrict__

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

using std::max;
using std::min;

static unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return (hi << s) | (lo >> (32 - s)); }
static double __hiloint2double(int hi, int lo)
{
    const unsigned long long b = (unsigned long long)(unsigned)hi << 32 | (unsigned)lo;
    double d;
    std::memcpy(&d, &b, sizeof d);
    return d;
}
static unsigned long long __ldg(const unsigned long long* p) { return *p; }

#include "moments_fixed.cuh"

using namespace gsis;

template <int NM>
static void cells(const MomQuad* quads, int nq, const double* I, int n, double* out, unsigned char* ok)
{
    std::vector<MomQuad> tab(quads, quads + nq);
    for (MomQuad& q : tab)
        for (auto& c : q.c) c[1] >>= 32 - FixedMoments<NM>::kFrac;   // as moments_quad_body loads it
    for (int c = 0; c < n; ++c) {
        FixedMoments<NM> f;
        ok[c] = f.run(tab.data(), nq, I, (size_t)n, c, out + (size_t)NM * c);
    }
}

extern "C" {

// The moments that may be summed in fixed point; quads: [K/4][16] words
int set_quads(int K, const double* mu, const double* eta, const double* w, void* quads)
{
    std::vector<MomQuad> q;
    const int n = mom_quads(K, mu, eta, w, q);
    std::memcpy(quads, q.data(), std::min(q.size(), (size_t)K / 4) * sizeof(MomQuad));
    return n;
}

// First directions of equal |mu|, |eta| and chains
int chains(int K, const double* mu, const double* eta, int* rep, int* next)
{
    return reflection_chains(K, mu, eta, rep, next);
}

// quads: [nq][16] words (4 directions, 6 coefficients in two halves); I: [K][n]; out: [n][nm]
void fixed_cells(int nm, const void* quads, int nq, const double* I, int n, double* out, unsigned char* ok)
{
    const MomQuad* q = static_cast<const MomQuad*>(quads);
    if (nm == 1) cells<1>(q, nq, I, n, out, ok);
    else if (nm == 3) cells<3>(q, nq, I, n, out, ok);
    else cells<6>(q, nq, I, n, out, ok);
}

// The FP64 loop: fused multiply-adds in the order of the directions; coef: [6][K]; out: [n][6]
void loop_cells(int K, const double* coef, const double* I, int n, double* out)
{
    for (int c = 0; c < n; ++c)
        for (int m = 0; m < 6; ++m) {
            double s = 0.0;
            for (int k = 0; k < K; ++k) s = std::fma(coef[(size_t)m * K + k], I[(size_t)k * n + c], s);
            out[(size_t)6 * c + m] = s;
        }
}
}
