// Directions of a quadrature that are reflections of one another, on the host.
// Sorted, not compared pairwise: of 4096 directions that took 10 ms of every
// call (and of each problem of a batch), sorting takes 0.6.
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

namespace gsis {

// The directions in order of |mu|, |eta|, w (unless null) and index.
inline std::vector<int> by_magnitude(int K, const double* mu, const double* eta, const double* w)
{
    std::vector<int> at(K);
    for (int s = 0; s < K; ++s) at[s] = s;
    std::sort(at.begin(), at.end(), [&](int a, int b) {
        const double ma = std::fabs(mu[a]), mb = std::fabs(mu[b]), ea = std::fabs(eta[a]), eb = std::fabs(eta[b]);
        if (ma != mb) return ma < mb;
        if (ea != eb) return ea < eb;
        if (w && w[a] != w[b]) return w[a] < w[b];
        return a < b;
    });
    return at;
}

// Directions of equal |mu| and |eta|: the first ones in rep, ascending, and from
// each the next one in next (-1: none).  Returns the number of first ones.
inline int reflection_chains(int K, const double* mu, const double* eta, int* rep, int* next)
{
    const std::vector<int> at = by_magnitude(K, mu, eta, nullptr);
    int n = 0;
    for (int i = 0; i < K; ++i) {
        const int s = at[i], p = i > 0 ? at[i - 1] : -1;
        next[s] = -1;
        if (p >= 0 && std::fabs(mu[p]) == std::fabs(mu[s]) && std::fabs(eta[p]) == std::fabs(eta[s])) next[p] = s;
        else rep[n++] = s;
    }
    std::sort(rep, rep + n);
    return n;
}

}  // namespace gsis
