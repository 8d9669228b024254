// The two mirror sectors of a far pair's M2L.
//
// The dyad between two boxes is symmetric under the reflection through the
// vertical plane that holds both centres.  In the frame of that plane the
// reflection exchanges the helical components a and b and flips the orders m,
// so with F the flip m -> -m the five tables satisfy T_s1 = F T_s1 F, T_s5 = F T_s5 F,
// and the 3P x 3P helical operator splits into an even and an odd block.  With
//   G[d] = i^d e^{i d phi}, phi the azimuth of c_s - c_t,
// the inputs of sector e (e = +1 even, -1 odd) are
//   W entries (n', m'):       G[m'-1] a(n', m') - e conj(G[m'-1]) b(n', -m'),
//   C entries (n', m' >= 0):  G[m'] c(n', m') + e conj(G[m']) c(n', -m')      (m' = 0 even only),
// the products y_e = M_e x_e, and the outputs (y = y_+ + y_-, y' = y_+ - y_-)
//   W (nu, mu):      a(nu, mu) += conj(G[mu-1]) y,   b(nu, -mu) -= G[mu-1] y',
//   C (nu, mu >= 0): c(nu, mu) += conj(G[mu]) y,     c(nu, -mu) += G[mu] y'   (mu > 0).
// M_e carries everything that depends on degrees, orders and the component: the
// level scaling, (i f_s)^n' and (-i f_t)^nu with the remaining powers of i, and the
// parities f^(n+m) of downward components and mirrored boxes.  Both blocks
// have about 3P/2 rows, so a pair costs 4.5 P^2 complex products instead of the
// 9 P^2 of the nine table applications, and its expansions are read and its outputs
// written once instead of three times.
#pragma once
#include "kernels.cuh"

namespace lmf {

// rows (= columns) of the sector blocks: P W entries, the C entries of order m > 0,
// then, in the even sector alone, the C entries of order 0
__host__ __device__ inline int sec_dim(int p, int odd)
{
    return (p + 1) * (p + 1) + p * (p + 1) / 2 + (odd ? 0 : p + 1);
}

struct SecEntry {
    int c, n, m;   // c = 0: W entry, 1: C entry
};

__host__ __device__ inline SecEntry sec_entry(int p, int j)
{
    const int P = (p + 1) * (p + 1);
    if (j < P) {
        int n = (int)sqrtf((float)j + 0.5f);
        while ((n + 1) * (n + 1) <= j) ++n;
        while (n * n > j) --n;
        return SecEntry{0, n, j - n * n - n};
    }
    j -= P;
    if (j >= p * (p + 1) / 2) return SecEntry{1, j - p * (p + 1) / 2, 0};
    int n = (int)((1.f + sqrtf(1.f + 8.f * (float)j)) * 0.5f);
    while (n * (n + 1) / 2 <= j) ++n;
    while (n * (n - 1) / 2 > j) --n;
    return SecEntry{1, n, j - n * (n - 1) / 2 + 1};
}

// where entry j reads and adds: offsets into [3][P] of its two coefficients, the index
// d of its phase shifted by p + 1, and what its type does with them
//   bits 0-9 off1, 10-19 off2, 20-25 d + p + 1, 26: C entry, 27: one coefficient only (C, m = 0)
__host__ __device__ inline uint32_t sec_word(int p, int j)
{
    const int P = (p + 1) * (p + 1);
    const SecEntry e = sec_entry(p, j);
    const int up = e.n * e.n + e.n + e.m, dn = e.n * e.n + e.n - e.m;
    const uint32_t o1 = e.c ? 2 * P + up : up, o2 = e.c ? 2 * P + dn : P + dn;
    return o1 | (o2 << 10) | ((uint32_t)((e.c ? e.m : e.m - 1) + p + 1) << 20) | (e.c ? 1u << 26 : 0u) |
           ((e.c && e.m == 0) ? 1u << 27 : 0u);
}

// M_e[r][k] without the row and column factors, from the five tables of the geometry
// (order s1, s5, s2, s4, s3)
__device__ inline cd sec_value(int p, int odd, const SecEntry &r, const SecEntry &k, const cd *tab)
{
    const int64_t P = (p + 1) * (p + 1), PP = P * P;
    const double e = odd ? -1.0 : 1.0;
    const int64_t ru = r.n * r.n + r.n + r.m, rd = r.n * r.n + r.n - r.m;
    const int64_t ku = k.n * k.n + k.n + k.m, kd = k.n * k.n + k.n - k.m;
    if (!r.c && !k.c) return mkd(0.0, 0.25) * (tab[ru * P + ku] + e * tab[4 * PP + ru * P + kd]);
    if (!r.c) {
        cd v = tab[2 * PP + ru * P + ku];
        if (k.m > 0) v += e * tab[2 * PP + ru * P + kd];
        return -0.5 * v;
    }
    if (!k.c) return (-0.25 * e) * (tab[3 * PP + ru * P + kd] + e * tab[3 * PP + rd * P + kd]);
    cd v = tab[PP + ru * P + ku];
    if (k.m > 0) v += e * tab[PP + ru * P + kd];
    return mkd(0.0, 0.5) * v;
}

// row and column factors: (-i)^(nu + [W]) f_t^(nu + mu) s_t^nu and i^(n' + [W]) f_s^(n' + m') s_s^n',
// pt / ps: powers of the level scales
__device__ inline cd sec_scaled(const SecEntry &r, const SecEntry &k, bool flip_in, bool flip_out, const double *pt,
                                const double *ps, cd v)
{
    double f = pt[r.n] * ps[k.n];
    if ((flip_out && ((r.n + r.m) & 1)) != (flip_in && ((k.n + k.m) & 1))) f = -f;
    return ipow<double>(k.n + 1 - k.c - (r.n + 1 - r.c)) * (f * v);
}

}  // namespace lmf
