// Setup kernels: density functions, M2L tabulation by the Chebyshev route of
// Section 3.4, and the M2M / L2L translation matrices.
#include "kernels.cuh"
#include "quad.cuh"
#include "specfun.cuh"

namespace lmf {

// ------------------------------------------------------------- densities
__global__ void k_densities(MediumDev M, int l, int lp, int64_t n, const cd *kr, cd *out)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    cd ph[4], ps[4];
    densities_dev(M, kr[i], l, lp, 0, ph);
    densities_dev(M, kr[i], l, lp, 1, ps);
    for (int c = 0; c < 4; ++c) {
        out[i * 8 + c] = ph[c];
        out[i * 8 + 4 + c] = ps[c];
    }
}

void launch_densities(const MediumDev &M, int l, int lp, int64_t n, const cd *kr, cd *out,
                      cudaStream_t st)
{
    if (n <= 0) return;
    k_densities<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(M, l, lp, n, kr, out);
}

// ---------------------------------------------------------- quadrature nodes
// per-node factors for the Chebyshev integrals:
//   base_t = w Z sigma_t   (5 tables), tau_src[4], tau_tgt[4], T_l(x_prim), J_d(k rho)
__global__ void k_tab_nodes(const GeomDev *G, int g0, MediumDev M, const CompDev *comps,
                            int LM, int DJ, cd *Fb, cd *Fs, cd *Ft, cd *FT, cd *FJ, int *flag)
{
    const GeomDev &g = G[g0 + blockIdx.y];
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    int Q = g.plan.n1 + g.plan.nmid + 2 * g.plan.nray;
    if (q >= Q) return;
    int64_t o = g.node0 + q;
    const CompDev c = comps[g.comp];
    cd kr, w;
    int kind = plan_node(g.plan, q, kr, w);
    cd k = M.k[c.l], kp = M.k[c.lp];
    cd kz = kz_of(k, kr), kzp = kz_of(kp, kr);
    cd sg[5];
    sigmas_dev(M, kr, c.l, c.lp, c.tu, c.su, sg);
    cd Z = cexpd(mul_i(c.s * (kz * g.zs - kzp * g.zt)));
    cd wZ = w * Z;
    const int64_t S = g.stride;
    Fb[0 * S + o] = wZ * sg[0];
    Fb[1 * S + o] = wZ * sg[4];
    Fb[2 * S + o] = wZ * sg[1];
    Fb[3 * S + o] = wZ * sg[3];
    Fb[4 * S + o] = wZ * sg[2];
    Fs[0 * S + o] = mkd(1.0);
    Fs[1 * S + o] = k / kz;
    Fs[2 * S + o] = kr / k;
    Fs[3 * S + o] = kr / kz;
    Ft[0 * S + o] = mkd(1.0);
    Ft[1 * S + o] = kp / kzp;
    Ft[2 * S + o] = kr / kp;
    Ft[3 * S + o] = kr / kzp;
    cd kprim = g.src_primary ? k : kp;
    cd x = mkd(1.0) - 2.0 * (kr * kr) / (kprim * kprim);
    cd t0 = mkd(1.0), t1 = x;
    FT[0 * S + o] = t0;
    if (LM > 1) FT[1 * S + o] = t1;
    for (int l = 2; l < LM; ++l) {
        cd t2 = 2.0 * (x * t1) - t0;
        FT[l * S + o] = t2;
        t0 = t1;
        t1 = t2;
    }
    cd J[64];
    if (kind == 0) {
        if (bessel_j_seq<64>(kr * g.rho, DJ - 1, J)) atomicOr(flag, 1);
        for (int dd = 0; dd < DJ; ++dd) FJ[dd * S + o] = J[dd];
    } else {
        // H^(2)_n(z) = conj(H^(1)_n(conj z)) for integer n
        cd z = kr * g.rho;
        if (kind == 2) z = conj(z);
        hankel1_seq(z, DJ - 1, J);
        for (int dd = 0; dd < DJ; ++dd) FJ[dd * S + o] = 0.5 * (kind == 2 ? conj(J[dd]) : J[dd]);
    }
}

// Bessel orders of I-breve that an entry can ask for: tau types 0, 1 belong to even orders m
// and 2, 3 to odd ones, so d = m' - mu + kappa_t has one parity per (t, ts, tt) and only
// every second order is formed: |d| = par + 2 h, h < tab_dh(DJ)
__host__ __device__ inline int tab_par(int t, int ts, int tt)
{
    const int kap = t < 2 ? 0 : t < 4 ? 1 : 2;
    return ((ts >> 1) + (tt >> 1) + kap) & 1;
}
__host__ __device__ inline int tab_dh(int DJ) { return (DJ + 1) / 2; }

// I-breve[t][ts][tt][l][h] = sum_q base_t tau_s tau_t T_l J_d  for one
// geometry, table t and source tau-type ts (blockIdx = (geometry, t*4+ts)).  In a
// same-layer component the tau of both sides are the same functions: tt < ts is
// the (tt, ts) block, which the assembly reads instead.
__global__ void k_tab_contract(const GeomDev *G, int g0, const CompDev *comps, int LM, int DJ, const cd *Fb,
                               const cd *Fs, const cd *Ft, const cd *FT, const cd *FJ,
                               cd *Ibr, int64_t ibr_stride)
{
    extern __shared__ unsigned char smraw[];
    const int CH = 32, DH = tab_dh(DJ);
    cd *W = (cd *)smraw;                 // [CH][4][LM]
    cd *Jc = W + CH * 4 * LM;            // [CH][DJ]
    cd *Bq = Jc + CH * DJ;               // [CH][4]: base_t tau_s tau_t
    const GeomDev &g = G[g0 + blockIdx.x];
    int t = blockIdx.y / 4, ts = blockIdx.y % 4;
    const CompDev c = comps[g.comp];
    const int tt0 = c.l == c.lp ? ts : 0, ntt = 4 - tt0;
    int Q = g.plan.n1 + g.plan.nmid + 2 * g.plan.nray;
    const int64_t S = g.stride;
    int64_t o0 = g.node0;
    const int NOUT = ntt * LM * DH;
    const int PER = 6;    // 4 LM DH <= 6 * 256 for p <= 16
    cd acc[PER];
    int wi[PER], ji[PER];                // an output's W row and Bessel order
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        acc[i] = mkd(0.0);
        const int out = min((int)(threadIdx.x + i * blockDim.x), NOUT - 1);
        const int r = out / DH, tt = tt0 + r / LM;
        wi[i] = r;
        ji[i] = min(tab_par(t, ts, tt) + 2 * (out - r * DH), DJ - 1);
    }
    for (int q0 = 0; q0 < Q; q0 += CH) {
        int nq = min(CH, Q - q0);
        for (int e = threadIdx.x; e < nq * ntt; e += blockDim.x) {
            const int q = e % nq, k = e / nq;
            const int64_t o = o0 + q0 + q;
            Bq[q * 4 + k] = Fb[t * S + o] * Fs[ts * S + o] * Ft[(tt0 + k) * S + o];
        }
        for (int e = threadIdx.x; e < nq * DJ; e += blockDim.x) {
            int q = e / DJ, dd = e % DJ;
            Jc[e] = FJ[dd * S + o0 + q0 + q];
        }
        __syncthreads();
        for (int e = threadIdx.x; e < nq * ntt * LM; e += blockDim.x) {
            int q = e / (ntt * LM), r = e % (ntt * LM), k = r / LM, l = r % LM;
            W[q * 4 * LM + r] = Bq[q * 4 + k] * FT[l * S + o0 + q0 + q];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if ((int)(threadIdx.x + i * blockDim.x) >= NOUT) break;
            cd a = acc[i];
            for (int q = 0; q < nq; ++q) a += W[q * 4 * LM + wi[i]] * Jc[q * DJ + ji[i]];
            acc[i] = a;
        }
        __syncthreads();
    }
    cd *dst = Ibr + (int64_t)blockIdx.x * ibr_stride + (int64_t)((t * 4 + ts) * 4 + tt0) * LM * DH;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        int out = threadIdx.x + i * blockDim.x;
        if (out < NOUT) dst[out] = acc[i];
    }
}

__device__ inline int tau_type(int n, int am)
{
    bool no = n & 1, mo = am & 1;
    if (!no && !mo) return 0;   // 1
    if (no && !mo) return 1;    // sec
    if (no && mo) return 2;     // sin
    return 3;                   // tan
}

// I-hat[t][row=(nu,mu)][col=(n',m')] = sgn(m') sgn(mu) sum_l G[(n',|m'|),(nu,|mu|)][l]
//   * I-breve[t][tau(n',m')][tau(nu,mu)][l][|d|] * (-1)^d [d<0],  d = m' - mu + kappa_t
__global__ void k_tab_assemble(const GeomDev *G, int g0, const CompDev *comps, int p, int LM, int DJ, const cd *Gten,
                               const int *comp_gidx, const cd *Ibr, int64_t ibr_stride,
                               cd *tab)
{
    const int P = (p + 1) * (p + 1), T = (p + 1) * (p + 2) / 2;
    const GeomDev &g = G[g0 + blockIdx.z];
    int t = blockIdx.y;
    const int kap[5] = {0, 0, 1, 1, 2};
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= P * P) return;
    int row = e / P, col = e % P;
    int nu = (int)sqrt((double)row + 0.5), mu;
    int n1 = (int)sqrt((double)col + 0.5), m1;
    while ((nu + 1) * (nu + 1) <= row) ++nu;
    while (nu * nu > row) --nu;
    mu = row - nu * nu - nu;
    while ((n1 + 1) * (n1 + 1) <= col) ++n1;
    while (n1 * n1 > col) --n1;
    m1 = col - n1 * n1 - n1;
    int am1 = m1 < 0 ? -m1 : m1, amu = mu < 0 ? -mu : mu;
    int dd = m1 - mu + kap[t];
    int ad = dd < 0 ? -dd : dd;
    double sgn = 1.0;
    if (m1 < 0 && (am1 & 1)) sgn = -sgn;
    if (mu < 0 && (amu & 1)) sgn = -sgn;
    if (dd < 0 && (ad & 1)) sgn = -sgn;
    int ts = tau_type(n1, am1), tt = tau_type(nu, amu);
    const cd *Gp = Gten + ((int64_t)comp_gidx[g.comp] * T * T + (int64_t)(((n1 * (n1 + 1)) / 2 + am1) * T
                           + (nu * (nu + 1)) / 2 + amu)) * LM;
    if (comps[g.comp].l == comps[g.comp].lp && tt < ts) {   // formed as (tt, ts)
        const int x = tt;
        tt = ts;
        ts = x;
    }
    const int DH = tab_dh(DJ);
    const cd *Ib = Ibr + (int64_t)blockIdx.z * ibr_stride + (int64_t)((t * 4 + ts) * 4 + tt) * LM * DH
                   + ((ad - tab_par(t, ts, tt)) >> 1);
    cd s = mkd(0.0);
    for (int l = 0; l < LM; ++l) s += Gp[l] * Ib[l * DH];
    tab[((int64_t)g.tab_index * NTAB + t) * P * P + e] = sgn * s;
}

// Chebyshev integrals of one geometry: [table][tau][tau'][l][h]
int64_t tab_integrals(int p) { return (int64_t)NTAB * 16 * (p + 2) * tab_dh(2 * p + 3); }

// One batch of geometries [g0, g0+nb): node factors, I-breve, I-hat.  The
// scratch holds (5+4+4+LM+DJ) * stride node factors followed by nb I-breve
// blocks; stride is the batch's total node count.
void launch_tab_batch(const GeomDev *dG, int g0, int nb, int qmax, const MediumDev &M,
                      const CompDev *dcomps, int p, const cd *dGten, const int *dcgidx,
                      cd *scratch, int64_t stride, cd *tab, int *dflag, cudaStream_t st)
{
    const int LM = p + 2, DJ = 2 * p + 3, P = (p + 1) * (p + 1);
    const int64_t ibr_stride = tab_integrals(p);
    const int64_t S = stride;
    cd *Fb = scratch, *Fs = Fb + 5 * S, *Ft = Fs + 4 * S, *FT = Ft + 4 * S, *FJ = FT + LM * S;
    cd *Ibr = FJ + DJ * S;
    dim3 gn((qmax + 127) / 128, nb);
    k_tab_nodes<<<gn, 128, 0, st>>>(dG, g0, M, dcomps, LM, DJ, Fb, Fs, Ft, FT, FJ, dflag);
    size_t sm = (size_t)(32 * 4 * LM + 32 * DJ + 32 * 4) * sizeof(cd);
    dim3 gc(nb, NTAB * 4);
    k_tab_contract<<<gc, 256, sm, st>>>(dG, g0, dcomps, LM, DJ, Fb, Fs, Ft, FT, FJ, Ibr, ibr_stride);
    dim3 ga((P * P + 255) / 256, NTAB, nb);
    k_tab_assemble<<<ga, 256, 0, st>>>(dG, g0, dcomps, p, LM, DJ, dGten, dcgidx, Ibr, ibr_stride, tab);
}

}  // namespace lmf

namespace lmf {
cudaError_t configure_tab_kernels()
{
    return cudaFuncSetAttribute(k_tab_contract, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                160 * 1024);
}
// ---------------------------------------------------- translation matrices
// Sums and products of double-doubles (Dekker, Numer. Math. 18 (1971); Knuth's two-sum):
// some 100 bits, so that an entry below is rounded once, like the long double of the host's
// translation_matrix.  In plain FP64 the quadrature and the sum over l left 5e-16 of a degree
// block's largest entry instead of 1.1e-16.
__device__ __forceinline__ dd dd_norm(double h, double l)   // |h| >= |l|
{
    const double s = h + l;
    return dd{s, l - (s - h)};
}

__device__ __forceinline__ dd dd_add(dd a, dd b)
{
    const double s = a.h + b.h, t = s - a.h;
    return dd_norm(s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l));
}

__device__ __forceinline__ dd dd_mul(dd a, dd b)
{
    const double q = a.h * b.h;
    return dd_norm(q, fma(a.h, b.h, -q) + fma(a.h, b.l, a.l * b.h));
}

__device__ __forceinline__ dd dd_neg(dd a) { return dd{-a.h, -a.l}; }

// Gaunt coefficients G(l; n', n) = int Y_l^(m-m') Y_n'^m' conj(Y_n^m) for l = |n - n'|,
// |n - n'| + 2, ... (zero where l < |m - m'|), p + 1 per entry, by the Gauss-Legendre rule
// that is exact for them.  One thread per coefficient: the quadrature is some 10^7 products
// at p = 12, which took the host (whose long double is software there) a second.
__global__ void k_gaunt(int p, int nq, const dd *w, const dd *Pq, double *G)
{
    const int P = (p + 1) * (p + 1), nt = (2 * p + 1) * (2 * p + 2) / 2;
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= P * P * (p + 1)) return;
    const int e = id / (p + 1), j = id % (p + 1), r = e / P, c = e % P;
    int n = (int)sqrtf((float)r + 0.5f), n1 = (int)sqrtf((float)c + 0.5f);
    while ((n + 1) * (n + 1) <= r) ++n;
    while (n * n > r) --n;
    while ((n1 + 1) * (n1 + 1) <= c) ++n1;
    while (n1 * n1 > c) --n1;
    const int m = r - n * n - n, m1 = c - n1 * n1 - n1, mu = m - m1;
    const int am = abs(m), am1 = abs(m1), amu = abs(mu);
    // P~_n^m = (-1)^m P~_n^|m| for m < 0
    const int neg = ((m < 0 ? am : 0) + (m1 < 0 ? am1 : 0) + (mu < 0 ? amu : 0)) & 1;
    const int l = abs(n - n1) + 2 * j;
    dd s{0.0, 0.0};
    if (l <= n + n1 && l >= amu) {
        for (int q = 0; q < nq; ++q) {
            const dd *Q = Pq + (int64_t)q * nt;
            s = dd_add(s, dd_mul(dd_mul(w[q], Q[l * (l + 1) / 2 + amu]),
                                 dd_mul(Q[n1 * (n1 + 1) / 2 + am1], Q[n * (n + 1) / 2 + am])));
        }
    }
    G[id] = neg ? -s.h : s.h;
}

// M2M = i^(n'-n) W(t) and L2L = i^(n-n') W(t) of every translation group, with the level
// scaling M~ = M / s^n, L~ = L s^nu: W = sum_l i^l j_l(k |t|) P~_l^mu(t^) 4 pi e^{-i mu phi} G(l).
// fac: trans_factors of the groups
__global__ void k_trans_build(int p, const double *G, const dd *fac, int nfac, cd *up, cd *dn)
{
    const int P = (p + 1) * (p + 1);
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= P * P) return;
    const int64_t g = blockIdx.y;
    const int r = e / P, c = e % P;
    int n = (int)sqrtf((float)r + 0.5f), n1 = (int)sqrtf((float)c + 0.5f);
    while ((n + 1) * (n + 1) <= r) ++n;
    while (n * n > r) --n;
    while ((n1 + 1) * (n1 + 1) <= c) ++n1;
    while (n1 * n1 > c) --n1;
    const int mu = (r - n * n - n) - (c - n1 * n1 - n1), amu = abs(mu);
    const dd *jl = fac + g * nfac, *Pt = jl + 2 * (2 * p + 1), *ep = Pt + (2 * p + 1) * (2 * p + 2) / 2;
    const dd *sc = ep + 2 * (4 * p + 1), *sp = sc + (p + 1);   // powers of the child and the parent scale
    dd sx{0.0, 0.0}, sy{0.0, 0.0};
    for (int j = 0; j <= p; ++j) {
        const int l = abs(n - n1) + 2 * j;
        if (l > n + n1) break;
        if (l < amu) continue;
        const dd f = dd_mul(Pt[l * (l + 1) / 2 + amu], dd{G[(int64_t)e * (p + 1) + j], 0.0});
        sx = dd_add(sx, dd_mul(f, jl[2 * l]));
        sy = dd_add(sy, dd_mul(f, jl[2 * l + 1]));
    }
    const dd ex = ep[2 * (mu + 2 * p)], ey = ep[2 * (mu + 2 * p) + 1];
    cd s{dd_add(dd_mul(sx, ex), dd_neg(dd_mul(sy, ey))).h, dd_add(dd_mul(sx, ey), dd_mul(sy, ex)).h};
    if (mu < 0 && (amu & 1)) s = -s;
    const int64_t o = g * P * P + e;
    up[o] = (sc[n1].h / sp[n].h) * (ipow<double>(n1 - n) * s);
    dn[o] = (sc[n].h / sp[n1].h) * (ipow<double>(n - n1) * s);
}

// out = in (T != double: rounded once), transposed per matrix if tr
template <typename T>
__global__ void k_trans_copy(int P, int tr, const cd *in, cx<T> *out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= P * P) return;
    const int64_t g = (int64_t)blockIdx.y * P * P;
    const cd v = in[g + (tr ? (e % P) * P + e / P : e)];
    out[g + e] = cx<T>{(T)v.x, (T)v.y};
}

void launch_trans_build(int p, int nq, const dd *w, const dd *Pq, double *G, int64_t ng, const dd *fac, cd *up, cd *dn,
                        cudaStream_t st)
{
    const int P = (p + 1) * (p + 1), nb = (P * P + 127) / 128;
    k_gaunt<<<(P * P * (p + 1) + 127) / 128, 128, 0, st>>>(p, nq, w, Pq, G);
    if (ng > 0) k_trans_build<<<dim3(nb, (unsigned)ng), 128, 0, st>>>(p, G, fac, trans_factor_count(p), up, dn);
}

template <typename T>
void launch_trans_copy(int p, int64_t ng, bool tr, const cd *in, cx<T> *out, cudaStream_t st)
{
    const int P = (p + 1) * (p + 1);
    if (ng > 0) k_trans_copy<T><<<dim3((P * P + 255) / 256, (unsigned)ng), 256, 0, st>>>(P, tr ? 1 : 0, in, out);
}
template void launch_trans_copy<float>(int, int64_t, bool, const cd *, cf *, cudaStream_t);
template void launch_trans_copy<double>(int, int64_t, bool, const cd *, cd *, cudaStream_t);

}  // namespace lmf
