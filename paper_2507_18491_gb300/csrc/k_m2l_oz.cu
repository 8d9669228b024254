// M2L of the FP64 form, and its transpose, on the 5th-generation tensor cores (tcgen05), on
// the mirror sectors of sector.cuh.
//
// The chip has 2 FP64 multiply-adds per clock and SM but 4096 bf16 ones, so the contraction
// runs on integers (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59 (2012), with digits on a common grid per row): every operand is a 64-bit
// fixed-point number, written as eight signed base-256 digits (a bf16 holds every integer
// up to 256), and the products of digits i and j are summed per diagonal d = i + j in an FP32
// accumulator of its own, which holds integers exactly below 2^24.  Digits are at most
// 128 in size, leading ones at most 64 (the matrix) or 64 on average over an input's two parts, so
// the sum over K real inputs is below K 2^14 for d = 1 and K 2^15 for d = 2: exact whatever the
// operands for d <= 1 at every p <= 16 (K = 884) and for d = 2 up to p = 11.  Beyond, exactness rests
// on digits that do not conspire: spread evenly over +-128, a sum's standard deviation is
// sqrt((d + 1) K) 2^14 / 3, a 36th of 2^24 at d = 7, p = 16, a 48th at p = 12; nothing detects
// a sum beyond (a rounding at d = 2 would be 2^-30 of the largest product).
// The 36 products with d <= 7 are formed; what is left out is 2^-64 of the row's and the pair's
// largest entries.  The eight sums are put together as 64-bit integers and converted once.
// Measured against the M2L in double-double, rms error per degree block: 3.2 to 16e-16 over two
// to four layers and p = 6 to 16, the FP64 SIMT kernels 7.8 to 24e-16.
//
// Grids: the matrix rows carry their own power of two, the inputs one per pair, after the
// degrees have been brought to one size by 2^a_n, which the matrix columns take out.  A product
// then misses the bits by which max |M| 2^-a max |x| 2^a exceeds max |M x| of its row.  Entries grow
// like C(n + nu, n) (2n + 1)!! (2 nu + 1)!! (S / R)^(n + nu), S the cell size, R the distance of the
// centres; the scaled expansions fall like (r / S)^n / (2n + 1)!!, r the points' radius, or stop falling
// at what the truncated translations leave.  r may be far below S, and then R too (a cell's centre
// next to an interface), so a_n comes from the matrix alone, per geometry: of the sum e_nu + a_n
// closest to the binary exponents of its degree blocks, the column part, in the mean over the rows
// of degree p / 2 and more (k_oz_degrees).  Whatever the inputs, the missing bits are then at most the
// spread of log2 C(n + nu, n) about that sum: 2 to 5 (p = 6 to 16) in the rows of the upper degrees; in those
// of degree 0, if the inputs' highest degree dominates there, 11 at p = 8, 18 at p = 12 and 25 at p = 16.  A 64-bit
// grid has 11 more than FP64, before the roundings of FP64's own sums.  Other choices of a_n: (2n + 1)!!
// alone lost a row's grid to columns whose inputs are tiny (r = S / 200, R = S / 25, p = 12: 46% of the
// result), (S / r)^n the inputs' to the translations' remainders (74%).
//
// One CTA per SM walks the work items (up to 64 pairs of one geometry).  Per sector: all
// threads form the inputs (FP64 phases, digits by integer operations) into a per-CTA image
// in global memory (L2), then per tile of 64 matrix rows one thread streams input and matrix
// K-steps through a shared ring, one issues the MMAs (8 accumulators x 64 columns: all of
// tensor memory; consecutive MMAs go to different accumulators), and all threads turn the
// accumulators into FP64 sums in a scratch.  At the end one warp per pair combines the two
// sectors and adds [3][P] with one bulk reduction.  The FP64 pipe (phases, conversions) and
// the ring's traffic bound it, not the MMAs.  Every wait is bounded; a wait that gives up
// sets bit 4 of the status word.
//
// Measured (GB300, M2L stage; before: the SIMT five-table kernel at 73% of the FP64 peak): 140593
// pairs at p = 10 142.8 -> 5.77 ms, 658907 pairs at p = 12 1469 -> 48.7 ms, 3583 pairs at p = 6
// 0.90 -> 0.11 ms.
#include <algorithm>

#include "sector.cuh"
#include "tc.cuh"

namespace lmf {

namespace {

constexpr int OZ_S = 8;            // digits
constexpr int OZ_BN = 64;          // pairs per work item
constexpr int OZ_NT = 64;          // matrix rows per tile
constexpr int OZ_T = 512;          // threads
constexpr int OZ_W = OZ_T / 32;
constexpr int OZ_ST = 3;           // ring slots
constexpr uint32_t OZ_A = OZ_S * 128 * 32;          // bytes of an input K-step (8 complex inputs)
constexpr uint32_t OZ_SLOT = OZ_A + OZ_S * OZ_NT * 32;
constexpr int OZ_POLLS = 1 << 22;
constexpr int OZ_PMAX = 16;

struct OzPlan {
    int p, P, D[2], nk[2], rows;   // rows: D0 + D1
    uint32_t sec_img[2], img_bytes;
    uint32_t o_ph, o_ent, o_adj, o_pair, o_exp, o_bars, smem, ph_bytes, stage_bytes;
    int out_warps;
};

__host__ __device__ inline int oz_tile_rows(int D, int t)
{
    const int r = D - t * OZ_NT;
    return r >= OZ_NT ? OZ_NT : (r + 15) & ~15;
}

OzPlan oz_plan(int p)
{
    OzPlan s{};
    s.p = p;
    s.P = (p + 1) * (p + 1);
    uint32_t img = 0;
    for (int e = 0; e < 2; ++e) {
        s.D[e] = sec_dim(p, e);
        s.nk[e] = (s.D[e] + 7) / 8;
        s.sec_img[e] = img;
        for (int t = 0; t * OZ_NT < s.D[e]; ++t) img += (uint32_t)(s.nk[e] * OZ_S * oz_tile_rows(s.D[e], t) * 32);
    }
    s.img_bytes = img;
    s.rows = s.D[0] + s.D[1];
    s.ph_bytes = (uint32_t)(2 * p + 2) * 16 + 16;      // padded against bank conflicts
    s.stage_bytes = (uint32_t)(3 * s.P) * 16;
    s.o_ph = OZ_ST * OZ_SLOT;
    s.o_ent = s.o_ph + OZ_BN * s.ph_bytes;
    s.o_adj = s.o_ent + (uint32_t)s.nk[0] * 8 * 4;
    s.o_pair = (s.o_adj + (uint32_t)s.nk[0] * 8 * 4 + 15) & ~15u;
    s.o_exp = s.o_pair + OZ_BN * (uint32_t)sizeof(M2LPair);
    s.o_bars = s.o_exp + OZ_BN * 4;
    s.smem = s.o_bars + (2 * OZ_ST + 2) * 8 + 16;
    s.out_warps = std::min<int>(OZ_W, (OZ_ST * OZ_SLOT) / s.stage_bytes);
    return s;
}

constexpr int OZ_ZERO = -(1 << 14), OZ_BAD = 1 << 14;   // exponents of a degree of zeros, of one that is not finite

struct __align__(16) OzIn {        // one input: its two coefficients
    double x, y, z, w;
};

// the eight digits of x 2^adj, below 1 - 2^-8 in size (the first digit would leave a byte beyond):
// sum_j s_j 2^(-7 - 8 j), s_j in [-128, 127], as floats' upper halves (bf16, exact).  The
// fixed-point number comes from the bits of x; adding 128 to every digit but the first makes the
// bytes of the sum the digits plus 128.
__device__ __forceinline__ void oz_digits(double x, int adj, uint32_t (&w)[OZ_S])
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)(u >> 52) & 0x7ff;
    const unsigned long long man = (u & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
    const int sh = max(ex, 1) - 1012 + adj;         // x 2^adj 2^63 = man 2^sh
    long long q = sh >= 0 ? (long long)(man << (sh > 10 ? 10 : sh)) : (long long)(sh > -64 ? man >> -sh : 0ull);
    if (u >> 63) q = -q;
    const unsigned long long t = (unsigned long long)q + 0x8080808080808080ull;   // first digit too: its byte is signed + 128
    const uint32_t hi = (uint32_t)(t >> 32), lo = (uint32_t)t;
#pragma unroll
    for (int j = 0; j < OZ_S; ++j) {
        const uint32_t b = __byte_perm(j < 4 ? hi : lo, 0x4b000000u, 0x7440 + (3 - (j & 3)));   // 2^23 + byte
        w[j] = __float_as_uint(__uint_as_float(b) - 8388736.f);                                 // - (2^23 + 128)
    }
}

// c (hi + 2^-32 lo), c a power of two, |hi| and |lo| below 2^51, rounded once.  Two operations of
// the FP64 pipe (conversions run there too): an integer added to the bits of 1.5 2^52 is a
// double, the offsets of both terms come off in one subtraction, and c is an exponent.
__device__ __forceinline__ double oz_value(long long hi, long long lo, double c)
{
    constexpr long long B = 0x4338000000000000ll;              // bits of 1.5 2^52
    const double h = __longlong_as_double(B + hi), l = __longlong_as_double(B + lo);
    const double v = fma(0x1p-32, l, h - (0x1.8p52 + 0x1.8p20));
    const int ev = (int)(__double_as_longlong(v) >> 52) & 0x7ff, ec = (int)(__double_as_longlong(c) >> 52) & 0x7ff;
    const int e = ev + ec - 1023;
    if (ev == 0 || ec == 0 || e <= 0 || e >= 0x7ff) return c * v;   // zero, or beyond the normal range
    return __longlong_as_double(__double_as_longlong(v) + ((long long)(ec - 1023) << 52));
}

__device__ __forceinline__ void mma_f16_ss(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
        "l"(da), "l"(db), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ double2 lds_d2(uint32_t a)
{
    double2 v;
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
    return v;
}

// transposed: the same walk with the matrices transposed, the phases conjugated and the roles
// of the pair's boxes exchanged (in: local, out: multipole expansions)
__global__ void __launch_bounds__(OZ_T, 1)
    k_m2l_oz(const __grid_constant__ OzPlan sp, int transposed, int64_t nwork, const M2LWork *work, const M2LPair *pairs,
             const unsigned char *img, const double *rscale, const int *dexp, const OzIn *packed, const int *bexp, cd *out,
             unsigned char *xscr, double *yscr, int *status)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    const int p = sp.p, P = sp.P, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t *ent = (uint32_t *)(smraw + sp.o_ent);
    // exponents per input and per pair
    int *adj = (int *)(smraw + sp.o_adj), *pexp = (int *)(smraw + sp.o_exp);
    M2LPair *pr = (M2LPair *)(smraw + sp.o_pair);
    uint64_t *full = (uint64_t *)(smraw + sp.o_bars), *empty = full + OZ_ST, *accfull = empty + OZ_ST;
    uint32_t *tslot = (uint32_t *)(accfull + 1);
    const uint32_t ph0 = tc::smem_u32(smraw + sp.o_ph);
    unsigned char *X = xscr + (size_t)blockIdx.x * sp.nk[0] * OZ_A;
    double2 *Y = (double2 *)yscr + (size_t)blockIdx.x * OZ_BN * sp.rows;   // [pair][row]
    const int D0e = sp.nk[0] * 8;

    if (warp == 0) tc::tmem_alloc(tslot, 512);
    if (tid == 0) {
        for (int s = 0; s < OZ_ST; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(accfull, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    for (int j = tid; j < D0e; j += OZ_T) ent[j] = j < sp.D[0] ? sec_word(p, j) : 0u;
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    bool failed = false;
    uint32_t g = 0;        // K-steps through the ring so far (producer and MMA thread count alike)
    uint32_t ntile = 0;    // tiles so far

    for (int64_t it = blockIdx.x; it < nwork && !failed; it += gridDim.x) {
        const M2LWork w = work[it];
        // the inputs' exponents: adj takes the degrees to one size, pexp the pair below 2^-2 (two
        // coefficients of parts below 2^(pexp - adj - 2): below 2^-1.5 of it each)
        const int *an = dexp + (int64_t)w.geom * (p + 1);
        for (int j = tid; j < D0e; j += OZ_T) adj[j] = an[j < sp.D[0] ? sec_entry(p, j).n : 0];
        // pair records and phases G[d] (conjugated for the transpose), d = -(p+1)..p
        if (tid < w.npair) {
            const M2LPair q = pairs[w.pair0 + tid];
            pr[tid] = q;
            const int *be = bexp + (transposed ? q.tgt : q.src) * (p + 1);
            int top = OZ_ZERO;
            for (int n = 0; n <= p; ++n) {
                const int e = be[n];
                if (e != OZ_ZERO) top = max(top, e == OZ_BAD ? OZ_BAD : e + an[n]);
            }
            pexp[tid] = top == OZ_ZERO ? 0 : top == OZ_BAD ? OZ_BAD : top + 2;
            cd b = mul_i(cd{q.cphi, q.sphi}), e{1.0, 0.0};
            if (transposed) b = conj(b);
            double2 *row = (double2 *)(smraw + sp.o_ph + tid * sp.ph_bytes) + (p + 1);
            for (int d = 0; d <= p + 1; ++d) {
                if (d <= p) row[d] = double2{e.x, e.y};
                row[-d] = double2{e.x, -e.y};
                e = e * b;
            }
        }
        __syncthreads();
        for (int sec = 0; sec < 2 && !failed; ++sec) {
            const int D = sp.D[sec], nk = sp.nk[sec];
            // ---- inputs: thread -> (pair, four inputs = 16 bytes of both rows of the pair)
            for (int e = tid; e < OZ_BN * 2 * nk; e += OZ_T) {
                const int c = e & (OZ_BN - 1), hk = e / OZ_BN;       // hk: half K-step
                uint32_t rr[OZ_S][4], ri[OZ_S][4];                    // rows 2c and 2c + 1, one word per input
                const int64_t box = c < w.npair ? (transposed ? pr[c].tgt : pr[c].src) : 0;
                const OzIn *src = packed + box * D0e + 4 * hk;
                const int4 ad = *(const int4 *)(adj + 4 * hk);
                const int pe = c < w.npair ? pexp[c] : 0;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    cd y{0.0, 0.0};
                    if (c < w.npair) {
                        const OzIn v = src[h];
                        const uint32_t we = ent[4 * hk + h];
                        const double2 G = lds_d2(ph0 + c * sp.ph_bytes + 16 * ((we >> 20) & 63));
                        // W entries subtract conj(G) b in the even sector, C entries add conj(G) c
                        const long long neg = (int)((we >> 26) & 1) == sec ? (long long)(1ull << 63) : 0ll;   // off the FP64 pipe
                        const double bx = __longlong_as_double(__double_as_longlong(v.z) ^ neg);
                        const double by = __longlong_as_double(__double_as_longlong(v.w) ^ neg);
                        y.x = fma(G.x, v.x + bx, G.y * (by - v.y));
                        y.y = fma(G.x, v.y + by, G.y * (v.x - bx));
                    }
                    uint32_t wr[OZ_S], wi[OZ_S];
                    const int sc = (h == 0 ? ad.x : h == 1 ? ad.y : h == 2 ? ad.z : ad.w) - pe;
                    oz_digits(y.x, sc, wr);
                    oz_digits(y.y, sc, wi);
#pragma unroll
                    for (int j = 0; j < OZ_S; ++j) {
                        rr[j][h] = __byte_perm(wr[j], wi[j] ^ 0x80000000u, 0x7632);   // (Re, -Im)
                        ri[j][h] = __byte_perm(wi[j], wr[j], 0x7632);                 // (Im, Re)
                    }
                }
                unsigned char *o = X + (size_t)(hk >> 1) * OZ_A + (hk & 1) * 128;
                const int r0 = 2 * c;
                const uint32_t off = (r0 >> 3) * 256 + (r0 & 7) * 16;   // row 2c + 1 follows 16 bytes on
#pragma unroll
                for (int j = 0; j < OZ_S; ++j) {
                    *(uint4 *)(o + j * 4096 + off) = make_uint4(rr[j][0], rr[j][1], rr[j][2], rr[j][3]);
                    *(uint4 *)(o + j * 4096 + off + 16) = make_uint4(ri[j][0], ri[j][1], ri[j][2], ri[j][3]);
                }
            }
            asm volatile("fence.proxy.async;" ::: "memory");   // the bulk copies read what was written here
            __syncthreads();
            const unsigned char *tile = img + (size_t)w.geom * sp.img_bytes + sp.sec_img[sec];
            const double *rs = rscale + (size_t)w.geom * sp.rows + (sec ? sp.D[0] : 0);
            for (int t = 0; t * OZ_NT < D && !failed; ++t, ++ntile) {
                const int N = oz_tile_rows(D, t);
                const uint32_t bb = (uint32_t)(OZ_S * N * 32);
                if (warp == 0 && lane == 0) {
                    for (int s = 0; s < nk; ++s) {
                        const uint32_t q = g + s, sl = q % OZ_ST;
                        if (q >= OZ_ST && !tc::mbar_wait(&empty[sl], (q / OZ_ST - 1) & 1, OZ_POLLS)) {
                            failed = true;
                            break;
                        }
                        tc::mbar_expect_tx(&full[sl], OZ_A + bb);
                        tc::bulk_g2s(smraw + sl * OZ_SLOT, X + (size_t)s * OZ_A, OZ_A, &full[sl]);
                        tc::bulk_g2s(smraw + sl * OZ_SLOT + OZ_A, tile + (size_t)s * bb, bb, &full[sl]);
                    }
                } else if (warp == 1 && tc::elect_one()) {
                    const uint32_t idesc = tc::idesc_bf16(128, N);
                    const uint64_t pa = 4096 >> 4, pb = (uint32_t)(N * 32) >> 4;
                    for (int s = 0; s < nk; ++s) {
                        const uint32_t q = g + s, sl = q % OZ_ST;
                        if (!tc::mbar_wait(&full[sl], (q / OZ_ST) & 1, OZ_POLLS)) {
                            failed = true;
                            break;
                        }
                        tc::fence_after();
                        const uint64_t da = tc::sdesc(tc::smem_u32(smraw + sl * OZ_SLOT), 128, 256);
                        const uint64_t db = tc::sdesc(tc::smem_u32(smraw + sl * OZ_SLOT + OZ_A), 128, 256);
#pragma unroll
                        for (int j = 0; j < OZ_S; ++j)
#pragma unroll
                            for (int i = 0; i + j < OZ_S; ++i)
                                mma_f16_ss(tbase + (i + j) * OZ_NT, da + i * pa, db + j * pb, idesc,
                                           (s > 0 || j > 0) ? 1u : 0u);
                        tc::commit(&empty[sl]);
                    }
                    tc::commit(accfull);
                }
                __syncwarp();
                g += nk;
                if (!tc::mbar_wait(accfull, ntile & 1, OZ_POLLS)) failed = true;
                tc::fence_after();
                // ---- accumulators -> FP64: warp -> lane quadrant warp % 4, 16 columns
                const int q4 = warp & 3, cg = warp >> 2, row = 32 * q4 + lane;
                if (32 * q4 < 2 * w.npair) {
                    for (int c0 = 16 * cg; c0 < 16 * cg + 16 && c0 < N; c0 += 8) {
                        uint32_t v[OZ_S][8];
#pragma unroll
                        for (int d = 0; d < OZ_S; ++d)
                            tc::tmem_ld8(tbase + ((uint32_t)(32 * q4) << 16) + d * OZ_NT + c0, v[d]);
                        tc::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int r = t * OZ_NT + c0 + i;
                            if (r >= D) break;
                            auto a = [&](int d) { return __float2int_rn(__uint_as_float(v[d][i])); };
                            const long long hi = (((long long)a(0) << 16) + ((long long)a(1) << 8) + a(2)) * 256 + a(3);
                            const long long lo = (((long long)a(4) << 16) + ((long long)a(5) << 8) + a(6)) * 256 + a(7);
                            const double y = oz_value(hi, lo, rs[r]);
                            ((double *)(Y + (size_t)(row >> 1) * sp.rows + (sec ? sp.D[0] : 0) + r))[row & 1] = y;
                        }
                    }
                }
                tc::fence_before();
                if (__syncthreads_or(failed)) failed = true;
                tc::fence_after();
                tile += (size_t)nk * bb;
            }
        }
        if (failed) break;
        // ---- outputs: the phases take the pair's power of two (not a number where an input is none)
        for (int e = tid; e < w.npair * (2 * p + 2); e += OZ_T) {
            const int c = e / (2 * p + 2), d = e - c * (2 * p + 2);
            double2 *G = (double2 *)(smraw + sp.o_ph + c * sp.ph_bytes) + d;
            const double f = pexp[c] == OZ_BAD ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(1.0, pexp[c]);
            *G = double2{f * G->x, f * G->y};
        }
        __syncthreads();
        if (warp < sp.out_warps) {
            double2 *sg = (double2 *)(smraw + warp * sp.stage_bytes);   // the ring is idle here
            for (int c = warp; c < w.npair; c += sp.out_warps) {
                const double2 *y0 = Y + (size_t)c * sp.rows, *y1 = y0 + sp.D[0];
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
                for (int r = lane; r < sp.D[0]; r += 32) {
                    const double2 ye = y0[r], yo = r < sp.D[1] ? y1[r] : double2{0.0, 0.0};
                    const uint32_t we = ent[r];
                    const double2 G = lds_d2(ph0 + c * sp.ph_bytes + 16 * ((we >> 20) & 63));
                    const double2 s{ye.x + yo.x, ye.y + yo.y};
                    double2 d{ye.x - yo.x, ye.y - yo.y};
                    sg[we & 1023] = double2{fma(G.x, s.x, G.y * s.y), fma(G.x, s.y, -G.y * s.x)};
                    if (!(we >> 26 & 1)) d = double2{-d.x, -d.y};
                    if (!(we >> 27 & 1))
                        sg[(we >> 10) & 1023] = double2{fma(G.x, d.x, -G.y * d.y), fma(G.x, d.y, G.y * d.x)};
                }
                tc::fence_smem_async();
                __syncwarp();
                if (lane == 0)
                    asm volatile(
                        "cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f64 [%0], [%1], %2;\n\t"
                        "cp.async.bulk.commit_group;" ::"l"(out + (transposed ? pr[c].src : pr[c].tgt) * 3 * P),
                        "r"(tc::smem_u32(sg)), "r"(sp.stage_bytes)
                        : "memory");
            }
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
        tc::fence_smem_async();   // the next bulk copies write where the staging rows were
        __syncthreads();
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (failed) {
        // copies and MMAs still in flight land before the CTA leaves
        if (tid == 0)
            for (int s = 0; s < OZ_ST; ++s) tc::mbar_wait(&full[s], 0, 1 << 12), tc::mbar_wait(&full[s], 1, 1 << 12);
        atomicOr(status, 4);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, 512);
}

// exponents a_n (0 <= n <= p, a_0 = 0) of the degrees of a geometry's columns: source degrees into
// dexp, target degrees (the transpose's columns) into dexpT.  Of the binary exponents l[nu][n] of the
// largest entry of every degree block of the five tables: the mean over the rows of degree p / 2 and
// more of l less the row's own mean.  The upper rows, whose blocks spread most, have it fit them
// closest: rms errors per degree block at p = 12, three layers, N = 1503, 0.9e-15 (SIMT 1.7e-15), with
// the mean over all rows 1.9e-15.  One block per geometry; a thread takes a table's row.
__global__ void __launch_bounds__(256) k_oz_degrees(int p, const GeomDev *geoms, const cd *tab64, int *dexp, int *dexpT)
{
    constexpr int NONE = -(1 << 20);
    __shared__ int l[OZ_PMAX + 1][OZ_PMAX + 1];
    __shared__ float mean[2][OZ_PMAX + 1];
    const int P = (p + 1) * (p + 1);
    const int64_t gi = blockIdx.x;
    for (int e = threadIdx.x; e < (OZ_PMAX + 1) * (OZ_PMAX + 1); e += blockDim.x) (&l[0][0])[e] = NONE;
    __syncthreads();
    for (int tr = threadIdx.x; tr < NTAB * P; tr += blockDim.x) {
        const cd *row = tab64 + (gi * NTAB * P + tr) * P;
        int nu = (int)sqrtf((float)(tr % P) + 0.5f);
        while ((nu + 1) * (nu + 1) <= tr % P) ++nu;
        while (nu * nu > tr % P) --nu;
        for (int n = 0, k = 0; n <= p; ++n) {
            int ex = 0;
            for (; k < (n + 1) * (n + 1); ++k)
                ex = max(ex, max((int)(__double_as_longlong(row[k].x) >> 52) & 0x7ff,
                                 (int)(__double_as_longlong(row[k].y) >> 52) & 0x7ff));
            if (ex > 0) atomicMax(&l[nu][n], ex - 1023);
        }
    }
    __syncthreads();
    // means over what is there of a row, then over the differences in a column
    const int i = threadIdx.x;
    auto at = [&](int c, int a, int b) { return c ? l[b][a] : l[a][b]; };   // c = 0: rows are target degrees
    for (int c = 0; c < 2; ++c)
        if (i <= p) {
            float s = 0.f;
            int n = 0;
            for (int b = 0; b <= p; ++b)
                if (at(c, i, b) != NONE) {
                    s += (float)at(c, i, b);
                    ++n;
                }
            mean[c][i] = n ? s / n : 0.f;
        }
    __syncthreads();
    if (i <= p)
        for (int c = 0; c < 2; ++c) {
            auto part = [&](int b) {           // of column b
                float s = 0.f;
                int n = 0;
                for (int a = (p + 1) / 2; a <= p; ++a)
                    if (at(c, a, b) != NONE) {
                        s += (float)at(c, a, b) - mean[c][a];
                        ++n;
                    }
                return n ? s / n : 0.f;
            };
            const GeomDev &g = geoms[gi];
            const float lg = (float)log2(c ? g.scale_t : g.scale_s);
            const float v = part(i) - part(0) + (float)i * lg;
            (c ? dexpT : dexp)[gi * (p + 1) + i] = (int)rintf(fminf(fmaxf(v, -900.f), 900.f));
        }
}

// one warp per row of a geometry's sector block (transposed: of its transpose, with the C
// entries of order 0 doubled as outputs and halved as inputs, as the shared input and output
// maps count them): the row's power of two, then its digits in the K-step images
__global__ void __launch_bounds__(256) k_oz_image(const __grid_constant__ OzPlan sp, int transposed,
                                                  const GeomDev *geoms, const CompDev *comps, const cd *tab64,
                                                  const int *dexp, unsigned char *img, double *rscale)
{
    __shared__ double ps[OZ_PMAX + 1], pt[OZ_PMAX + 1], cs[OZ_PMAX + 1];
    const int64_t gi = blockIdx.y;
    const GeomDev &gm = geoms[gi];
    if (threadIdx.x <= sp.p) {
        double a = 1.0, b = 1.0;
        for (int i = 0; i < (int)threadIdx.x; ++i) {
            a *= gm.scale_s;
            b *= gm.scale_t;
        }
        ps[threadIdx.x] = a;
        pt[threadIdx.x] = b;
        cs[threadIdx.x] = ldexp(1.0, -dexp[gi * (sp.p + 1) + threadIdx.x]);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= sp.rows) return;
    const int sec = row >= sp.D[0], r = row - (sec ? sp.D[0] : 0), D = sp.D[sec];
    const CompDev cp = comps[gm.comp];
    const bool fi = (cp.s < 0) != (cp.has_src_refl != 0), fo = (cp.s < 0) != (cp.has_tgt_refl != 0);
    const cd *tab = tab64 + gi * NTAB * (int64_t)sp.P * sp.P;
    const SecEntry er = sec_entry(sp.p, r);
    auto value = [&](int k) {
        const SecEntry ek = sec_entry(sp.p, k);
        cd v;
        if (!transposed) {
            v = sec_scaled(er, ek, fi, fo, pt, ps, sec_value(sp.p, sec, er, ek, tab));
        } else {
            v = sec_scaled(ek, er, fi, fo, pt, ps, sec_value(sp.p, sec, ek, er, tab));
            if (er.c && er.m == 0) v = 2.0 * v;
            if (ek.c && ek.m == 0) v = 0.5 * v;
        }
        return cs[ek.n] * v;
    };
    double mx = 0.0;
    for (int k = lane; k < D; k += 32) {
        const cd v = value(k);
        mx = fmax(mx, fmax(fabs(v.x), fabs(v.y)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    int e = 0;
    if (mx > 0.0) {
        frexp(mx, &e);
        ++e;                                   // mx < 2^(e - 1)
    }
    if (lane == 0) rscale[gi * sp.rows + row] = ldexp(1.0, e - 38);
    const double f = ldexp(1.0, -e);
    const int t = r / OZ_NT, rl = r - t * OZ_NT, N = oz_tile_rows(D, t), nk = sp.nk[sec];
    // the tiles before this one are full
    unsigned char *o = img + gi * (size_t)sp.img_bytes + sp.sec_img[sec] + (size_t)t * nk * OZ_S * OZ_NT * 32 +
                       (rl >> 3) * 256 + (rl & 7) * 16;
    for (int k = lane; k < nk * 8; k += 32) {
        cd v{0.0, 0.0};
        if (k < D) v = f * value(k);
        uint32_t wr[OZ_S], wi[OZ_S];
        oz_digits(v.x, 0, wr);
        oz_digits(v.y, 0, wi);
        unsigned char *q = o + (size_t)(k >> 3) * (OZ_S * N * 32) + ((k & 7) >> 2) * 128 + (k & 3) * 4;
#pragma unroll
        for (int j = 0; j < OZ_S; ++j) *(uint32_t *)(q + (size_t)j * N * 32) = __byte_perm(wr[j], wi[j], 0x7632);
    }
}

// packed inputs of every box: entry j's two coefficients side by side, and per degree the
// exponent e of its largest part, |part| < 2^e; clears the box's output expansion
__global__ void __launch_bounds__(128) k_oz_pack(int p, int n8, int D0, const cd *in, OzIn *pk, int *bexp, cd *out)
{
    __shared__ int top[OZ_PMAX + 1];
    const int P = (p + 1) * (p + 1), P3 = 3 * P;
    const int64_t box = blockIdx.x;
    const cd *m = in + box * P3;
    if (threadIdx.x <= p) top[threadIdx.x] = OZ_ZERO;
    __syncthreads();
    for (int j = threadIdx.x; j < P3; j += blockDim.x) {
        const cd v = m[j];
        const int ex = max((int)(__double_as_longlong(v.x) >> 52) & 0x7ff, (int)(__double_as_longlong(v.y) >> 52) & 0x7ff);
        int n = (int)sqrtf((float)(j % P) + 0.5f);
        while ((n + 1) * (n + 1) <= j % P) ++n;
        while (n * n > j % P) --n;
        if (ex == 0x7ff) atomicMax(&top[n], OZ_BAD);
        else if (v.x != 0.0 || v.y != 0.0) atomicMax(&top[n], max(ex, 1) - 1022);
        out[box * P3 + j] = cd{0.0, 0.0};
    }
    for (int j = threadIdx.x; j < n8; j += blockDim.x) {
        OzIn v{0.0, 0.0, 0.0, 0.0};
        if (j < D0) {
            const uint32_t w = sec_word(p, j);
            const cd a = m[w & 1023], b = m[(w >> 10) & 1023];
            v = OzIn{a.x, a.y, b.x, b.y};
        }
        pk[box * n8 + j] = v;
    }
    __syncthreads();
    if (threadIdx.x <= p) bexp[box * (p + 1) + threadIdx.x] = top[threadIdx.x];
}

}  // namespace

bool m2l_oz_supported(int p) { return p >= 1 && p <= OZ_PMAX; }
int m2l_oz_pairs() { return OZ_BN; }
size_t m2l_oz_image_bytes(int p, int64_t ngeom)
{
    const OzPlan sp = oz_plan(p);
    return (size_t)ngeom * (sp.img_bytes + (size_t)sp.rows * sizeof(double) + (p + 1) * sizeof(int));
}
size_t m2l_oz_packed_bytes(int p, int64_t nbox) { return (size_t)nbox * (oz_plan(p).nk[0] * 8 * sizeof(OzIn) + (p + 1) * sizeof(int)); }
size_t m2l_oz_scratch_bytes(int p, int ncta)
{
    const OzPlan sp = oz_plan(p);
    return (size_t)ncta * ((size_t)sp.nk[0] * OZ_A + (size_t)OZ_BN * sp.rows * sizeof(double2));
}

// behind the images: the rows' powers of two, the degrees' exponents
static double *oz_rscale(const OzPlan &sp, const void *img, int64_t ng) { return (double *)((unsigned char *)img + (size_t)ng * sp.img_bytes); }
static int *oz_dexp(const OzPlan &sp, const void *img, int64_t ng) { return (int *)(oz_rscale(sp, img, ng) + (size_t)ng * sp.rows); }

void launch_oz_images(int p, int64_t ng, const GeomDev *geoms, const CompDev *comps, const cd *tab64, void *img, void *imgT,
                      cudaStream_t st)
{
    const OzPlan sp = oz_plan(p);
    if (ng <= 0) return;
    k_oz_degrees<<<(unsigned)ng, 256, 0, st>>>(p, geoms, tab64, oz_dexp(sp, img, ng), oz_dexp(sp, imgT, ng));
    for (int tr = 0; tr < 2; ++tr) {
        void *q = tr ? imgT : img;
        cudaMemsetAsync(q, 0, (size_t)ng * sp.img_bytes, st);     // rows beyond the block stay zero
        for (int64_t g0 = 0; g0 < ng; g0 += 32768) {              // grid.y is limited to 65535
            const int64_t nb = std::min<int64_t>(32768, ng - g0);
            k_oz_image<<<dim3((sp.rows + 7) / 8, (unsigned)nb), 256, 0, st>>>(
                sp, tr, geoms + g0, comps, tab64 + g0 * NTAB * (int64_t)sp.P * sp.P, oz_dexp(sp, q, ng) + g0 * (p + 1),
                (unsigned char *)q + (size_t)g0 * sp.img_bytes, oz_rscale(sp, q, ng) + g0 * sp.rows);
        }
    }
}

cudaError_t launch_m2l_oz(int p, bool transposed, int64_t ngeom, int64_t nwork, const M2LWork *work, const M2LPair *pairs,
                          const void *img, int64_t nbox, const cd *in, cd *out, void *packed, void *scratch, int ncta,
                          int *status, cudaStream_t st)
{
    if (!m2l_oz_supported(p) || ncta < 1) return cudaErrorInvalidValue;
    const OzPlan sp = oz_plan(p);
    const int n8 = sp.nk[0] * 8;
    int *be = (int *)((unsigned char *)packed + (size_t)nbox * n8 * sizeof(OzIn));
    if (nbox > 0) k_oz_pack<<<(unsigned)nbox, 128, 0, st>>>(p, n8, sp.D[0], in, (OzIn *)packed, be, out);
    if (nwork <= 0) return cudaGetLastError();
    unsigned char *x = (unsigned char *)scratch;
    k_m2l_oz<<<(unsigned)std::min<int64_t>(nwork, ncta), OZ_T, std::max<size_t>(sp.smem, 116 * 1024), st>>>(
        sp, transposed ? 1 : 0, nwork, work, pairs, (const unsigned char *)img, oz_rscale(sp, img, ngeom),
        oz_dexp(sp, img, ngeom), (const OzIn *)packed, be, out, x,
        (double *)(x + (size_t)ncta * sp.nk[0] * OZ_A), status);
    return cudaGetLastError();
}

cudaError_t configure_m2l_oz()
{
    return cudaFuncSetAttribute(k_m2l_oz, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

}  // namespace lmf
