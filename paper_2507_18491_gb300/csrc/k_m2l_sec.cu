// M2L of the mixed form on the 5th-generation tensor cores (tcgen05), p <= 12, on the
// mirror sectors of sector.cuh.
//
// A work item is up to 64 pairs of one geometry.  For each sector block M_e it forms
//   D (128 x N) = X (128 x K) M_e'^T,
// whose 128 rows are real columns -- rows 2c, 2c+1 hold (Re x, -Im x) and (Im x, Re x)
// of the sector vector of pair c, giving Re (M x) and Im (M x) -- and whose N columns are
// the block's rows.  The block is the B operand (K = interleaved Re / Im input index),
// stored once per build as three bf16 planes (x ~ x1 + x2 + x3, each the bf16 rounding
// of what the previous pieces leave: 24 bits, FP32's exponent range) in exactly the
// shared-memory image of each K-step.  Of the nine products of pieces the six of size
// 2^-16 and more are formed: X1 T1 in one accumulator and the other five in further ones
// (the tensor core truncates small addends against a large accumulator).
//
// Blocks of up to 192 padded rows (p <= 10) take one tile, larger ones two, so that the
// accumulators leave tensor memory for the X ring.  The five small products alternate
// between two accumulators where three fit (N <= 128, p <= 8), so that fewer MMAs follow one
// into the same accumulator.
// Roles (864 threads, one CTA per SM):
//   warps 0-7   X producers, two groups of four warps (one per tensor-memory lane
//               quadrant), group g writing K-step g of every chunk: the two coefficients of
//               an input lie side by side in the packed expansions (k_sec_pack), so that a
//               K-step of a pair is one 128-byte line; asynchronous copies bring the lines of
//               the warp's 16 pairs into its shared ring two chunks ahead (a load per
//               coefficient touches 32 lines per instruction: 0.95 against 0.76 ms for 397328
//               pairs at p = 7); then one phase per input, the split into three pieces (the
//               two rows of a pair share them) and the store into the tensor-memory ring;
//   warps 8-23  epilogue: accumulators -> a per-CTA scratch in global memory (L2-resident)
//               ([pair][row], through a tile in shared memory), so that tensor memory is free
//               again at once; after the item's last tile one warp per pair combines the two
//               sectors, applies the output phases into a shared staging row [3][P] and
//               adds it to the pair's local expansions with one bulk reduction;
//   warp 24     one bulk copy per matrix chunk into a shared-memory ring;
//   warp 25     MMA issue;
//   warp 26     bulk copies of the pair records and phases, one item ahead.
// Every wait is bounded; a wait that gives up sets bit 4 of the status word and its role
// stops.
//
// Measured (GB300, M2L stage; before: nine applications of five P x P tables per pair on the
// same pipeline): 1.70M pairs at p = 8 14.1 -> 3.31 ms, 397328 pairs at p = 7 2.9 -> 0.65 ms,
// 136292 pairs at p = 12 1.8 -> 1.17 ms.  Per 64-pair item at p = 8 the MMAs take 12 thousand
// cycles, the producers 32, the scatter 18.
#include <algorithm>

#include <cuda_bf16.h>

#include "sector.cuh"
#include "tc.cuh"

namespace lmf {

namespace {

constexpr int SC_BN = 64;          // pairs per work item
constexpr int SC_KS = 2;           // MMA K-steps (16 real K, 8 complex inputs) per chunk
constexpr int SC_KC = 8 * SC_KS;   // complex inputs per chunk
constexpr int SC_NPC = 3;          // bf16 pieces per value
constexpr int SC_XW = 8 * SC_NPC * SC_KS;   // tensor-memory columns of an X chunk
constexpr int SC_SX_MAX = 4;       // X ring slots
constexpr int SC_ST_MAX = 12;      // matrix ring slots
constexpr int SC_XD = 3;           // stages of a producer warp's shared ring of packed inputs
constexpr uint32_t SC_XROW = 144;  // bytes of a pair's K-step there: 8 inputs of 16 bytes, padded against bank conflicts
constexpr uint32_t SC_XST = 16 * SC_XROW;
constexpr int SC_PT = 256, SC_ET = 512;     // producer, epilogue threads
constexpr int SC_EW = SC_ET / 32;
constexpr int SC_DS = 34;          // row stride (words) of an epilogue warp's 16-row drain tile
constexpr uint32_t SC_TILE = 16 * SC_DS * 4;
constexpr int SC_WTMA = (SC_PT + SC_ET) / 32, SC_WMMA = SC_WTMA + 1, SC_WMETA = SC_WTMA + 2;
constexpr int SC_THREADS = (SC_WMETA + 1) * 32;
constexpr int SC_PMAX = 12;
constexpr int SC_MAXT = 4;
constexpr uint32_t SC_SMEM_MAX = 227 * 1024;
constexpr int SC_POLLS = 1 << 22;

struct SecTile {
    int sec, row0, N, nchunk;      // sector, first row, padded rows, K chunks
    uint32_t cb, img;              // bytes of a chunk; offset of the tile in a geometry's image
    int y0;                        // first row of the tile in the scratch
};

struct SecPlan {
    int p, P, D0, D1, ntile, nmax, nacc, SX, ST, nchunk0, yrows, ews;
    uint32_t slot, img_bytes, ph_bytes, meta_bytes, stage_bytes;
    uint32_t o_meta, o_ent, o_xsrc, o_stage, o_bars, smem;
    SecTile t[SC_MAXT];
};

SecPlan sec_plan(int p)
{
    SecPlan s{};
    s.p = p;
    s.P = (p + 1) * (p + 1);
    s.D0 = sec_dim(p, 0);
    s.D1 = sec_dim(p, 1);
    auto r16 = [](int v) { return (v + 15) & ~15; };
    const bool split = r16(s.D0) > 192;
    uint32_t img = 0;
    for (int e = 0; e < 2; ++e) {
        const int D = e ? s.D1 : s.D0;
        const int first = split ? 16 * ((D + 16) / 32) : D;   // half of the rows, to a multiple of 16
        for (int r0 = 0; r0 < D; r0 += first) {
            SecTile &t = s.t[s.ntile++];
            t.sec = e;
            t.row0 = r0;
            t.N = r16(std::min(first, D - r0));
            if (split && r0 > 0) t.N = r16(D - r0);
            t.nchunk = (D + SC_KC - 1) / SC_KC;
            t.cb = (uint32_t)(SC_KS * SC_NPC * t.N * 32);
            t.img = img;
            img += t.cb * t.nchunk;
            t.y0 = s.yrows;
            s.yrows += t.N;
            s.nmax = std::max(s.nmax, t.N);
            s.slot = std::max(s.slot, t.cb);
            if (split && r0 > 0) break;
        }
    }
    s.img_bytes = img;
    s.nchunk0 = s.t[0].nchunk;
    s.nacc = 3 * s.nmax + 2 * SC_XW <= 512 ? 3 : 2;
    s.SX = std::min(SC_SX_MAX, (512 - s.nmax * s.nacc) / SC_XW);
    s.ph_bytes = (uint32_t)m2l_sec_phases(p) * 8;
    s.meta_bytes = SC_BN * (s.ph_bytes + (uint32_t)sizeof(M2LPair));
    s.stage_bytes = ((uint32_t)(3 * s.P + 2) * 8 + 15) & ~15u;
    s.ews = s.D0 <= 128 ? SC_EW : SC_EW / 2;   // epilogue warps that scatter: their staging rows take shared memory
    const uint32_t bars = (2 * SC_ST_MAX + 2 * SC_SX_MAX + 12) * 8 + 16;
    const uint32_t ent = (uint32_t)s.nchunk0 * SC_KC * 4;
    // staging rows of the scatter; the drain tiles of all epilogue warps lie there too
    const uint32_t stages = std::max(s.ews * s.stage_bytes, (uint32_t)SC_EW * SC_TILE);
    const uint32_t fixed = 2 * s.meta_bytes + ent + SC_PT / 32 * SC_XD * SC_XST + stages + bars;
    s.ST = (int)std::min<uint32_t>(SC_ST_MAX, (SC_SMEM_MAX - fixed) / s.slot);
    s.o_meta = s.ST * s.slot;
    s.o_ent = s.o_meta + 2 * s.meta_bytes;
    s.o_xsrc = s.o_ent + ent;
    s.o_stage = s.o_xsrc + SC_PT / 32 * SC_XD * SC_XST;
    s.o_bars = s.o_stage + stages;
    s.smem = s.o_bars + bars;
    return s;
}

__device__ __forceinline__ cf lds_c(uint32_t a)
{
    cf v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}

// three-piece bf16 split of a pair of floats; word j holds piece j, lo in the low half
__device__ __forceinline__ void split_bf16(float lo, float hi, uint32_t (&w)[SC_NPC])
{
    float2 r{lo, hi};
#pragma unroll
    for (int j = 0; j < SC_NPC; ++j) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(r.x, r.y);
        w[j] = *(const uint32_t *)&h;
        if (j + 1 < SC_NPC) {
            const float2 f = __bfloat1622float2(h);
            r = float2{r.x - f.x, r.y - f.y};
        }
    }
}

// RJ: rows of the even sector per lane of an epilogue warp (32 RJ >= D0)
template <int RJ>
__global__ void __launch_bounds__(SC_THREADS, 1)
    k_m2l_sec(const __grid_constant__ SecPlan sp, int64_t nwork, const M2LWork *work, TcProb one, const TcProb *probs,
              float *yscr, int *status)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    const int p = sp.p, P = sp.P, ST = sp.ST, SX = sp.SX;
    uint32_t *ent = (uint32_t *)(smraw + sp.o_ent);
    uint64_t *bars = (uint64_t *)(smraw + sp.o_bars);
    uint64_t *tfull = bars, *tempty = bars + SC_ST_MAX, *xfull = bars + 2 * SC_ST_MAX, *xempty = xfull + SC_SX_MAX;
    uint64_t *accfull = xempty + SC_SX_MAX, *accempty = accfull + 1, *metafull = accfull + 2, *metaempty = accfull + 4,
             *fin = accfull + 6, *ydone = accfull + 7, *yfree = accfull + 8;
    uint32_t *tslot = (uint32_t *)(accfull + 9);
    auto meta_ph = [&](int slot) { return smraw + sp.o_meta + slot * sp.meta_bytes; };
    auto meta_pair = [&](int slot) { return (const M2LPair *)(meta_ph(slot) + SC_BN * sp.ph_bytes); };
    auto prob = [&](const M2LWork &w) { return probs ? probs[w.prob] : one; };

    float2 *Y = (float2 *)(yscr + (size_t)blockIdx.x * sp.yrows * 128);   // [pair][row]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) tc::tmem_alloc(tslot, 512);
    if (tid == 0) {
        for (int s = 0; s < ST; ++s) {
            tc::mbar_init(&tfull[s], 1);
            tc::mbar_init(&tempty[s], 1);
        }
        for (int s = 0; s < SX; ++s) {
            tc::mbar_init(&xfull[s], SC_PT);   // both producer groups (one K-step each)
            tc::mbar_init(&xempty[s], 1);
        }
        tc::mbar_init(accfull, 1);
        tc::mbar_init(accempty, SC_ET);
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&metafull[i], 1);
            tc::mbar_init(&metaempty[i], (SC_PT + SC_ET) / 32);
        }
        tc::mbar_init(fin, 1);
        tc::mbar_init(ydone, SC_ET);
        tc::mbar_init(yfree, SC_ET);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    for (int j = tid; j < sp.nchunk0 * SC_KC; j += SC_THREADS) ent[j] = j < sp.D0 ? sec_word(p, j) : 0u;
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = *tslot;
    const uint32_t xb = tbase + (uint32_t)(sp.nmax * sp.nacc);   // tensor-memory address of the X ring
    bool failed = false;

    if (warp == SC_WTMA) {
        // ------------------------------------------------ matrix chunks
        if (lane == 0) {
            uint32_t g = 0, ph = 0;   // chunks issued; parity of the current pass over the ring
            int s = 0;
            for (int64_t it = blockIdx.x; it < nwork && !failed; it += gridDim.x) {
                const M2LWork w = work[it];
                const unsigned char *src = (const unsigned char *)prob(w).img + (size_t)w.geom * sp.img_bytes;
                for (int t = 0; t < sp.ntile && !failed; ++t) {
                    const uint32_t cb = sp.t[t].cb;
                    const unsigned char *ts = src + sp.t[t].img;
                    for (int c = 0; c < sp.t[t].nchunk; ++c) {
                        if (g >= (uint32_t)ST && !tc::mbar_wait(&tempty[s], ph ^ 1, SC_POLLS)) {
                            failed = true;
                            break;
                        }
                        tc::mbar_expect_tx(&tfull[s], cb);
                        tc::bulk_g2s(smraw + s * sp.slot, ts + (size_t)c * cb, cb, &tfull[s]);
                        ++g;
                        if (++s == ST) {
                            s = 0;
                            ph ^= 1;
                        }
                    }
                }
            }
            // copies still in flight land before the CTA leaves
            for (uint32_t q = g > (uint32_t)ST ? g - ST : 0; q < g; ++q)
                tc::mbar_wait(&tfull[q % ST], (q / ST) & 1, SC_POLLS);
        }
    } else if (warp == SC_WMETA) {
        // ------------------------------------------------ pair records and phases
        if (lane == 0) {
            uint32_t li = 0;
            for (int64_t it = blockIdx.x; it < nwork; it += gridDim.x, ++li) {
                const M2LWork w = work[it];
                const TcProb pd = prob(w);
                const int slot = li & 1;
                if (li >= 2 && !tc::mbar_wait(&metaempty[slot], ((li >> 1) - 1) & 1, SC_POLLS)) {
                    failed = true;
                    break;
                }
                const uint32_t b0 = w.npair * sp.ph_bytes, b1 = w.npair * (uint32_t)sizeof(M2LPair);
                tc::mbar_expect_tx(&metafull[slot], b0 + b1);
                tc::bulk_g2s(meta_ph(slot), (const unsigned char *)pd.ephase + (size_t)w.pair0 * sp.ph_bytes, b0,
                             &metafull[slot]);
                tc::bulk_g2s((void *)meta_pair(slot), pd.pairs + w.pair0, b1, &metafull[slot]);
            }
            for (uint32_t q = li > 2 ? li - 2 : 0; q < li; ++q) tc::mbar_wait(&metafull[q & 1], (q >> 1) & 1, SC_POLLS);
        }
    } else if (warp == SC_WMMA) {
        // ------------------------------------------------ MMA issue
        if (tc::elect_one()) {
            // descriptor of ring slot 0; the address field counts 16-byte units
            const uint64_t dring0 = tc::sdesc(tc::smem_u32(smraw), 128, 256);
            const uint64_t d_slot = sp.slot >> 4;
            uint64_t dslot = dring0;
            uint32_t aslot = xb;
            uint32_t tph = 0, xph = 0, tc_n = 0;   // ring parities; tiles so far
            int st = 0, sx = 0;
            for (int64_t it = blockIdx.x; it < nwork && !failed; it += gridDim.x) {
                for (int t = 0; t < sp.ntile && !failed; ++t, ++tc_n) {
                    if (tc_n >= 1 && !tc::mbar_wait(accempty, (tc_n - 1) & 1, SC_POLLS)) {
                        failed = true;
                        break;
                    }
                    tc::fence_after();
                    const int N = sp.t[t].N;
                    const uint32_t idesc = tc::idesc_bf16(128, N);
                    const uint64_t d_pl = (uint32_t)(N * 32) >> 4, d_sb = SC_NPC * d_pl;
                    // big products; small ones in two accumulators, or in one where three do not fit
                    const uint32_t big = tbase, s1 = tbase + sp.nmax, s2 = tbase + (sp.nacc - 1) * sp.nmax;
                    const uint32_t own = sp.nacc == 3 ? 0u : 1u;   // s2 is s1: its first product adds
                    for (int c = 0; c < sp.t[t].nchunk; ++c) {
                        if (!tc::mbar_wait(&tfull[st], tph, SC_POLLS) || !tc::mbar_wait(&xfull[sx], xph, SC_POLLS)) {
                            failed = true;
                            break;
                        }
                        tc::fence_after();
#pragma unroll
                        for (int u = 0; u < SC_KS; ++u) {
                            // pieces 1, 2, 3 of X (tensor memory) and of the matrix (shared memory)
                            const uint32_t a1 = aslot + 8 * SC_NPC * u, a2 = a1 + 8, a3 = a1 + 16;
                            const uint64_t b1 = dslot + u * d_sb, b2 = b1 + d_pl, b3 = b2 + d_pl;
                            const uint32_t acc = (c > 0 || u > 0) ? 1u : 0u;
                            tc::mma_f16_ta(s1, a1, b2, idesc, acc);
                            tc::mma_f16_ta(s2, a2, b1, idesc, acc | own);
                            tc::mma_f16_ta(big, a1, b1, idesc, acc);
                            tc::mma_f16_ta(s1, a1, b3, idesc, 1u);
                            tc::mma_f16_ta(s2, a3, b1, idesc, 1u);
                            tc::mma_f16_ta(s1, a2, b2, idesc, 1u);
                        }
                        tc::commit(&tempty[st]);
                        tc::commit(&xempty[sx]);
                        dslot += d_slot;
                        aslot += SC_XW;
                        if (++st == ST) {
                            st = 0;
                            tph ^= 1;
                            dslot = dring0;
                        }
                        if (++sx == SX) {
                            sx = 0;
                            xph ^= 1;
                            aslot = xb;
                        }
                    }
                    if (failed) break;
                    tc::commit(accfull);
                }
            }
            tc::commit(fin);   // every MMA issued above has completed once fin flips
            tc::mbar_wait(fin, 0, SC_POLLS);
        }
    } else if (warp < SC_PT / 32) {
        // ------------------------------------------------ X producers
        // the two lanes of a pair's rows (b = 0: Re, -Im; b = 1: Im, Re) each form and split
        // four of the K-step's eight inputs, swap the pieces with the partner lane and store
        // the K-step's 24 columns of their own row
        constexpr int KQ = 4;                  // inputs per lane and chunk
        const int pg = warp / 4, pq = 16 * (warp & 3);   // K-step; first pair of the warp
        const int cc = pq + (lane >> 1), b = lane & 1;
        const int kk0 = 8 * pg + KQ * b;       // the lane's first input within the chunk
        const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
        const uint32_t ent0 = tc::smem_u32(ent) + 4 * kk0;
        const uint32_t ring = tc::smem_u32(smraw + sp.o_xsrc) + warp * (SC_XD * SC_XST);
        const int64_t box_units = sp.nchunk0 * SC_KC;
        // fetch side: lane copies 16-byte unit lane % 8 of the lines of pairs lane / 8 + 4 i
        const uint32_t dst0 = ring + (lane >> 3) * SC_XROW + 16 * (lane & 7);
        int64_t fit = blockIdx.x;
        uint32_t fli = 0;
        int ft = sp.ntile, fc = 0, fst = 0;    // no tile open yet; next stage to fill
        const float4 *fme = nullptr;           // packed expansions of the item's problem
        constexpr uint32_t NONE = 0xffffffffu;
        uint32_t fsrc[4] = {NONE, NONE, NONE, NONE};   // boxes; none: no such pair
        auto fetch = [&]() -> bool {
            if (ft == sp.ntile && fit < nwork) {      // open the next item
                const int slot = fli & 1;
                if (!__all_sync(0xffffffffu, tc::mbar_wait(&metafull[slot], (fli >> 1) & 1, SC_POLLS))) return false;
                const M2LWork w = work[fit];
                fme = (const float4 *)prob(w).me + 8 * pg + (lane & 7);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int c = pq + (lane >> 3) + 4 * i;
                    fsrc[i] = c < w.npair ? (uint32_t)meta_pair(slot)[c].src : NONE;
                }
                ft = fc = 0;
                ++fli;
                fit += gridDim.x;
            }
            if (ft < sp.ntile) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (fsrc[i] != NONE)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                         dst0 + fst * SC_XST + 4 * i * SC_XROW),
                                     "l"(fme + ((int64_t)fsrc[i] * box_units + fc * SC_KC))
                                     : "memory");
                if (++fc == sp.t[ft].nchunk) {
                    fc = 0;
                    ++ft;
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            fst = fst + 1 == SC_XD ? 0 : fst + 1;
            return true;
        };
        const uint32_t sel_lo = b ? 0x5476u : 0x3210u, sel_hi = b ? 0x1032u : 0x7654u, sgn = b ? 0u : 0x80000000u;
        uint32_t li = 0, g = 0, xph = 0;       // items, chunks of this CTA so far
        int xs = 0, cst = 0;                   // tensor-memory slot and stage of chunk g
        for (int u = 0; u < SC_XD - 1 && !failed; ++u) failed = !fetch();
        for (int64_t it = blockIdx.x; it < nwork && !failed; it += gridDim.x, ++li) {
            const int slot = li & 1;
            const M2LWork w = work[it];
            const bool valid = cc < w.npair;
            const uint32_t gr = tc::smem_u32(meta_ph(slot)) + (valid ? cc : 0) * sp.ph_bytes;
            for (int t = 0; t < sp.ntile && !failed; ++t) {
                const int odd = sp.t[t].sec, nch = sp.t[t].nchunk;
                for (int ch = 0; ch < nch; ++ch) {
                    // wait_group covers a lane's own copies only, and the rows read below came with other
                    // lanes'; the stage that fetch fills was read by the whole warp in the last chunk
                    asm volatile("cp.async.wait_group %0;" ::"n"(SC_XD - 2) : "memory");
                    __syncwarp();
                    if (!fetch()) {
                        failed = true;
                        break;
                    }
                    const bool okw = g < (uint32_t)SX || tc::mbar_wait(&xempty[xs], xph ^ 1, SC_POLLS);
                    if (__any_sync(0xffffffffu, !okw)) {
                        failed = true;
                        break;
                    }
                    tc::fence_after();
                    uint32_t ew[KQ], own[KQ][SC_NPC], oth[KQ][SC_NPC];
                    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(ew[0]), "=r"(ew[1]), "=r"(ew[2]), "=r"(ew[3])
                                 : "r"(ent0 + 4 * SC_KC * ch));
                    const uint32_t xr = ring + cst * SC_XST + (lane >> 1) * SC_XROW + 64 * b;
#pragma unroll
                    for (int h = 0; h < KQ; ++h) {
                        float4 v;   // the input's two coefficients
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                                     : "r"(xr + 16 * h));
                        const cf G = lds_c(gr + 8 * ((ew[h] >> 20) & 63));
                        // W entries subtract conj(G) b in the even sector, C entries add conj(G) c
                        const float s = (int)((ew[h] >> 26) & 1) == odd ? -1.f : 1.f;
                        const float cx = s * v.z, cy = s * v.w;
                        cf y{fmaf(G.x, v.x + cx, G.y * (cy - v.y)), fmaf(G.x, v.y + cy, G.y * (v.x - cx))};
                        if (!valid) y = cf{0.f, 0.f};
                        split_bf16(y.x, y.y, own[h]);
                    }
#pragma unroll
                    for (int h = 0; h < KQ; ++h)
#pragma unroll
                        for (int pc = 0; pc < SC_NPC; ++pc) oth[h][pc] = __shfl_xor_sync(0xffffffffu, own[h][pc], 1);
                    // the K-step's eight inputs in this lane's row: (Re, -Im) = negated high
                    // half, (Im, Re) = swapped halves; columns piece-major, even K in the low
                    // half.  One byte permutation picks own or partner's word and swaps
                    uint32_t rw[8 * SC_NPC];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
#pragma unroll
                        for (int pc = 0; pc < SC_NPC; ++pc)
                            rw[i + 8 * pc] =
                                __byte_perm(own[i & (KQ - 1)][pc], oth[i & (KQ - 1)][pc], i < KQ ? sel_lo : sel_hi) ^ sgn;
                    const uint32_t ta = lane_base + xb + SC_XW * xs + 8 * SC_NPC * pg;
                    static_assert(SC_KS == 2 && SC_NPC == 3, "two K-steps of 24 columns per chunk");
                    if (pg == 0) {
                        tc::tmem_st16(ta, rw);
                        tc::tmem_st8(ta + 16, rw + 16);
                    } else {
                        tc::tmem_st8(ta, rw);
                        tc::tmem_st16(ta + 8, rw + 8);
                    }
                    tc::tmem_st_wait();
                    tc::fence_before();
                    tc::mbar_arrive(&xfull[xs]);
                    ++g;
                    cst = cst + 1 == SC_XD ? 0 : cst + 1;
                    if (++xs == SX) {
                        xs = 0;
                        xph ^= 1;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&metaempty[slot]);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    } else if (warp < SC_WTMA) {
        // ------------------------------------------------ epilogue
        const int ea = tid - SC_PT, ew = ea >> 5;     // epilogue warp 0 .. SC_EW-1
        const int q4 = warp & 3, part = ea / 128;     // lane quadrant, first slab
        const uint32_t lane_base = tbase + ((uint32_t)(32 * q4) << 16);
        constexpr int RB = RJ == 4 ? 2 : 3;
        constexpr int EWS = RJ <= 4 ? SC_EW : SC_EW / 2;   // sec_plan's ews
        float2 *stage = (float2 *)(smraw + sp.o_stage + ew * sp.stage_bytes);
        const int yodd = sp.t[sp.ntile / 2].y0;       // scratch row of the odd sector
        uint32_t li = 0, tc_n = 0;
        for (int64_t it = blockIdx.x; it < nwork && !failed; it += gridDim.x, ++li) {
            const M2LWork w = work[it];
            const int slot = li & 1;
            // the previous item's scatter has read the scratch, and its reductions the staging rows
            bool ok = li == 0 || tc::mbar_wait(yfree, (li - 1) & 1, SC_POLLS);
            if (__any_sync(0xffffffffu, !ok)) {
                failed = true;
                break;
            }
            for (int t = 0; t < sp.ntile; ++t, ++tc_n) {
                ok = tc::mbar_wait(accfull, tc_n & 1, SC_POLLS);
                if (__any_sync(0xffffffffu, !ok)) {
                    failed = true;
                    break;
                }
                tc::fence_after();
                const int N = sp.t[t].N;
                // a 16-row slab of the warp's 16 pairs goes through its tile, so that a store
                // instruction writes four whole 128-byte lines (lane: pair 4h + lane / 8, rows
                // 2 (lane % 8), + 1) and the scatter reads whole lines
                float *T = (float *)(smraw + sp.o_stage + ew * SC_TILE);
                const int lr = 2 * (lane & 7), lc = lane >> 3;
                float4 *Yt = (float4 *)(Y + (size_t)(16 * q4) * sp.yrows + sp.t[t].y0);
                for (int c0 = 16 * part; c0 < N; c0 += SC_ET / 8) {   // N is a multiple of 16
                    uint32_t va[16], vb[16];
                    tc::tmem_ld16(lane_base + sp.nmax + c0, va);
                    if (sp.nacc == 3) {
                        tc::tmem_ld16(lane_base + 2 * sp.nmax + c0, vb);
                        tc::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            va[i] = __float_as_uint(__uint_as_float(va[i]) + __uint_as_float(vb[i]));
                    }
                    tc::tmem_ld16(lane_base + c0, vb);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) T[i * SC_DS + lane] = __uint_as_float(va[i]) + __uint_as_float(vb[i]);
                    __syncwarp();
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int cl = 4 * h + lc;
                        const float2 x0 = *(const float2 *)(T + lr * SC_DS + 2 * cl);
                        const float2 x1 = *(const float2 *)(T + (lr + 1) * SC_DS + 2 * cl);
                        Yt[((size_t)cl * sp.yrows + c0 + lr) >> 1] = make_float4(x0.x, x0.y, x1.x, x1.y);
                    }
                    __syncwarp();
                }
                tc::fence_before();
                tc::mbar_arrive(accempty);
            }
            if (failed) break;
            tc::mbar_arrive(ydone);
            ok = tc::mbar_wait(ydone, li & 1, SC_POLLS) && tc::mbar_wait(&metafull[slot], (li >> 1) & 1, SC_POLLS);
            if (__any_sync(0xffffffffu, !ok)) {
                failed = true;
                break;
            }
            cf *const le = prob(w).le;
            const uint32_t gr = tc::smem_u32(meta_ph(slot));
            for (int c = ew; ew < EWS && c < w.npair; c += EWS) {
                // RB rows per lane and step
                auto load = [&](int i0, float2 (&ye)[RB], float2 (&yo)[RB]) {
#pragma unroll
                    for (int i = 0; i < RB; ++i) {
                        const int r = min(lane + 32 * (i0 + i), sp.D0 - 1), ro = yodd + min(r, sp.D1 - 1);
                        ye[i] = Y[(size_t)c * sp.yrows + r];
                        yo[i] = Y[(size_t)c * sp.yrows + ro];
                    }
                };
                float2 ye[RB], yo[RB];
                load(0, ye, yo);
                cf *dst = le + meta_pair(slot)[c].tgt * 3 * P;
                // the reduction wants 16-byte alignment on both sides: an odd first element and the
                // last one left over are added by an atomic
                const int head = (int)(((uintptr_t)dst >> 3) & 1), body = (3 * P - head) & ~1;
                float2 *sg = stage + head;
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
#pragma unroll 1
                for (int i0 = 0; i0 < RJ; i0 += RB) {
                    if (i0 > 0) load(i0, ye, yo);
                    // no branch between the rows: their entry words and phases are fetched together
                    uint32_t we[RB];
                    cf G[RB];
#pragma unroll
                    for (int i = 0; i < RB; ++i) we[i] = ent[min(lane + 32 * (i0 + i), sp.D0 - 1)];
#pragma unroll
                    for (int i = 0; i < RB; ++i) G[i] = lds_c(gr + c * sp.ph_bytes + 8 * ((we[i] >> 20) & 63));
#pragma unroll
                    for (int i = 0; i < RB; ++i) {
                        const int r = lane + 32 * (i0 + i);
                        const float ko = r < sp.D1 ? 1.f : 0.f, kd = (we[i] >> 26 & 1) ? 1.f : -1.f;
                        const float2 o{ko * yo[i].x, ko * yo[i].y};
                        const float2 s{ye[i].x + o.x, ye[i].y + o.y};
                        const float2 d{kd * (ye[i].x - o.x), kd * (ye[i].y - o.y)};
                        const cf g = G[i];
                        if (r < sp.D0) sg[we[i] & 1023] = float2{fmaf(g.x, s.x, g.y * s.y), fmaf(g.x, s.y, -g.y * s.x)};
                        if (r < sp.D0 && !(we[i] >> 27 & 1))
                            sg[(we[i] >> 10) & 1023] = float2{fmaf(g.x, d.x, -g.y * d.y), fmaf(g.x, d.y, g.y * d.x)};
                    }
                }
                tc::fence_smem_async();
                __syncwarp();
                if (lane == 0) {
                    asm volatile(
                        "cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;\n\t"
                        "cp.async.bulk.commit_group;" ::"l"(dst + head),
                        "r"(tc::smem_u32(sg + head)), "r"((uint32_t)body * 8)
                        : "memory");
                } else if (lane == 1 && head) {
                    atomicAdd((float2 *)dst, sg[0]);
                } else if (lane == 2 && head + body < 3 * P) {
                    atomicAdd((float2 *)dst + head + body, sg[head + body]);
                }
            }
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
            tc::mbar_arrive(yfree);
            if (lane == 0) tc::mbar_arrive(&metaempty[slot]);
        }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // every reduction has landed
    }
    if (failed) atomicOr(status, 4);
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, 512);
}

// three-piece bf16 split of a double
__device__ inline void split3(double v, uint16_t (&o)[SC_NPC])
{
    double r = v;
#pragma unroll
    for (int j = 0; j < SC_NPC; ++j) {
        const __nv_bfloat16 h = __float2bfloat16_rn((float)r);
        o[j] = *(const uint16_t *)&h;
        r -= (double)__bfloat162float(h);
    }
}

// image of the sector matrices: per geometry and tile the K-steps of 8 complex inputs (zero
// beyond the sector's dimension), each SC_NPC planes of N rows x 16 real K in K-major core
// matrices of 8 rows x 8 values (the two K halves 128 B apart, 8-row groups 256 B apart)
__global__ void __launch_bounds__(256) k_sec_image(const __grid_constant__ SecPlan sp, const GeomDev *geoms,
                                                   const CompDev *comps, const cd *tab64, unsigned char *img)
{
    __shared__ double ps[SC_PMAX + 1], pt[SC_PMAX + 1];
    const SecTile &t = sp.t[blockIdx.y];
    const int64_t gi = blockIdx.z;
    const GeomDev &g = geoms[gi];
    if (threadIdx.x <= sp.p) {
        double a = 1.0, b = 1.0;
        for (int i = 0; i < (int)threadIdx.x; ++i) {
            a *= g.scale_s;
            b *= g.scale_t;
        }
        ps[threadIdx.x] = a;
        pt[threadIdx.x] = b;
    }
    __syncthreads();
    const int D = t.sec ? sp.D1 : sp.D0, N = t.N;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= t.nchunk * SC_KS * N * 8) return;
    const int c = e / (N * 8), rem = e % (N * 8), rl = rem >> 3, i = rem & 7;
    const int r = t.row0 + rl, k = 8 * c + i;
    cd v{0.0, 0.0};
    if (r < D && k < D) {
        const CompDev cp = comps[g.comp];
        const SecEntry er = sec_entry(sp.p, r), ek = sec_entry(sp.p, k);
        v = sec_scaled(er, ek, (cp.s < 0) != (cp.has_src_refl != 0), (cp.s < 0) != (cp.has_tgt_refl != 0), pt, ps,
                       sec_value(sp.p, t.sec, er, ek, tab64 + gi * NTAB * (int64_t)sp.P * sp.P));
    }
    uint16_t re[SC_NPC], im[SC_NPC];
    split3(v.x, re);
    split3(v.y, im);
    unsigned char *sub = img + (size_t)gi * sp.img_bytes + t.img + (size_t)c * (SC_NPC * N * 32);
    const int off = (rl >> 3) * 256 + (i >> 2) * 128 + (rl & 7) * 16 + (i & 3) * 4;
#pragma unroll
    for (int pc = 0; pc < SC_NPC; ++pc)
        *(uint32_t *)(sub + (size_t)pc * N * 32 + off) = (uint32_t)re[pc] | ((uint32_t)im[pc] << 16);
}

__host__ __device__ inline int phase_row(int p) { return 2 * ((p + 1) | 1); }

// phases of every pair: powers in FP64, rounded once to FP32
__global__ void k_pair_phases(int p, int64_t npair, const M2LPair *pairs, cf *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= npair) return;
    cf *row = out + i * phase_row(p) + (p + 1);
    const cd b = mul_i(cd{pairs[i].cphi, pairs[i].sphi});
    cd e{1.0, 0.0};
    for (int d = 0; d <= p + 1; ++d) {
        if (d <= p) row[d] = cf{(float)e.x, (float)e.y};
        row[-d] = cf{(float)e.x, (float)-e.y};
        e = e * b;
    }
}

// packed multipole expansions: per box the inputs of the sector vectors, entry j's two
// coefficients side by side ([nchunk0 * 16][2], zero beyond D0); clears the box's local
// expansion on the way (the M2L adds into it)
__global__ void __launch_bounds__(128) k_sec_pack(int p, int n16, int D0, const cf *me, float4 *pk, cf *le)
{
    const int P3 = 3 * (p + 1) * (p + 1);
    const int64_t box = blockIdx.x;
    const cf *m = me + box * P3;
    for (int j = threadIdx.x; j < n16; j += blockDim.x) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j < D0) {
            const uint32_t w = sec_word(p, j);
            const cf a = m[w & 1023], b = m[(w >> 10) & 1023];
            v = make_float4(a.x, a.y, b.x, b.y);
        }
        pk[box * n16 + j] = v;
    }
    for (int j = threadIdx.x; j < P3; j += blockDim.x) le[box * P3 + j] = cf{0.f, 0.f};
}

template <int RJ>
cudaError_t launch_rj(const SecPlan &sp, int64_t nwork, const M2LWork *work, const TcProb &one, const TcProb *probs,
                      float *yscr, int ncta, int *status, cudaStream_t st)
{
    // each CTA takes all 512 tensor-memory columns: ask for more than half of an SM's
    // shared memory so that no two CTAs are resident on one SM
    const size_t smem = std::max<size_t>(sp.smem, 116 * 1024);
    k_m2l_sec<RJ><<<(unsigned)std::min<int64_t>(nwork, ncta), SC_THREADS, smem, st>>>(sp, nwork, work, one, probs, yscr,
                                                                                     status);
    return cudaGetLastError();
}

}  // namespace

bool m2l_sec_supported(int p) { return p >= 1 && p <= SC_PMAX; }
int m2l_sec_pairs() { return SC_BN; }
// d = -(p+1)..p; rows of an odd number of 16-byte units, so that the phases of neighbouring
// pairs lie in different shared-memory banks
int m2l_sec_phases(int p) { return phase_row(p); }
size_t m2l_sec_image_bytes(int p, int64_t ngeom) { return (size_t)ngeom * sec_plan(p).img_bytes; }
size_t m2l_sec_scratch_floats(int p, int ncta) { return (size_t)ncta * 128 * sec_plan(p).yrows; }

void launch_sec_image(int p, int64_t ng, const GeomDev *geoms, const CompDev *comps, const cd *tab64, void *img,
                      cudaStream_t st)
{
    const SecPlan sp = sec_plan(p);
    int most = 0;
    for (int t = 0; t < sp.ntile; ++t) most = std::max(most, sp.t[t].nchunk * SC_KS * sp.t[t].N * 8);
    // grid.z is limited to 65535
    for (int64_t g0 = 0; g0 < ng; g0 += 32768) {
        const int64_t nb = std::min<int64_t>(32768, ng - g0);
        k_sec_image<<<dim3((most + 255) / 256, sp.ntile, (unsigned)nb), 256, 0, st>>>(
            sp, geoms + g0, comps, tab64 + g0 * NTAB * (int64_t)sp.P * sp.P,
            (unsigned char *)img + (size_t)g0 * sp.img_bytes);
    }
}

void launch_pair_phases(int p, int64_t npair, const M2LPair *pairs, cf *out, cudaStream_t st)
{
    if (npair > 0) k_pair_phases<<<(unsigned)((npair + 255) / 256), 256, 0, st>>>(p, npair, pairs, out);
}

size_t m2l_sec_packed_bytes(int p, int64_t nbox) { return (size_t)nbox * sec_plan(p).nchunk0 * SC_KC * 16; }

void launch_sec_pack(int p, int64_t nbox, const cf *me, void *packed, cf *le, cudaStream_t st)
{
    const SecPlan sp = sec_plan(p);
    if (nbox > 0)
        k_sec_pack<<<(unsigned)nbox, 128, 0, st>>>(p, sp.nchunk0 * SC_KC, sp.D0, me, (float4 *)packed, le);
}

cudaError_t launch_m2l_sec(int p, int64_t nwork, const M2LWork *work, const TcProb &one, const TcProb *probs,
                           float *yscr, int ncta, int *status, cudaStream_t st)
{
    if (nwork <= 0) return cudaSuccess;
    if (!m2l_sec_supported(p) || ncta < 1) return cudaErrorInvalidValue;
    const SecPlan sp = sec_plan(p);
    switch ((sp.D0 + 31) / 32) {
    case 1:
    case 2:
    case 3: return launch_rj<3>(sp, nwork, work, one, probs, yscr, ncta, status, st);   // p <= 6
    case 4: return launch_rj<4>(sp, nwork, work, one, probs, yscr, ncta, status, st);   // p <= 8
    case 5:
    case 6: return launch_rj<6>(sp, nwork, work, one, probs, yscr, ncta, status, st);   // p <= 10
    default: return launch_rj<9>(sp, nwork, work, one, probs, yscr, ncta, status, st);  // p <= 12
    }
}

cudaError_t configure_m2l_sec()
{
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_m2l_sec<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, SC_SMEM_MAX))) return e;
    if ((e = cudaFuncSetAttribute(k_m2l_sec<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, SC_SMEM_MAX))) return e;
    if ((e = cudaFuncSetAttribute(k_m2l_sec<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, SC_SMEM_MAX))) return e;
    return cudaFuncSetAttribute(k_m2l_sec<9>, cudaFuncAttributeMaxDynamicSharedMemorySize, SC_SMEM_MAX);
}

}  // namespace lmf
