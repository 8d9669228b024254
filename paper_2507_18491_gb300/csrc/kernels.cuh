// Device-side records and kernel launchers.
#pragma once
#include <cuda_runtime.h>

#include <vector>

#include "gauss.cuh"
#include "internal.h"

#define LMF_PMAX 20

namespace lmf {

// k_rho nodes of one Sommerfeld integral (Section 3.5):
//   [0, n1)                Gamma_1 from 0 to a (Gauss-Legendre 16 per panel)
//   [n1, n1+nmid)          real segment [a, x1] with J_d (Gauss-Legendre 8)
//   then, when nray > 0, the rays Gamma_2+ and Gamma_2- from x1,
//   k = x1 + t (dz +- i rho)/r, t in [0, tend], with H^(1)_d/2 and H^(2)_d/2.
struct QuadPlanDev {
    int n1, nmid, nray, pad;
    double a, kp, x1;   // Gamma_1 end, its shape parameter, end of the real segment
    double cr, sr, tend;// ray direction (dz/r, rho/r) and length
};

struct GeomDev {
    int comp, src_primary;
    double rho, zs, zt;
    double scale_s, scale_t;  // |k| S_level of the source and target layers
    QuadPlanDev plan;
    int64_t node0;      // first node within its tabulation batch
    int64_t stride;     // node count of its batch (factor-array stride)
    int64_t tab_index;  // table slot
    int batch, pad;
};

struct LayerScale {      // |k_l| S_leaf per layer (expansion scaling at the leaves)
    double s[LMF_MAXL + 1];
};

struct TransGroupDev {
    int layer, level;
    double t[3];
};

struct BoxDev {
    int64_t p0, p1;
    double c[3];
    int layer, pad;
};

struct LeafUnit {       // P2M work of one warp: points [i0, i1) (at most 128) of leaf box
    int64_t i0, i1;
    int box, whole;     // whole: the unit covers the leaf (plain stores, else atomics)
};


struct GemmWork {       // M2M / L2L: pairs [pair0, pair0 + npair) of one translation group
    int group, npair;
    int64_t pair0;
};

struct M2LWork {        // one M2L table, or both sector blocks, applied to a chunk of pairs of one geometry
    int geom, t, npair;
    int flags;          // bit 0: odd input degrees change sign, bit 1: odd output degrees
    int64_t pair0;
    int prob, pad;      // problem of a batched launch (TcProb index), else 0
};

// per-problem arrays of a persistent M2L launch (k_m2l_sec): one problem's pairs,
// pair phases and matrix image (one block per geometry), its packed multipole expansions
// and its local expansions
struct TcProb {
    const M2LPair *pairs;
    const cf *ephase;
    const void *img;
    const void *me;
    cf *le;
};

// k_tab.cu
void launch_densities(const MediumDev &M, int l, int lp, int64_t n, const cd *kr, cd *out,
                      cudaStream_t st);
int64_t tab_integrals(int p);   // complex numbers of scratch per geometry, beside the node factors
void launch_tab_batch(const GeomDev *dG, int g0, int nb, int qmax, const MediumDev &M,
                      const CompDev *dcomps, int p, const cd *dGten, const int *dcgidx,
                      cd *scratch, int64_t stride, cd *tab, int *dflag, cudaStream_t st);

// translation matrices of ng groups on the device: the Gaunt coefficients (G: P^2 (p + 1)
// doubles) from the nodes of gaunt_nodes, then M2M (up) and L2L (dn), [group][P][P]; fac
// from trans_factors
void launch_trans_build(int p, int nq, const dd *w, const dd *Pq, double *G, int64_t ng, const dd *fac, cd *up, cd *dn,
                        cudaStream_t st);
template <typename T>
void launch_trans_copy(int p, int64_t ng, bool tr, const cd *in, cx<T> *out, cudaStream_t st);

// k_fmm.cu
cudaError_t configure_fmm_kernels();
cudaError_t configure_tab_kernels();
// J / Phi: caller's [N][3] complex128 (LMFMM_C128) or complex64 (LMFMM_C64)
void launch_gather_in(int64_t N, const int64_t *perm, const void *J, int dtype, cd *qh, bool conj_in,
                      cudaStream_t st);
void launch_scatter_out(int64_t N, const int64_t *perm, const cd *phih, void *Phi, int dtype, bool conj_out,
                        cudaStream_t st);
// P2M of the helical charges qh into me at the leaves; with l2p_basis the
// coefficients are taken against L2P's functions instead (transpose of L2P)
template <typename T>
void launch_p2m(int p, int64_t nleaf, const int64_t *leaves, const BoxDev *boxes,
                const double *xyz, const cd *qh, const MediumDev &M, const LayerScale &ls,
                cx<T> *me, cudaStream_t st, bool l2p_basis = false);
// L2P of le at the leaf points into phih; with p2m_basis the expansions are
// evaluated with P2M's functions (transpose of P2M); accumulate adds into phih
template <typename T>
void launch_l2p(int p, int64_t nleaf, const int64_t *leaves, const BoxDev *boxes,
                const double *xyz, const cx<T> *le, const MediumDev &M, const LayerScale &ls,
                cd *phih, cudaStream_t st, bool p2m_basis = false, bool accumulate = false);

// k_leaf.cu: P2M and L2P of the mixed form for p <= 15 (FP32 expansions), one thread per
// sorted point (pt_box: its leaf box): ph (cd [N][3]) = the expansions le (cf
// [box][3][P]) evaluated at the points (added with accumulate).  conj_basis /
// scale select P2M's functions (conj Y, 4 pi: the transpose of P2M) or L2P's (Y, 1).
bool leaf_fast_supported(int p);
cudaError_t configure_leaf_fast();
void launch_l2p_fast(int p, int64_t N, const int *pt_box, const BoxDev *boxes, const double *xyz, const cf *le,
                     const MediumDev &M, const LayerScale &ls, cd *ph, bool conj_basis, double scale, bool accumulate,
                     cudaStream_t st);
// P2M of the mixed form for p <= 15: one warp per unit, me (cf [box][3][P], zeroed
// beforehand) += the coefficients of the helical charges qh (cd, sorted)
// (many: the kernel for units of many points)
void launch_p2m_fast(int p, int64_t nunit, bool many, const LeafUnit *units, const BoxDev *boxes, const double *xyz,
                     const cd *qh, const MediumDev &M, const LayerScale &ls, cf *me, bool conj_basis, double scale,
                     cudaStream_t st);

// k_trans.cu
cudaError_t configure_trans_kernels();
template <typename T> int gemm_cols();
template <typename T>
void launch_group_gemm_t(int p, int64_t nwork, const GemmWork *work, const cx<T> *mats,
                         const int64_t *src, const int64_t *dst, const cx<T> *in, cx<T> *out,
                         bool atomic, cudaStream_t st);
// M2M / L2L of the FP64 form: matsT holds the transposed matrices
void launch_trans_fp64(int p, int64_t nwork, const GemmWork *work, const cd *matsT, const int64_t *src,
                       const int64_t *dst, const cd *in, cd *out, cudaStream_t st);
template <typename T>
void launch_m2l_t(int p, int64_t nwork, const M2LWork *work, const GeomDev *geoms,
                  const CompDev *comps, const M2LPair *pairs, const cx<T> *tab, const cx<T> *me,
                  cx<T> *le, cudaStream_t st);
// transpose of the SIMT M2L: me_bar[src] += (M2L)^T le_bar[tgt], same work items
template <typename T>
void launch_m2l_tr(int p, int64_t nwork, const M2LWork *work, const GeomDev *geoms,
                   const CompDev *comps, const M2LPair *pairs, const cx<T> *tab, const cx<T> *le_bar,
                   cx<T> *me_bar, cudaStream_t st);
// k_m2l_tc.cu: mixed-form M2L on tcgen05 tensor cores (3xTF32), p <= 15;
// status gets bit 4 if a tensor-core wait gave up
bool m2l_tc_supported(int p);
int m2l_tc_cols();
// M2L work items of a context whose host structures are built, cut to at most bn
// helical columns, in the order the matvec launches them (api.cu)
int64_t plan_work_items(const lmfmm_ctx *ctx, int bn, std::vector<M2LWork> &mw);
// ... and those of the sector kernels, runs of at most `pairs` pairs of a geometry
void plan_sector_items(const lmfmm_ctx *ctx, int pairs, std::vector<M2LWork> &mw);
cudaError_t configure_m2l_tc();
cudaError_t launch_m2l_tc(int p, int64_t nwork, const M2LWork *work, const GeomDev *geoms,
                          const CompDev *comps, const M2LPair *pairs, const cf *tab, const cf *me,
                          cf *le, int *status, cudaStream_t st);
// k_m2l_sec.cu: persistent tensor-core M2L of the mixed form (p <= 12) on the mirror
// sectors of sector.cuh.  Items M2LWork{geom, npair <= 64, pair0, prob}; img is the
// image of the sector matrices in three bf16 pieces (launch_sec_image from the FP64
// tables); ephase holds G[d] = i^d e^{i d phi} of every pair, d = -(p+1)..p, in rows of
// m2l_sec_phases(p) entries (FP32 from FP64); yscr holds m2l_sec_scratch_floats(p, ncta)
// floats, ncta = the most CTAs that the launch may have (at most the SM count: one per SM)
bool m2l_sec_supported(int p);
int m2l_sec_pairs();             // pairs of a full work item
int m2l_sec_phases(int p);
size_t m2l_sec_image_bytes(int p, int64_t ngeom);
size_t m2l_sec_scratch_floats(int p, int ncta);
cudaError_t configure_m2l_sec();
void launch_sec_image(int p, int64_t ng, const GeomDev *geoms, const CompDev *comps, const cd *tab64, void *img,
                      cudaStream_t st);
void launch_pair_phases(int p, int64_t npair, const M2LPair *pairs, cf *out, cudaStream_t st);
// packs the multipole expansions me into what the kernel reads (TcProb::me,
// m2l_sec_packed_bytes) and clears the local expansions le
size_t m2l_sec_packed_bytes(int p, int64_t nbox);
void launch_sec_pack(int p, int64_t nbox, const cf *me, void *packed, cf *le, cudaStream_t st);
// probs: the problems of a batched launch (device array), or null with one problem in `one`
cudaError_t launch_m2l_sec(int p, int64_t nwork, const M2LWork *work, const TcProb &one, const TcProb *probs,
                           float *yscr, int ncta, int *status, cudaStream_t st);
// k_m2l_oz.cu: M2L of the FP64 form on the tensor cores, operands as eight base-256 digits.
// out is cleared, then out[tgt] += M in[src] over the items' pairs (transposed: in over the
// targets, out over the sources); img from launch_oz_images (m2l_oz_image_bytes), packed and
// scratch of the sizes below
bool m2l_oz_supported(int p);
int m2l_oz_pairs();
size_t m2l_oz_image_bytes(int p, int64_t ngeom);   // with the exponents of rows and degrees
size_t m2l_oz_packed_bytes(int p, int64_t nbox);
size_t m2l_oz_scratch_bytes(int p, int ncta);
cudaError_t configure_m2l_oz();
// the images of the blocks and of their transposes
void launch_oz_images(int p, int64_t ng, const GeomDev *geoms, const CompDev *comps, const cd *tab64, void *img, void *imgT,
                      cudaStream_t st);
cudaError_t launch_m2l_oz(int p, bool transposed, int64_t ngeom, int64_t nwork, const M2LWork *work, const M2LPair *pairs,
                          const void *img, int64_t nbox, const cd *in, cd *out, void *packed, void *scratch, int ncta,
                          int *status, cudaStream_t st);
// M2M or L2L on a persistent tensor-core kernel (k_m2l_tc.cu, p <= 12): items M2LWork{geom = translation group, t = 0,
// npair, pair0} over pairs (tsrc[q], tdst[q]), 3 helical columns each; img holds
// one tiled matrix per group (launch_tile_matrices, tc2_matrix_bytes(p) each)
cudaError_t launch_trans_tc2(int p, int64_t nwork, const M2LWork *work, const int64_t *tsrc,
                             const int64_t *tdst, const void *img, const cf *in, cf *out, float *yscr, int ncta,
                             int *status, cudaStream_t st);
bool trans_tc2_supported(int p);
size_t trans_tc2_scratch_floats(int p, int ncta);
size_t tc2_matrix_bytes(int p);
void launch_tile_matrices(int p, int64_t ng, const cd *M, void *img, cudaStream_t st);   // [ng][P][P], row = output index
template <typename T>
void launch_scale_tables(int p, int64_t g0, int64_t ng, const GeomDev *geoms, const cd *tab64,
                         cx<T> *tab, cudaStream_t st);
// five Sommerfeld integrals per point pair of every near pair; a pair whose
// k_rho rule needs more than node_cap nodes sets bit 2 of *dflag (clamped rule)
void launch_s2t_pre(int64_t nnear, const NearPair *near, const BoxDev *boxes, const double *xyz,
                    const MediumDev &M, const CompDev *comps, double a, int node_cap, cd *coef,
                    int *dflag, cudaStream_t st);
// matvec near field: 8 combined coefficients per point pair ([j][8][i] per near pair)
void launch_s2t_combine(int64_t nnear, const NearPair *near, const BoxDev *boxes, const double *xyz,
                        const cd *coef5, cd *coef8, cudaStream_t st);
// one target row of the matvec near field: target ii of near pair `pair`
// against the pair's sources [s0, s0 + S2T_SRC); rows are ordered by pair,
// then source block, then ii
constexpr int S2T_SRC = 64;
struct S2TRow {
    int64_t pair;
    int ii, s0;
};
void launch_s2t_apply8(int64_t nrow, const S2TRow *rows, const NearPair *near, const BoxDev *boxes,
                       const cd *coef8, const cd *qh, cd *phih, cudaStream_t st);
// transposed near field: one row per (near pair, source jj), all targets
struct S2TRowT {
    int64_t pair;
    int jj, pad;
};
void launch_s2t_apply8_tr(int64_t nrow, const S2TRowT *rows, const NearPair *near, const BoxDev *boxes,
                          const cd *coef8, const cd *phb, cd *qhb, cudaStream_t st);
// free-space near field: per leaf box b the runs [roff[b], roff[b + 1]) of sorted points
// near it, one warp per sorted point (pt_box: its leaf).  Forward: points are targets, out =
// ph; transposed: points are sources, out = qh_bar
struct FreeRun {
    int64_t p0;
    int n, pad;
};
void launch_p2p_free(int64_t N, const int *pt_box, const int *roff, const FreeRun *runs, const BoxDev *boxes,
                     const double *xyz, const MediumDev &M, const cd *in, cd *out, bool transposed, cudaStream_t st);
// transposes of the helical maps: ph_bar = S^T y (caller order -> sorted),
// out = G^T qh_bar (sorted -> caller order), optional conjugation of y / out
void launch_gather_tr(int64_t N, const int64_t *perm, const void *y, int dtype, cd *phb, bool conj_in,
                      cudaStream_t st);
void launch_scatter_tr(int64_t N, const int64_t *perm, const cd *qhb, void *out, int dtype, bool conj_out,
                       cudaStream_t st);
void launch_s2t_apply(int64_t nnear, const NearPair *near, const BoxDev *boxes,
                      const double *xyz, const cd *coef, const cd *qh, cd *phih,
                      cudaStream_t st);

// k_grad.cu: position gradient of the FP64 form (see the file's header).
// grad (caller order, [N][3] real) is accumulated: zero it first.
void launch_grad_leaf(int p, int64_t N, int64_t nleaf, const int64_t *leaves, const BoxDev *boxes, const double *xyz,
                      const int64_t *perm, const cd *le, const cd *meb, const cd *qh, const cd *nu, const MediumDev &M,
                      const LayerScale &ls, double *grad, cudaStream_t st);
// 20 derivative integrals per near point pair (coef: [pair coef0 + e][20])
void launch_s2t_pre_grad(int64_t nnear, const NearPair *near, const BoxDev *boxes, const double *xyz,
                         const MediumDev &M, const CompDev *comps, double a, int node_cap, cd *coef, cudaStream_t st);
void launch_grad_near(int64_t nnear, const NearPair *near, const BoxDev *boxes, const double *xyz, const int64_t *perm,
                      const CompDev *comps, const cd *coefg, const cd *qh, const cd *nu, double *grad, cudaStream_t st);

}  // namespace lmf
