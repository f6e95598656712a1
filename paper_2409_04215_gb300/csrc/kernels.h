// Internal host-side entry points of the libmfs kernels (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "common.cuh"

namespace mfs {

// ---- pair sums (pair_kernel.cu) ----
struct PairVariant {
    int D, nrhs, T, NT, tile_targets;
    int packed;  // 1: f32x2 Stokes policy with duplicated source records
    int grad;    // not a pair sum: 1 the adjoint's centre-gradient kernel, 2 pressure and traction (D = 4 outputs)
    int comp;    // 1: compensated double-FP32 arithmetic (precision = 3), records from pack_sources_comp
    const char *name;  // policy and template arguments, e.g. "PackedStokes<1,3,128>"
};
const PairVariant *pair_variants(int *count);
int pair_occupancy(int variant);  // resident CTAs per SM
int pair_record_floats(int D, int nrhs, int packed);
cudaError_t pair_launch(int variant, const PairGeom &geo, const PairWork &work, int *err, cudaStream_t st);
cudaError_t pair_epilogue(int D, int nrhs, const PairWork &work, const double *base, double beta, double scale,
                          double *out, int ntargets, cudaStream_t st);
cudaError_t pack_sources(int D, int nrhs, int packed, const float4 *src_pos, const int *src_pt_of_rec,
                         const double *strength, int nsrc, int nrec, float *records, cudaStream_t st);
// Records of several point sets in one launch: set q's n[q] points at pos[q] with strengths
// strength[q] [nrhs][n[q]][D] to rec[q].
struct PackSets {
    static constexpr int MAX = 8;
    int sets = 0;
    int n[MAX] = {};
    const float4 *pos[MAX] = {};
    const double *strength[MAX] = {};
    float *rec[MAX] = {};
    void add(int count, const float4 *p, const double *s, float *r) {
        n[sets] = count;
        pos[sets] = p;
        strength[sets] = s;
        rec[sets++] = r;
    }
};
cudaError_t pack_sets(int D, int nrhs, int packed, const PackSets &a, cudaStream_t st);
// Records of the compensated kernels from FP64 body-local positions [nsrc][3] and strengths.
cudaError_t pack_sources_comp(int D, int nrhs, const double *src_local64, const int *src_pt_of_rec,
                              const double *strength, int nsrc, int nrec, float *records, cudaStream_t st);

// FP64 sums (precision = 1), one thread per target and source chunk: raw sums (no 1/(4 pi) factor) in
// `chunks` partials [chunks][nrhs][ntargets][D], to be added in chunk order (fp64_pair_chunks gives the
// count for targets whose smallest suspension has min_sources sources).
int fp64_pair_chunks(int ntargets, int min_sources, int sm_count);
cudaError_t pair_sum_fp64(int D, int nrhs, int chunks, const double *tgt_local, const int *tgt_body, int ntargets,
                          const double *src_local4, int nsrc, const int *susp_src_begin, const int *susp_src_end,
                          const int *body_src_off, const double *centres, const double *strength, int include_self,
                          double *out_raw, cudaStream_t st);
// The adjoint's pair gradient in FP64, per target: sum over the other bodies' sources of
// grad_r (tw^T G(r) strength), raw (no 1/(8 pi mu)); tw [nrhs][ntargets][3], out [chunks][ntargets][3];
// the other arguments as pair_sum_fp64.
cudaError_t grad_pair_fp64(int nrhs, int chunks, const double *tgt_local, const int *tgt_body, int ntargets,
                           const double *tw, const double *src_local4, int nsrc, const int *susp_src_begin,
                           const int *susp_src_end, const int *body_src_off, const double *centres,
                           const double *strength, double *out, cudaStream_t st);

// ---- preconditioner and setup (precond.cu) ----
struct ShapeDev {
    int M, N, dM, dN, r;  // r = dN (rank kept; truncated sigmas give zero columns)
    float *U;             // [dM][r]  left singular vectors (GEMM 1: t = U^T g)
    float *Wp;            // [r][dN]  ((I - L0) V Sigma^+)^T (projected apply, matvec)
    float *Wr;            // [r][dN]  (V Sigma^+)^T (recovery apply)
    double *U64, *Wp64, *Wr64;  // FP64 copies (precision = 1)
    double *UT64 = nullptr, *WpT64 = nullptr, *WrT64 = nullptr;  // their transposes (the FP64 adjoint)
    double sigma1, sigma_min;   // largest / smallest kept singular value
};

// Build S_L = S0 (I - L) + L_r column-major (dM x dN) in FP64 on the device (Sec. 3.3); with bare,
// the self block S0 itself (the Dirichlet problems, Sec. 2.3).
cudaError_t build_SL(int kind, int M, int N, const double *X0, const double *Y0, double mu, const double *G0inv,
                     int bare, double *SL, cudaStream_t st);
// From the SVD (U col-major dM x r, sigma, VT col-major r x dN) write the FP32 / FP64 apply factors;
// with bare, Wp = Wr = (V Sigma^+)^T (no projector).
cudaError_t build_apply_factors(int kind, int M, int N, const double *Ucm, const double *sigma, const double *VTcm,
                                const double *Y0, const double *G0inv, double eps_trunc, int bare, ShapeDev &sd,
                                cudaStream_t st);

// Gather: A[col][i] = (R_k^T gamma_k)[i] as FP32 for the columns (body, rhs) of one shape.
cudaError_t gather_rotate(int D, const double *gamma, int sum_MD, const int *col_body, const int *col_rhs,
                          const int *body_tgt_off, const double *rot, int ncols, int dM, float *A, double *A64,
                          cudaStream_t st);
// Split-K FP32 GEMM with TwoSum-compensated slices; chunk results (FP64, P [S][m][n]) summed in FP64
// into C32 (FP32) or C64 (FP64).  S from gemm_splitk_chunks; P must hold S*m*n doubles.
int gemm_splitk_chunks(int m, int n, int k, int sm_count);
cudaError_t splitk_reduce(int S, size_t mn, const double *P, float *C32, double *C64, cudaStream_t st);

// ---- tensor-core one-body apply (tc_gemm.cu): split-K multi-piece TF32 tcgen05 GEMM ----
struct alignas(64) TcMap {
    unsigned char bytes[128];  // an encoded CUtensorMap
};
struct TcOperands {  // kernel parameter: the factor as FP32 (hi, lo) planes (b[0], b[1]), the columns' TF32 pieces (a)
    TcMap b[3];
    TcMap a[3];
};
// 2-D FP32 tensor [rows][ld], ld % 32 == 0, box 32 x box_rows, 128-byte swizzle; false if not encodable.
bool make_tc_map(TcMap &out, const float *ptr, int rows, int ld, int box_rows);
int tc_gemm_bn(int m, int pieces);
int tc_gemm_chunks(int m, int n, int k, int sm_count, int pieces);
int tc_gemm_sz(int k, int S);
// P[z][m][n] = sum_{k in chunk z} A[m][k] B[n][k] as (hi, lo) float pairs, products of `pieces` (2 or 3)
// TF32 pieces per operand: the factor B given as FP32 (hi, lo) planes (maps b[0], b[1]; cut into pieces
// in shared memory), the columns A as pieces (maps a[0..pieces)); S from tc_gemm_chunks, P holds
// tc_gemm_sz(k, S) * m * n pairs.
cudaError_t tc_gemm(int pieces, const TcMap *b, const TcMap *a, int m, int n, int k, int S, float2 *P, int *err,
                    cudaStream_t st);
// FP64 [rows][cols] -> FP32 (hi, lo) planes dst[0 or 1][cols][ld_dst] (transposed, zero K padding).
cudaError_t split_hilo_transpose(const double *src, int rows, int cols, float *dst, int ld_dst, size_t pstride,
                                 cudaStream_t st);
// pieces src[p][rows][ld_src] (first cols valid) -> dst[p][cols][ld_dst] (transposed, zero padding to
// ld_dst >= rows), p at offsets p * sstride and p * dstride.
cudaError_t transpose_pieces(const float *src, int rows, int cols, int ld_src, size_t sstride, float *dst, int ld_dst,
                             size_t dstride, int pieces, cudaStream_t st);
// sum_z P[z] ([rows][cols], (hi, lo) pairs, double-float sums) -> pieces dst[p][rows][ld_dst].
cudaError_t reduce_pieces(int S, int rows, int cols, const float2 *P, float *dst, int ld_dst, size_t pstride,
                          int pieces, cudaStream_t st);
// gather_rotate with the FP64 values written as pieces dst[p][ncols][ld_dst].
cudaError_t gather_rotate_pieces(int D, const double *gamma, int sum_MD, const int *col_body, const int *col_rhs,
                                 const int *body_tgt_off, const double *rot, int ncols, int dM, float *dst, int ld_dst,
                                 size_t pstride, int pieces, cudaStream_t st);
cudaError_t gemm_splitk(int m, int n, int k, int S, const float *A, const float *B, double *P, float *C32,
                        double *C64, cudaStream_t st, bool trans_b = false);  // trans_b: B stored [n][k]
// FP64 C[m][n] = sum_k A[m][k] B[k][n] (row-major) split over K into S chunks (gemm_rm64_chunks),
// partials P [S][m][n] (unused when S = 1) summed in chunk order into C (deterministic).
int gemm_rm64_chunks(int m, int n, int k, int sm_count);
cudaError_t gemm_rm64_splitk(int m, int n, int k, int S, const double *A, const double *B, double *P, double *C,
                             cudaStream_t st);
// ---- one-body apply for few columns, and the scatter of every apply (apply_few.cu) ----
constexpr int FC_MAX = 8;
// Whether `ncols` columns of a dM x dN factor go to the warps instead of the tensor cores.  The warps'
// time grows with columns times elements, the tensor cores' with the factor's bytes from a base of 15 us a
// product; both sides of the line, whole apply (call included): 600 x 300 points, 8 columns 35 us
// against 38 on the tensor cores; 1200 x 600, 2 columns 33 against 48, 4 columns 47 against 48, 6 columns 52
// against 48; 2000 x 1000, 2 columns 62 against 76, 4 columns 87 against 76.  Stokes only: the potentials
// of a few conductors would move by 1.5e-7 (towards the exact ones, from 1.7e-7 off to 2e-8), which is
// more than FP64 callers that compare results between versions expect of this path.
inline bool fc_takes(int D, int ncols, int dM, int dN) {
    return D == 3 && ncols <= FC_MAX && (ncols <= 2 || (double)ncols * dM * dN <= 16777216.0);
}
// out[c][row] = sum_k F[row][k] G[c][k] as (hi, lo) pairs; F the factor's (hi, lo) planes [2][rows][ldk] at
// pstride, G [ncols][ldk], out [ncols][ldo]; ldk a multiple of 4.
cudaError_t fc_apply(int ncols, int rows, int ldk, const float *F, size_t pstride, const float2 *G, float2 *out, int ldo,
                     cudaStream_t st);
// gather_rotate with the values as (hi, lo) pairs [ncols][ld].
cudaError_t gather_rotate_hl(int D, const double *gamma, int sum_MD, const int *col_body, const int *col_rhs,
                             const int *body_off, const double *rot, int ncols, int dM, float2 *out, int ld,
                             cudaStream_t st);
struct ScatterArgs {
    const float2 *P = nullptr;     // (hi, lo) chunk partials [S][ncols][dN], or
    int S = 0;
    const double *L64 = nullptr;   // FP64 values [ncols][dN]
    const int *col_body = nullptr, *col_rhs = nullptr;
    const int *body_off = nullptr;    // each body's first output point
    const double *rot64 = nullptr;
    int ncols = 0, dN = 0, sum_N = 0;
    double *out = nullptr;         // [nrhs][sum_N][D] at the columns' bodies
    const double *base = nullptr;  // added when given
    // source records of the outputs for the pair kernel (layout packed or plain), or null
    float *rec = nullptr;
    int rec_floats = 0, packed = 0, nrhs = 1;
    const int *rec_off = nullptr;
    const float4 *src_pos = nullptr;
};
// out = base + R_k (column values), and the records.
cudaError_t scatter_rotate(int D, const ScatterArgs &a, cudaStream_t st);

// Completion strengths (Eq. lambda01-02 / Eq. al0) and extraction (Eq. getU / Eq. vkal).
cudaError_t completion_stokes(const double *F, const double *T, int nrhs, int P, const double *rot64,
                              const double *G0inv_shapes, const int *shape_id, const double *src_local64,
                              const int *body_src_off, int sum_N, double *lam0, cudaStream_t st);
cudaError_t completion_laplace(const double *Q, int nrhs, int P, const int *body_src_off, int sum_N, double *alpha0,
                               cudaStream_t st);
// sign -1: velocities (Eq. getU); +1: forces and torques (Eq. force_def).
cudaError_t extract_stokes(const double *lam, int nrhs, int P, const double *src_local64, const int *body_src_off,
                           int sum_N, double *U, double *Om, cudaStream_t st, double sign = -1.0);
// sum 0: potentials -mean(alpha) (Eq. vkal); 1: net charges sum(alpha) (Eq. qkgauss).
cudaError_t extract_laplace(const double *alpha, int nrhs, int P, const int *body_src_off, int sum_N, double *V,
                            cudaStream_t st, int sum = 0);
// Dirichlet data: rigid motion K_M U at the collocation points (Sec. 2.2) / phi 1_M (Sec. 2.1).
cudaError_t dirichlet_rhs_stokes(const double *U, const double *Om, int nrhs, int P, const double *tgt_local64,
                                 const int *body_tgt_off, int sum_M, double *b, cudaStream_t st);
cudaError_t dirichlet_rhs_laplace(const double *phi, int nrhs, int P, const int *body_tgt_off, int sum_M, double *b,
                                  cudaStream_t st);

// ---- evaluation points grouped by body (eval_group.cu) ----
// Device pointers.  A point's key is its owner body, or key_of_body[owner] (body_of_key its inverse)
// when given; grouped point j is the caller's point order[j], keys ascending, the caller's order kept
// within a key; toff[q] the first grouped point of key q.
int eval_chunks(int np);
struct EvalGroup {
    int np = 0, P = 0;
    const double *points = nullptr, *normals = nullptr;  // [np][3]; normals may be null
    const int *owner = nullptr;                          // [np] or null: the nearest centre
    const double *centres = nullptr;                     // [P][3] by body
    const int *key_of_body = nullptr, *body_of_key = nullptr;
    int *key = nullptr, *counts = nullptr, *total = nullptr;  // scratch [np], [eval_chunks(np)][P], [P]
    int *toff = nullptr, *order = nullptr;               // [P + 1], [np]
    float4 *t4 = nullptr;                                // [np] relative to the owner's centre, w = key (int bits)
    float *n32 = nullptr;                                // [np][3] grouped normals (with normals)
    double *t64 = nullptr, *n64 = nullptr;               // [np][3] FP64 copies, or null
    int *tbody = nullptr;                                // [np] keys, or null
    unsigned long long *radius = nullptr;                // [P] largest distance per key (double bits), or null
    int *err = nullptr;                                  // |= MFS_DEVERR_BADARG
};
cudaError_t eval_group(const EvalGroup &e, cudaStream_t st);

// ---- pressure and traction at evaluation points (stress.cu, Eq. traction), FP64 reference ----
// Points tgt_local (owner-relative) with owners tbody, unit normals nrm [np][3] or null (no traction),
// FP64 body-local sources and strengths, per-body suspension body range [sb0, sb1); outputs p
// [nrhs][np], traction [nrhs][np][3] (either may be null).  The FP32 path is the pair kernel's stress
// entry (StressStokes).
cudaError_t stress_f64(int nrhs, const double *tgt_local, const int *tbody, const double *nrm, int np,
                       const double *src_local, const int *src_off, int sum_N, const double *lam, const int *sb0,
                       const int *sb1, const double *centres, double *p_out, double *t_out, cudaStream_t st);

// ---- far field of the pair sums: equivalent-source treecode (farfield.cu) ----
constexpr int FF_NE = 196;            // equivalent points per node (a Fibonacci sphere of radius r_e)
// Check points per node and their radius over r_e, least-squares fit: 256 at 2.6 leave a field error of
// 1.2e-7 at 3 radii where 392 at 2.5 left 1.6e-7 (white-noise sources), fill two target pairs of every
// thread of an upward tile exactly and take a third off the FP64 fit.
constexpr int FF_NC = 256;
constexpr double FF_CHECK = 2.6;
constexpr double FF_MIN_SEPARATION = 2.5;  // the smallest mfs_options.farfield_separation
constexpr double FF_SRC_RATIO = 0.83; // a node's source radius / its equivalent radius
// (a target at least mfs_options.farfield_separation equivalent radii from a node's centre sees the node
// through its equivalent points)
// Lower orders of the same equivalent sources, for targets further away: order o has FF_ORD_N[o] points
// on the node's equivalent sphere and serves targets at least FF_ORD_KAPPA[o] equivalent radii from the
// node's centre (order 0 from farfield_separation on).  Its strengths are the least-squares match of the
// next higher order's field at FF_ORD_NC[o] points at FF_ORD_CHECK[o] radii, where the high-degree part
// that the smaller set cannot hold has already decayed.  White-noise sources at the edge of the node,
// relative field error: 196 points 1.2e-7 at 3 radii and 3e-8 at 4; 128 points 6e-8 at 4; 96 points
// 5e-8 at 5; 64 points 3e-8 at 8 (each falling further out).
constexpr int FF_NORD = 4;
constexpr int FF_ORD_N[FF_NORD] = {FF_NE, 128, 96, 64};
constexpr int FF_ORD_NC[FF_NORD] = {FF_NC, 192, 160, 128};
constexpr double FF_ORD_CHECK[FF_NORD] = {FF_CHECK, 4.0, 5.0, 8.0};
constexpr double FF_ORD_KAPPA[FF_NORD] = {3.0, 4.0, 5.0, 8.0};
// Singular values kept relative to the largest.  The last order's and the local match are cut at 1e-8:
// below it they only amplify FP32 rounding of the check field into strengths twice as large, whose own
// FP32 rounding then shows (field of 400 ellipsoids, white-noise strengths: 3.6e-7 uncut, 2.0e-7 cut,
// 2.1e-7 without local expansions or lower orders).
constexpr double FF_ORD_TRUNC[FF_NORD] = {1e-12, 1e-12, 1e-12, 1e-8}, FF_LOC_TRUNC = 1e-8;
// Local expansions: the field of the sources whose equivalent spheres stay FF_LOC_GAP target radii
// (rt, a body's farthest target point) away from a body's centre is evaluated at FF_LOC_NC points at
// FF_LOC_CHECK rt, matched by FF_LOC_N sources at FF_LOC_EQ rt around the body, and those are summed at
// the body's targets (1.5e-7 at the gap's edge, 3e-8 one radius further, 1e-8 at twice the distance).
constexpr int FF_LOC_N = 96, FF_LOC_NC = 128;
constexpr double FF_LOC_CHECK = 1.1, FF_LOC_EQ = 6.0, FF_LOC_GAP = 5.0;
// The match of one body's local sources (3 FF_LOC_NC x 3 FF_LOC_N FP64 FMAs at 2 per clock per SM) in
// pairs of the pair kernel (5.8 per clock per SM).
constexpr double FF_LOC_FIT_PAIRS = 3.2e5;
struct FFNode {
    double c[3] = {0, 0, 0};  // centre
    double rs = 0.0;          // radius of the node's proxy sources about c
    double re = 0.0;          // equivalent radius rs / FF_SRC_RATIO
    int body = -1;            // the body of a leaf, -1 for a group
    int first = 0, count = 0; // descendant bodies: order[first .. first + count)
    int nchild = 0;
    int child[8] = {0, 0, 0, 0, 0, 0, 0, 0};
};
struct FFTree {
    std::vector<FFNode> nodes;
    std::vector<int> order;  // bodies in tree (depth-first leaf) order
    std::vector<int> pos;    // pos[body] = its index in `order`
    std::vector<int> roots;  // one per suspension
};
// The 8-ary median-split tree of each suspension's bodies (centres [P][3], source radii rsrc [P]).
void ff_build_tree(int P, const double *centres, const double *rsrc, int S, const int *body_off, FFTree &t);
// Interaction list of the target bodies `tbodies` (original ids; target radii rtgt): segment ids, a
// body's proxy points as its tree position q < P, a node's equivalent points as P + node.  With
// self_skip, a single target body's own proxy points are left out.
void ff_interaction_list(const FFTree &t, int root, const std::vector<int> &tbodies, const double *centres,
                         const double *rtgt, double kappa, int self_skip, std::vector<int> &segs);
// Segment ids of the sums over several orders: proxies of tree position q: q; order o of node n:
// P + o nodes + n; local sources of tree position q: P + FF_NORD nodes + q.
// The highest order index whose distance rule holds at `ratio` = distance to the nearest target over
// r_e, -1 when none does; kappa0 = farfield_separation (orders keep their distances when it is below 3
// and move out in proportion above).
int ff_order(double ratio, double kappa0);
// Segments of the targets of the body set `tbodies` (one list for all of them): near bodies' proxies,
// far nodes at their order; self_skip as ff_interaction_list.
void ff_ordered_list(const FFTree &t, int root, const std::vector<int> &tbodies, const double *centres,
                     const double *rtgt, double kappa0, int self_skip, std::vector<int> &segs);
// The same cover split for local expansions: `local` gets the nodes that every body of the cell
// `tbodies` sees through its local expansion; direct[i] the remaining segments of tbodies[i] itself (its
// own proxies left out), among them its own local segment when `local` is not empty.  `local` stays
// empty where summing those nodes at the bodies' targets (targets_per_body of them) is less work.
void ff_cell_lists(const FFTree &t, int root, const std::vector<int> &tbodies, const double *centres,
                   const double *rtgt, double kappa0, double targets_per_body, std::vector<int> &local,
                   std::vector<std::vector<int>> &direct);
// mu[h][node][e][d] *= re[node] (the fit was made on the unit sphere; the kernels are homogeneous of
// degree -1).
cudaError_t ff_scale(double *mu, const double *re, int nodes, int per_node, int nrhs, cudaStream_t st);
// The constant and linear part of a local check field u [nrhs][bodies][FF_LOC_NC][D] at each body's points
// (chk [bodies][FF_LOC_NC] about its centre, target radii radius[bodies]) to far [nrhs][bodies][4][D] and out of
// u: these are fields that the local sources need not carry (mfs_api.cu, ff_pair_apply).
cudaError_t ff_take_linear(int D, double *u, const float4 *chk, const double *radius, int bodies, int nrhs, double *far,
                           cudaStream_t st);

// ---- GMRES (gmres.cu): L independent lanes, lane l owns vector entries [seg[l], seg[l+1]) ----
struct GmresDev {
    int L, m;                  // lanes, Krylov basis capacity (m <= 1023)
    long long n;               // vector length (all lanes)
    int sms;                   // SMs of the device
    int nblk;                  // blocks of the long-lane kernels, each within one lane
    const int *blk_lane;       // [nblk] the block's lane
    const long long *blk_off;  // [nblk+1] its first entry (blocks are contiguous)
    const int *lane_blk;       // [L+1] the lane's first block
    int clusters;              // 1: the lanes are short and few enough for the one-launch Arnoldi step
    double *V;                 // [(m+1)][n] basis
    double *H;                 // [L][m+1][m] Hessenberg, rotated to upper triangular
    double *cs, *sn, *g;       // [L][m], [L][m], [L][m+1]
    double *ibeta;             // [L] 1 / ||b||
    double *hbuf;              // [L][m+1] current column
    double *part;              // [2][nblk][m+1] block partials of the two passes' dots
    double *normp;             // [nblk] block partials of the norm
    unsigned *arrive;          // [1] blocks done (wraps to 0)
    int *active;               // [L] 1 while the lane iterates
    int *iters;                // [L] iterations done
    int *status;               // [L] 0 ok, 2 breakdown (non-finite)
    double *resid;             // [L] |g_k| / ||b||
    int *done;                 // [1] 1 when no lane is active
    int *jcur;                 // [1] the current Arnoldi column j (device-side, so a graph can loop)
    double tol;
};
// The blocks of lanes seg[0..L]: about equal lengths, whole waves of the SMs; returns whether every lane
// is short enough for the one-launch step.
bool gmres_plan_blocks(const std::vector<long long> &seg, int sm_count, std::vector<int> &blk_lane,
                       std::vector<long long> &blk_off, std::vector<int> &lane_blk);
// Kernel attributes for this basis; clears gd.clusters when the device does not hold the lanes' clusters
// at about one time.
cudaError_t gmres_prepare(GmresDev &gd);
// Start (two launches): v_0 = b / ||b|| per lane, also to vin (the matvec's input at a fixed address),
// lanes with b = 0 inactive, j = 0, done = (no lane active).
cudaError_t gmres_init(GmresDev &gd, const double *b, double *vin, cudaStream_t st);
// Orthogonalise w = A v_j against v_0..v_j (CGS2), append v_{j+1} (also to vin), Givens-update every
// active lane; j is read from gd.jcur and, with advance, increased unless done or the basis is full.
cudaError_t gmres_arnoldi(GmresDev &gd, double *w, double *vin, int advance, cudaStream_t st);
int gmres_arnoldi_launches(const GmresDev &gd);
// The advance as a kernel of its own that also sets a while node's condition to whether another
// iteration follows.
cudaError_t gmres_advance(GmresDev &gd, cudaGraphConditionalHandle cond, cudaStream_t st);
// x = V y with H y = g per lane.
cudaError_t gmres_solution(GmresDev &gd, double *x, cudaStream_t st);

}  // namespace mfs
