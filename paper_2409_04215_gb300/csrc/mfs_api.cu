// libmfs host runtime and C ABI (see include/mfs.h).
#include <cusolverDn.h>

#include <algorithm>
#include <array>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/mfs.h"
#include "common.cuh"
#include "kernels.h"

using namespace mfs;

namespace {

thread_local std::string g_setup_error;

struct DevBuf {
    void *p = nullptr;
    size_t bytes = 0;
};

// The treecode's matrices on the unit sphere (FP64, device): check field -> order-0 strengths, each
// order's strengths -> the next lower order's, local check field -> local sources.  They depend on the
// kernel's dimension only; the contexts of a process that are alive together share one set per device
// (ff_matrices), freed with the last of them.
struct FFMatrices {
    double *PinvT = nullptr;              // [D FF_NC][D FF_NE]
    double *ordT[FF_NORD] = {};           // [D FF_ORD_N[o - 1]][D FF_ORD_N[o]], o >= 1
    double *locT = nullptr;               // [D FF_LOC_NC][D FF_LOC_N]
    FFMatrices() = default;
    FFMatrices(const FFMatrices &) = delete;
    ~FFMatrices() {
        cudaFree(PinvT);
        cudaFree(locT);
        for (double *p : ordT) cudaFree(p);
    }
};

// Where the scratch of single calls comes from: one pool per device, shared by the contexts of a process
// that are alive together, so that what it keeps between calls does not grow with their number; given back
// with the last of them.  It keeps 256 MB: an evaluation takes from 50 bytes a point (velocities, one
// right-hand side, device inputs) to 350 (pressure and traction, four of them, host inputs).  More goes back
// to the device, where the next context may need it and the calls are long enough to allocate again.
struct CallPool {
    cudaMemPool_t pool = nullptr;
    CallPool() = default;
    CallPool(const CallPool &) = delete;
    ~CallPool() {
        if (pool) cudaMemPoolDestroy(pool);
    }
};

cudaError_t call_pool(int dev, std::shared_ptr<CallPool> &out) {
    static std::mutex mu;
    static std::weak_ptr<CallPool> kept[64];
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 64) out = kept[dev].lock();
    if (out) return cudaSuccess;
    auto p = std::make_shared<CallPool>();
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    unsigned long long keep = 256ull << 20;
    int no = 0;  // one stream's call never waits for another's to reuse its memory
    cudaError_t e = cudaMemPoolCreate(&p->pool, &props);
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(p->pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(p->pool, cudaMemPoolReuseAllowInternalDependencies, &no);
    if (e != cudaSuccess) return e;
    out = p;
    if (dev < 64) kept[dev] = p;
    return cudaSuccess;
}

struct PairPlan {
    int variant = -1;
    int include_self = 0;
    int tile_targets = 0;
    int G = 0;
    int ntiles = 0;
    long long total_units = 0;
    PairTile *tiles = nullptr;
    double *partial = nullptr;
    double *direct = nullptr;
    size_t partial_bytes = 0, direct_bytes = 0;
    int max_share = 1;  // the most CTAs that share one tile (sizes the epilogue)
};

// The one-body apply factors of one formulation for one shape, FP32 / FP64 and as tensor-core pieces.
struct FactorSet {
    bool built = false;
    ShapeDev dev{};
    bool tc_ready = false;
    float *Utp = nullptr, *Wptp = nullptr, *Wrtp = nullptr;  // FP32 (hi, lo) planes [2][r or dN][ld]
    size_t ut_stride = 0, wt_stride = 0;
    TcMap mU[3], mWp[3], mWr[3];
    // the transposed apply (adjoint), built on first use: (hi, lo) planes of U [dM][ld2] and of W^T [r][ld2]
    bool tcT_ready = false;
    float *Un = nullptr, *WpT = nullptr, *WrT = nullptr;
    size_t un_stride = 0;
    TcMap mUn[3], mWpT[3], mWrT[3];
};

struct ShapeHost {
    int M = 0, N = 0;
    std::vector<double> X0, Y0;  // body frame
    double G0inv[36];
    std::vector<int> bodies;     // bodies of this shape
    int *col_body = nullptr, *col_rhs = nullptr;  // device, [max_rhs * nbodies]
    float *A = nullptr, *Tm = nullptr;  // GEMM buffers
    double *Pk = nullptr;                              // split-K chunk results
    size_t Pk_count = 0;
    double *O64 = nullptr, *PkT = nullptr;             // adjoint: transposed-apply output and chunks
    float2 *PtcT = nullptr;                            // adjoint: tensor-core chunk results
    // tensor-core apply scratch: K-major TF32 pieces of the columns, chunk results
    int pieces = 0;        // TF32 pieces per operand (3: 6xTF32 products, 2: 3xTF32)
    int ld1 = 0, ld2 = 0;  // K extents padded to 32: roundup(dM, 32), roundup(r, 32)
    float *Ap = nullptr, *Tp = nullptr;  // [piece][columns][ld1 or ld2]
    size_t ap_stride = 0, tp_stride = 0;
    float2 *Ptc = nullptr;  // chunk results as (hi, lo) pairs
    std::map<int, std::array<TcMap, 6>> amaps;  // per column count: A pieces, T pieces
    double *A64 = nullptr, *T64 = nullptr, *L64 = nullptr;
    double *Pk64 = nullptr;  // FP64 apply: split-K partials
    // few columns: [FC_MAX][ld1], [FC_MAX][ld2] twice (forward and transposed), [FC_MAX][dM]
    float2 *Gf = nullptr, *Tf = nullptr, *Xf = nullptr, *Lf = nullptr;
    // one-body factors per formulation: [0] recompleted S_L (Sec. 3.3), [1] bare self block S^(00)
    // of the Dirichlet problems (Sec. 2.3), built on first use
    FactorSet fs[2];
};

}  // namespace

struct mfs_ctx {
    int kind = 0, D = 1;
    int fset = 0;  // factor set of the one-body apply: 0 recompleted (Sec. 3.3), 1 bare self block (Sec. 2.3)
    // GMRES iteration loops captured as CUDA graphs, by nrhs * 4 + fset * 2 + transposed
    struct SolveGraph {
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        int launches = 0, pair_launches = 0;  // per iteration
    };
    std::map<int, SolveGraph> graphs;
    double *vin_d = nullptr;  // matvec input of every iteration (v_j at a fixed address)
    cudaStream_t cap_stream = nullptr;  // capture only (the legacy stream cannot capture); launches use the caller's
    void drop_graphs() {
        for (auto &kv : graphs) {
            if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
            if (kv.second.graph) cudaGraphDestroy(kv.second.graph);
        }
        graphs.clear();
    }
    mfs_options opt{};
    int P = 0, S = 0, nshapes = 0;
    std::vector<double> centres, quats;
    std::vector<int> shape_id, body_off;
    std::vector<int> tgt_off, src_off, rec_off;  // [P+1] point / padded-record offsets
    std::vector<long long> blk_off;
    std::vector<int> tgt_body;                     // [sum_M]
    int sumM = 0, sumN = 0, nrec = 0;
    std::vector<double> rot;                       // [P][9]
    std::vector<ShapeHost> shapes;

    // device geometry
    double *centres_d = nullptr, *rot64_d = nullptr, *G0inv_d = nullptr;
    float *rot_d = nullptr;
    int *shape_id_d = nullptr;
    float4 *tgt_pos_d = nullptr, *src_pos_d = nullptr;
    float4 *tgt_hi_d = nullptr, *tgt_lo_d = nullptr;  // precision 3: grid-split body-local targets
    double *tgt_local64_d = nullptr, *src_local64_d = nullptr, *src_local4_d = nullptr;
    int *tgt_body_d = nullptr, *rec_pt_d = nullptr, *rec_off_d = nullptr, *tgt_off_d = nullptr,
        *src_off_d = nullptr, *susp_src_begin_d = nullptr, *susp_src_end_d = nullptr;
    long long *blk_off_d = nullptr;
    int *err_d = nullptr;

    // work buffers
    float *rec_d = nullptr;      // packed source records (max_rhs)
    int rec_floats = 0;          // floats per record allocated in rec_d (and recT_floats in recT_d)
    int recT_floats = 0;
    double *lam_d = nullptr;     // [max_rhs][sumN][D]
    double *raw_d = nullptr;     // FP64 pair sums: source-chunk partials [chunks][max_rhs][sumM or sumN][D]
    std::map<int, PairPlan> plans;  // key: variant * 4 + include_self * 2 + transposed
    int best_variant[2][5] = {{-1, -1, -1, -1, -1}, {-1, -1, -1, -1, -1}};  // [D==3][nrhs]

    // GMRES
    GmresDev gd{};
    size_t gd_n = 0;
    int gd_L = 0, gd_m = 0;
    double *w_d = nullptr, *b_d = nullptr, *x_d = nullptr;
    unsigned char *stat_d = nullptr, *stat_h = nullptr;  // the solve's statistics, device and pinned host
    static size_t stat_bytes(int L) { return sizeof(double) * L + sizeof(int) * (2 * (size_t)L + 4); }
    int *done_h = nullptr;   // pinned: [0] done, [1] the device error flag

    // solution kept for the adjoint
    // the last solve, for mfs_mobility_vjp and mfs_evaluate: which problem, its GMRES solution gamma
    // [max_rhs][sum_M][D] and its inputs (F then T [nrhs][P][3], or Q [nrhs][P])
    int last_solve = 0;  // 0 none, 1 mobility, 2 elastance, 3 resistance, 4 capacitance
    double *keep_gamma = nullptr;
    double *keep_lam0 = nullptr;  // [max_rhs][P][6]
    int last_nrhs = 0;

    // adjoint: the transposed direction (proxy targets, collocation sources)
    bool trans_ready = false;
    std::vector<int> src_body, recT_off;
    std::vector<long long> blkT_off;
    int nrecT = 0;
    float4 *tgtT_pos_d = nullptr;
    // the FP64 transposed sums (precision = 1): proxy -> body, collocation points [sum_M][4] (body-local
    // x, y, z and the body id), each body's suspension as a collocation range
    int *src_body_d = nullptr, *colT_begin_d = nullptr, *colT_end_d = nullptr;
    double *colloc4_d = nullptr;
    float *recT_d = nullptr;
    int *recT_off_d = nullptr, *rec_ptT_d = nullptr;
    long long *blkT_off_d = nullptr;
    double *tmpM_d = nullptr;     // [max_rhs][sum_M][3]
    double *gradT_d = nullptr;    // [sum_M][3] per-target gradient sums
    double *src_grad_d = nullptr; // [P][3]
    double *six_d = nullptr;      // [max_rhs][P][6] scratch for -K_N^T z
    float *w32_d = nullptr;       // [max_rhs][sum_M][3] FP32 adjoint strengths
    double *eye6_d = nullptr;     // [nshapes][36] identity (K_N [u; w] expansion)

    // far field of the pair sums (opt.farfield = 1): equivalent-source treecode (farfield.cu)
    struct FarField {
        bool ready = false;
        // the roles of the point sets: forward sums (proxy sources, collocation targets) or the
        // adjoint's transposed sums (collocation sources, proxy targets)
        bool src_colloc = false;
        const float4 *src_pos = nullptr;             // [nsrc] body-local source positions
        const int *rec_pt = nullptr;                 // [nrec] source record -> point (-1: padding)
        const float4 *tgt_pos = nullptr;             // [ntgt] body-local target positions
        const std::vector<int> *rec_off = nullptr;   // [P + 1] padded record offsets of the sources
        const std::vector<int> *tgt_off = nullptr;   // [P + 1] target offsets
        int nsrc = 0, nrec = 0, ntgt = 0;
        FFTree tree;
        int nodes = 0;
        std::vector<double> rsrc, rtgt;              // per body: radius of its proxy / collocation points
        std::shared_ptr<const FFMatrices> mat;       // the fits' matrices
        double *centres = nullptr;                   // [P + nodes][3]: bodies in tree order, then the nodes
        double *re = nullptr;                        // [nodes] equivalent radii
        float4 *eq_pos = nullptr;                    // [nodes FF_NE] equivalent points about their node's centre
        int *eq_pt = nullptr;                        // identity record -> point map (packing)
        float4 *chk_pos = nullptr;                   // [nodes FF_NC] check points, w = P + node
        float4 *tgt = nullptr;                       // [sum_M] targets in tree order, w = tree position
        int *pos = nullptr, *order = nullptr;        // [P] body -> tree position and back (device)
        int *tperm = nullptr;                        // [sum_M] tree-order target -> caller's target index
        int *seg_rec0 = nullptr, *seg_rec1 = nullptr;  // [P + nodes] record range of every segment
        std::vector<int> seg_rec0_h, seg_rec1_h;
        float *rec = nullptr;                        // proxy records, then equivalent records
        int rec_floats = 0;
        double *ucheck = nullptr;                    // [max_rhs][nodes FF_NC][D]
        double *mu = nullptr;                        // [max_rhs][nodes FF_NE][D]
        double *fit_chunks = nullptr;                // split-K partials of the fit products
        float *wt = nullptr;                         // [max_rhs][ntgt][3] target weights in tree order (gradient)
        // lower orders of the equivalent sources (index 1 .. FF_NORD - 1): the points about their node's
        // centre, the strengths
        float4 *ord_pos[FF_NORD] = {};               // [nodes FF_ORD_N[o]]
        double *ord_mu[FF_NORD] = {};                // [max_rhs][nodes FF_ORD_N[o]][D]
        size_t ord_rec[FF_NORD] = {};                // first record of the order's segments
        // local expansions of the bodies (tree order)
        bool use_local = false;
        double *rloc = nullptr;                      // [P] target radii
        float4 *loc_pos = nullptr, *lchk_pos = nullptr;  // [P FF_LOC_N], [P FF_LOC_NC] about the body's centre
        double *ulocal = nullptr, *nu = nullptr;     // [max_rhs][P FF_LOC_NC][D], [max_rhs][P FF_LOC_N][D]
        double *ufar = nullptr;                      // [max_rhs][P][4][D]
        size_t loc_rec = 0;
        struct ListPlan {
            PairPlan p;
            int *seg = nullptr;
            long long *cum = nullptr;
            double pairs = 0.0;                      // target-source pairs one application evaluates
            int orders = 0;                          // bit o: the lists hold segments of order o
        };
        std::map<int, ListPlan> up;                  // upward sums, key: variant
        std::map<int, ListPlan> ev;                  // order-0 lists at the targets (gradient), key: variant
        std::map<int, ListPlan> loc;                 // local check points, key: variant
        std::map<int, ListPlan> direct;              // targets, all orders, key: variant * 2 + include_self
        struct Cells {                               // ff_cell_lists of every cell of consecutive tree positions
            std::vector<int> first;                  // first tree position of each cell, then P
            std::vector<int> cell_of;                // tree position -> cell
            std::vector<std::vector<int>> local;     // per cell
            std::vector<std::vector<int>> direct;    // per tree position
            bool any_local = false;
        };
        Cells cells;
    } ff, ffT;                                       // forward sums; transposed sums (adjoint)

    int sm_count = 0;
    std::shared_ptr<CallPool> pool;  // scratch of single calls (Scratch)
    std::string last_error;
    std::vector<void *> allocs;
    double ms_setup = 0.0;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr, evp0 = nullptr, evp1 = nullptr;
    double pair_ms_acc = 0.0;
    int launches = 0;        // kernels + memsets enqueued by the current call
    int pair_launches = 0;   // pair-kernel launches of the current call
    std::vector<cudaEvent_t> pev;  // profile: event pairs around pair-kernel launches

    int fail_alloc = 0;      // mfs_selftest_fail_alloc: the allocation from now that is refused (1 = the next; 0 = none)
    bool refuse_alloc() {    // a request that no device can serve, so that the runtime reports what it does in earnest
        void *p = nullptr;
        return fail_alloc > 0 && --fail_alloc == 0 && cudaMalloc(&p, (size_t)1 << 60) != cudaSuccess;
    }

    template <typename T>
    cudaError_t alloc(T **p, size_t count) {
        *p = nullptr;
        if (refuse_alloc()) return cudaErrorMemoryAllocation;
        if (count == 0) count = 1;
        cudaError_t e = cudaMalloc((void **)p, sizeof(T) * count);
        if (e == cudaErrorMemoryAllocation && pool) {  // what the pool keeps may be enough
            cudaGetLastError();
            e = cudaMemPoolTrimTo(pool->pool, 0);
            if (e == cudaSuccess) e = cudaMalloc((void **)p, sizeof(T) * count);
        }
        if (e == cudaSuccess) allocs.push_back((void *)*p);
        return e;
    }
    void release(void *p) {
        if (!p) return;
        auto it = std::find(allocs.begin(), allocs.end(), p);
        if (it != allocs.end()) allocs.erase(it);
        cudaFree(p);
    }
    ~mfs_ctx() {
        drop_graphs();
        if (cap_stream) cudaStreamDestroy(cap_stream);
        for (void *p : allocs) cudaFree(p);
        if (done_h) cudaFreeHost(done_h);
        if (stat_h) cudaFreeHost(stat_h);
        if (ev0) cudaEventDestroy(ev0);
        if (ev1) cudaEventDestroy(ev1);
        if (evp0) cudaEventDestroy(evp0);
        if (evp1) cudaEventDestroy(evp1);
        for (cudaEvent_t e : pev) cudaEventDestroy(e);
    }
};

static mfs_status ff_setup(mfs_ctx *ctx, mfs_ctx::FarField &F, cudaStream_t st);  // far-field structures

namespace {

#define CK(call)                                                                             \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess) {                                                             \
            ctx->last_error = std::string(#call) + ": " + cudaGetErrorString(e_);            \
            cudaGetLastError(); /* the next call's launch checks are not to find it */       \
            return e_ == cudaErrorMemoryAllocation ? MFS_ERR_OOM : MFS_ERR_CUDA;              \
        }                                                                                    \
    } while (0)

#define CKS(call)                                  \
    do {                                           \
        mfs_status s_ = (call);                    \
        if (s_ != MFS_OK) return s_;               \
    } while (0)

bool is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Device scratch of one call on one stream: allocations from the device's call pool, freed in stream order
// when the call returns (no device synchronisation; a cudaMalloc and cudaFree pair per buffer took most
// of a small evaluation).
struct Scratch {
    mfs_ctx *ctx;
    cudaStream_t st;
    std::vector<void *> ps;
    std::vector<std::shared_ptr<void>> host;  // host arrays whose uploads may still be in flight
    Scratch(mfs_ctx *c, cudaStream_t s) : ctx(c), st(s) {}
    Scratch(const Scratch &) = delete;
    ~Scratch() {
        if (!host.empty()) cudaStreamSynchronize(st);
        for (void *p : ps) cudaFreeAsync(p, st);
    }
    // Upload of a host array that is kept until the stream is done with it.
    template <typename T>
    cudaError_t upload(T *dst, std::vector<T> &&src) {
        auto kept = std::make_shared<std::vector<T>>(std::move(src));
        host.push_back(kept);
        return cudaMemcpyAsync(dst, kept->data(), sizeof(T) * kept->size(), cudaMemcpyHostToDevice, st);
    }
    template <typename T>
    cudaError_t alloc(T **p, size_t count) {
        *p = nullptr;
        const cudaError_t e =
            cudaMallocFromPoolAsync((void **)p, sizeof(T) * std::max<size_t>(count, 1), ctx->pool->pool, st);
        if (e == cudaSuccess) ps.push_back((void *)*p);
        return e;
    }
};

// A device view of a user pointer: either the pointer itself or a staged copy.
struct Staged {
    mfs_ctx *ctx = nullptr;
    double *d = nullptr;
    const void *user = nullptr;
    size_t count = 0;
    bool owned = false;
    bool reading = false;  // the copy from the user's host memory may be in flight (pinned memory)
    cudaStream_t st = nullptr;
    ~Staged() {
        if (reading) cudaStreamSynchronize(st);  // the caller may reuse its memory once the call returns
        if (owned && d) cudaFreeAsync(d, st);
    }
};

mfs_status stage_in(mfs_ctx *ctx, Staged &s, const double *user, size_t count, cudaStream_t st) {
    s.ctx = ctx;
    s.user = user;
    s.count = count;
    if (is_device_ptr(user)) {
        s.d = const_cast<double *>(user);
        return MFS_OK;
    }
    s.st = st;
    CK(cudaMallocFromPoolAsync((void **)&s.d, sizeof(double) * std::max<size_t>(count, 1), ctx->pool->pool, st));
    s.owned = true;
    s.reading = true;
    CK(cudaMemcpyAsync(s.d, user, sizeof(double) * count, cudaMemcpyHostToDevice, st));
    return MFS_OK;
}

mfs_status stage_out_alloc(mfs_ctx *ctx, Staged &s, double *user, size_t count, cudaStream_t st) {
    s.ctx = ctx;
    s.user = user;
    s.count = count;
    if (is_device_ptr(user)) {
        s.d = user;
        return MFS_OK;
    }
    s.st = st;
    CK(cudaMallocFromPoolAsync((void **)&s.d, sizeof(double) * std::max<size_t>(count, 1), ctx->pool->pool, st));
    s.owned = true;
    return MFS_OK;
}

mfs_status stage_out_finish(mfs_ctx *ctx, Staged &s, cudaStream_t st) {
    if (s.owned) {
        CK(cudaMemcpyAsync(const_cast<void *>(s.user), s.d, sizeof(double) * s.count, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
    }
    return MFS_OK;
}

mfs_status check_device_error(mfs_ctx *ctx, cudaStream_t st) {
    int h = 0;
    CK(cudaMemcpyAsync(&h, ctx->err_d, sizeof(int), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (h) {
        ctx->last_error = (h & MFS_DEVERR_TIMEOUT) ? "a device-side bounded wait gave up" : "device argument error";
        cudaMemsetAsync(ctx->err_d, 0, sizeof(int), st);
        return MFS_ERR_DEVICE_TIMEOUT;
    }
    return MFS_OK;
}

void quat_to_rot(const double *q, double *R) {
    const double w = q[0], x = q[1], y = q[2], z = q[3];
    R[0] = 1 - 2 * (y * y + z * z); R[1] = 2 * (x * y - w * z); R[2] = 2 * (x * z + w * y);
    R[3] = 2 * (x * y + w * z); R[4] = 1 - 2 * (x * x + z * z); R[5] = 2 * (y * z - w * x);
    R[6] = 2 * (x * z - w * y); R[7] = 2 * (y * z + w * x); R[8] = 1 - 2 * (x * x + y * y);
}

// 6x6 inverse by Gauss-Jordan with partial pivoting; returns false when singular.
bool invert6(const double *A, double *Ainv) {
    double a[6][12];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 12; ++j) a[i][j] = j < 6 ? A[i * 6 + j] : (j - 6 == i ? 1.0 : 0.0);
    for (int c = 0; c < 6; ++c) {
        int p = c;
        for (int r = c + 1; r < 6; ++r)
            if (std::fabs(a[r][c]) > std::fabs(a[p][c])) p = r;
        if (a[p][c] == 0.0) return false;
        for (int j = 0; j < 12; ++j) std::swap(a[c][j], a[p][j]);
        const double inv = 1.0 / a[c][c];
        for (int j = 0; j < 12; ++j) a[c][j] *= inv;
        for (int r = 0; r < 6; ++r)
            if (r != c) {
                const double f = a[r][c];
                for (int j = 0; j < 12; ++j) a[r][j] -= f * a[c][j];
            }
    }
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) Ainv[i * 6 + j] = a[i][j + 6];
    return true;
}

// G0 = K_N0^T K_N0 for body-frame proxy points (Eq. lambda02 with Eq. Kdef).
void gram6(const std::vector<double> &Y0, double *G) {
    std::memset(G, 0, sizeof(double) * 36);
    const int n = (int)Y0.size() / 3;
    for (int q = 0; q < n; ++q) {
        const double *d = &Y0[3 * q];
        const double cm[3][3] = {{0.0, d[2], -d[1]}, {-d[2], 0.0, d[0]}, {d[1], -d[0], 0.0}};
        for (int b = 0; b < 3; ++b) {
            double row[6];
            for (int m = 0; m < 3; ++m) row[m] = (b == m) ? 1.0 : 0.0;
            for (int m = 0; m < 3; ++m) row[3 + m] = cm[b][m];
            for (int i = 0; i < 6; ++i)
                for (int j = 0; j < 6; ++j) G[i * 6 + j] += row[i] * row[j];
        }
    }
}

int default_variant(int D, int nrhs, int comp = 0) {
    int count = 0;
    const PairVariant *v = pair_variants(&count);
    // preferred variant per kind and nrhs when not autotuned: packed f32x2 for Stokes, scalar for Laplace
    const int wantT = (D == 3) ? (nrhs == 1 ? 4 : 2) : 4;
    const int wantNT = 128, wantPacked = (D == 3 && nrhs != 3) ? 1 : 0;
    if (!comp)
        for (int i = 0; i < count; ++i)
            if (!v[i].grad && !v[i].comp && v[i].D == D && v[i].nrhs == nrhs && v[i].T == wantT &&
                v[i].NT == wantNT && v[i].packed == wantPacked)
                return i;
    for (int i = 0; i < count; ++i)
        if (!v[i].grad && v[i].comp == comp && v[i].D == D && v[i].nrhs == nrhs) return i;
    return -1;
}

// The forward pair-sum variant of this context for nrhs: compensated kernels with precision = 3.
int forward_variant(const mfs_ctx *ctx, int nrhs) {
    const int tuned = ctx->best_variant[ctx->D == 3][nrhs];
    return tuned >= 0 ? tuned : default_variant(ctx->D, nrhs, ctx->opt.precision == 3);
}

// An FP32 (not compensated) variant for the sums that have no compensated form (transposed sums,
// evaluation at arbitrary points).
int fp32_variant(const mfs_ctx *ctx, int D, int nrhs) {
    if (ctx->opt.precision == 3) return default_variant(D, nrhs, 0);
    const int tuned = ctx->best_variant[D == 3][nrhs];
    return tuned >= 0 ? tuned : default_variant(D, nrhs, 0);
}

// Tiles and CTA shares for one pair-kernel variant.  transposed = 0: collocation targets, proxy
// sources (the matvec and u_0); transposed = 1: proxy targets, collocation sources (the adjoint's
// S^T sums).
// Work list of a pair sum over any target set grouped by body: targets of body k are
// [toff[k], toff[k+1]); source blocks per body from boff.  With `tmp` the plan's device arrays are that
// call's scratch.
mfs_status build_plan_for(mfs_ctx *ctx, int variant, int include_self, const std::vector<int> &toff,
                          const std::vector<long long> &boff, int ntargets, PairPlan &plan, Scratch *tmp = nullptr) {
    int count = 0;
    const PairVariant *vv = pair_variants(&count);
    const PairVariant &v = vv[variant];
    const int TT = v.tile_targets;
    const int C = v.grad == 1 ? 3 : v.D * v.nrhs;  // the gradient kernel: one 3-vector per target
    std::vector<PairTile> tiles;
    long long units = 0;
    for (int s = 0; s < ctx->S; ++s) {
        const int B0 = ctx->body_off[s], B1 = ctx->body_off[s + 1];
        const int t_end = toff[B1];
        int t = toff[B0], kb0 = B0;
        while (t < t_end) {
            int t1 = std::min(t + TT, t_end);
            while (toff[kb0 + 1] <= t) ++kb0;  // the body of target t, then of target t1 - 1
            int kb1 = kb0;
            while (toff[kb1 + 1] < t1) ++kb1;
            if (kb1 - kb0 + 1 > MFS_MAX_TILE_BODIES) {
                kb1 = kb0 + MFS_MAX_TILE_BODIES - 1;
                t1 = toff[kb1 + 1];
            }
            PairTile tl;
            tl.t0 = t;
            tl.t1 = t1;
            tl.kb0 = kb0;
            tl.nb = kb1 - kb0 + 1;
            tl.skip = (!include_self && tl.nb == 1) ? kb0 : -1;
            tl.B0 = B0;
            tl.B1 = B1;
            tl.L0 = tl.L1 = -1;
            long long u = 0;
            for (int b = B0; b < B1; ++b)
                if (b != tl.skip) u += boff[b + 1] - boff[b];
            tl.u0 = units;
            tl.u1 = units + u;
            units += u;
            tiles.push_back(tl);
            t = t1;
        }
    }
    const int occ = pair_occupancy(variant);
    if (occ <= 0) {
        ctx->last_error = "pair kernel variant cannot be resident on this GPU";
        return MFS_ERR_CUDA;
    }
    long long G = (long long)occ * ctx->sm_count;
    if (G > units) G = std::max<long long>(units, 1);
    const long long W = units;
    int max_share = 1;
    for (auto &tl : tiles) {
        if (tl.u1 == tl.u0) {
            tl.gA = tl.gB = -1;
            continue;
        }
        auto owner = [&](long long u) { return (int)(((u + 1) * G - 1) / W); };
        tl.gA = owner(tl.u0);
        tl.gB = owner(tl.u1 - 1);
        tl.slotA = (long long)tl.gA * W / G >= tl.u0 ? 0 : 1;
        max_share = std::max(max_share, tl.gB - tl.gA + 1);
    }
    plan.variant = variant;
    plan.include_self = include_self;
    plan.tile_targets = TT;
    plan.G = (int)G;
    plan.ntiles = (int)tiles.size();
    plan.max_share = max_share;
    plan.total_units = units;
    if (tmp) {
        CK(tmp->alloc(&plan.tiles, tiles.size()));
        CK(tmp->alloc(&plan.partial, (size_t)G * 2 * TT * C));
        CK(tmp->alloc(&plan.direct, (size_t)std::max(ntargets, 1) * C));
        CK(tmp->upload(plan.tiles, std::move(tiles)));
        return MFS_OK;
    }
    CK(ctx->alloc(&plan.tiles, tiles.size()));
    CK(cudaMemcpy(plan.tiles, tiles.data(), sizeof(PairTile) * tiles.size(), cudaMemcpyHostToDevice));
    plan.partial_bytes = sizeof(double) * (size_t)G * 2 * TT * C;
    plan.direct_bytes = sizeof(double) * (size_t)ntargets * C;
    CK(ctx->alloc(&plan.partial, (size_t)G * 2 * TT * C));
    CK(ctx->alloc(&plan.direct, (size_t)std::max(ntargets, 1) * C));
    return MFS_OK;
}

mfs_status build_plan(mfs_ctx *ctx, int variant, int include_self, int transposed, PairPlan &plan) {
    return build_plan_for(ctx, variant, include_self, transposed ? ctx->src_off : ctx->tgt_off,
                          transposed ? ctx->blkT_off : ctx->blk_off, transposed ? ctx->sumN : ctx->sumM, plan);
}

void release_plan(mfs_ctx *ctx, PairPlan &plan) {
    ctx->release(plan.tiles);
    ctx->release(plan.partial);
    ctx->release(plan.direct);
    plan = PairPlan{};
}

mfs_status get_plan(mfs_ctx *ctx, int variant, int include_self, PairPlan **out, int transposed = 0) {
    const int key = variant * 4 + include_self * 2 + transposed;
    auto it = ctx->plans.find(key);
    if (it == ctx->plans.end()) {
        PairPlan p;
        CKS(build_plan(ctx, variant, include_self, transposed, p));
        it = ctx->plans.emplace(key, p).first;
    }
    *out = &it->second;
    return MFS_OK;
}

PairWork work_of(const PairPlan &p) {
    PairWork w;
    w.tiles = p.tiles;
    w.ntiles = p.ntiles;
    w.total_units = p.total_units;
    w.G = p.G;
    w.partial = p.partial;
    w.direct = p.direct;
    w.tile_targets = p.tile_targets;
    w.include_self = p.include_self;
    w.max_share = p.max_share;
    return w;
}

PairGeom geom_of(mfs_ctx *ctx) {
    PairGeom g;
    g.tgt = ctx->tgt_pos_d;
    g.src = ctx->rec_d;
    g.src_off = ctx->rec_off_d;
    g.blk_off = ctx->blk_off_d;
    g.centres = ctx->centres_d;
    g.ntargets = ctx->sumM;
    g.tgt_hi = ctx->tgt_hi_d;
    g.tgt_lo = ctx->tgt_lo_d;
    return g;
}

// Source records for `variant` from FP64 strengths [nrhs][sum_N][D].
cudaError_t pack_for(mfs_ctx *ctx, int variant, const double *strength, int nrhs, cudaStream_t st) {
    int vc = 0;
    const PairVariant *vv = pair_variants(&vc);
    // the record buffer holds every layout this context's entries use; anything else is refused
    if (pair_record_floats(ctx->D, nrhs, vv[variant].comp ? 2 : vv[variant].packed) > ctx->rec_floats)
        return cudaErrorInvalidValue;
    if (vv[variant].comp)
        return pack_sources_comp(ctx->D, nrhs, ctx->src_local64_d, ctx->rec_pt_d, strength, ctx->sumN, ctx->nrec,
                                 ctx->rec_d, st);
    return pack_sources(ctx->D, nrhs, vv[variant].packed, ctx->src_pos_d, ctx->rec_pt_d, strength, ctx->sumN,
                        ctx->nrec, ctx->rec_d, st);
}

double kernel_scale(mfs_ctx *ctx) {
    return ctx->kind == MFS_STOKES ? 1.0 / (8.0 * MFS_PI * ctx->opt.mu) : 1.0 / (4.0 * MFS_PI);
}

// out = beta * base + sign * (pair sum of strengths)  (strengths FP64 [nrhs][sumN][D] on device)
// (raw in S partials of n, added in order)
__global__ void combine_raw_kernel(const double *raw, const double *base, double beta, double scale, double *out,
                                   size_t n, int S) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v = raw[i];
    for (int z = 1; z < S; ++z) v += raw[(size_t)z * n + i];
    out[i] = (base ? beta * base[i] : 0.0) + scale * v;
}

// Source chunks of the FP64 sums over ntargets targets (transposed: the collocation points are the sources).
int fp64_chunks(const mfs_ctx *ctx, int ntargets, bool transposed = false) {
    const std::vector<int> &off = transposed ? ctx->tgt_off : ctx->src_off;
    int least = off.back();
    for (int s = 0; s < ctx->S; ++s) least = std::min(least, off[ctx->body_off[s + 1]] - off[ctx->body_off[s]]);
    return fp64_pair_chunks(ntargets, least, ctx->sm_count);
}

mfs_status ff_pair_apply(mfs_ctx *ctx, mfs_ctx::FarField &F, int variant, const double *strength, double *out,
                         const double *base, double beta, double scale, int nrhs, int include_self, cudaStream_t st);

mfs_status pair_apply(mfs_ctx *ctx, const double *strength, double *out, const double *base, double beta,
                      double sign, int nrhs, int include_self, cudaStream_t st, bool packed = false) {
    const double scale = sign * kernel_scale(ctx);
    if (ctx->opt.precision == 1) {
        const int S = fp64_chunks(ctx, ctx->sumM);
        CK(pair_sum_fp64(ctx->D, nrhs, S, ctx->tgt_local64_d, ctx->tgt_body_d, ctx->sumM, ctx->src_local4_d,
                         ctx->sumN, ctx->susp_src_begin_d, ctx->susp_src_end_d, ctx->src_off_d, ctx->centres_d,
                         strength, include_self, ctx->raw_d, st));
        const size_t n = (size_t)nrhs * ctx->sumM * ctx->D;
        combine_raw_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ctx->raw_d, base, beta, scale, out, n, S);
        CK(cudaGetLastError());
        ctx->launches += 2;
        ctx->pair_launches += 1;
        return MFS_OK;
    }
    const int variant = forward_variant(ctx, nrhs);
    if (variant < 0) {
        ctx->last_error = "no pair-kernel variant for this nrhs";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->ff.ready)
        return ff_pair_apply(ctx, ctx->ff, variant, strength, out, base, beta, scale, nrhs, include_self, st);
    PairPlan *plan = nullptr;
    CKS(get_plan(ctx, variant, include_self, &plan));
    if (!packed) CK(pack_for(ctx, variant, strength, nrhs, st));
    const PairWork w = work_of(*plan);
    ctx->launches += packed ? 1 : 2;
    if (w.total_units > 0) {
        const size_t slot = 2 * (size_t)ctx->pair_launches;
        if (ctx->opt.profile) {
            while (ctx->pev.size() < slot + 2) {
                cudaEvent_t e;
                CK(cudaEventCreate(&e));
                ctx->pev.push_back(e);
            }
            CK(cudaEventRecord(ctx->pev[slot], st));
        }
        CK(pair_launch(variant, geom_of(ctx), w, ctx->err_d, st));
        if (ctx->opt.profile) CK(cudaEventRecord(ctx->pev[slot + 1], st));
        ctx->launches += 1;
        ctx->pair_launches += 1;
    }
    CK(pair_epilogue(ctx->D, nrhs, w, base, beta, scale, out, ctx->sumM, st));
    return MFS_OK;
}

// Tiles over targets grouped into consecutive groups (group g: targets [toff[g], toff[g+1]), its id in
// the geometry's centre table gid0 + g), never crossing a group boundary listed in `cuts`, each tile
// with the interaction list that list_of(g0, g1) gives for its groups g0..g1; seg_blocks[s] blocks of
// MFS_BS records per segment s.  Uploads the tiles and the lists (PairGeom::lst_seg, lst_cum).
template <class ListFn>
mfs_status build_plan_lists(mfs_ctx *ctx, int variant, int include_self, const std::vector<int> &toff, int gid0,
                            const std::vector<int> &cuts, const std::vector<long long> &seg_blocks,
                            const std::vector<int> &seg_recs, ListFn list_of, PairPlan &plan, int **lst_seg_d,
                            long long **lst_cum_d, double &pairs, Scratch *tmp = nullptr) {
    int count = 0;
    const PairVariant *vv = pair_variants(&count);
    const PairVariant &v = vv[variant];
    const int TT = v.tile_targets;
    const int C = v.grad == 1 ? 3 : v.D * v.nrhs;  // the gradient kernel: one 3-vector per target
    std::vector<PairTile> tiles;
    std::vector<int> lst;
    std::vector<long long> cum{0};
    std::vector<int> segs;
    long long units = 0;
    pairs = 0.0;
    const int ngroups = (int)toff.size() - 1;
    std::vector<int> tgroup(toff.back());
    for (int g = 0; g < ngroups; ++g)
        for (int t = toff[g]; t < toff[g + 1]; ++t) tgroup[t] = g;
    for (size_t ci = 0; ci + 1 < cuts.size(); ++ci) {
        const int t_end = toff[cuts[ci + 1]];
        int t = toff[cuts[ci]];
        while (t < t_end) {
            // as few tiles as the range needs, of about equal length in whole target pairs: 839 targets as
            // 512 + 327 (4 and 3 pairs a thread) rather than 768 + 71 (6 and 1, whose one pair hides no latency).
            // 2000 ellipsoids, one treecode matvec with tiles of 512 / 768 targets: 32.5 / 33.2 ms after this and
            // the epilogue's grid cap, 33-34 ms before
            const int left = (t_end - t + TT - 1) / TT, unit = 2 * v.NT;
            const int size = std::min(TT, ((t_end - t + left - 1) / left + unit - 1) / unit * unit);
            int t1 = std::min(t + size, t_end);
            const int g0 = tgroup[t];
            int g1 = tgroup[t1 - 1];
            if (g1 - g0 + 1 > MFS_MAX_TILE_BODIES) {
                g1 = g0 + MFS_MAX_TILE_BODIES - 1;
                t1 = toff[g1 + 1];
            }
            PairTile tl;
            tl.t0 = t;
            tl.t1 = t1;
            tl.kb0 = gid0 + g0;
            tl.nb = g1 - g0 + 1;
            tl.skip = -1;
            tl.B0 = tl.B1 = 0;
            segs.clear();
            list_of(g0, g1, segs);
            tl.L0 = (int)lst.size();
            long long u = 0;
            for (int sgi : segs) {
                lst.push_back(sgi);
                u += seg_blocks[sgi];
                cum.push_back(units + u);
                pairs += (double)(t1 - t) * seg_recs[sgi];
            }
            tl.L1 = (int)lst.size();
            tl.u0 = units;
            tl.u1 = units + u;
            units += u;
            tiles.push_back(tl);
            t = t1;
        }
    }
    const int occ = pair_occupancy(variant);
    if (occ <= 0) {
        ctx->last_error = "pair kernel variant cannot be resident on this GPU";
        return MFS_ERR_CUDA;
    }
    long long G = (long long)occ * ctx->sm_count;
    if (G > units) G = std::max<long long>(units, 1);
    const long long W = std::max<long long>(units, 1);
    int max_share = 1;
    for (auto &tl : tiles) {
        if (tl.u1 == tl.u0) {
            tl.gA = tl.gB = -1;
            continue;
        }
        auto owner = [&](long long u) { return (int)(((u + 1) * G - 1) / W); };
        tl.gA = owner(tl.u0);
        tl.gB = owner(tl.u1 - 1);
        tl.slotA = (long long)tl.gA * W / G >= tl.u0 ? 0 : 1;
        max_share = std::max(max_share, tl.gB - tl.gA + 1);
    }
    plan.variant = variant;
    plan.include_self = include_self;
    plan.tile_targets = TT;
    plan.G = (int)G;
    plan.ntiles = (int)tiles.size();
    plan.max_share = max_share;
    plan.total_units = units;
    auto alloc_all = [&](auto &&from) -> cudaError_t {
        cudaError_t e = from.alloc(&plan.tiles, tiles.size());
        if (e == cudaSuccess) e = from.alloc(&plan.partial, (size_t)G * 2 * TT * C);
        if (e == cudaSuccess) e = from.alloc(&plan.direct, (size_t)std::max(toff.back(), 1) * C);
        if (e == cudaSuccess) e = from.alloc(lst_seg_d, lst.size());
        if (e == cudaSuccess) e = from.alloc(lst_cum_d, cum.size());
        return e;
    };
    CK(tmp ? alloc_all(*tmp) : alloc_all(*ctx));
    if (tmp) {
        CK(tmp->upload(plan.tiles, std::move(tiles)));
        CK(tmp->upload(*lst_seg_d, std::move(lst)));
        CK(tmp->upload(*lst_cum_d, std::move(cum)));
        return MFS_OK;
    }
    CK(cudaMemcpy(plan.tiles, tiles.data(), sizeof(PairTile) * tiles.size(), cudaMemcpyHostToDevice));
    if (!lst.empty()) CK(cudaMemcpy(*lst_seg_d, lst.data(), sizeof(int) * lst.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(*lst_cum_d, cum.data(), sizeof(long long) * cum.size(), cudaMemcpyHostToDevice));
    return MFS_OK;
}

// Records and blocks of every far-field segment.
static void ff_segments(const mfs_ctx::FarField &F, std::vector<long long> &blocks, std::vector<int> &recs) {
    const size_t n = F.seg_rec0_h.size();
    blocks.resize(n);
    recs.resize(n);
    for (size_t sg = 0; sg < n; ++sg) {
        recs[sg] = F.seg_rec1_h[sg] - F.seg_rec0_h[sg];
        blocks[sg] = (recs[sg] + MFS_BS - 1) / MFS_BS;
    }
}

// The orders of equivalent sources among the segments (bit o: order o).
static int ff_orders(const mfs_ctx *ctx, const mfs_ctx::FarField &F, const std::vector<int> &segs) {
    int mask = 0;
    for (int sg : segs)
        if (sg >= ctx->P && sg < ctx->P + FF_NORD * F.nodes) mask |= 1 << ((sg - ctx->P) / F.nodes);
    return mask;
}

static std::vector<int> suspension_of_bodies(const mfs_ctx *ctx) {
    std::vector<int> sus(ctx->P);
    for (int sp = 0; sp < ctx->S; ++sp)
        for (int b = ctx->body_off[sp]; b < ctx->body_off[sp + 1]; ++b) sus[b] = sp;
    return sus;
}

using FFListPlan = mfs_ctx::FarField::ListPlan;

// The plan of the upward sums for one pair-kernel variant: each node's check points against its
// descendant bodies' proxy points (one group per node, tiles never span two nodes).
mfs_status ff_up_plan(mfs_ctx *ctx, mfs_ctx::FarField &F, int variant, FFListPlan **out) {
    auto it = F.up.find(variant);
    if (it == F.up.end()) {
        FFListPlan lp;
        const int nodes = F.nodes;
        std::vector<long long> blocks;
        std::vector<int> recs, toff(nodes + 1), cuts(nodes + 1);
        ff_segments(F, blocks, recs);
        for (int n = 0; n <= nodes; ++n) {
            toff[n] = n * FF_NC;
            cuts[n] = n;
        }
        CKS(build_plan_lists(ctx, variant, 1, toff, ctx->P, cuts, blocks, recs,
                             [&](int g0, int g1, std::vector<int> &segs) {
                                 for (int n = g0; n <= g1; ++n)
                                     for (int q = F.tree.nodes[n].first;
                                          q < F.tree.nodes[n].first + F.tree.nodes[n].count; ++q)
                                         segs.push_back(q);
                             },
                             lp.p, &lp.seg, &lp.cum, lp.pairs));
        it = F.up.emplace(variant, lp).first;
    }
    *out = &it->second;
    return MFS_OK;
}

// The order-0 plan at the targets in tree order (the centre gradient's kernels): tiles stay inside a
// suspension and may span bodies, self pairs left out.
mfs_status ff_ev_plan(mfs_ctx *ctx, mfs_ctx::FarField &F, int variant, FFListPlan **out) {
    auto it = F.ev.find(variant);
    if (it == F.ev.end()) {
        FFListPlan lp;
        const int P = ctx->P;
        std::vector<long long> blocks;
        std::vector<int> recs, toff(P + 1, 0), cuts(ctx->body_off.begin(), ctx->body_off.end()), tb;
        ff_segments(F, blocks, recs);
        for (int q = 0; q < P; ++q) {
            const int b = F.tree.order[q];
            toff[q + 1] = toff[q] + ((*F.tgt_off)[b + 1] - (*F.tgt_off)[b]);
        }
        const std::vector<int> sus = suspension_of_bodies(ctx);
        CKS(build_plan_lists(ctx, variant, 0, toff, 0, cuts, blocks, recs,
                             [&](int g0, int g1, std::vector<int> &segs) {
                                 tb.clear();
                                 for (int q = g0; q <= g1; ++q) tb.push_back(F.tree.order[q]);
                                 ff_interaction_list(F.tree, F.tree.roots[sus[tb[0]]], tb, ctx->centres.data(),
                                                     F.rtgt.data(), ctx->opt.farfield_separation, 1, segs);
                             },
                             lp.p, &lp.seg, &lp.cum, lp.pairs));
        it = F.ev.emplace(variant, lp).first;
    }
    *out = &it->second;
    return MFS_OK;
}

// Bodies that share a cell (one list, one tile of FF_LOC_NC check points each).  More bodies fill a tile
// better (5 or 6 of them with the widest policies), but a node must be far from all of them: with 6 the
// bodies' own lists take 6.2e6 pairs a body (2000 ellipsoids, near bodies apart), with 2 they take 3.5e6
// and the two active target pairs per thread cost the cells' sums little (matvec 38.7 ms with 6, 36.4 with
// 2, 36.8 with 1; 37.3, 35.8 and 36.3 with the 5-pair policy: before the 256-target entry and equal tiles).
constexpr int FF_CELL = 2;

// The cells of FF_CELL consecutive tree positions (cut at suspensions) and their lists.
static const mfs_ctx::FarField::Cells &ff_cells(mfs_ctx *ctx, mfs_ctx::FarField &F) {
    mfs_ctx::FarField::Cells &c = F.cells;
    if (!c.first.empty()) return c;
    c.cell_of.resize(ctx->P);
    c.direct.resize(ctx->P);
    std::vector<int> tb;
    std::vector<std::vector<int>> direct;
    for (int sp = 0; sp < ctx->S; ++sp)
        for (int q0 = ctx->body_off[sp]; q0 < ctx->body_off[sp + 1]; q0 += FF_CELL) {
            const int q1 = std::min(q0 + FF_CELL, ctx->body_off[sp + 1]);
            tb.clear();
            for (int q = q0; q < q1; ++q) tb.push_back(F.tree.order[q]);
            c.local.emplace_back();
            ff_cell_lists(F.tree, F.tree.roots[sp], tb, ctx->centres.data(), F.rtgt.data(),
                          ctx->opt.farfield_separation, (double)F.ntgt / ctx->P, c.local.back(), direct);
            c.any_local = c.any_local || !c.local.back().empty();
            for (int q = q0; q < q1; ++q) {
                c.cell_of[q] = (int)c.first.size();
                c.direct[q].swap(direct[q - q0]);
            }
            c.first.push_back(q0);
        }
    c.first.push_back(ctx->P);
    return c;
}

// The plan of the sums at the bodies' local check points (one tile and one list per cell).
mfs_status ff_loc_plan(mfs_ctx *ctx, mfs_ctx::FarField &F, int variant, FFListPlan **out) {
    auto it = F.loc.find(variant);
    if (it == F.loc.end()) {
        FFListPlan lp;
        const int P = ctx->P;
        const auto &cells = ff_cells(ctx, F);
        std::vector<long long> blocks;
        std::vector<int> recs, toff(P + 1);
        ff_segments(F, blocks, recs);
        for (int q = 0; q <= P; ++q) toff[q] = q * FF_LOC_NC;
        CKS(build_plan_lists(ctx, variant, 1, toff, 0, cells.first, blocks, recs,
                             [&](int g0, int, std::vector<int> &segs) {
                                 segs = cells.local[cells.cell_of[g0]];
                                 lp.orders |= ff_orders(ctx, F, segs);
                             },
                             lp.p, &lp.seg, &lp.cum, lp.pairs));
        it = F.loc.emplace(variant, lp).first;
    }
    *out = &it->second;
    return MFS_OK;
}

// The plan of the final sums at the targets (tree order).  With local expansions every tile holds one
// body's targets and that body's own list; without, tiles span bodies and share the list of them all.
mfs_status ff_direct_plan(mfs_ctx *ctx, mfs_ctx::FarField &F, int variant, int include_self, FFListPlan **out) {
    const int key = variant * 2 + include_self;
    auto it = F.direct.find(key);
    if (it == F.direct.end()) {
        FFListPlan lp;
        const int P = ctx->P;
        std::vector<long long> blocks;
        std::vector<int> recs, toff(P + 1, 0), cuts, tb;
        ff_segments(F, blocks, recs);
        for (int q = 0; q < P; ++q) {
            const int b = F.tree.order[q];
            toff[q + 1] = toff[q] + ((*F.tgt_off)[b + 1] - (*F.tgt_off)[b]);
        }
        if (F.use_local) {
            const auto &cells = ff_cells(ctx, F);
            for (int q = 0; q <= P; ++q) cuts.push_back(q);
            CKS(build_plan_lists(ctx, variant, include_self, toff, 0, cuts, blocks, recs,
                                 [&](int g0, int, std::vector<int> &segs) {
                                     segs = cells.direct[g0];
                                     if (include_self) segs.push_back(g0);
                                     lp.orders |= ff_orders(ctx, F, segs);
                                 },
                                 lp.p, &lp.seg, &lp.cum, lp.pairs));
        } else {
            cuts.assign(ctx->body_off.begin(), ctx->body_off.end());
            const std::vector<int> sus = suspension_of_bodies(ctx);
            CKS(build_plan_lists(ctx, variant, include_self, toff, 0, cuts, blocks, recs,
                                 [&](int g0, int g1, std::vector<int> &segs) {
                                     tb.clear();
                                     for (int q = g0; q <= g1; ++q) tb.push_back(F.tree.order[q]);
                                     ff_ordered_list(F.tree, F.tree.roots[sus[tb[0]]], tb, ctx->centres.data(),
                                                     F.rtgt.data(), ctx->opt.farfield_separation, !include_self,
                                                     segs);
                                     lp.orders |= ff_orders(ctx, F, segs);
                                 },
                                 lp.p, &lp.seg, &lp.cum, lp.pairs));
        }
        it = F.direct.emplace(key, lp).first;
    }
    *out = &it->second;
    return MFS_OK;
}

// One pair-kernel launch on the far-field geometry, bracketed by profiling events like pair_apply's.
mfs_status ff_launch(mfs_ctx *ctx, int variant, const PairGeom &g, const PairWork &w, cudaStream_t st) {
    if (w.total_units == 0) return MFS_OK;
    const size_t slot = 2 * (size_t)ctx->pair_launches;
    if (ctx->opt.profile) {
        while (ctx->pev.size() < slot + 2) {
            cudaEvent_t e;
            CK(cudaEventCreate(&e));
            ctx->pev.push_back(e);
        }
        CK(cudaEventRecord(ctx->pev[slot], st));
    }
    CK(pair_launch(variant, g, w, ctx->err_d, st));
    if (ctx->opt.profile) CK(cudaEventRecord(ctx->pev[slot + 1], st));
    ctx->launches += 1;
    ctx->pair_launches += 1;
    return MFS_OK;
}

// The geometry of a far-field launch: the tree-ordered centres and the segments' record ranges.
static PairGeom ff_geom(const mfs_ctx::FarField &F, const FFListPlan &lp) {
    PairGeom g;
    g.lst_seg = lp.seg;
    g.lst_cum = lp.cum;
    g.src = F.rec;
    g.src_off = nullptr;
    g.blk_off = nullptr;
    g.centres = F.centres;
    g.seg_rec0 = F.seg_rec0;
    g.seg_rec1 = F.seg_rec1;
    return g;
}

// C [rows][D n] = A [rows][D k] B [D k][D n] in FP64 (the far field's fits; the context's D).
static cudaError_t ff_fit(mfs_ctx *ctx, mfs_ctx::FarField &F, int rows, int n, int k, const double *A, const double *B,
                          double *C, cudaStream_t st) {
    const int D = ctx->D;
    return gemm_rm64_splitk(rows, D * n, D * k, gemm_rm64_chunks(rows, D * n, D * k, ctx->sm_count), A, B,
                            F.fit_chunks, C, st);
}

// The pair-kernel entry for the sums at check points, whose tiles hold 256 targets (a node, a cell): the
// packed entry of exactly that tile where the table has one (1, 2 and 4 right-hand sides), whose warps have
// no inactive target pairs; else the entry of the other sums.  One right-hand side: 12 warps per SM where
// the widest entries keep 8 with two of their six target pairs active; one matvec of 2000 ellipsoids 33.2 ->
// 31.7 ms (entry <1,6,64> for the rest), 600: 5.52 -> 5.26 ms.  Two and four, one pair sum: 500 ellipsoids
// (M = 839) 11.48 -> 11.24 and 20.25 -> 20.07 ms, 400 spheres (M = 600) 4.73 -> 4.62 and 8.34 -> 8.26 ms.
static int ff_check_variant(int D, int nrhs, int variant) {
    int count = 0;
    const PairVariant *vv = pair_variants(&count);
    if (!vv[variant].packed) return variant;
    for (int i = 0; i < count; ++i)
        if (!vv[i].grad && !vv[i].comp && vv[i].packed && vv[i].D == D && vv[i].nrhs == nrhs && D == 3 &&
            vv[i].NT == 64 && vv[i].tile_targets == FF_NC)
            return i;
    return variant;
}

// The upward step of the treecode: the sources (records in the layout of `variant`, packed into
// F.rec) summed at every node's check points over the node's descendant bodies, then the node's
// equivalent strengths F.mu = (FP64 product with the pseudo-inverse) scaled by the radius.
static mfs_status ff_upward(mfs_ctx *ctx, mfs_ctx::FarField &F, int variant, const double *strength, int nrhs,
                            cudaStream_t st) {
    FFListPlan *pl = nullptr;
    const int cv = ff_check_variant(ctx->D, nrhs, variant);
    CKS(ff_up_plan(ctx, F, cv, &pl));
    int vc = 0;
    const PairVariant *vv = pair_variants(&vc);
    const int D = ctx->D, nodes = F.nodes;
    if (pair_record_floats(D, nrhs, vv[variant].packed) > F.rec_floats) {
        ctx->last_error = "far field: record layout larger than its buffer";
        return MFS_ERR_INVALID_ARG;
    }
    CK(pack_sources(D, nrhs, vv[variant].packed, F.src_pos, F.rec_pt, strength, F.nsrc, F.nrec, F.rec, st));
    PairGeom g = ff_geom(F, *pl);
    g.tgt = F.chk_pos;
    g.ntargets = nodes * FF_NC;
    const PairWork wu = work_of(pl->p);
    CKS(ff_launch(ctx, cv, g, wu, st));
    CK(pair_epilogue(D, nrhs, wu, nullptr, 0.0, 1.0, F.ucheck, nodes * FF_NC, st));
    CK(ff_fit(ctx, F, nrhs * nodes, FF_NE, FF_NC, F.ucheck, F.mat->PinvT, F.mu, st));
    CK(ff_scale(F.mu, F.re, nodes, D * FF_NE, nrhs, st));
    ctx->launches += 4;
    return MFS_OK;
}

// out = beta * base + scale * (pair sum of strengths) through the treecode, results in the caller's
// target order: the upward step, the lower orders of the equivalent strengths, the far cells' field at
// the bodies' local check points and the local sources that match it, then the sums at the targets.
//
// What bounds it is the number of pairs.  With order-0 lists at all targets a body of 2000 Type T
// ellipsoids (839 targets) saw about 850 nodes x 196 points: 1.4e8 pairs, 96 % of a matvec's 162 ms.
// Fewer points for distant nodes (FF_ORD_*) and 128 check points in place of the body's targets for
// everything beyond FF_LOC_GAP leave 2.1e10 pairs per sum for 1000 ellipsoids (1.0e11 before), and a
// matvec of 2000 takes 31.4 ms (162); the result is as close to the exact sums as before (400
// ellipsoids: white-noise strengths 1.13e-7, 1.28e-7 before; of one direction 1.8e-8, 2.0e-8 before).
mfs_status ff_pair_apply(mfs_ctx *ctx, mfs_ctx::FarField &F, int variant, const double *strength, double *out,
                         const double *base, double beta, double scale, int nrhs, int include_self, cudaStream_t st) {
    FFListPlan *pl = nullptr, *ll = nullptr;
    CKS(ff_direct_plan(ctx, F, variant, include_self, &pl));
    int vc = 0;
    const PairVariant *vv = pair_variants(&vc);
    const int D = ctx->D, nodes = F.nodes, P = ctx->P, layout = vv[variant].packed;
    const size_t REC = pair_record_floats(D, nrhs, layout);
    // local expansions, and the orders that the lists hold (a small cluster needs few of them)
    const bool local = F.use_local && F.cells.any_local;
    const int cv = ff_check_variant(D, nrhs, variant);
    if (local) CKS(ff_loc_plan(ctx, F, cv, &ll));
    const int orders = pl->orders | (local ? ll->orders : 0);
    CKS(ff_upward(ctx, F, variant, strength, nrhs, st));
    PackSets sets;
    for (int o = 0; o < FF_NORD && (orders >> o) != 0; ++o) {
        const int n = FF_ORD_N[o];
        if (o > 0) {
            CK(ff_fit(ctx, F, nrhs * nodes, n, FF_ORD_N[o - 1], o == 1 ? F.mu : F.ord_mu[o - 1], F.mat->ordT[o],
                      F.ord_mu[o], st));
            ctx->launches += 1;
        }
        if ((orders >> o) & 1)
            sets.add(nodes * n, o == 0 ? F.eq_pos : F.ord_pos[o], o == 0 ? F.mu : F.ord_mu[o],
                     F.rec + F.ord_rec[o] * REC);
    }
    CK(pack_sets(D, nrhs, layout, sets, st));
    ctx->launches += 1;
    if (local) {
        PairGeom g = ff_geom(F, *ll);
        g.tgt = F.lchk_pos;
        g.ntargets = P * FF_LOC_NC;
        const PairWork wl = work_of(ll->p);
        CKS(ff_launch(ctx, cv, g, wl, st));
        CK(pair_epilogue(D, nrhs, wl, nullptr, 0.0, 1.0, F.ulocal, P * FF_LOC_NC, st));
        // The constant and linear part of the far field at a body stay FP64 and go to the targets in the last
        // epilogue; the local sources carry the rest.  Strengths of one direction or in long waves give a far
        // field of little else, and its sum over 96 FP32 records rounded every target by about 5e-8 of it
        // (one direction, 400 ellipsoids: 5.3e-8 off the exact sums; with this 1.8e-8, without local sources 2.0e-8).
        CK(ff_take_linear(D, F.ulocal, F.lchk_pos, F.rloc, P, nrhs, F.ufar, st));
        CK(ff_fit(ctx, F, nrhs * P, FF_LOC_N, FF_LOC_NC, F.ulocal, F.mat->locT, F.nu, st));
        CK(ff_scale(F.nu, F.rloc, P, D * FF_LOC_N, nrhs, st));
        PackSets loc;
        loc.add(P * FF_LOC_N, F.loc_pos, F.nu, F.rec + F.loc_rec * REC);
        CK(pack_sets(D, nrhs, layout, loc, st));
        ctx->launches += 5;
    }
    PairGeom g = ff_geom(F, *pl);
    g.tgt = F.tgt;
    g.ntargets = F.ntgt;
    PairWork we = work_of(pl->p);
    we.tperm = F.tperm;
    if (local) {
        we.far = F.ufar;  // every tile holds one body's targets (ff_direct_plan)
        we.far_tgt = F.tgt;
        we.nfar = P;
    }
    CKS(ff_launch(ctx, variant, g, we, st));
    CK(pair_epilogue(D, nrhs, we, base, beta, scale, out, F.ntgt, st));
    ctx->launches += 2;
    return MFS_OK;
}

// wt[h][t][c] = (float) v[h][perm[t]][c]: per-target weights in the tree's target order.
static __global__ void ff_gather_weights_kernel(const double *v, const int *perm, int n, int nrhs, float *wt) {
    const size_t total = (size_t)nrhs * n * 3;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const size_t h = e / ((size_t)n * 3), r = e % ((size_t)n * 3);
        const int t = (int)(r / 3), c = (int)(r % 3);
        wt[e] = (float)v[(h * n + perm[t]) * 3 + c];
    }
}

// The adjoint's pair gradient through the treecode, per target of F (scaled, FP64, caller's order):
//   out_t = scale * sum_h sum_{s not on t's body} grad_r (tw_h(t)^T G(r) sigma_h(s)),  r = x_t - y_s,
// with sigma the sources' strengths (near bodies directly, far nodes through the equivalent
// strengths fitted to sigma) and tw the targets' weights.  On the forward tree (targets the
// collocation points, tw = w, sigma = mu) it is the target side of the centre gradient; on the
// transposed tree (targets the proxy points, tw = mu, sigma = w) its source side with the sign
// reversed (G symmetric and even, so its gradient is odd).
mfs_status ff_grad_apply(mfs_ctx *ctx, mfs_ctx::FarField &F, int gv, const double *sigma, const double *tw, int nrhs,
                         double *out, cudaStream_t st) {
    const int fv = fp32_variant(ctx, 3, nrhs);  // the upward sums: the forward pair kernel
    FFListPlan *pg = nullptr;
    CKS(ff_ev_plan(ctx, F, gv, &pg));
    CKS(ff_upward(ctx, F, fv, sigma, nrhs, st));
    // records of the gradient kernel (plain layout): the sources, then the equivalent points
    const int REC = pair_record_floats(3, nrhs, 0), nodes = F.nodes;
    CK(pack_sources(3, nrhs, 0, F.src_pos, F.rec_pt, sigma, F.nsrc, F.nrec, F.rec, st));
    CK(pack_sources(3, nrhs, 0, F.eq_pos, F.eq_pt, F.mu, nodes * FF_NE, nodes * FF_NE, F.rec + (size_t)F.nrec * REC,
                    st));
    if (!F.wt) CK(ctx->alloc(&F.wt, (size_t)ctx->opt.max_rhs * F.ntgt * 3));
    ff_gather_weights_kernel<<<1024, 256, 0, st>>>(tw, F.tperm, F.ntgt, nrhs, F.wt);
    CK(cudaGetLastError());
    PairGeom g = ff_geom(F, *pg);
    g.tgt = F.tgt;
    g.ntargets = F.ntgt;
    g.tgt_w = F.wt;
    PairWork we = work_of(pg->p);
    we.tperm = F.tperm;
    we.src_grad = nullptr;  // segments are bodies and nodes here: no per-source-body reduction
    CKS(ff_launch(ctx, gv, g, we, st));
    CK(pair_epilogue(3, 1, we, nullptr, 0.0, kernel_scale(ctx), out, F.ntgt, st));
    ctx->launches += 5;
    return MFS_OK;
}

// pairs evaluated per right-hand side by one pair sum
double pair_count(mfs_ctx *ctx, int include_self) {
    double total = 0.0;
    for (int s = 0; s < ctx->S; ++s) {
        double sm = 0, sn = 0, self = 0;
        for (int k = ctx->body_off[s]; k < ctx->body_off[s + 1]; ++k) {
            const double m = ctx->tgt_off[k + 1] - ctx->tgt_off[k], n = ctx->src_off[k + 1] - ctx->src_off[k];
            sm += m;
            sn += n;
            self += m * n;
        }
        total += sm * sn - (include_self ? 0.0 : self);
    }
    return total;
}

// C [cols][n] = A [cols][k] B [k][n] in FP64 with the shape's split-K scratch.
cudaError_t gemm64(mfs_ctx *ctx, ShapeHost &sh, int cols, int n, int k, const double *A, const double *B, double *C,
                   cudaStream_t st) {
    return gemm_rm64_splitk(cols, n, k, gemm_rm64_chunks(cols, n, k, ctx->sm_count), A, B, sh.Pk64, C, st);
}

// lambda = (I - L) S_L^+ gamma (project) or S_L^+ gamma  (Eq. pseudo, Remark congruent)
// With pack_variant >= 0 the strengths' source records for that pair-kernel entry too (as pack_for).
mfs_status precond_apply_dev(mfs_ctx *ctx, const double *gamma, double *lambda, int project, int nrhs,
                             cudaStream_t st, int pack_variant = -1) {
    const int D = ctx->D;
    int vc = 0;
    const PairVariant *vv = pair_variants(&vc);
    for (auto &sh : ctx->shapes) {
        const int nb = (int)sh.bodies.size();
        if (nb == 0) continue;
        const int ncols = nb * nrhs;
        const FactorSet &fx = sh.fs[ctx->fset];
        const ShapeDev &sd = fx.dev;
        ScatterArgs sc;
        sc.col_body = sh.col_body;
        sc.col_rhs = sh.col_rhs;
        sc.body_off = ctx->src_off_d;
        sc.rot64 = ctx->rot64_d;
        sc.ncols = ncols;
        sc.dN = sd.dN;
        sc.sum_N = ctx->sumN;
        sc.out = lambda;
        if (pack_variant >= 0) {
            sc.rec = ctx->rec_d;
            sc.packed = vv[pack_variant].packed;
            sc.rec_floats = pair_record_floats(D, nrhs, sc.packed);
            sc.nrhs = nrhs;
            sc.rec_off = ctx->rec_off_d;
            sc.src_pos = ctx->src_pos_d;
            if (sc.rec_floats > ctx->rec_floats) {
                ctx->last_error = "source records larger than their buffer";
                return MFS_ERR_INVALID_ARG;
            }
        }
        if (ctx->opt.precision >= 1) {  // FP64 one-body apply (reference and mixed modes)
            CK(gather_rotate(D, gamma, ctx->sumM * D, sh.col_body, sh.col_rhs, ctx->tgt_off_d, ctx->rot64_d, ncols,
                             sd.dM, sh.A, sh.A64, st));
            CK(gemm64(ctx, sh, ncols, sd.r, sd.dM, sh.A64, sd.U64, sh.T64, st));
            CK(gemm64(ctx, sh, ncols, sd.dN, sd.r, sh.T64, project ? sd.Wp64 : sd.Wr64, sh.L64, st));
            sc.L64 = sh.L64;
        } else if (fx.tc_ready && fc_takes(D, ncols, sd.dM, sd.dN)) {  // few columns: warps on the factor rows
            CK(gather_rotate_hl(D, gamma, ctx->sumM * D, sh.col_body, sh.col_rhs, ctx->tgt_off_d, ctx->rot64_d, ncols,
                                sd.dM, sh.Gf, sh.ld1, st));
            CK(fc_apply(ncols, sd.r, sh.ld1, fx.Utp, fx.ut_stride, sh.Gf, sh.Tf, sh.ld2, st));
            CK(fc_apply(ncols, sd.dN, sh.ld2, project ? fx.Wptp : fx.Wrtp, fx.wt_stride, sh.Tf, sh.Lf, sd.dN, st));
            sc.P = sh.Lf;
            sc.S = 1;
        } else if (fx.tc_ready) {  // tensor cores: multi-piece TF32 tcgen05 GEMMs, double-float chunk sums
            const int np = sh.pieces;
            auto it = sh.amaps.find(ncols);
            if (it == sh.amaps.end()) {
                std::array<TcMap, 6> mp;
                const int bn = tc_gemm_bn(ncols, np);
                bool enc = true;
                for (int p = 0; p < np; ++p)
                    enc = enc && make_tc_map(mp[p], sh.Ap + p * sh.ap_stride, ncols, sh.ld1, bn) &&
                          make_tc_map(mp[3 + p], sh.Tp + p * sh.tp_stride, ncols, sh.ld2, bn);
                if (!enc) {
                    ctx->last_error = "tensor-map encoding for the tensor-core apply failed";
                    return MFS_ERR_CUDA;
                }
                it = sh.amaps.emplace(ncols, mp).first;
            }
            const std::array<TcMap, 6> &mp = it->second;
            // t = U^T g (Eq. pseudo): gathered columns as pieces, chunk sums re-cut into pieces of t
            CK(gather_rotate_pieces(D, gamma, ctx->sumM * D, sh.col_body, sh.col_rhs, ctx->tgt_off_d, ctx->rot64_d,
                                    ncols, sd.dM, sh.Ap, sh.ld1, sh.ap_stride, np, st));
            const int S1 = tc_gemm_chunks(ncols, sd.r, sd.dM, ctx->sm_count, np);
            CK(tc_gemm(np, fx.mU, mp.data(), ncols, sd.r, sd.dM, S1, sh.Ptc, ctx->err_d, st));
            CK(reduce_pieces(tc_gemm_sz(sd.dM, S1), ncols, sd.r, sh.Ptc, sh.Tp, sh.ld2, sh.tp_stride, np, st));
            // lambda = W t, the chunk sums added by the scatter
            const int S2 = tc_gemm_chunks(ncols, sd.dN, sd.r, ctx->sm_count, np);
            CK(tc_gemm(np, project ? fx.mWp : fx.mWr, mp.data() + 3, ncols, sd.dN, sd.r, S2, sh.Ptc, ctx->err_d, st));
            sc.P = sh.Ptc;
            sc.S = tc_gemm_sz(sd.r, S2);
            ctx->launches += 1;
        } else {
            CK(gather_rotate(D, gamma, ctx->sumM * D, sh.col_body, sh.col_rhs, ctx->tgt_off_d, ctx->rot64_d, ncols,
                             sd.dM, sh.A, nullptr, st));
            // t = U^T g (FP32 result), then lambda = W t kept in FP64 (split-K, compensated; Eq. pseudo)
            const int S1 = gemm_splitk_chunks(ncols, sd.r, sd.dM, ctx->sm_count);
            const int S2 = gemm_splitk_chunks(ncols, sd.dN, sd.r, ctx->sm_count);
            CK(gemm_splitk(ncols, sd.r, sd.dM, S1, sh.A, sd.U, sh.Pk, sh.Tm, nullptr, st));
            CK(gemm_splitk(ncols, sd.dN, sd.r, S2, sh.Tm, project ? sd.Wp : sd.Wr, sh.Pk, nullptr, sh.L64, st));
            sc.L64 = sh.L64;
            ctx->launches += 2;
        }
        CK(scatter_rotate(D, sc, st));
        ctx->launches += 4;
    }
    return MFS_OK;
}

// y = gamma + sum_{k' != k} S^(kk') (I - L^(k')) S_L^(k')+ gamma^(k')  (Eq. 2esysprec)
mfs_status matvec_dev(mfs_ctx *ctx, const double *gamma, double *y, int nrhs, cudaStream_t st) {
    // direct FP32 sums: the apply's scatter writes the pair kernel's records
    const bool direct = (ctx->opt.precision == 0 || ctx->opt.precision == 2) && !ctx->ff.ready;
    const int pack = direct ? forward_variant(ctx, nrhs) : -1;
    CKS(precond_apply_dev(ctx, gamma, ctx->lam_d, 1, nrhs, st, pack));
    CKS(pair_apply(ctx, ctx->lam_d, y, gamma, 1.0, 1.0, nrhs, 0, st, pack >= 0));
    return MFS_OK;
}

mfs_status ensure_gmres(mfs_ctx *ctx, int nrhs) {
    const long long n = (long long)nrhs * ctx->sumM * ctx->D;
    const int L = nrhs * ctx->S;
    const int m = std::min(ctx->opt.restart, ctx->opt.max_iter);
    if (ctx->gd.V && ctx->gd_n == (size_t)n && ctx->gd_L == L && ctx->gd_m == m) return MFS_OK;
    GmresDev &gd = ctx->gd;
    void *olds[] = {gd.V, gd.H, gd.cs, gd.sn, gd.g, gd.ibeta, gd.hbuf, gd.part, gd.normp, gd.active, (void *)gd.blk_lane,
                    (void *)gd.blk_off, (void *)gd.lane_blk, ctx->stat_d, ctx->w_d, ctx->b_d, ctx->x_d, ctx->vin_d};
    ctx->drop_graphs();  // they hold the old buffers' addresses
    for (void *p : olds) ctx->release(p);
    if (ctx->stat_h) cudaFreeHost(ctx->stat_h);
    ctx->vin_d = ctx->w_d = ctx->b_d = ctx->x_d = nullptr;
    ctx->stat_d = ctx->stat_h = nullptr;
    gd = GmresDev{};
    ctx->gd_n = 0;  // until every buffer below exists: a build that runs out of memory half-way is not taken for a whole one
    ctx->gd_L = ctx->gd_m = 0;
    gd.L = L;
    gd.m = m;
    gd.n = n;
    gd.tol = ctx->opt.gmres_tol;
    std::vector<long long> seg(L + 1), blk_off;
    std::vector<int> blk_lane, lane_blk;
    for (int h = 0; h < nrhs; ++h)
        for (int s = 0; s < ctx->S; ++s) {
            const int l = h * ctx->S + s;
            seg[l] = (long long)h * ctx->sumM * ctx->D + (long long)ctx->tgt_off[ctx->body_off[s]] * ctx->D;
        }
    seg[L] = n;
    gd.clusters = gmres_plan_blocks(seg, ctx->sm_count, blk_lane, blk_off, lane_blk) ? 1 : 0;
    gd.sms = ctx->sm_count;
    gd.nblk = (int)blk_lane.size();
    int *bl = nullptr, *lb = nullptr;
    long long *bo = nullptr;
    CK(ctx->alloc(&bl, blk_lane.size()));
    gd.blk_lane = bl;
    CK(ctx->alloc(&bo, blk_off.size()));
    gd.blk_off = bo;
    CK(ctx->alloc(&lb, lane_blk.size()));
    gd.lane_blk = lb;
    CK(cudaMemcpy(bl, blk_lane.data(), sizeof(int) * blk_lane.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(bo, blk_off.data(), sizeof(long long) * blk_off.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(lb, lane_blk.data(), sizeof(int) * lane_blk.size(), cudaMemcpyHostToDevice));
    CK(ctx->alloc(&gd.V, (size_t)(m + 1) * n));
    CK(ctx->alloc(&gd.H, (size_t)L * (m + 1) * m));
    CK(ctx->alloc(&gd.cs, (size_t)L * m));
    CK(ctx->alloc(&gd.sn, (size_t)L * m));
    CK(ctx->alloc(&gd.g, (size_t)L * (m + 1)));
    CK(ctx->alloc(&gd.ibeta, L));
    CK(ctx->alloc(&gd.hbuf, (size_t)L * (m + 1)));
    CK(ctx->alloc(&gd.part, 2 * (size_t)gd.nblk * (m + 1)));
    CK(ctx->alloc(&gd.normp, gd.nblk));
    CK(ctx->alloc(&gd.active, L));
    // what a solve reports, in one block (one copy back): resid [L], iters [L], status [L], done, jcur,
    // and the blocks' arrival counter
    CK(ctx->alloc(&ctx->stat_d, ctx->stat_bytes(L)));
    CK(ctx->refuse_alloc() ? cudaErrorMemoryAllocation : cudaMallocHost((void **)&ctx->stat_h, ctx->stat_bytes(L)));
    CK(cudaMemset(ctx->stat_d, 0, ctx->stat_bytes(L)));
    gd.resid = reinterpret_cast<double *>(ctx->stat_d);
    gd.iters = reinterpret_cast<int *>(gd.resid + L);
    gd.status = gd.iters + L;
    gd.done = gd.status + L;
    gd.jcur = gd.done + 1;
    gd.arrive = reinterpret_cast<unsigned *>(gd.jcur + 1);
    CK(gmres_prepare(gd));
    CK(ctx->alloc(&ctx->vin_d, n));
    CK(ctx->alloc(&ctx->w_d, n));
    CK(ctx->alloc(&ctx->b_d, n));
    CK(ctx->alloc(&ctx->x_d, n));
    ctx->gd_n = n;
    ctx->gd_L = L;
    ctx->gd_m = m;
    return MFS_OK;
}

// ---------------------------------------------------------------------------
// Adjoint (transposed) operators
// ---------------------------------------------------------------------------
// dst[c][r] = src[r][c], FP64 (setup of the FP64 adjoint's factor transposes).
static __global__ void transpose64_kernel(const double *src, int rows, int cols, double *dst) {
    const size_t n = (size_t)rows * cols;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        dst[(i % cols) * rows + i / cols] = src[i];
}

// The transposed geometry: proxy points as targets (float4 with body bits), collocation points
// as sources packed into records with their own padded offsets; plus adjoint scratch; with
// farfield = 1 the treecode of the transposed sums (collocation sources, proxy targets).
mfs_status ensure_transposed(mfs_ctx *ctx) {
    if (ctx->trans_ready) return MFS_OK;
    const int P = ctx->P, R = ctx->opt.max_rhs;
    ctx->src_body.resize(ctx->sumN);
    for (int k = 0; k < P; ++k)
        for (int q = ctx->src_off[k]; q < ctx->src_off[k + 1]; ++q) ctx->src_body[q] = k;
    ctx->recT_off.assign(P + 1, 0);
    ctx->blkT_off.assign(P + 1, 0);
    for (int k = 0; k < P; ++k) {
        const int mpad = (ctx->tgt_off[k + 1] - ctx->tgt_off[k] + 3) / 4 * 4;
        ctx->recT_off[k + 1] = ctx->recT_off[k] + mpad;
        ctx->blkT_off[k + 1] = ctx->blkT_off[k] + (mpad + MFS_BS - 1) / MFS_BS;
    }
    ctx->nrecT = ctx->recT_off[P];
    std::vector<int> rec_pt(ctx->nrecT, -1);
    for (int k = 0; k < P; ++k)
        for (int i = 0; i < ctx->tgt_off[k + 1] - ctx->tgt_off[k]; ++i) rec_pt[ctx->recT_off[k] + i] = ctx->tgt_off[k] + i;
    // proxy targets: rotated local coordinates with the body id in w
    std::vector<float4> tp(ctx->sumN);
    std::vector<float> s4(4 * (size_t)ctx->sumN);
    CK(cudaMemcpy(tp.data(), ctx->src_pos_d, sizeof(float4) * ctx->sumN, cudaMemcpyDeviceToHost));
    for (int q = 0; q < ctx->sumN; ++q) {
        int k = ctx->src_body[q];
        float kb;
        std::memcpy(&kb, &k, sizeof(float));
        tp[q].w = kb;
    }
    const int recf = std::max(pair_record_floats(3, R, 0), pair_record_floats(3, R, 1));
    ctx->recT_floats = recf;
    CK(ctx->alloc(&ctx->tgtT_pos_d, ctx->sumN));
    CK(ctx->alloc(&ctx->recT_d, (size_t)ctx->nrecT * recf));
    CK(ctx->alloc(&ctx->recT_off_d, P + 1));
    CK(ctx->alloc(&ctx->rec_ptT_d, ctx->nrecT));
    CK(ctx->alloc(&ctx->blkT_off_d, P + 1));
    CK(ctx->alloc(&ctx->tmpM_d, (size_t)R * ctx->sumM * 3));
    CK(ctx->alloc(&ctx->gradT_d, (size_t)ctx->sumM * 3));
    CK(ctx->alloc(&ctx->src_grad_d, (size_t)P * 3));
    CK(ctx->alloc(&ctx->six_d, (size_t)R * P * 6));
    CK(ctx->alloc(&ctx->w32_d, (size_t)R * ctx->sumM * 3));
    CK(ctx->alloc(&ctx->eye6_d, (size_t)ctx->nshapes * 36));
    CK(cudaMemcpy(ctx->tgtT_pos_d, tp.data(), sizeof(float4) * ctx->sumN, cudaMemcpyHostToDevice));
    CK(cudaMemset(ctx->recT_d, 0, sizeof(float) * (size_t)ctx->nrecT * recf));
    CK(cudaMemcpy(ctx->recT_off_d, ctx->recT_off.data(), sizeof(int) * (P + 1), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->rec_ptT_d, rec_pt.data(), sizeof(int) * ctx->nrecT, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->blkT_off_d, ctx->blkT_off.data(), sizeof(long long) * (P + 1), cudaMemcpyHostToDevice));
    std::vector<double> eye(36 * (size_t)ctx->nshapes, 0.0);
    for (int s = 0; s < ctx->nshapes; ++s)
        for (int i = 0; i < 6; ++i) eye[36 * s + 7 * i] = 1.0;
    CK(cudaMemcpy(ctx->eye6_d, eye.data(), sizeof(double) * eye.size(), cudaMemcpyHostToDevice));
    for (auto &sh : ctx->shapes) {  // transposed-apply buffers
        const int nb = (int)sh.bodies.size();
        if (nb == 0) continue;
        const int m = sh.fs[0].dev.dM, n = sh.fs[0].dev.dN;
        size_t need = 0;
        for (int h = 1; h <= R; ++h) {
            const int rows = h * nb;
            need = std::max(need, (size_t)gemm_splitk_chunks(rows, n, n, ctx->sm_count) * rows * n);
            need = std::max(need, (size_t)gemm_splitk_chunks(rows, m, n, ctx->sm_count) * rows * m);
        }
        CK(ctx->alloc(&sh.PkT, need));
        FactorSet &fx = sh.fs[0];
        if (!fx.tc_ready) CK(ctx->alloc(&sh.O64, (size_t)R * nb * m));
        if (fx.tc_ready) {  // tensor cores: the factor planes transposed (exact), their maps, chunk results
            const int np = sh.pieces;
            fx.un_stride = (size_t)m * sh.ld2;
            CK(ctx->alloc(&fx.Un, 2 * fx.un_stride));
            CK(ctx->alloc(&fx.WpT, 2 * fx.wt_stride));
            CK(ctx->alloc(&fx.WrT, 2 * fx.wt_stride));
            // U^T planes [r][ld1] -> U planes [dM][ld2]; W planes [dN][ld2] -> W^T planes [r][ld2]
            CK(transpose_pieces(fx.Utp, n, m, sh.ld1, fx.ut_stride, fx.Un, sh.ld2, fx.un_stride, 2, 0));
            CK(transpose_pieces(fx.Wptp, n, n, sh.ld2, fx.wt_stride, fx.WpT, sh.ld2, fx.wt_stride, 2, 0));
            CK(transpose_pieces(fx.Wrtp, n, n, sh.ld2, fx.wt_stride, fx.WrT, sh.ld2, fx.wt_stride, 2, 0));
            CK(cudaDeviceSynchronize());
            bool enc = true;
            for (int p = 0; p < 2; ++p)
                enc = enc && make_tc_map(fx.mUn[p], fx.Un + p * fx.un_stride, m, sh.ld2, 128) &&
                      make_tc_map(fx.mWpT[p], fx.WpT + p * fx.wt_stride, n, sh.ld2, 128) &&
                      make_tc_map(fx.mWrT[p], fx.WrT + p * fx.wt_stride, n, sh.ld2, 128);
            if (!enc) {
                ctx->last_error = "tensor-map encoding for the transposed tensor-core apply failed";
                return MFS_ERR_CUDA;
            }
            size_t needT = 0;
            for (int h = 1; h <= R; ++h) {
                const int cols = h * nb;
                needT = std::max(needT, (size_t)tc_gemm_sz(n, tc_gemm_chunks(cols, n, n, ctx->sm_count, np)) * cols * n);
                needT = std::max(needT, (size_t)tc_gemm_sz(n, tc_gemm_chunks(cols, m, n, ctx->sm_count, np)) * cols * m);
            }
            CK(ctx->alloc(&sh.PtcT, needT));
            fx.tcT_ready = true;
        }
    }
    if (ctx->opt.precision == 1) {  // the FP64 transposed sums and one-body apply
        std::vector<double> tl(3 * (size_t)ctx->sumM), c4(4 * (size_t)ctx->sumM);
        CK(cudaMemcpy(tl.data(), ctx->tgt_local64_d, sizeof(double) * tl.size(), cudaMemcpyDeviceToHost));
        for (int i = 0; i < ctx->sumM; ++i) {
            for (int a = 0; a < 3; ++a) c4[4 * (size_t)i + a] = tl[3 * (size_t)i + a];
            c4[4 * (size_t)i + 3] = (double)ctx->tgt_body[i];
        }
        std::vector<int> cb(P), ce(P);
        for (int sp = 0; sp < ctx->S; ++sp)
            for (int k = ctx->body_off[sp]; k < ctx->body_off[sp + 1]; ++k) {
                cb[k] = ctx->tgt_off[ctx->body_off[sp]];
                ce[k] = ctx->tgt_off[ctx->body_off[sp + 1]];
            }
        CK(ctx->alloc(&ctx->src_body_d, ctx->sumN));
        CK(ctx->alloc(&ctx->colloc4_d, c4.size()));
        CK(ctx->alloc(&ctx->colT_begin_d, P));
        CK(ctx->alloc(&ctx->colT_end_d, P));
        CK(cudaMemcpy(ctx->src_body_d, ctx->src_body.data(), sizeof(int) * ctx->sumN, cudaMemcpyHostToDevice));
        CK(cudaMemcpy(ctx->colloc4_d, c4.data(), sizeof(double) * c4.size(), cudaMemcpyHostToDevice));
        CK(cudaMemcpy(ctx->colT_begin_d, cb.data(), sizeof(int) * P, cudaMemcpyHostToDevice));
        CK(cudaMemcpy(ctx->colT_end_d, ce.data(), sizeof(int) * P, cudaMemcpyHostToDevice));
        for (auto &sh : ctx->shapes) {
            if (sh.bodies.empty()) continue;
            ShapeDev &sd = sh.fs[0].dev;
            CK(ctx->alloc(&sd.UT64, (size_t)sd.dM * sd.r));
            CK(ctx->alloc(&sd.WpT64, (size_t)sd.r * sd.dN));
            CK(ctx->alloc(&sd.WrT64, (size_t)sd.r * sd.dN));
            transpose64_kernel<<<1024, 256>>>(sd.U64, sd.dM, sd.r, sd.UT64);
            transpose64_kernel<<<1024, 256>>>(sd.Wp64, sd.r, sd.dN, sd.WpT64);
            transpose64_kernel<<<1024, 256>>>(sd.Wr64, sd.r, sd.dN, sd.WrT64);
            CK(cudaGetLastError());
        }
        CK(cudaDeviceSynchronize());
    }
    if (ctx->opt.farfield) {
        auto &F = ctx->ffT;
        F.src_colloc = true;
        F.src_pos = ctx->tgt_pos_d;
        F.rec_pt = ctx->rec_ptT_d;
        F.nsrc = ctx->sumM;
        F.nrec = ctx->nrecT;
        F.rec_off = &ctx->recT_off;
        F.tgt_pos = ctx->tgtT_pos_d;
        F.tgt_off = &ctx->src_off;
        F.ntgt = ctx->sumN;
        CKS(ff_setup(ctx, F, 0));
    }
    ctx->trans_ready = true;
    return MFS_OK;
}

// z^(k') = sum_k S^(kk')^T w^(k) at the proxy points (the Stokeslet is symmetric and even in r),
// self pairs included or not.  w: [nrhs][sum_M][3], z: [nrhs][sum_N][3], both FP64 on the device.
mfs_status pair_apply_T(mfs_ctx *ctx, const double *w, double *z, int nrhs, int include_self, cudaStream_t st) {
    if (ctx->opt.precision == 1) {  // FP64 reference: the plain FP64 loops with the roles swapped
        const int S = fp64_chunks(ctx, ctx->sumN, true);
        CK(pair_sum_fp64(3, nrhs, S, ctx->src_local64_d, ctx->src_body_d, ctx->sumN, ctx->colloc4_d, ctx->sumM,
                         ctx->colT_begin_d, ctx->colT_end_d, ctx->tgt_off_d, ctx->centres_d, w, include_self,
                         ctx->raw_d, st));
        const size_t n = (size_t)nrhs * ctx->sumN * 3;
        combine_raw_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ctx->raw_d, nullptr, 0.0, kernel_scale(ctx), z,
                                                                        n, S);
        CK(cudaGetLastError());
        ctx->launches += 2;
        return MFS_OK;
    }
    const int variant = fp32_variant(ctx, 3, nrhs);
    if (ctx->ffT.ready)
        return ff_pair_apply(ctx, ctx->ffT, variant, w, z, nullptr, 0.0, kernel_scale(ctx), nrhs, include_self, st);
    int vc = 0;
    const PairVariant *vv = pair_variants(&vc);
    if (pair_record_floats(3, nrhs, vv[variant].packed) > ctx->recT_floats) {
        ctx->last_error = "transposed pair sum: record layout larger than its buffer";
        return MFS_ERR_INVALID_ARG;
    }
    PairPlan *plan = nullptr;
    CKS(get_plan(ctx, variant, include_self, &plan, 1));
    CK(pack_sources(3, nrhs, vv[variant].packed, ctx->tgt_pos_d, ctx->rec_ptT_d, w, ctx->sumM, ctx->nrecT,
                    ctx->recT_d, st));
    PairGeom g;
    g.tgt = ctx->tgtT_pos_d;
    g.src = ctx->recT_d;
    g.src_off = ctx->recT_off_d;
    g.blk_off = ctx->blkT_off_d;
    g.centres = ctx->centres_d;
    g.ntargets = ctx->sumN;
    const PairWork wk = work_of(*plan);
    if (wk.total_units > 0) {
        CK(pair_launch(variant, g, wk, ctx->err_d, st));
        ctx->launches += 1;
    }
    CK(pair_epilogue(3, nrhs, wk, nullptr, 0.0, kernel_scale(ctx), z, ctx->sumN, st));
    ctx->launches += 2;
    return MFS_OK;
}

// out^(k) = ((I - L^(k)) S_L^(k)+)^T z^(k) = R_M U W_p R_N^T z (project) or (S_L^(k)+)^T z = R_M U W_r R_N^T z,
// z [nrhs][sum_N][3] -> out [nrhs][sum_M][3] (transposes of the two-step apply, Eq. pseudo).
// base + that, when base [nrhs][sum_M][3] is given.
mfs_status precondT_dev(mfs_ctx *ctx, const double *z, double *out, int project, int nrhs, cudaStream_t st,
                        const double *base = nullptr) {
    for (auto &sh : ctx->shapes) {
        const int nb = (int)sh.bodies.size();
        if (nb == 0) continue;
        const int ncols = nb * nrhs;
        const FactorSet &fx = sh.fs[0];
        const ShapeDev &sd = fx.dev;
        ScatterArgs sc;
        sc.col_body = sh.col_body;
        sc.col_rhs = sh.col_rhs;
        sc.body_off = ctx->tgt_off_d;
        sc.rot64 = ctx->rot64_d;
        sc.ncols = ncols;
        sc.dN = sd.dM;
        sc.sum_N = ctx->sumM;
        sc.out = out;
        sc.base = base;
        if (ctx->opt.precision == 1) {
            // FP64 reference: out = R_M U (W (R_N^T z)) with the transposed FP64 factors
            CK(gather_rotate(3, z, ctx->sumN * 3, sh.col_body, sh.col_rhs, ctx->src_off_d, ctx->rot64_d, ncols, sd.dN,
                             sh.A, sh.A64, st));
            CK(gemm64(ctx, sh, ncols, sd.r, sd.dN, sh.A64, project ? sd.WpT64 : sd.WrT64, sh.T64, st));
            CK(gemm64(ctx, sh, ncols, sd.dM, sd.r, sh.T64, sd.UT64, sh.O64, st));
            sc.L64 = sh.O64;
        } else if (fx.tcT_ready && ctx->opt.precision == 0 && fc_takes(3, ncols, sd.dM, sd.dN)) {
            // few columns, as the forward apply: x = W^T (R_N^T z), out = R_M U x
            CK(gather_rotate_hl(3, z, ctx->sumN * 3, sh.col_body, sh.col_rhs, ctx->src_off_d, ctx->rot64_d, ncols, sd.dN,
                                sh.Tf, sh.ld2, st));
            CK(fc_apply(ncols, sd.r, sh.ld2, project ? fx.WpT : fx.WrT, fx.wt_stride, sh.Tf, sh.Xf, sh.ld2, st));
            CK(fc_apply(ncols, sd.dM, sh.ld2, fx.Un, fx.un_stride, sh.Xf, sh.Lf, sd.dM, st));
            sc.P = sh.Lf;
            sc.S = 1;
        } else if (fx.tcT_ready && ctx->opt.precision == 0) {
            // tensor cores, as the forward apply: x = W^T (R_N^T z) with the K = dN column pieces in Tp,
            // x cut back into pieces (same layout, Tp reused), out = R_M U x
            const int np = sh.pieces;
            auto it = sh.amaps.find(ncols);
            if (it == sh.amaps.end()) {
                std::array<TcMap, 6> mp;
                const int bn = tc_gemm_bn(ncols, np);
                bool enc = true;
                for (int p = 0; p < np; ++p)
                    enc = enc && make_tc_map(mp[p], sh.Ap + p * sh.ap_stride, ncols, sh.ld1, bn) &&
                          make_tc_map(mp[3 + p], sh.Tp + p * sh.tp_stride, ncols, sh.ld2, bn);
                if (!enc) {
                    ctx->last_error = "tensor-map encoding for the tensor-core apply failed";
                    return MFS_ERR_CUDA;
                }
                it = sh.amaps.emplace(ncols, mp).first;
            }
            const TcMap *colmaps = it->second.data() + 3;
            CK(gather_rotate_pieces(3, z, ctx->sumN * 3, sh.col_body, sh.col_rhs, ctx->src_off_d, ctx->rot64_d, ncols,
                                    sd.dN, sh.Tp, sh.ld2, sh.tp_stride, np, st));
            const int S1 = tc_gemm_chunks(ncols, sd.r, sd.dN, ctx->sm_count, np);
            CK(tc_gemm(np, project ? fx.mWpT : fx.mWrT, colmaps, ncols, sd.r, sd.dN, S1, sh.PtcT, ctx->err_d, st));
            CK(reduce_pieces(tc_gemm_sz(sd.dN, S1), ncols, sd.r, sh.PtcT, sh.Tp, sh.ld2, sh.tp_stride, np, st));
            const int S2 = tc_gemm_chunks(ncols, sd.dM, sd.r, ctx->sm_count, np);
            CK(tc_gemm(np, fx.mUn, colmaps, ncols, sd.dM, sd.r, S2, sh.PtcT, ctx->err_d, st));
            sc.P = sh.PtcT;
            sc.S = tc_gemm_sz(sd.r, S2);
            ctx->launches += 1;
        } else {
            CK(gather_rotate(3, z, ctx->sumN * 3, sh.col_body, sh.col_rhs, ctx->src_off_d, ctx->rot64_d, ncols, sd.dN,
                             sh.A, nullptr, st));
            const int S1 = gemm_splitk_chunks(ncols, sd.r, sd.dN, ctx->sm_count);
            const int S2 = gemm_splitk_chunks(ncols, sd.dM, sd.r, ctx->sm_count);
            CK(gemm_splitk(ncols, sd.r, sd.dN, S1, sh.A, project ? sd.Wp : sd.Wr, sh.PkT, sh.Tm, nullptr, st, true));
            CK(gemm_splitk(ncols, sd.dM, sd.r, S2, sh.Tm, sd.U, sh.PkT, nullptr, sh.O64, st, true));
            sc.L64 = sh.O64;
            ctx->launches += 2;
        }
        CK(scatter_rotate(3, sc, st));
        ctx->launches += 4;
    }
    return MFS_OK;
}

// y = A^T w = w + [((I - L^(k')) S_L^(k')+)^T sum_{k != k'} S^(kk')^T w^(k)]_k'
mfs_status matvec_T_dev(mfs_ctx *ctx, const double *w, double *y, int nrhs, cudaStream_t st) {
    CKS(pair_apply_T(ctx, w, ctx->lam_d, nrhs, 0, st));
    return precondT_dev(ctx, ctx->lam_d, y, 1, nrhs, st, w);
}

struct SolveStats {
    int iters = 0, converged = 1, matvecs = 0, breakdown = 0;
    double resid = 0.0;
    int host_iters = 0;                              // iterations the host enqueued one by one
    const mfs_ctx::SolveGraph *graph = nullptr;      // the rest ran in it
};

// One GMRES iteration's matvec: w = A vin (or A^T vin).
mfs_status iteration_matvec(mfs_ctx *ctx, const double *vin, int nrhs, bool transposed, cudaStream_t st) {
    if (transposed) return matvec_T_dev(ctx, vin, ctx->w_d, nrhs, st);
    return matvec_dev(ctx, vin, ctx->w_d, nrhs, st);
}

// The loop of iterations as a CUDA graph: a while node whose body applies the matvec to vin,
// orthogonalises (Arnoldi, Givens; v_{j+1} to vin) and advances j, clearing the node's condition when
// every lane stopped or the basis is full.  Built on first use (the first iteration of that solve ran on
// the host loop, so every plan and tensor map the body needs exists) and kept per key; later solves run
// all their iterations in it.
mfs_status solve_graph(mfs_ctx *ctx, int nrhs, bool transposed, mfs_ctx::SolveGraph **out) {
    const int key = nrhs * 4 + ctx->fset * 2 + (transposed ? 1 : 0);
    auto it = ctx->graphs.find(key);
    if (it != ctx->graphs.end()) {
        *out = &it->second;
        return MFS_OK;
    }
    if (!ctx->cap_stream) CK(cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
    cudaStream_t st = ctx->cap_stream;  // records the body; nothing executes on it
    mfs_ctx::SolveGraph g;
    GmresDev &gd = ctx->gd;
    CK(cudaGraphCreate(&g.graph, 0));
    auto fail = [&](cudaError_t e) {
        cudaGetLastError();
        if (g.graph) cudaGraphDestroy(g.graph);
        ctx->last_error = std::string("CUDA graph of the GMRES loop: ") + cudaGetErrorString(e);
        return MFS_ERR_CUDA;
    };
    cudaGraphConditionalHandle cond;
    cudaError_t e = cudaGraphConditionalHandleCreate(&cond, g.graph, 1, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) return fail(e);
    // the parameter union has no default constructor: zeroed storage, then the conditional member
    alignas(cudaGraphNodeParams) unsigned char cp_raw[sizeof(cudaGraphNodeParams)];
    std::memset(cp_raw, 0, sizeof(cp_raw));
    cudaGraphNodeParams &cp = *reinterpret_cast<cudaGraphNodeParams *>(cp_raw);
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = cond;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    e = cudaGraphAddNode(&node, g.graph, nullptr, nullptr, 0, &cp);
    if (e != cudaSuccess) return fail(e);
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    const int l0 = ctx->launches, p0 = ctx->pair_launches;
    e = cudaStreamBeginCaptureToGraph(st, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
    if (e != cudaSuccess) return fail(e);
    mfs_status ms = MFS_OK;
    cudaError_t ce = cudaSuccess;
    ms = iteration_matvec(ctx, ctx->vin_d, nrhs, transposed, st);
    if (ms == MFS_OK) ce = gmres_arnoldi(gd, ctx->w_d, ctx->vin_d, 0, st);
    if (ce == cudaSuccess && ms == MFS_OK) ce = gmres_advance(gd, cond, st);
    cudaGraph_t captured = nullptr;
    e = cudaStreamEndCapture(st, &captured);
    g.launches = ctx->launches - l0 + gmres_arnoldi_launches(gd) + 1;
    g.pair_launches = ctx->pair_launches - p0;
    ctx->launches = l0;
    ctx->pair_launches = p0;
    if (ms != MFS_OK) {
        cudaGraphDestroy(g.graph);
        return ms;
    }
    if (ce != cudaSuccess) return fail(ce);
    if (e != cudaSuccess) return fail(e);
    e = cudaGraphInstantiate(&g.exec, g.graph, 0);
    if (e != cudaSuccess) return fail(e);
    it = ctx->graphs.emplace(key, g).first;
    *out = &it->second;
    return MFS_OK;
}

// Enqueue the solve of A x = b (or A^T x = b) with b = ctx->b_d for all lanes, x to `x`; gmres_finish
// waits for it.  Once a solve of this kind has run, its whole iteration loop is one graph launch and
// nothing here waits for the device.
mfs_status gmres_solve(mfs_ctx *ctx, int nrhs, cudaStream_t st, double *x, SolveStats &stats,
                       bool transposed = false) {
    GmresDev &gd = ctx->gd;
    CK(gmres_init(gd, ctx->b_d, ctx->vin_d, st));
    ctx->launches += 2;
    const bool use_graph = ctx->opt.graphs && !ctx->opt.profile;
    const auto have = ctx->graphs.find(nrhs * 4 + ctx->fset * 2 + (transposed ? 1 : 0));
    if (use_graph && have != ctx->graphs.end()) {
        stats.graph = &have->second;
        CK(cudaGraphLaunch(have->second.exec, st));
    } else {
        for (int j = 0; j < gd.m; ++j) {
            CKS(iteration_matvec(ctx, ctx->vin_d, nrhs, transposed, st));
            CK(gmres_arnoldi(gd, ctx->w_d, ctx->vin_d, 1, st));
            ctx->launches += gmres_arnoldi_launches(gd);
            CK(cudaMemcpyAsync(ctx->done_h, gd.done, sizeof(int), cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            stats.host_iters = j + 1;
            if (*ctx->done_h || j + 1 >= gd.m) break;
            if (use_graph) {  // the remaining iterations as one graph launch
                mfs_ctx::SolveGraph *g = nullptr;
                CKS(solve_graph(ctx, nrhs, transposed, &g));
                stats.graph = g;
                CK(cudaGraphLaunch(g->exec, st));
                break;
            }
        }
    }
    CK(gmres_solution(gd, x, st));
    ctx->launches += 1;
    CK(cudaMemcpyAsync(ctx->stat_h, ctx->stat_d, ctx->stat_bytes(gd.L), cudaMemcpyDeviceToHost, st));
    return MFS_OK;
}

// Wait for the stream and read the solve's statistics and the device error flag.
mfs_status gmres_finish(mfs_ctx *ctx, cudaStream_t st, SolveStats &stats) {
    const GmresDev &gd = ctx->gd;
    CK(cudaMemcpyAsync(ctx->done_h + 1, ctx->err_d, sizeof(int), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    const double *res = reinterpret_cast<const double *>(ctx->stat_h);
    const int *it = reinterpret_cast<const int *>(res + gd.L), *status = it + gd.L, jend = status[gd.L + 1];
    for (int l = 0; l < gd.L; ++l) {
        stats.iters = std::max(stats.iters, it[l]);
        stats.resid = std::max(stats.resid, res[l]);
        if (status[l] == 2) stats.breakdown = 1;
        if (!(res[l] <= gd.tol)) stats.converged = 0;
    }
    stats.matvecs = jend + 1;
    if (stats.graph) {
        ctx->launches += (stats.matvecs - stats.host_iters) * stats.graph->launches;
        ctx->pair_launches += (stats.matvecs - stats.host_iters) * stats.graph->pair_launches;
    }
    if (ctx->done_h[1]) return check_device_error(ctx, st);
    return MFS_OK;
}

}  // namespace

// ===========================================================================
// C ABI
// ===========================================================================
extern "C" {

void mfs_default_options(mfs_options *opt) {
    if (!opt) return;
    opt->mu = 1.0;
    opt->gmres_tol = 1e-7;
    opt->max_iter = 200;
    opt->restart = 200;
    opt->eps_trunc = 0.0;
    opt->precision = 0;
    opt->autotune = 1;
    opt->max_rhs = 4;
    opt->profile = 0;
    opt->tensor_cores = 1;
    opt->pair_variant = -1;
    opt->graphs = 1;
    opt->farfield = 0;
    opt->farfield_separation = 3.0;
}

int32_t mfs_abi_version(void) { return MFS_ABI_VERSION; }

const char *mfs_pair_variant_info(int32_t index, int32_t *d, int32_t *nrhs, int32_t *grad) {
    int count = 0;
    const PairVariant *vv = pair_variants(&count);
    if (index < 0 || index >= count) return nullptr;
    if (d) *d = vv[index].D;
    if (nrhs) *nrhs = vv[index].nrhs;
    if (grad) *grad = vv[index].grad;
    return vv[index].name;
}

const char *mfs_pair_variant(const mfs_ctx *ctx, int32_t nrhs) {
    if (!ctx || nrhs < 1 || nrhs > 4 || nrhs > ctx->opt.max_rhs) return "";
    const int v = forward_variant(ctx, nrhs);
    int count = 0;
    const PairVariant *vv = pair_variants(&count);
    return (v >= 0 && v < count) ? vv[v].name : "";
}

const char *mfs_last_error(const mfs_ctx *ctx) { return ctx ? ctx->last_error.c_str() : ""; }

mfs_status mfs_selftest_fail_alloc(mfs_ctx *ctx, int32_t nth) {
    if (!ctx || nth < 0) return MFS_ERR_INVALID_ARG;
    ctx->fail_alloc = nth;
    return MFS_OK;
}

mfs_status mfs_selftest_device_error(mfs_ctx *ctx, void *stream) {
    if (!ctx) return MFS_ERR_INVALID_ARG;
    const int flag = MFS_DEVERR_TIMEOUT;
    CK(cudaMemcpyAsync(ctx->err_d, &flag, sizeof(int), cudaMemcpyHostToDevice, (cudaStream_t)stream));
    CK(cudaStreamSynchronize((cudaStream_t)stream));
    return MFS_OK;
}

const char *mfs_setup_error(void) { return g_setup_error.c_str(); }

void mfs_destroy(mfs_ctx *ctx) { delete ctx; }

}  // extern "C"

// One formulation's one-body factors for shape s: the block (S_L, or the bare S^(00) when set = 1),
// its thin SVD in FP64 (cuSOLVER gesvd, Eq. pseudo), the FP32 / FP64 apply factors and, for the
// tensor cores, their TF32 pieces and tensor maps.
static mfs_status build_shape_factors(mfs_ctx *ctx, cusolverDnHandle_t solver, int s, int set, cudaStream_t st) {
    ShapeHost &sh = ctx->shapes[s];
    FactorSet &fx = sh.fs[set];
    ShapeDev &sd = fx.dev;
    const int D = ctx->D, kind = ctx->kind;
    sd.M = sh.M;
    sd.N = sh.N;
    sd.dM = D * sh.M;
    sd.dN = D * sh.N;
    sd.r = sd.dN;
    const int m = sd.dM, n = sd.dN;
    double *X0 = nullptr, *Y0 = nullptr, *G0i = nullptr, *SL = nullptr, *Ucm = nullptr, *sig = nullptr, *VT = nullptr,
           *work = nullptr;
    int *info_d = nullptr;
    auto cleanup = [&]() {
        cudaFree(X0); cudaFree(Y0); cudaFree(G0i); cudaFree(SL); cudaFree(Ucm); cudaFree(sig); cudaFree(VT);
        cudaFree(work); cudaFree(info_d);
    };
    auto fail = [&](const std::string &msg, mfs_status code) {
        cleanup();
        cudaGetLastError();
        ctx->last_error = msg;
        return code;
    };
    if (cudaMalloc(&X0, sizeof(double) * 3 * sh.M) != cudaSuccess ||
        cudaMalloc(&Y0, sizeof(double) * 3 * sh.N) != cudaSuccess ||
        cudaMalloc(&G0i, sizeof(double) * 36) != cudaSuccess ||
        cudaMalloc(&SL, sizeof(double) * (size_t)m * n) != cudaSuccess ||
        cudaMalloc(&Ucm, sizeof(double) * (size_t)m * n) != cudaSuccess ||
        cudaMalloc(&sig, sizeof(double) * n) != cudaSuccess ||
        cudaMalloc(&VT, sizeof(double) * (size_t)n * n) != cudaSuccess ||
        cudaMalloc(&info_d, sizeof(int)) != cudaSuccess)
        return fail("device allocation for the one-body SVD failed", MFS_ERR_OOM);
    cudaMemcpy(X0, sh.X0.data(), sizeof(double) * 3 * sh.M, cudaMemcpyHostToDevice);
    cudaMemcpy(Y0, sh.Y0.data(), sizeof(double) * 3 * sh.N, cudaMemcpyHostToDevice);
    cudaMemcpy(G0i, sh.G0inv, sizeof(double) * 36, cudaMemcpyHostToDevice);
    cudaError_t ce = build_SL(kind, sh.M, sh.N, X0, Y0, ctx->opt.mu, G0i, set, SL, st);
    int lwork = 0;
    if (ce == cudaSuccess && cusolverDnDgesvd_bufferSize(solver, m, n, &lwork) != CUSOLVER_STATUS_SUCCESS)
        ce = cudaErrorUnknown;
    if (ce == cudaSuccess) ce = cudaMalloc(&work, sizeof(double) * std::max(lwork, 1));
    if (ce == cudaSuccess) {
        signed char jobu = 'S', jobvt = 'S';
        cusolverStatus_t cs =
            cusolverDnDgesvd(solver, jobu, jobvt, m, n, SL, m, sig, Ucm, m, VT, n, work, lwork, nullptr, info_d);
        if (cs != CUSOLVER_STATUS_SUCCESS) ce = cudaErrorUnknown;
    }
    int info_h = 0;
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(&info_h, info_d, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
    if (ce != cudaSuccess || info_h != 0)
        return fail(std::string("one-body SVD failed: ") + (ce != cudaSuccess ? cudaGetErrorString(ce) : "gesvd info != 0"),
                    MFS_ERR_CUDA);
    // apply factors
    const bool want_tc = ctx->opt.tensor_cores != 0 && ctx->opt.precision == 0;
    bool ok = ctx->alloc(&sd.U, (size_t)m * n) == cudaSuccess && ctx->alloc(&sd.Wp, (size_t)n * n) == cudaSuccess &&
              ctx->alloc(&sd.Wr, (size_t)n * n) == cudaSuccess;
    if (ok && (ctx->opt.precision >= 1 || want_tc))  // the tensor-core pieces are cut from FP64 factors
        ok = ctx->alloc(&sd.U64, (size_t)m * n) == cudaSuccess && ctx->alloc(&sd.Wp64, (size_t)n * n) == cudaSuccess &&
             ctx->alloc(&sd.Wr64, (size_t)n * n) == cudaSuccess;
    if (!ok) return fail("device allocation for the apply factors failed", MFS_ERR_OOM);
    ce = build_apply_factors(kind, sh.M, sh.N, Ucm, sig, VT, Y0, G0i, ctx->opt.eps_trunc, set, sd, st);
    cleanup();
    if (ce != cudaSuccess) {
        ctx->last_error = std::string("apply factors: ") + cudaGetErrorString(ce);
        return MFS_ERR_CUDA;
    }
    if (!(sd.sigma1 > 0.0) || !std::isfinite(sd.sigma1)) {
        ctx->last_error = "one-body SVD returned a non-finite or zero largest singular value";
        return MFS_ERR_ILL_CONDITIONED;
    }
    if (want_tc) {
        // K-major FP32 (hi, lo) planes: U^T [r][ld1], Wp^T and Wr^T [dN][ld2], from the FP64 factors; zero
        // K padding.  The kernel cuts them into TF32 pieces in shared memory.
        sh.pieces = ctx->opt.tensor_cores == 2 ? 2 : 3;
        sh.ld1 = (m + 31) / 32 * 32;
        sh.ld2 = (n + 31) / 32 * 32;
        fx.ut_stride = (size_t)n * sh.ld1;
        fx.wt_stride = (size_t)n * sh.ld2;
        ok = ctx->alloc(&fx.Utp, 2 * fx.ut_stride) == cudaSuccess &&
             ctx->alloc(&fx.Wptp, 2 * fx.wt_stride) == cudaSuccess &&
             ctx->alloc(&fx.Wrtp, 2 * fx.wt_stride) == cudaSuccess;
        if (!ok) {
            ctx->last_error = "device allocation for the tensor-core factors failed";
            return MFS_ERR_OOM;
        }
        CK(split_hilo_transpose(sd.U64, m, n, fx.Utp, sh.ld1, fx.ut_stride, st));
        CK(split_hilo_transpose(sd.Wp64, n, n, fx.Wptp, sh.ld2, fx.wt_stride, st));
        CK(split_hilo_transpose(sd.Wr64, n, n, fx.Wrtp, sh.ld2, fx.wt_stride, st));
        CK(cudaStreamSynchronize(st));
        const int box = 128;  // factor rows per CTA (MMA M)
        bool enc = true;
        for (int p = 0; p < 2; ++p)
            enc = enc && make_tc_map(fx.mU[p], fx.Utp + p * fx.ut_stride, n, sh.ld1, box) &&
                  make_tc_map(fx.mWp[p], fx.Wptp + p * fx.wt_stride, n, sh.ld2, box) &&
                  make_tc_map(fx.mWr[p], fx.Wrtp + p * fx.wt_stride, n, sh.ld2, box);
        if (!enc) {
            ctx->last_error = "tensor-map encoding for the tensor-core apply failed";
            return MFS_ERR_CUDA;
        }
        fx.tc_ready = true;
        if (ctx->opt.precision == 0) {  // the FP64 factors were only the source of the pieces
            ctx->release(sd.U64);
            ctx->release(sd.Wp64);
            ctx->release(sd.Wr64);
            sd.U64 = sd.Wp64 = sd.Wr64 = nullptr;
        }
    }
    fx.built = true;
    return MFS_OK;
}

// Column lists and GEMM scratch of one shape's one-body apply (shared by the formulations).
static mfs_status alloc_apply_scratch(mfs_ctx *ctx, ShapeHost &sh, cudaStream_t st) {
    const int R = ctx->opt.max_rhs;
    const int m = sh.fs[0].dev.dM, n = sh.fs[0].dev.dN;
    const int nb = (int)sh.bodies.size();
    if (nb == 0) return MFS_OK;
    std::vector<int> cb(R * nb), cr(R * nb);
    for (int h = 0; h < R; ++h)
        for (int i = 0; i < nb; ++i) {
            cb[h * nb + i] = sh.bodies[i];
            cr[h * nb + i] = h;
        }
    bool ok = ctx->alloc(&sh.col_body, R * nb) == cudaSuccess && ctx->alloc(&sh.col_rhs, R * nb) == cudaSuccess &&
              ctx->alloc(&sh.A, (size_t)R * nb * m) == cudaSuccess &&
              ctx->alloc(&sh.Tm, (size_t)R * nb * n) == cudaSuccess;
    if (ok && ctx->opt.precision >= 1) {
        size_t need = 1;  // both GEMMs, and the adjoint's second one (n -> m)
        for (int h = 1; h <= R; ++h) {
            const int rows = h * nb;
            need = std::max(need, (size_t)gemm_rm64_chunks(rows, n, m, ctx->sm_count) * rows * n);
            need = std::max(need, (size_t)gemm_rm64_chunks(rows, n, n, ctx->sm_count) * rows * n);
            need = std::max(need, (size_t)gemm_rm64_chunks(rows, m, n, ctx->sm_count) * rows * m);
        }
        ok = ctx->alloc(&sh.A64, (size_t)R * nb * m) == cudaSuccess &&
             ctx->alloc(&sh.T64, (size_t)R * nb * n) == cudaSuccess && ctx->alloc(&sh.Pk64, need) == cudaSuccess;
    }
    if (ok && sh.pieces == 0) ok = ctx->alloc(&sh.L64, (size_t)R * nb * n) == cudaSuccess;
    if (ok) {  // split-K chunk results: the largest S * rows * cols over nrhs = 1..R and both GEMMs
        size_t need = 0;
        for (int h = 1; h <= R; ++h) {
            const int rows = h * nb;
            need = std::max(need, (size_t)gemm_splitk_chunks(rows, n, m, ctx->sm_count) * rows * n);
            need = std::max(need, (size_t)gemm_splitk_chunks(rows, n, n, ctx->sm_count) * rows * n);
        }
        sh.Pk_count = need;
        ok = ctx->alloc(&sh.Pk, need) == cudaSuccess;
    }
    if (ok && sh.pieces > 0) {  // tensor cores: column pieces and chunk results
        const int np = sh.pieces;
        const size_t cap = (size_t)R * nb;
        sh.ap_stride = cap * sh.ld1;
        sh.tp_stride = cap * sh.ld2;
        size_t need = 0;
        for (int h = 1; h <= R; ++h) {
            const int cols = h * nb;
            need = std::max(need, (size_t)tc_gemm_sz(m, tc_gemm_chunks(cols, n, m, ctx->sm_count, np)) * cols * n);
            need = std::max(need, (size_t)tc_gemm_sz(n, tc_gemm_chunks(cols, n, n, ctx->sm_count, np)) * cols * n);
        }
        ok = ctx->alloc(&sh.Ap, np * sh.ap_stride) == cudaSuccess &&
             ctx->alloc(&sh.Tp, np * sh.tp_stride) == cudaSuccess && ctx->alloc(&sh.Ptc, need) == cudaSuccess;
        // the padding columns of the column pieces stay zero: the kernels write only the first dM / r
        if (ok)
            ok = cudaMemsetAsync(sh.Ap, 0, sizeof(float) * np * sh.ap_stride, st) == cudaSuccess &&
                 cudaMemsetAsync(sh.Tp, 0, sizeof(float) * np * sh.tp_stride, st) == cudaSuccess;
    }
    if (ok && sh.pieces > 0) {  // few columns (their K padding stays zero, as the pieces')
        ok = ctx->alloc(&sh.Gf, (size_t)FC_MAX * sh.ld1) == cudaSuccess &&
             ctx->alloc(&sh.Tf, (size_t)FC_MAX * sh.ld2) == cudaSuccess &&
             ctx->alloc(&sh.Xf, (size_t)FC_MAX * sh.ld2) == cudaSuccess &&
             ctx->alloc(&sh.Lf, (size_t)FC_MAX * m) == cudaSuccess &&
             cudaMemsetAsync(sh.Xf, 0, sizeof(float2) * FC_MAX * sh.ld2, st) == cudaSuccess &&
             cudaMemsetAsync(sh.Gf, 0, sizeof(float2) * FC_MAX * sh.ld1, st) == cudaSuccess &&
             cudaMemsetAsync(sh.Tf, 0, sizeof(float2) * FC_MAX * sh.ld2, st) == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        ctx->last_error = "device allocation for the preconditioner buffers failed";
        return MFS_ERR_OOM;
    }
    CK(cudaMemcpy(sh.col_body, cb.data(), sizeof(int) * cb.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(sh.col_rhs, cr.data(), sizeof(int) * cr.size(), cudaMemcpyHostToDevice));
    return MFS_OK;
}

// The Dirichlet formulation's factors (bare self blocks), built on the first capacitance or
// resistance solve: one more SVD per shape.
static mfs_status ensure_dirichlet(mfs_ctx *ctx, cudaStream_t st) {
    bool all = true;
    for (auto &sh : ctx->shapes) all = all && sh.fs[1].built;
    if (all) return MFS_OK;
    cusolverDnHandle_t solver = nullptr;
    if (cusolverDnCreate(&solver) != CUSOLVER_STATUS_SUCCESS) {
        ctx->last_error = "cusolverDnCreate failed";
        return MFS_ERR_CUDA;
    }
    cusolverDnSetStream(solver, st);
    mfs_status status = MFS_OK;
    for (int s = 0; s < (int)ctx->shapes.size() && status == MFS_OK; ++s)
        if (!ctx->shapes[s].fs[1].built) status = build_shape_factors(ctx, solver, s, 1, st);
    cusolverDnDestroy(solver);
    return status;
}

// n points of the Fibonacci lattice on the unit sphere (z_i = 1 - (2i+1)/n, golden-angle longitudes).
static void unit_fibonacci(int n, std::vector<double> &p) {
    const double ga = 2.0 * MFS_PI / (((1.0 + std::sqrt(5.0)) / 2.0) * ((1.0 + std::sqrt(5.0)) / 2.0));
    p.resize(3 * (size_t)n);
    for (int i = 0; i < n; ++i) {
        const double z = 1.0 - (2.0 * i + 1.0) / n, rho = std::sqrt(std::max(0.0, 1.0 - z * z));
        p[3 * i] = rho * std::cos(ga * i);
        p[3 * i + 1] = rho * std::sin(ga * i);
        p[3 * i + 2] = z;
    }
}

// The raw kernel (1/r or (I + r r^T / r^2) / r) between two scaled point sets, column-major
// [D nt][D ns] (read row-major: its transpose).
static std::vector<double> ff_map(int D, const std::vector<double> &tgt, double rt, const std::vector<double> &src,
                                  double rs) {
    const int nt = (int)tgt.size() / 3, ns = (int)src.size() / 3;
    const int m = D * nt;
    std::vector<double> A((size_t)m * D * ns);
    for (int j = 0; j < ns; ++j)
        for (int i = 0; i < nt; ++i) {
            double r[3], r2 = 0.0;
            for (int a = 0; a < 3; ++a) {
                r[a] = rt * tgt[3 * i + a] - rs * src[3 * j + a];
                r2 += r[a] * r[a];
            }
            const double ri = 1.0 / std::sqrt(r2);
            for (int b = 0; b < D; ++b)
                for (int a = 0; a < D; ++a)
                    A[(size_t)(D * j + b) * m + (D * i + a)] =
                        D == 1 ? ri : ((a == b ? ri : 0.0) + r[a] * r[b] * ri * ri * ri);
        }
    return A;
}

// V[j][k] *= 1 / s_k over the singular values kept (s_k > trunc s_0), 0 for the others.
static __global__ void ff_scale_columns_kernel(double *V, const double *s, int n, double trunc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * n) return;
    const int k = i % n;
    V[i] *= s[k] > trunc * s[0] ? 1.0 / s[k] : 0.0;
}

// The transposed pseudo-inverse [m][n] (device, row-major, cudaMalloc'ed, the caller's) of a
// column-major m x n matrix, m >= n, in FP64, truncated at `trunc` of the largest singular value.
static mfs_status ff_pinvT(mfs_ctx *ctx, cusolverDnHandle_t solver, int m, int n, const std::vector<double> &A,
                           double trunc, double **out, cudaStream_t st) {
    double *A_d = nullptr, *U_d = nullptr, *S_d = nullptr, *VT_d = nullptr, *work = nullptr, *P_d = nullptr;
    int *info_d = nullptr, lwork = 0, info_h = 0;
    double s0 = 0.0;
    CK(cudaMalloc(out, sizeof(double) * (size_t)m * n));
    bool ok = cudaMalloc(&A_d, sizeof(double) * A.size()) == cudaSuccess &&
              cudaMalloc(&U_d, sizeof(double) * (size_t)m * n) == cudaSuccess &&
              cudaMalloc(&S_d, sizeof(double) * n) == cudaSuccess &&
              cudaMalloc(&VT_d, sizeof(double) * (size_t)n * n) == cudaSuccess &&
              cudaMalloc(&P_d, sizeof(double) * (size_t)n * m) == cudaSuccess &&
              cudaMalloc(&info_d, sizeof(int)) == cudaSuccess &&
              cudaMemcpyAsync(A_d, A.data(), sizeof(double) * A.size(), cudaMemcpyHostToDevice, st) == cudaSuccess &&
              cusolverDnDgesvd_bufferSize(solver, m, n, &lwork) == CUSOLVER_STATUS_SUCCESS &&
              cudaMalloc(&work, sizeof(double) * std::max(lwork, 1)) == cudaSuccess;
    signed char jobu = 'S', jobvt = 'S';
    ok = ok && cusolverDnDgesvd(solver, jobu, jobvt, m, n, A_d, m, S_d, U_d, m, VT_d, n, work, lwork, nullptr,
                                info_d) == CUSOLVER_STATUS_SUCCESS;
    if (ok) {  // pinv [n][m] = (V S^+) U^T: column-major V^T read row-major is V, column-major U is U^T
        ff_scale_columns_kernel<<<(n * n + 255) / 256, 256, 0, st>>>(VT_d, S_d, n, trunc);
        ok = gemm_rm64_splitk(n, m, n, 1, VT_d, U_d, nullptr, P_d, st) == cudaSuccess;
        transpose64_kernel<<<1024, 256, 0, st>>>(P_d, n, m, *out);
        ok = ok && cudaGetLastError() == cudaSuccess &&
             cudaMemcpyAsync(&info_h, info_d, sizeof(int), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
             cudaMemcpyAsync(&s0, S_d, sizeof(double), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
             cudaStreamSynchronize(st) == cudaSuccess && info_h == 0;
    }
    cudaFree(A_d); cudaFree(U_d); cudaFree(S_d); cudaFree(VT_d); cudaFree(P_d); cudaFree(work); cudaFree(info_d);
    if (!ok || !(s0 > 0.0)) {
        cudaGetLastError();
        ctx->last_error = "far field: SVD of a check <- equivalent map failed";
        return MFS_ERR_CUDA;
    }
    return MFS_OK;
}

static mfs_status ff_build_matrices(mfs_ctx *ctx, FFMatrices &M, cudaStream_t st) {
    const int D = ctx->D;
    cusolverDnHandle_t solver = nullptr;
    if (cusolverDnCreate(&solver) != CUSOLVER_STATUS_SUCCESS) {
        ctx->last_error = "cusolverDnCreate failed";
        return MFS_ERR_CUDA;
    }
    cusolverDnSetStream(solver, st);
    auto build = [&]() -> mfs_status {
        std::vector<double> e[FF_NORD], c;
        for (int o = 0; o < FF_NORD; ++o) {
            unit_fibonacci(FF_ORD_N[o], e[o]);
            unit_fibonacci(FF_ORD_NC[o], c);
            const int m = D * FF_ORD_NC[o], n = D * FF_ORD_N[o];
            double *pinvT = nullptr, *G_d = nullptr;
            const mfs_status s = ff_pinvT(ctx, solver, m, n, ff_map(D, c, FF_ORD_CHECK[o], e[o], 1.0),
                                          FF_ORD_TRUNC[o], o == 0 ? &M.PinvT : &pinvT, st);
            if (s != MFS_OK || o == 0) {
                cudaFree(pinvT);
                CKS(s);
                continue;
            }
            // ordT = (previous order's field at this order's check points)^T pinvT
            const int np = D * FF_ORD_N[o - 1];
            const std::vector<double> G = ff_map(D, c, FF_ORD_CHECK[o], e[o - 1], 1.0);
            const bool ok =
                cudaMalloc(&G_d, sizeof(double) * G.size()) == cudaSuccess &&
                cudaMalloc(&M.ordT[o], sizeof(double) * (size_t)np * n) == cudaSuccess &&
                cudaMemcpyAsync(G_d, G.data(), sizeof(double) * G.size(), cudaMemcpyHostToDevice, st) == cudaSuccess &&
                gemm_rm64_splitk(np, n, m, 1, G_d, pinvT, nullptr, M.ordT[o], st) == cudaSuccess &&
                cudaStreamSynchronize(st) == cudaSuccess;
            cudaFree(G_d);
            cudaFree(pinvT);
            if (!ok) CK(cudaErrorMemoryAllocation);
        }
        std::vector<double> l;
        unit_fibonacci(FF_LOC_N, l);
        unit_fibonacci(FF_LOC_NC, c);
        return ff_pinvT(ctx, solver, D * FF_LOC_NC, D * FF_LOC_N, ff_map(D, c, FF_LOC_CHECK, l, FF_LOC_EQ),
                        FF_LOC_TRUNC, &M.locT, st);
    };
    const mfs_status rc = build();
    cusolverDnDestroy(solver);
    return rc;
}

// The matrices of this context's kernel on the current device: those of another live context, or built
// (five small FP64 SVDs, 0.1 s) under the lock and complete on the device before anyone else sees them.
static mfs_status ff_matrices(mfs_ctx *ctx, std::shared_ptr<const FFMatrices> &out, cudaStream_t st) {
    static std::mutex mu;
    static std::weak_ptr<const FFMatrices> kept[64][2];
    int dev = 0;
    CK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 64) out = kept[dev][ctx->D == 3].lock();
    if (out) return MFS_OK;
    auto M = std::make_shared<FFMatrices>();
    CKS(ff_build_matrices(ctx, *M, st));
    CK(cudaStreamSynchronize(st));
    out = M;
    if (dev < 64) kept[dev][ctx->D == 3] = out;
    return MFS_OK;
}

// Frees the far-field structures that depend on the body centres (all but the pseudo-inverse) and
// drops the captured graphs that hold their addresses.
static void ff_release_geometry(mfs_ctx *ctx, mfs_ctx::FarField &F) {
    ctx->drop_graphs();
    for (auto *plans : {&F.up, &F.ev, &F.loc, &F.direct}) {
        for (auto &kv : *plans) {
            release_plan(ctx, kv.second.p);
            ctx->release(kv.second.seg);
            ctx->release(kv.second.cum);
        }
        plans->clear();
    }
    F.cells = mfs_ctx::FarField::Cells{};
    for (int o = 1; o < FF_NORD; ++o) {
        ctx->release(F.ord_pos[o]);
        ctx->release(F.ord_mu[o]);
        F.ord_pos[o] = nullptr;
        F.ord_mu[o] = nullptr;
    }
    for (void *p : {(void *)F.rloc, (void *)F.loc_pos, (void *)F.lchk_pos, (void *)F.ulocal, (void *)F.nu,
                    (void *)F.ufar})
        ctx->release(p);
    F.rloc = F.ulocal = F.nu = F.ufar = nullptr;
    F.loc_pos = F.lchk_pos = nullptr;
    ctx->release(F.centres);
    ctx->release(F.re);
    ctx->release(F.eq_pos);
    ctx->release(F.eq_pt);
    ctx->release(F.chk_pos);
    ctx->release(F.tgt);
    ctx->release(F.tperm);
    ctx->release(F.pos);
    ctx->release(F.order);
    F.pos = F.order = nullptr;
    ctx->release(F.seg_rec0);
    ctx->release(F.seg_rec1);
    ctx->release(F.rec);
    ctx->release(F.ucheck);
    ctx->release(F.mu);
    ctx->release(F.fit_chunks);
    F.centres = F.ucheck = F.mu = F.fit_chunks = F.re = nullptr;
    F.eq_pos = F.chk_pos = F.tgt = nullptr;
    F.eq_pt = F.tperm = F.seg_rec0 = F.seg_rec1 = nullptr;
    F.rec = nullptr;
    F.ready = false;
}

// The far-field structures (opt.farfield = 1): the tree, the FP64 pseudo-inverse of the map from
// equivalent strengths on the unit sphere to the field at the check points (ff_matrices, once per
// process and device), and the tree-ordered geometry (again after every mfs_update_centers).
static mfs_status ff_setup(mfs_ctx *ctx, mfs_ctx::FarField &F, cudaStream_t st) {
    const int P = ctx->P, D = ctx->D;
    F.rsrc.assign(P, 0.0);
    F.rtgt.assign(P, 0.0);
    for (int k = 0; k < P; ++k) {
        const ShapeHost &sh = ctx->shapes[ctx->shape_id[k]];
        double rp = 0.0, rc = 0.0;  // radii of the proxy and collocation points about the centre
        for (int j = 0; j < sh.N; ++j)
            rp = std::max(rp, std::sqrt(sh.Y0[3 * j] * sh.Y0[3 * j] + sh.Y0[3 * j + 1] * sh.Y0[3 * j + 1] +
                                        sh.Y0[3 * j + 2] * sh.Y0[3 * j + 2]));
        for (int i = 0; i < sh.M; ++i)
            rc = std::max(rc, std::sqrt(sh.X0[3 * i] * sh.X0[3 * i] + sh.X0[3 * i + 1] * sh.X0[3 * i + 1] +
                                        sh.X0[3 * i + 2] * sh.X0[3 * i + 2]));
        F.rsrc[k] = F.src_colloc ? rc : rp;
        F.rtgt[k] = F.src_colloc ? rp : rc;
    }
    ff_build_tree(P, ctx->centres.data(), F.rsrc.data(), ctx->S, ctx->body_off.data(), F.tree);
    const int nodes = F.nodes = (int)F.tree.nodes.size();

    std::vector<double> ue, uc;
    unit_fibonacci(FF_NE, ue);
    unit_fibonacci(FF_NC, uc);
    if (!F.mat) CKS(ff_matrices(ctx, F.mat, st));  // independent of the centres
    // Local expansions where a body has clearly more targets than check points: with fewer, the check
    // sums, the match and six more launches cost more than the lower orders at the targets themselves
    // (150 ellipsoids with 200 targets each: 1.15 ms with them, 1.08 without); ff_cell_lists then
    // weighs each cell.
    F.use_local = F.ntgt >= 2LL * FF_LOC_NC * P;
    for (int k = 0; k < P; ++k) F.use_local = F.use_local && F.rtgt[k] > 0.0;
    // tree-ordered geometry and segments: proxy segment q (tree position) = body order[q], node segment
    // P + o nodes + node = order o of its equivalent points, local segment P + FF_NORD nodes + q
    const int nseg = P + FF_NORD * nodes + (F.use_local ? P : 0);
    std::vector<double> cen(3 * (size_t)nseg), re(nodes), rloc(P);
    for (int q = 0; q < P; ++q) {
        rloc[q] = F.rtgt[F.tree.order[q]];
        for (int a = 0; a < 3; ++a) {
            cen[3 * (size_t)q + a] = ctx->centres[3 * F.tree.order[q] + a];
            if (F.use_local) cen[3 * (size_t)(P + FF_NORD * nodes + q) + a] = ctx->centres[3 * F.tree.order[q] + a];
        }
    }
    for (int nd = 0; nd < nodes; ++nd) {
        for (int o = 0; o < FF_NORD; ++o)
            for (int a = 0; a < 3; ++a) cen[3 * (size_t)(P + o * nodes + nd) + a] = F.tree.nodes[nd].c[a];
        re[nd] = F.tree.nodes[nd].re;
    }
    // unit points scaled by r[i] about their centres, w = id0 + i (int bits)
    auto scaled = [](const std::vector<double> &unit, double f, const std::vector<double> &r, int id0) {
        const int n = (int)unit.size() / 3;
        std::vector<float4> out(r.size() * n);
        for (size_t i = 0; i < r.size(); ++i) {
            float w;
            const int id = id0 + (int)i;
            std::memcpy(&w, &id, sizeof(float));
            for (int e = 0; e < n; ++e)
                out[i * n + e] = make_float4((float)(f * r[i] * unit[3 * e]), (float)(f * r[i] * unit[3 * e + 1]),
                                             (float)(f * r[i] * unit[3 * e + 2]), w);
        }
        return out;
    };
    const std::vector<float4> eq = scaled(ue, 1.0, re, 0), chk = scaled(uc, FF_CHECK, re, P);
    std::vector<int> eq_pt((size_t)nodes * FF_NE);  // identity (packing); long enough for every order
    for (size_t i = 0; i < eq_pt.size(); ++i) eq_pt[i] = (int)i;
    std::vector<float4> tpos(F.ntgt), tff(F.ntgt);
    CK(cudaMemcpy(tpos.data(), F.tgt_pos, sizeof(float4) * F.ntgt, cudaMemcpyDeviceToHost));
    std::vector<int> tperm(F.ntgt);
    int t = 0;
    for (int q = 0; q < P; ++q) {
        const int b = F.tree.order[q];
        float w;
        std::memcpy(&w, &q, sizeof(float));
        for (int i = (*F.tgt_off)[b]; i < (*F.tgt_off)[b + 1]; ++i, ++t) {
            tff[t] = make_float4(tpos[i].x, tpos[i].y, tpos[i].z, w);
            tperm[t] = i;
        }
    }
    F.seg_rec0_h.resize(nseg);
    F.seg_rec1_h.resize(nseg);
    for (int q = 0; q < P; ++q) {
        const int b = F.tree.order[q];
        F.seg_rec0_h[q] = (*F.rec_off)[b];
        F.seg_rec1_h[q] = (*F.rec_off)[b + 1];  // padded to a multiple of 4 (zero-strength padding records)
    }
    size_t nrec_all = F.nrec;
    for (int o = 0; o < FF_NORD; ++o) {
        F.ord_rec[o] = nrec_all;
        for (int nd = 0; nd < nodes; ++nd) {
            F.seg_rec0_h[P + o * nodes + nd] = (int)nrec_all + nd * FF_ORD_N[o];
            F.seg_rec1_h[P + o * nodes + nd] = (int)nrec_all + (nd + 1) * FF_ORD_N[o];
        }
        nrec_all += (size_t)nodes * FF_ORD_N[o];
    }
    F.loc_rec = nrec_all;
    if (F.use_local) {
        for (int q = 0; q < P; ++q) {
            F.seg_rec0_h[P + FF_NORD * nodes + q] = (int)nrec_all + q * FF_LOC_N;
            F.seg_rec1_h[P + FF_NORD * nodes + q] = (int)nrec_all + (q + 1) * FF_LOC_N;
        }
        nrec_all += (size_t)P * FF_LOC_N;
    }
    const int R = ctx->opt.max_rhs;
    F.rec_floats = std::max(pair_record_floats(D, R, 0), pair_record_floats(D, R, 1));  // plain or f32x2 policies
    CK(ctx->alloc(&F.centres, cen.size()));
    CK(ctx->alloc(&F.re, re.size()));
    CK(ctx->alloc(&F.eq_pos, eq.size()));
    CK(ctx->alloc(&F.eq_pt, eq_pt.size()));
    CK(ctx->alloc(&F.chk_pos, chk.size()));
    CK(ctx->alloc(&F.tgt, tff.size()));
    CK(ctx->alloc(&F.tperm, tperm.size()));
    CK(ctx->alloc(&F.pos, P));
    CK(ctx->alloc(&F.order, P));
    CK(cudaMemcpy(F.pos, F.tree.pos.data(), sizeof(int) * P, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.order, F.tree.order.data(), sizeof(int) * P, cudaMemcpyHostToDevice));
    CK(ctx->alloc(&F.seg_rec0, F.seg_rec0_h.size()));
    CK(ctx->alloc(&F.seg_rec1, F.seg_rec1_h.size()));
    CK(ctx->alloc(&F.rec, nrec_all * F.rec_floats));
    auto upload4 = [&](float4 **dst, const std::vector<float4> &v) -> cudaError_t {
        const cudaError_t e = ctx->alloc(dst, v.size());
        return e != cudaSuccess ? e
                                : cudaMemcpy(*dst, v.data(), sizeof(float4) * v.size(), cudaMemcpyHostToDevice);
    };
    for (int o = 1; o < FF_NORD; ++o) {
        std::vector<double> u;
        unit_fibonacci(FF_ORD_N[o], u);
        CK(upload4(&F.ord_pos[o], scaled(u, 1.0, re, 0)));
        CK(ctx->alloc(&F.ord_mu[o], (size_t)R * nodes * FF_ORD_N[o] * D));
    }
    if (F.use_local) {
        std::vector<double> u;
        unit_fibonacci(FF_LOC_N, u);
        CK(upload4(&F.loc_pos, scaled(u, FF_LOC_EQ, rloc, 0)));
        unit_fibonacci(FF_LOC_NC, u);
        CK(upload4(&F.lchk_pos, scaled(u, FF_LOC_CHECK, rloc, 0)));
        CK(ctx->alloc(&F.rloc, rloc.size()));
        CK(cudaMemcpy(F.rloc, rloc.data(), sizeof(double) * P, cudaMemcpyHostToDevice));
        CK(ctx->alloc(&F.ulocal, (size_t)R * P * FF_LOC_NC * D));
        CK(ctx->alloc(&F.nu, (size_t)R * P * FF_LOC_N * D));
        CK(ctx->alloc(&F.ufar, (size_t)R * P * 4 * D));
    }
    CK(ctx->alloc(&F.ucheck, (size_t)R * nodes * FF_NC * D));
    CK(ctx->alloc(&F.mu, (size_t)R * nodes * FF_NE * D));
    {
        size_t chunk_doubles = 1;
        auto fit_size = [&](int rows, int n, int k) {
            const int S = gemm_rm64_chunks(rows, D * n, D * k, ctx->sm_count);
            if (S > 1) chunk_doubles = std::max(chunk_doubles, (size_t)S * rows * n * D);
        };
        for (int h = 1; h <= R; ++h) {
            fit_size(h * nodes, FF_NE, FF_NC);
            for (int o = 1; o < FF_NORD; ++o) fit_size(h * nodes, FF_ORD_N[o], FF_ORD_N[o - 1]);
            fit_size(h * P, FF_LOC_N, FF_LOC_NC);
        }
        CK(ctx->alloc(&F.fit_chunks, chunk_doubles));
    }
    CK(cudaMemcpy(F.centres, cen.data(), sizeof(double) * cen.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.re, re.data(), sizeof(double) * re.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.eq_pos, eq.data(), sizeof(float4) * eq.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.eq_pt, eq_pt.data(), sizeof(int) * eq_pt.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.chk_pos, chk.data(), sizeof(float4) * chk.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.tgt, tff.data(), sizeof(float4) * tff.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.tperm, tperm.data(), sizeof(int) * tperm.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.seg_rec0, F.seg_rec0_h.data(), sizeof(int) * F.seg_rec0_h.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(F.seg_rec1, F.seg_rec1_h.data(), sizeof(int) * F.seg_rec1_h.size(), cudaMemcpyHostToDevice));
    CK(cudaMemset(F.rec, 0, sizeof(float) * nrec_all * F.rec_floats));
    F.ready = true;
    return MFS_OK;
}

static mfs_status setup_impl(mfs_ctx *ctx, mfs_kind kind, const mfs_bodies *bodies, int32_t num_shapes,
                             const mfs_pointset *proxy, const mfs_pointset *colloc, cudaStream_t st) {
    auto t0 = std::chrono::steady_clock::now();
    ctx->kind = kind;
    ctx->D = kind == MFS_STOKES ? 3 : 1;
    const int P = bodies->num_bodies;
    ctx->P = P;
    ctx->nshapes = num_shapes;
    ctx->S = bodies->num_suspensions > 0 && bodies->body_offsets ? bodies->num_suspensions : 1;
    ctx->centres.assign(bodies->centers, bodies->centers + 3 * P);
    ctx->shape_id.resize(P);
    for (int k = 0; k < P; ++k) ctx->shape_id[k] = bodies->shape_id ? bodies->shape_id[k] : 0;
    if (bodies->body_offsets && bodies->num_suspensions > 0)
        ctx->body_off.assign(bodies->body_offsets, bodies->body_offsets + ctx->S + 1);
    else
        ctx->body_off = {0, P};
    // validation
    if (ctx->body_off.front() != 0 || ctx->body_off.back() != P) {
        ctx->last_error = "body_offsets must start at 0 and end at num_bodies";
        return MFS_ERR_INVALID_ARG;
    }
    for (int s = 0; s < ctx->S; ++s)
        if (ctx->body_off[s + 1] <= ctx->body_off[s]) {
            ctx->last_error = "every suspension needs at least one body";
            return MFS_ERR_INVALID_ARG;
        }
    for (int k = 0; k < P; ++k) {
        if (ctx->shape_id[k] < 0 || ctx->shape_id[k] >= num_shapes) {
            ctx->last_error = "shape_id out of range";
            return MFS_ERR_INVALID_ARG;
        }
        for (int c = 0; c < 3; ++c)
            if (!std::isfinite(ctx->centres[3 * k + c])) {
                ctx->last_error = "non-finite body centre";
                return MFS_ERR_INVALID_ARG;
            }
    }
    ctx->rot.resize(9 * P);
    for (int k = 0; k < P; ++k) {
        if (bodies->quats) {
            double q[4];
            double nq = 0.0;
            for (int c = 0; c < 4; ++c) {
                q[c] = bodies->quats[4 * k + c];
                nq += q[c] * q[c];
            }
            if (!(nq > 0.0) || !std::isfinite(nq)) {
                ctx->last_error = "quaternion must be non-zero and finite";
                return MFS_ERR_INVALID_ARG;
            }
            nq = std::sqrt(nq);
            for (int c = 0; c < 4; ++c) q[c] /= nq;
            quat_to_rot(q, &ctx->rot[9 * k]);
        } else {
            const double I[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};
            std::memcpy(&ctx->rot[9 * k], I, sizeof(I));
        }
    }
    ctx->shapes.resize(num_shapes);
    for (int s = 0; s < num_shapes; ++s) {
        ShapeHost &sh = ctx->shapes[s];
        sh.M = colloc[s].n;
        sh.N = proxy[s].n;
        if (sh.N <= 0 || sh.M <= sh.N || !colloc[s].pts || !proxy[s].pts) {
            ctx->last_error = "each shape needs 0 < N < M points";
            return MFS_ERR_INVALID_ARG;
        }
        sh.X0.assign(colloc[s].pts, colloc[s].pts + 3 * sh.M);
        sh.Y0.assign(proxy[s].pts, proxy[s].pts + 3 * sh.N);
        for (double v : sh.X0)
            if (!std::isfinite(v)) { ctx->last_error = "non-finite collocation point"; return MFS_ERR_INVALID_ARG; }
        for (double v : sh.Y0)
            if (!std::isfinite(v)) { ctx->last_error = "non-finite proxy point"; return MFS_ERR_INVALID_ARG; }
        double G0[36];
        gram6(sh.Y0, G0);
        if (kind == MFS_STOKES) {
            if (!invert6(G0, sh.G0inv)) {
                ctx->last_error = "proxy points do not span rigid-body motions (singular K_N^T K_N)";
                return MFS_ERR_INVALID_ARG;
            }
        } else {
            std::memset(sh.G0inv, 0, sizeof(sh.G0inv));
        }
    }
    for (int k = 0; k < P; ++k) ctx->shapes[ctx->shape_id[k]].bodies.push_back(k);

    // offsets
    ctx->tgt_off.assign(P + 1, 0);
    ctx->src_off.assign(P + 1, 0);
    ctx->rec_off.assign(P + 1, 0);
    ctx->blk_off.assign(P + 1, 0);
    for (int k = 0; k < P; ++k) {
        const ShapeHost &sh = ctx->shapes[ctx->shape_id[k]];
        const int npad = (sh.N + 3) / 4 * 4;
        ctx->tgt_off[k + 1] = ctx->tgt_off[k] + sh.M;
        ctx->src_off[k + 1] = ctx->src_off[k] + sh.N;
        ctx->rec_off[k + 1] = ctx->rec_off[k] + npad;
        ctx->blk_off[k + 1] = ctx->blk_off[k] + (npad + MFS_BS - 1) / MFS_BS;
    }
    ctx->sumM = ctx->tgt_off[P];
    ctx->sumN = ctx->src_off[P];
    ctx->nrec = ctx->rec_off[P];
    ctx->tgt_body.resize(ctx->sumM);
    for (int k = 0; k < P; ++k)
        for (int i = ctx->tgt_off[k]; i < ctx->tgt_off[k + 1]; ++i) ctx->tgt_body[i] = k;

    // rotated body-local points
    std::vector<float4> tgt_pos(ctx->sumM), src_pos(ctx->sumN);
    std::vector<double> tgt64(3 * (size_t)ctx->sumM), src64(3 * (size_t)ctx->sumN), src4(4 * (size_t)ctx->sumN);
    std::vector<int> rec_pt(ctx->nrec, -1), susp_b(P), susp_e(P);
    for (int s = 0; s < ctx->S; ++s)
        for (int k = ctx->body_off[s]; k < ctx->body_off[s + 1]; ++k) {
            susp_b[k] = ctx->src_off[ctx->body_off[s]];
            susp_e[k] = ctx->src_off[ctx->body_off[s + 1]];
        }
    for (int k = 0; k < P; ++k) {
        const ShapeHost &sh = ctx->shapes[ctx->shape_id[k]];
        const double *R = &ctx->rot[9 * k];
        for (int i = 0; i < sh.M; ++i) {
            double x[3];
            for (int a = 0; a < 3; ++a)
                x[a] = R[3 * a] * sh.X0[3 * i] + R[3 * a + 1] * sh.X0[3 * i + 1] + R[3 * a + 2] * sh.X0[3 * i + 2];
            const int t = ctx->tgt_off[k] + i;
            float kb;
            std::memcpy(&kb, &k, sizeof(float));  // body id stored as int bits
            tgt_pos[t] = make_float4((float)x[0], (float)x[1], (float)x[2], kb);
            for (int a = 0; a < 3; ++a) tgt64[3 * (size_t)t + a] = x[a];
        }
        for (int j = 0; j < sh.N; ++j) {
            double y[3];
            for (int a = 0; a < 3; ++a)
                y[a] = R[3 * a] * sh.Y0[3 * j] + R[3 * a + 1] * sh.Y0[3 * j + 1] + R[3 * a + 2] * sh.Y0[3 * j + 2];
            const int q = ctx->src_off[k] + j;
            src_pos[q] = make_float4((float)y[0], (float)y[1], (float)y[2], 0.f);
            for (int a = 0; a < 3; ++a) {
                src64[3 * (size_t)q + a] = y[a];
                src4[4 * (size_t)q + a] = y[a];
            }
            src4[4 * (size_t)q + 3] = (double)k;
            rec_pt[ctx->rec_off[k] + j] = q;
        }
    }
    // padding records point at the body centre: rec_pt = -1 packs (0,0,0) with zero strength
    std::vector<float> rot32(9 * (size_t)P);
    for (size_t i = 0; i < rot32.size(); ++i) rot32[i] = (float)ctx->rot[i];

    CK(ctx->alloc(&ctx->centres_d, 3 * (size_t)P));
    CK(ctx->alloc(&ctx->rot64_d, 9 * (size_t)P));
    CK(ctx->alloc(&ctx->rot_d, 9 * (size_t)P));
    CK(ctx->alloc(&ctx->shape_id_d, P));
    CK(ctx->alloc(&ctx->tgt_pos_d, ctx->sumM));
    CK(ctx->alloc(&ctx->src_pos_d, ctx->sumN));
    CK(ctx->alloc(&ctx->tgt_local64_d, 3 * (size_t)ctx->sumM));
    CK(ctx->alloc(&ctx->src_local64_d, 3 * (size_t)ctx->sumN));
    CK(ctx->alloc(&ctx->src_local4_d, 4 * (size_t)ctx->sumN));
    CK(ctx->alloc(&ctx->tgt_body_d, ctx->sumM));
    CK(ctx->alloc(&ctx->rec_pt_d, ctx->nrec));
    CK(ctx->alloc(&ctx->rec_off_d, P + 1));
    CK(ctx->alloc(&ctx->blk_off_d, P + 1));
    CK(ctx->alloc(&ctx->tgt_off_d, P + 1));
    CK(ctx->alloc(&ctx->src_off_d, P + 1));
    CK(ctx->alloc(&ctx->susp_src_begin_d, P));
    CK(ctx->alloc(&ctx->susp_src_end_d, P));
    CK(ctx->alloc(&ctx->err_d, 1));
    CK(cudaMemset(ctx->err_d, 0, sizeof(int)));
    CK(cudaMemcpy(ctx->centres_d, ctx->centres.data(), sizeof(double) * 3 * P, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->rot64_d, ctx->rot.data(), sizeof(double) * 9 * P, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->rot_d, rot32.data(), sizeof(float) * 9 * P, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->shape_id_d, ctx->shape_id.data(), sizeof(int) * P, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->tgt_pos_d, tgt_pos.data(), sizeof(float4) * ctx->sumM, cudaMemcpyHostToDevice));
    if (ctx->opt.precision == 3) {  // compensated pair sums: x = hi + lo, hi on the 1/MFS_XGRID grid
        std::vector<float4> hi(ctx->sumM), lo(ctx->sumM);
        for (int t = 0; t < ctx->sumM; ++t) {
            float h[3], l[3];
            for (int a = 0; a < 3; ++a) {
                const double x = tgt64[3 * (size_t)t + a], xh = std::rint(x * MFS_XGRID) / MFS_XGRID;
                h[a] = (float)xh;
                l[a] = (float)(x - xh);
            }
            hi[t] = make_float4(h[0], h[1], h[2], 0.f);
            lo[t] = make_float4(l[0], l[1], l[2], 0.f);
        }
        CK(ctx->alloc(&ctx->tgt_hi_d, ctx->sumM));
        CK(ctx->alloc(&ctx->tgt_lo_d, ctx->sumM));
        CK(cudaMemcpy(ctx->tgt_hi_d, hi.data(), sizeof(float4) * ctx->sumM, cudaMemcpyHostToDevice));
        CK(cudaMemcpy(ctx->tgt_lo_d, lo.data(), sizeof(float4) * ctx->sumM, cudaMemcpyHostToDevice));
    }
    CK(cudaMemcpy(ctx->src_pos_d, src_pos.data(), sizeof(float4) * ctx->sumN, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->tgt_local64_d, tgt64.data(), sizeof(double) * tgt64.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->src_local64_d, src64.data(), sizeof(double) * src64.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->src_local4_d, src4.data(), sizeof(double) * src4.size(), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->tgt_body_d, ctx->tgt_body.data(), sizeof(int) * ctx->sumM, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->rec_pt_d, rec_pt.data(), sizeof(int) * ctx->nrec, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->rec_off_d, ctx->rec_off.data(), sizeof(int) * (P + 1), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->blk_off_d, ctx->blk_off.data(), sizeof(long long) * (P + 1), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->tgt_off_d, ctx->tgt_off.data(), sizeof(int) * (P + 1), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->src_off_d, ctx->src_off.data(), sizeof(int) * (P + 1), cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->susp_src_begin_d, susp_b.data(), sizeof(int) * P, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->susp_src_end_d, susp_e.data(), sizeof(int) * P, cudaMemcpyHostToDevice));
    {
        std::vector<double> g0(36 * (size_t)num_shapes);
        for (int s = 0; s < num_shapes; ++s) std::memcpy(&g0[36 * s], ctx->shapes[s].G0inv, sizeof(double) * 36);
        CK(ctx->alloc(&ctx->G0inv_d, g0.size()));
        CK(cudaMemcpy(ctx->G0inv_d, g0.data(), sizeof(double) * g0.size(), cudaMemcpyHostToDevice));
    }

    // per-shape one-body factors: S_L and its SVD in FP64 (cuSOLVER), then the apply factors
    cusolverDnHandle_t solver = nullptr;
    if (cusolverDnCreate(&solver) != CUSOLVER_STATUS_SUCCESS) {
        ctx->last_error = "cusolverDnCreate failed";
        return MFS_ERR_CUDA;
    }
    cusolverDnSetStream(solver, st);
    const int D = ctx->D;
    const int R = ctx->opt.max_rhs;
    mfs_status status = MFS_OK;
    for (int s = 0; s < num_shapes && status == MFS_OK; ++s) status = build_shape_factors(ctx, solver, s, 0, st);
    for (int s = 0; s < num_shapes && status == MFS_OK; ++s) status = alloc_apply_scratch(ctx, ctx->shapes[s], st);
    cusolverDnDestroy(solver);
    if (status != MFS_OK) return status;

    // work buffers
    // every layout a forward pair-kernel entry of this kind may use: plain, f32x2 (Stokes and Laplace),
    // compensated
    const int recf = std::max({pair_record_floats(D, R, 0), pair_record_floats(D, R, 1),
                               ctx->opt.precision == 3 ? pair_record_floats(D, R, 2) : 0});
    ctx->rec_floats = recf;
    CK(ctx->alloc(&ctx->rec_d, (size_t)ctx->nrec * recf));
    CK(cudaMemset(ctx->rec_d, 0, sizeof(float) * (size_t)ctx->nrec * recf));
    CK(ctx->alloc(&ctx->lam_d, (size_t)R * ctx->sumN * D));
    if (ctx->opt.precision == 1)
        CK(ctx->alloc(&ctx->raw_d, R * D * std::max((size_t)fp64_chunks(ctx, ctx->sumM) * ctx->sumM,
                                                    (size_t)fp64_chunks(ctx, ctx->sumN, true) * ctx->sumN)));
    CK(cudaMallocHost(&ctx->done_h, 2 * sizeof(int)));
    CK(cudaEventCreate(&ctx->ev0));
    CK(cudaEventCreate(&ctx->ev1));
    CK(cudaEventCreate(&ctx->evp0));
    CK(cudaEventCreate(&ctx->evp1));
    if (ctx->opt.farfield) {  // forward sums: proxy sources, collocation targets
        auto &F = ctx->ff;
        F.src_colloc = false;
        F.src_pos = ctx->src_pos_d;
        F.rec_pt = ctx->rec_pt_d;
        F.nsrc = ctx->sumN;
        F.nrec = ctx->nrec;
        F.rec_off = &ctx->rec_off;
        F.tgt_pos = ctx->tgt_pos_d;
        F.tgt_off = &ctx->tgt_off;
        F.ntgt = ctx->sumM;
        CKS(ff_setup(ctx, F, st));
    }
    CK(cudaStreamSynchronize(st));
    ctx->ms_setup = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return MFS_OK;
}

// Time every pair-kernel variant for (D, nrhs) on the actual geometry and keep the fastest.
static mfs_status autotune(mfs_ctx *ctx, int nrhs, cudaStream_t st) {
    int count = 0;
    const PairVariant *v = pair_variants(&count);
    double best = 1e300;
    int best_i = -1;
    // zero strengths: the timing does not depend on the values
    CK(cudaMemsetAsync(ctx->lam_d, 0, sizeof(double) * (size_t)nrhs * ctx->sumN * ctx->D, st));
    // Large problems are timed on a sample: the targets of the first bodies of the first suspension
    // against all of its sources, about 4e10 pairs (tens of milliseconds, every SM busy), so that
    // trying every variant costs a fraction of one pair sum.
    const double sample_pairs = 4e10;
    bool sample = pair_count(ctx, 0) > 2.0 * sample_pairs;
    std::vector<int> toff_s;
    int nt_s = 0;
    if (sample) {
        const int B0 = ctx->body_off[0], B1 = ctx->body_off[1];
        const double ns = ctx->src_off[B1] - ctx->src_off[B0];
        int kb = B0;
        double acc = 0.0;
        while (kb < B1 && acc < sample_pairs) {
            acc += (double)(ctx->tgt_off[kb + 1] - ctx->tgt_off[kb]) * ns;
            ++kb;
        }
        toff_s.assign(ctx->tgt_off.begin(), ctx->tgt_off.end());
        for (int k = kb; k <= ctx->P; ++k) toff_s[k] = ctx->tgt_off[kb];
        nt_s = ctx->tgt_off[kb];
        sample = nt_s > 0;
    }
    for (int i = 0; i < count; ++i) {
        if (v[i].grad || v[i].D != ctx->D || v[i].nrhs != nrhs || v[i].comp != (ctx->opt.precision == 3)) continue;
        if (pair_occupancy(i) <= 0) continue;
        PairPlan local;
        PairPlan *plan = &local;
        if (sample)
            CKS(build_plan_for(ctx, i, 0, toff_s, ctx->blk_off, nt_s, local));
        else
            CKS(get_plan(ctx, i, 0, &plan));
        struct Release {
            mfs_ctx *c;
            PairPlan *p;
            ~Release() {
                if (p->tiles) release_plan(c, *p);
            }
        } release{ctx, &local};
        const PairWork w = work_of(*plan);
        if (w.total_units == 0) return MFS_OK;
        CK(pack_for(ctx, i, ctx->lam_d, nrhs, st));
        float ms_best = 1e30f;
        for (int rep = 0; rep < 3; ++rep) {
            CK(cudaEventRecord(ctx->ev0, st));
            CK(pair_launch(i, geom_of(ctx), w, ctx->err_d, st));
            CK(cudaEventRecord(ctx->ev1, st));
            CK(cudaEventSynchronize(ctx->ev1));
            float ms = 0.f;
            cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1);
            if (rep > 0) ms_best = std::min(ms_best, ms);
        }
        if (ms_best < best) {
            best = ms_best;
            best_i = i;
        }
    }
    ctx->best_variant[ctx->D == 3][nrhs] = best_i;
    return check_device_error(ctx, st);
}

extern "C" {

mfs_status mfs_setup(mfs_ctx **out, mfs_kind kind, const mfs_bodies *bodies, int32_t num_shapes,
                     const mfs_pointset *proxy, const mfs_pointset *colloc, const mfs_options *opt, void *stream) {
    g_setup_error.clear();
    if (!out || !bodies || !proxy || !colloc || num_shapes <= 0 || bodies->num_bodies <= 0 || !bodies->centers ||
        (kind != MFS_LAPLACE && kind != MFS_STOKES)) {
        g_setup_error = "mfs_setup: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    *out = nullptr;
    std::unique_ptr<mfs_ctx> ctx(new mfs_ctx());
    if (opt) ctx->opt = *opt; else mfs_default_options(&ctx->opt);
    if (ctx->opt.max_rhs < 1 || ctx->opt.max_rhs > 4 || ctx->opt.max_iter < 1 || ctx->opt.restart < 1 ||
        ctx->opt.restart > 1023 || !(ctx->opt.mu > 0.0) || !(ctx->opt.gmres_tol >= 0.0) ||
        ctx->opt.precision < 0 || ctx->opt.precision > 3 || !(ctx->opt.eps_trunc >= 0.0)) {
        g_setup_error = "mfs_setup: invalid options";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->opt.farfield != 0 && (ctx->opt.farfield != 1 || (ctx->opt.precision != 0 && ctx->opt.precision != 2))) {
        g_setup_error = "mfs_setup: farfield must be 0 or 1, and 1 needs precision 0 or 2 (FP32 pair sums)";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->opt.farfield == 1 && !(ctx->opt.farfield_separation >= FF_MIN_SEPARATION && ctx->opt.farfield_separation <= 10.0)) {
        g_setup_error = "mfs_setup: farfield_separation must lie in [2.5, 10]";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->opt.max_iter > ctx->opt.restart) {
        g_setup_error = "mfs_setup: max_iter above restart is not supported (no restarted GMRES)";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->opt.pair_variant >= 0) {  // a forced pair-kernel variant: a forward sum of this kind's d
        int count = 0;
        const PairVariant *vv = pair_variants(&count);
        const int pv = ctx->opt.pair_variant;
        if (pv >= count || vv[pv].grad || vv[pv].D != (kind == MFS_STOKES ? 3 : 1) ||
            vv[pv].nrhs > ctx->opt.max_rhs || vv[pv].comp != (ctx->opt.precision == 3)) {
            g_setup_error = "mfs_setup: pair_variant is not a forward pair-sum variant of this kind";
            return MFS_ERR_INVALID_ARG;
        }
        ctx->best_variant[kind == MFS_STOKES][vv[pv].nrhs] = pv;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        g_setup_error = "mfs_setup: no CUDA device";
        return MFS_ERR_CUDA;
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (call_pool(dev, ctx->pool) != cudaSuccess) {
        cudaGetLastError();
        g_setup_error = "mfs_setup: cannot create a memory pool";
        return MFS_ERR_CUDA;
    }
    mfs_status s = setup_impl(ctx.get(), kind, bodies, num_shapes, proxy, colloc, st);
    if (s == MFS_OK && ctx->opt.autotune && ctx->opt.precision != 1 && ctx->best_variant[kind == MFS_STOKES][1] < 0) {
        // tune the single-rhs variant now; other nrhs on first use
        s = autotune(ctx.get(), 1, st);
    }
    if (s != MFS_OK) {
        g_setup_error = ctx->last_error;
        return s;
    }
    *out = ctx.release();
    return MFS_OK;
}

mfs_status mfs_update_centers(mfs_ctx *ctx, const double *centers, void *stream) {
    if (!ctx || !centers) return MFS_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (is_device_ptr(centers)) {
        CK(cudaMemcpyAsync(ctx->centres.data(), centers, sizeof(double) * 3 * ctx->P, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
    } else {
        std::memcpy(ctx->centres.data(), centers, sizeof(double) * 3 * ctx->P);
    }
    for (double v : ctx->centres)
        if (!std::isfinite(v)) {
            ctx->last_error = "non-finite body centre";
            return MFS_ERR_INVALID_ARG;
        }
    CK(cudaMemcpyAsync(ctx->centres_d, ctx->centres.data(), sizeof(double) * 3 * ctx->P, cudaMemcpyHostToDevice, st));
    CK(cudaStreamSynchronize(st));
    for (auto *F : {&ctx->ff, &ctx->ffT}) {  // the treecodes' trees, node centres and lists follow the bodies
        if (!F->ready) continue;
        CK(cudaDeviceSynchronize());
        ff_release_geometry(ctx, *F);
        CKS(ff_setup(ctx, *F, st));
    }
    return MFS_OK;
}

mfs_status mfs_matvec(mfs_ctx *ctx, const double *gamma, double *y, int32_t nrhs, void *stream) {
    if (!ctx || !gamma || !y || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_matvec: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const size_t n = (size_t)nrhs * ctx->sumM * ctx->D;
    Staged gi, yo;
    CKS(stage_in(ctx, gi, gamma, n, st));
    CKS(stage_out_alloc(ctx, yo, y, n, st));
    CKS(matvec_dev(ctx, gi.d, yo.d, nrhs, st));
    CKS(stage_out_finish(ctx, yo, st));
    return check_device_error(ctx, st);
}

mfs_status mfs_matvec_transposed(mfs_ctx *ctx, const double *w, double *y, int32_t nrhs, void *stream) {
    if (!ctx || !w || !y || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_matvec_transposed: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->kind != MFS_STOKES) {
        ctx->last_error = "mfs_matvec_transposed: Stokes contexts only";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    CKS(ensure_transposed(ctx));
    const size_t n = (size_t)nrhs * ctx->sumM * 3;
    Staged wi, yo;
    CKS(stage_in(ctx, wi, w, n, st));
    CKS(stage_out_alloc(ctx, yo, y, n, st));
    CKS(matvec_T_dev(ctx, wi.d, yo.d, nrhs, st));
    CKS(stage_out_finish(ctx, yo, st));
    return check_device_error(ctx, st);
}

mfs_status mfs_precond_apply(mfs_ctx *ctx, const double *gamma, double *lambda, int32_t project, int32_t nrhs,
                             void *stream) {
    if (!ctx || !gamma || !lambda || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_precond_apply: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    Staged gi, lo;
    CKS(stage_in(ctx, gi, gamma, (size_t)nrhs * ctx->sumM * ctx->D, st));
    CKS(stage_out_alloc(ctx, lo, lambda, (size_t)nrhs * ctx->sumN * ctx->D, st));
    CKS(precond_apply_dev(ctx, gi.d, lo.d, project ? 1 : 0, nrhs, st));
    CKS(stage_out_finish(ctx, lo, st));
    return MFS_OK;
}

mfs_status mfs_pair_sum(mfs_ctx *ctx, const double *strengths, double *u, int32_t nrhs, int32_t include_self,
                        void *stream) {
    if (!ctx || !strengths || !u || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_pair_sum: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    Staged si, uo;
    CKS(stage_in(ctx, si, strengths, (size_t)nrhs * ctx->sumN * ctx->D, st));
    CKS(stage_out_alloc(ctx, uo, u, (size_t)nrhs * ctx->sumM * ctx->D, st));
    CKS(pair_apply(ctx, si.d, uo.d, nullptr, 0.0, 1.0, nrhs, include_self ? 1 : 0, st));
    CKS(stage_out_finish(ctx, uo, st));
    return check_device_error(ctx, st);
}

// Where a solve's gamma goes: it is kept for mfs_mobility_vjp and mfs_evaluate.
static mfs_status keep_buffers(mfs_ctx *ctx) {
    if (!ctx->keep_gamma) CK(ctx->alloc(&ctx->keep_gamma, (size_t)ctx->opt.max_rhs * ctx->sumM * ctx->D));
    if (!ctx->keep_lam0) CK(ctx->alloc(&ctx->keep_lam0, (size_t)ctx->opt.max_rhs * ctx->P * 6));
    ctx->last_solve = 0;  // until this one is done
    return MFS_OK;
}

// Keep the inputs a (and b), n doubles each, of the solve just enqueued (kind: 1 mobility, 2 elastance,
// 3 resistance, 4 capacitance), whose gamma is in keep_gamma, and wait for it.  It counts as the last
// solve only when the device reported no error: what a kernel that gave up left behind is not a solution.
static mfs_status keep_and_finish(mfs_ctx *ctx, int kind, int nrhs, const double *a, const double *b, size_t n,
                                  cudaStream_t st, SolveStats &ss) {
    if (a) CK(cudaMemcpyAsync(ctx->keep_lam0, a, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
    if (b) CK(cudaMemcpyAsync(ctx->keep_lam0 + n, b, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
    CKS(gmres_finish(ctx, st, ss));
    ctx->last_solve = kind;
    ctx->last_nrhs = nrhs;
    return MFS_OK;
}

static void begin_call(mfs_ctx *ctx) {
    ctx->launches = 0;
    ctx->pair_launches = 0;
    ctx->pair_ms_acc = 0.0;
}

static double pair_profile_ms(mfs_ctx *ctx) {
    if (!ctx->opt.profile) return 0.0;
    double total = 0.0;
    for (int i = 0; i < ctx->pair_launches && 2 * (size_t)i + 1 < ctx->pev.size(); ++i) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, ctx->pev[2 * i], ctx->pev[2 * i + 1]) == cudaSuccess) total += ms;
    }
    return total;
}

static mfs_status finish_info(mfs_ctx *ctx, mfs_solve_info *info, const SolveStats &ss, float ms, int nrhs,
                              bool rhs_pairs = true) {
    ctx->pair_ms_acc = pair_profile_ms(ctx);
    if (info) {
        info->launches = ctx->launches;
        info->pair_launches = ctx->pair_launches;
        info->iters = ss.iters;
        info->converged = ss.converged;
        info->matvecs = ss.matvecs;
        info->lanes = nrhs * ctx->S;
        info->rel_residual = ss.resid;
        info->ms_setup = ctx->ms_setup;
        info->ms_solve = ms;
        info->ms_pairs = ctx->pair_ms_acc;
        info->pairs = pair_count(ctx, 0) * ss.matvecs + (rhs_pairs ? pair_count(ctx, 1) : 0.0);
        info->pairs_evaluated = info->pairs;
        if (ctx->ff.ready) {  // what the treecode's launches evaluated for the same sums
            auto evaluated = [&](int include_self) {
                const int v = forward_variant(ctx, nrhs);
                const auto d = ctx->ff.direct.find(v * 2 + include_self);
                const int c = ff_check_variant(ctx->D, nrhs, v);
                const auto u = ctx->ff.up.find(c), l = ctx->ff.loc.find(c);
                return (d == ctx->ff.direct.end() ? 0.0 : d->second.pairs) +
                       (u == ctx->ff.up.end() ? 0.0 : u->second.pairs) +
                       (l == ctx->ff.loc.end() ? 0.0 : l->second.pairs);
            };
            info->pairs_evaluated = evaluated(0) * ss.matvecs + (rhs_pairs ? evaluated(1) : 0.0);
        }
    }
    if (ss.breakdown) {
        ctx->last_error = "GMRES breakdown: non-finite residual";
        return MFS_ERR_BREAKDOWN;
    }
    if (!ss.converged) {
        ctx->last_error = "GMRES did not reach the tolerance within max_iter";
        return MFS_ERR_NOT_CONVERGED;
    }
    return MFS_OK;
}

mfs_status mfs_solve_mobility(mfs_ctx *ctx, const double *F, const double *T, double *U, double *Omega, int32_t nrhs,
                              mfs_solve_info *info, void *stream) {
    if (!ctx || !F || !T || !U || !Omega || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_solve_mobility: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->kind != MFS_STOKES) {
        ctx->last_error = "mfs_solve_mobility needs a Stokes context";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const size_t nb = (size_t)nrhs * ctx->P * 3;
    Staged Fi, Ti, Uo, Oo;
    CKS(stage_in(ctx, Fi, F, nb, st));
    CKS(stage_in(ctx, Ti, T, nb, st));
    CKS(stage_out_alloc(ctx, Uo, U, nb, st));
    CKS(stage_out_alloc(ctx, Oo, Omega, nb, st));
    if (ctx->opt.autotune && ctx->opt.precision != 1 && ctx->best_variant[1][nrhs] < 0) CKS(autotune(ctx, nrhs, st));
    CKS(ensure_gmres(ctx, nrhs));
    CKS(keep_buffers(ctx));
    begin_call(ctx);
    CK(cudaEventRecord(ctx->ev0, st));
    ctx->launches += 1;
    // lambda_0 and b = -u_0 (all pairs, Eq. stou0)
    CK(completion_stokes(Fi.d, Ti.d, nrhs, ctx->P, ctx->rot64_d, ctx->G0inv_d, ctx->shape_id_d, ctx->src_local64_d,
                         ctx->src_off_d, ctx->sumN, ctx->lam_d, st));
    CKS(pair_apply(ctx, ctx->lam_d, ctx->b_d, nullptr, 0.0, -1.0, nrhs, 1, st));
    SolveStats ss;
    CKS(gmres_solve(ctx, nrhs, st, ctx->keep_gamma, ss));
    // lambda = S_L^+ gamma, [U; Omega] = -K_N^T lambda (Eq. getU)
    CKS(precond_apply_dev(ctx, ctx->keep_gamma, ctx->lam_d, 0, nrhs, st));
    CK(extract_stokes(ctx->lam_d, nrhs, ctx->P, ctx->src_local64_d, ctx->src_off_d, ctx->sumN, Uo.d, Oo.d, st));
    ctx->launches += 1;
    CK(cudaEventRecord(ctx->ev1, st));
    // keep gamma, F and T for mfs_mobility_vjp and mfs_evaluate (outside the timed region)
    CKS(keep_and_finish(ctx, 1, nrhs, Fi.d, Ti.d, nb, st, ss));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1);
    CKS(stage_out_finish(ctx, Uo, st));
    CKS(stage_out_finish(ctx, Oo, st));
    return finish_info(ctx, info, ss, ms, nrhs);
}

mfs_status mfs_solve_elastance(mfs_ctx *ctx, const double *Q, double *V, int32_t nrhs, mfs_solve_info *info,
                               void *stream) {
    if (!ctx || !Q || !V || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_solve_elastance: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->kind != MFS_LAPLACE) {
        ctx->last_error = "mfs_solve_elastance needs a Laplace context";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const size_t nb = (size_t)nrhs * ctx->P;
    Staged Qi, Vo;
    CKS(stage_in(ctx, Qi, Q, nb, st));
    CKS(stage_out_alloc(ctx, Vo, V, nb, st));
    if (ctx->opt.autotune && ctx->opt.precision != 1 && ctx->best_variant[0][nrhs] < 0) CKS(autotune(ctx, nrhs, st));
    CKS(ensure_gmres(ctx, nrhs));
    CKS(keep_buffers(ctx));
    begin_call(ctx);
    CK(cudaEventRecord(ctx->ev0, st));
    ctx->launches += 1;
    CK(completion_laplace(Qi.d, nrhs, ctx->P, ctx->src_off_d, ctx->sumN, ctx->lam_d, st));  // Eq. al0
    CKS(pair_apply(ctx, ctx->lam_d, ctx->b_d, nullptr, 0.0, -1.0, nrhs, 1, st));           // b = -u_0, Eq. erhsK
    SolveStats ss;
    CKS(gmres_solve(ctx, nrhs, st, ctx->keep_gamma, ss));
    CKS(precond_apply_dev(ctx, ctx->keep_gamma, ctx->lam_d, 0, nrhs, st));
    CK(extract_laplace(ctx->lam_d, nrhs, ctx->P, ctx->src_off_d, ctx->sumN, Vo.d, st));  // Eq. vkal
    ctx->launches += 1;
    CK(cudaEventRecord(ctx->ev1, st));
    CKS(keep_and_finish(ctx, 2, nrhs, Qi.d, nullptr, nb, st, ss));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1);
    CKS(stage_out_finish(ctx, Vo, st));
    return finish_info(ctx, info, ss, ms, nrhs);
}

}  // extern "C"

namespace {
// Selects the Dirichlet factor set for the duration of one solve, on every return path.
struct DirichletScope {
    mfs_ctx *ctx;
    explicit DirichletScope(mfs_ctx *c) : ctx(c) { ctx->fset = 1; }
    ~DirichletScope() { ctx->fset = 0; }
};

// Algorithm 1 SOLVE with the Dirichlet data already in ctx->b_d: gamma by GMRES on Eq. 2sysprec, then
// the strengths alpha = S^+ gamma in ctx->lam_d.
mfs_status dirichlet_solve(mfs_ctx *ctx, int nrhs, cudaStream_t st, SolveStats &ss) {
    DirichletScope scope(ctx);
    CKS(gmres_solve(ctx, nrhs, st, ctx->keep_gamma, ss));
    CKS(precond_apply_dev(ctx, ctx->keep_gamma, ctx->lam_d, 0, nrhs, st));
    return MFS_OK;
}
}  // namespace

extern "C" {

mfs_status mfs_dirichlet_matvec(mfs_ctx *ctx, const double *gamma, double *y, int32_t nrhs, void *stream) {
    if (!ctx || !gamma || !y || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_dirichlet_matvec: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    CKS(ensure_dirichlet(ctx, st));
    Staged gi, yo;
    const size_t n = (size_t)nrhs * ctx->sumM * ctx->D;
    CKS(stage_in(ctx, gi, gamma, n, st));
    CKS(stage_out_alloc(ctx, yo, y, n, st));
    {
        DirichletScope scope(ctx);
        CKS(matvec_dev(ctx, gi.d, yo.d, nrhs, st));
    }
    CKS(stage_out_finish(ctx, yo, st));
    return check_device_error(ctx, st);
}

mfs_status mfs_dirichlet_apply(mfs_ctx *ctx, const double *gamma, double *alpha, int32_t nrhs, void *stream) {
    if (!ctx || !gamma || !alpha || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_dirichlet_apply: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    CKS(ensure_dirichlet(ctx, st));
    Staged gi, ao;
    CKS(stage_in(ctx, gi, gamma, (size_t)nrhs * ctx->sumM * ctx->D, st));
    CKS(stage_out_alloc(ctx, ao, alpha, (size_t)nrhs * ctx->sumN * ctx->D, st));
    {
        DirichletScope scope(ctx);
        CKS(precond_apply_dev(ctx, gi.d, ao.d, 0, nrhs, st));
    }
    CKS(stage_out_finish(ctx, ao, st));
    return check_device_error(ctx, st);
}

mfs_status mfs_solve_resistance(mfs_ctx *ctx, const double *U, const double *Omega, double *F, double *T,
                                int32_t nrhs, mfs_solve_info *info, void *stream) {
    if (!ctx || !U || !Omega || !F || !T || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_solve_resistance: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->kind != MFS_STOKES) {
        ctx->last_error = "mfs_solve_resistance needs a Stokes context";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const size_t nb = (size_t)nrhs * ctx->P * 3;
    Staged Ui, Oi, Fo, To;
    CKS(stage_in(ctx, Ui, U, nb, st));
    CKS(stage_in(ctx, Oi, Omega, nb, st));
    CKS(stage_out_alloc(ctx, Fo, F, nb, st));
    CKS(stage_out_alloc(ctx, To, T, nb, st));
    CKS(ensure_dirichlet(ctx, st));
    if (ctx->opt.autotune && ctx->opt.precision != 1 && ctx->best_variant[1][nrhs] < 0) CKS(autotune(ctx, nrhs, st));
    CKS(ensure_gmres(ctx, nrhs));
    CKS(keep_buffers(ctx));
    begin_call(ctx);
    CK(cudaEventRecord(ctx->ev0, st));
    // b = K_M U (Sec. 2.2), then Algorithm 1 and [f; t] = K_N^T lambda (Eq. force_def)
    CK(dirichlet_rhs_stokes(Ui.d, Oi.d, nrhs, ctx->P, ctx->tgt_local64_d, ctx->tgt_off_d, ctx->sumM, ctx->b_d, st));
    SolveStats ss;
    CKS(dirichlet_solve(ctx, nrhs, st, ss));
    CK(extract_stokes(ctx->lam_d, nrhs, ctx->P, ctx->src_local64_d, ctx->src_off_d, ctx->sumN, Fo.d, To.d, st, 1.0));
    ctx->launches += 2;
    CK(cudaEventRecord(ctx->ev1, st));
    CKS(keep_and_finish(ctx, 3, nrhs, nullptr, nullptr, 0, st, ss));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1);
    CKS(stage_out_finish(ctx, Fo, st));
    CKS(stage_out_finish(ctx, To, st));
    return finish_info(ctx, info, ss, ms, nrhs, false);
}

mfs_status mfs_solve_capacitance(mfs_ctx *ctx, const double *phi, double *q, int32_t nrhs, mfs_solve_info *info,
                                 void *stream) {
    if (!ctx || !phi || !q || nrhs < 1 || nrhs > ctx->opt.max_rhs) {
        if (ctx) ctx->last_error = "mfs_solve_capacitance: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->kind != MFS_LAPLACE) {
        ctx->last_error = "mfs_solve_capacitance needs a Laplace context";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const size_t nb = (size_t)nrhs * ctx->P;
    Staged Pi, Qo;
    CKS(stage_in(ctx, Pi, phi, nb, st));
    CKS(stage_out_alloc(ctx, Qo, q, nb, st));
    CKS(ensure_dirichlet(ctx, st));
    if (ctx->opt.autotune && ctx->opt.precision != 1 && ctx->best_variant[0][nrhs] < 0) CKS(autotune(ctx, nrhs, st));
    CKS(ensure_gmres(ctx, nrhs));
    CKS(keep_buffers(ctx));
    begin_call(ctx);
    CK(cudaEventRecord(ctx->ev0, st));
    // eta = phi 1_M (Sec. 2.1), then Algorithm 1 and q = sum alpha (Eq. qkgauss)
    CK(dirichlet_rhs_laplace(Pi.d, nrhs, ctx->P, ctx->tgt_off_d, ctx->sumM, ctx->b_d, st));
    SolveStats ss;
    CKS(dirichlet_solve(ctx, nrhs, st, ss));
    CK(extract_laplace(ctx->lam_d, nrhs, ctx->P, ctx->src_off_d, ctx->sumN, Qo.d, st, 1));
    ctx->launches += 2;
    CK(cudaEventRecord(ctx->ev1, st));
    CKS(keep_and_finish(ctx, 4, nrhs, nullptr, nullptr, 0, st, ss));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1);
    CKS(stage_out_finish(ctx, Qo, st));
    return finish_info(ctx, info, ss, ms, nrhs, false);
}

}  // extern "C"

// FP64 -> FP32 (adjoint strengths for the gradient kernel)
static __global__ void to_f32_kernel(const double *x, float *y, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] = (float)x[i];
}

// dL/dc_k = scale * (source-side sum of body k) - (sum over the targets of body k of their gradient sums)
static __global__ void centre_grad_kernel(const double *gradT, const int *tgt_off, const double *src_grad, double scale,
                                          double *dc) {
    const int k = blockIdx.x;
    double acc[3] = {0.0, 0.0, 0.0};
    for (int i = tgt_off[k] + threadIdx.x; i < tgt_off[k + 1]; i += blockDim.x)
        for (int c = 0; c < 3; ++c) acc[c] += gradT[3 * (size_t)i + c];
    __shared__ double red[3][128];
    for (int c = 0; c < 3; ++c) red[c][threadIdx.x] = acc[c];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int c = 0; c < 3; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 3) dc[3 * k + threadIdx.x] = scale * src_grad[3 * k + threadIdx.x] - red[threadIdx.x][0];
}

// The centre gradient from the two treecode passes: dc_k = -(sum over body k's collocation points of gc)
// - (sum over its proxy points of gp), both already scaled.
static __global__ void centre_grad_ff_kernel(const double *gc, const int *tgt_off, const double *gp, const int *src_off,
                                             double *dc) {
    const int k = blockIdx.x;
    double acc[3] = {0.0, 0.0, 0.0};
    for (int i = tgt_off[k] + threadIdx.x; i < tgt_off[k + 1]; i += blockDim.x)
        for (int c = 0; c < 3; ++c) acc[c] += gc[3 * (size_t)i + c];
    for (int j = src_off[k] + threadIdx.x; j < src_off[k + 1]; j += blockDim.x)
        for (int c = 0; c < 3; ++c) acc[c] += gp[3 * (size_t)j + c];
    __shared__ double red[3][128];
    for (int c = 0; c < 3; ++c) red[c][threadIdx.x] = acc[c];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int c = 0; c < 3; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 3) dc[3 * k + threadIdx.x] = -red[threadIdx.x][0];
}

// [dF; dT]_k = G_k^{-1} v_k with G_k = R_2 G_0 R_2^T (v = -K_N^T z, given as its force and torque parts)
static __global__ void gram_solve_kernel(const double *vf, const double *vt, int P, int nrhs, const double *rot64,
                                         const double *G0inv_shapes, const int *shape_id, double *dF, double *dT) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P * nrhs) return;
    const int k = i % P;
    const double *R = rot64 + 9 * k;
    const double *f = vf + 3 * (size_t)i, *t = vt + 3 * (size_t)i;
    double b[6], a[6];
    for (int c = 0; c < 3; ++c) {
        b[c] = R[c] * f[0] + R[3 + c] * f[1] + R[6 + c] * f[2];
        b[3 + c] = R[c] * t[0] + R[3 + c] * t[1] + R[6 + c] * t[2];
    }
    const double *Gi = G0inv_shapes + 36 * shape_id[k];
    for (int m = 0; m < 6; ++m) {
        double s = 0.0;
        for (int n = 0; n < 6; ++n) s += Gi[m * 6 + n] * b[n];
        a[m] = s;
    }
    for (int c = 0; c < 3; ++c) {
        dF[3 * (size_t)i + c] = R[3 * c] * a[0] + R[3 * c + 1] * a[1] + R[3 * c + 2] * a[2];
        dT[3 * (size_t)i + c] = R[3 * c] * a[3] + R[3 * c + 1] * a[4] + R[3 * c + 2] * a[5];
    }
}

extern "C" {

// Reverse mode of the last mfs_solve_mobility.  With U = E gamma, E = -K_N^T S_L^+ and A gamma = -u_0:
//   g = E^T dL/dU = -(S_L^+)^T K_N [dU; dOmega];  A^T w = g;  mu = lambda_0 + (I - L) S_L^+ gamma;
//   dL/dc_k = -sum_{i in k, j not in k} d/dr[w_i^T G mu_j] + sum_{j in k, i not in k} d/dr[w_i^T G mu_j];
//   dL/d[f; t]_k = -G_k^{-1} K_N^T (S^T w)_k over all pairs (Eq. stou0, Eq. lambda01-02).
mfs_status mfs_mobility_vjp(mfs_ctx *ctx, const double *dU, const double *dOmega, int32_t nrhs, double *dcenters,
                            double *dF, double *dT, void *stream) {
    if (!ctx || !dU || !dOmega || !dcenters || nrhs < 1 || nrhs > ctx->opt.max_rhs || (!dF) != (!dT)) {
        if (ctx) ctx->last_error = "mfs_mobility_vjp: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->kind != MFS_STOKES || ctx->last_solve != 1 || ctx->last_nrhs != nrhs) {
        ctx->last_error = "mfs_mobility_vjp needs a preceding mfs_solve_mobility with the same nrhs";
        return MFS_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int P = ctx->P;
    const size_t nb = (size_t)nrhs * P * 3, nM = (size_t)nrhs * ctx->sumM * 3;
    Staged dUi, dWi, dco, dFo, dTo;
    CKS(stage_in(ctx, dUi, dU, nb, st));
    CKS(stage_in(ctx, dWi, dOmega, nb, st));
    CKS(stage_out_alloc(ctx, dco, dcenters, (size_t)P * 3, st));
    if (dF) {
        CKS(stage_out_alloc(ctx, dFo, dF, nb, st));
        CKS(stage_out_alloc(ctx, dTo, dT, nb, st));
    }
    CKS(ensure_transposed(ctx));
    CKS(ensure_gmres(ctx, nrhs));
    begin_call(ctx);
    // 1. seed g = -(S_L^+)^T K_N [dU; dOmega]
    CK(completion_stokes(dUi.d, dWi.d, nrhs, P, ctx->rot64_d, ctx->eye6_d, ctx->shape_id_d, ctx->src_local64_d,
                         ctx->src_off_d, ctx->sumN, ctx->lam_d, st));
    CKS(precondT_dev(ctx, ctx->lam_d, ctx->tmpM_d, 0, nrhs, st));
    combine_raw_kernel<<<(unsigned)((nM + 255) / 256), 256, 0, st>>>(ctx->tmpM_d, nullptr, 0.0, -1.0, ctx->b_d, nM, 1);
    CK(cudaGetLastError());
    // 2. A^T w = g
    SolveStats ss;
    CKS(gmres_solve(ctx, nrhs, st, ctx->x_d, ss, true));
    CKS(gmres_finish(ctx, st, ss));
    if (ss.breakdown || !ss.converged) {
        ctx->last_error = "adjoint GMRES did not converge";
        return ss.breakdown ? MFS_ERR_BREAKDOWN : MFS_ERR_NOT_CONVERGED;
    }
    // 3. mu = lambda_0 + (I - L) S_L^+ gamma  (lambda_0 rebuilt from the kept F, T)
    double *lam0 = ctx->tmpM_d;  // [nrhs][sum_N][3] fits: sum_N < sum_M
    CK(completion_stokes(ctx->keep_lam0, ctx->keep_lam0 + nb, nrhs, P, ctx->rot64_d, ctx->G0inv_d, ctx->shape_id_d,
                         ctx->src_local64_d, ctx->src_off_d, ctx->sumN, lam0, st));
    CKS(precond_apply_dev(ctx, ctx->keep_gamma, ctx->lam_d, 1, nrhs, st));
    const size_t nN = (size_t)nrhs * ctx->sumN * 3;
    combine_raw_kernel<<<(unsigned)((nN + 255) / 256), 256, 0, st>>>(lam0, ctx->lam_d, 1.0, 1.0, ctx->lam_d, nN, 1);
    CK(cudaGetLastError());
    // 4. centre gradient: pair kernel over off-diagonal pairs with target strengths w, source strengths mu
    int vc = 0, gv = -1;
    const PairVariant *vv = pair_variants(&vc);
    for (int i = 0; i < vc; ++i)
        if (vv[i].grad == 1 && vv[i].nrhs == nrhs) gv = i;  // the centre-gradient entry (not the stress one)
    if (gv < 0) {
        ctx->last_error = "no gradient kernel for this nrhs";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->ff.ready && ctx->ffT.ready) {
        // through the treecodes: the target side on the forward tree (weights w at the collocation
        // points, sources mu), the source side on the transposed tree (weights mu at the proxy
        // points, sources w); tmpM_d (free again) takes the proxy-side gradient
        CKS(ff_grad_apply(ctx, ctx->ff, gv, ctx->lam_d, ctx->x_d, nrhs, ctx->gradT_d, st));
        CKS(ff_grad_apply(ctx, ctx->ffT, gv, ctx->x_d, ctx->lam_d, nrhs, ctx->tmpM_d, st));
        centre_grad_ff_kernel<<<P, 128, 0, st>>>(ctx->gradT_d, ctx->tgt_off_d, ctx->tmpM_d, ctx->src_off_d, dco.d);
        CK(cudaGetLastError());
        ctx->launches += 1;
    } else if (ctx->opt.precision == 1) {
        // FP64 reference, the same two sides as the treecode's: weights w at the collocation points
        // against mu, weights mu at the proxy points against w (roles swapped, sign folded into dc)
        const double scale = kernel_scale(ctx);
        const size_t nc = (size_t)ctx->sumM * 3, np3 = (size_t)ctx->sumN * 3;
        const int Sc = fp64_chunks(ctx, ctx->sumM), Sp = fp64_chunks(ctx, ctx->sumN, true);
        CK(grad_pair_fp64(nrhs, Sc, ctx->tgt_local64_d, ctx->tgt_body_d, ctx->sumM, ctx->x_d, ctx->src_local4_d,
                          ctx->sumN, ctx->susp_src_begin_d, ctx->susp_src_end_d, ctx->src_off_d, ctx->centres_d,
                          ctx->lam_d, ctx->raw_d, st));
        combine_raw_kernel<<<(unsigned)((nc + 255) / 256), 256, 0, st>>>(ctx->raw_d, nullptr, 0.0, scale,
                                                                         ctx->gradT_d, nc, Sc);
        CK(grad_pair_fp64(nrhs, Sp, ctx->src_local64_d, ctx->src_body_d, ctx->sumN, ctx->lam_d, ctx->colloc4_d,
                          ctx->sumM, ctx->colT_begin_d, ctx->colT_end_d, ctx->tgt_off_d, ctx->centres_d, ctx->x_d,
                          ctx->raw_d, st));
        combine_raw_kernel<<<(unsigned)((np3 + 255) / 256), 256, 0, st>>>(ctx->raw_d, nullptr, 0.0, scale,
                                                                          ctx->tmpM_d, np3, Sp);
        centre_grad_ff_kernel<<<P, 128, 0, st>>>(ctx->gradT_d, ctx->tgt_off_d, ctx->tmpM_d, ctx->src_off_d, dco.d);
        CK(cudaGetLastError());
        ctx->launches += 5;
    } else {
        to_f32_kernel<<<1024, 256, 0, st>>>(ctx->x_d, ctx->w32_d, nM);
        CK(pack_sources(3, nrhs, 0, ctx->src_pos_d, ctx->rec_pt_d, ctx->lam_d, ctx->sumN, ctx->nrec, ctx->rec_d, st));
        CK(cudaMemsetAsync(ctx->src_grad_d, 0, sizeof(double) * 3 * P, st));
        PairPlan *plan = nullptr;
        CKS(get_plan(ctx, gv, 0, &plan));
        PairGeom g = geom_of(ctx);
        g.tgt_w = ctx->w32_d;
        PairWork wk = work_of(*plan);
        wk.src_grad = ctx->src_grad_d;
        if (wk.total_units > 0) CK(pair_launch(gv, g, wk, ctx->err_d, st));
        CK(pair_epilogue(3, 1, wk, nullptr, 0.0, kernel_scale(ctx), ctx->gradT_d, ctx->sumM, st));
        centre_grad_kernel<<<P, 128, 0, st>>>(ctx->gradT_d, ctx->tgt_off_d, ctx->src_grad_d, kernel_scale(ctx), dco.d);
        CK(cudaGetLastError());
        ctx->launches += 6;
    }
    // 5. force and torque cotangents
    if (dF) {
        CKS(pair_apply_T(ctx, ctx->x_d, ctx->lam_d, nrhs, 1, st));
        CK(extract_stokes(ctx->lam_d, nrhs, P, ctx->src_local64_d, ctx->src_off_d, ctx->sumN, ctx->six_d,
                          ctx->six_d + nb, st));
        gram_solve_kernel<<<(unsigned)((P * nrhs + 127) / 128), 128, 0, st>>>(
            ctx->six_d, ctx->six_d + nb, P, nrhs, ctx->rot64_d, ctx->G0inv_d, ctx->shape_id_d, dFo.d, dTo.d);
        CK(cudaGetLastError());
        ctx->launches += 2;
        CKS(stage_out_finish(ctx, dFo, st));
        CKS(stage_out_finish(ctx, dTo, st));
    }
    CKS(stage_out_finish(ctx, dco, st));
    CK(cudaStreamSynchronize(st));
    return check_device_error(ctx, st);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Evaluation of the last solve's representation at arbitrary points
// ---------------------------------------------------------------------------
static __global__ void add_kernel(double *a, const double *b, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        a[i] += b[i];
}

// (p, T_x, T_y, T_z) per point and rhs -> pressure [n] and traction [n][3] (the -3 of Eq. traction).
static __global__ void split_stress_kernel(const double *o4, size_t n, double *p, double *t) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        if (p) p[e] = o4[4 * e];
        if (t)
            for (int c = 0; c < 3; ++c) t[3 * e + c] = -3.0 * o4[4 * e + 1 + c];
    }
}

// The stress entry of the pair-kernel table for nrhs (grad = 2), -1 if none.
static int stress_variant(int nrhs) {
    int count = 0;
    const PairVariant *vv = pair_variants(&count);
    for (int i = 0; i < count; ++i)
        if (vv[i].grad == 2 && vv[i].nrhs == nrhs) return i;
    return -1;
}

// out[h][order[i]][c] = in[h][i][c]: back from owner-sorted to the caller's point order.
static __global__ void unsort_kernel(const double *in, const int *order, int np, int D, int nrhs, double *out) {
    const size_t n = (size_t)nrhs * np * D;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const size_t h = e / ((size_t)np * D), r = e % ((size_t)np * D);
        const int i = (int)(r / D), c = (int)(r % D);
        out[(h * np + order[i]) * D + c] = in[e];
    }
}

// Evaluation points grouped by owner body, or by tree position when `tree` (eval_group.cu); device
// arrays in the call's scratch, offsets and, for the tree, each key's largest distance on the host.
struct Grouped {
    std::vector<int> toff;
    std::vector<double> radius;
    float4 *t4 = nullptr;
    float *n32 = nullptr;
    double *t64 = nullptr, *n64 = nullptr;
    int *tbody = nullptr, *order = nullptr;
};

static mfs_status group_points(mfs_ctx *ctx, const double *points, const double *normals, const int32_t *owner, int np,
                               bool tree, bool want64, Scratch &tmp, Grouped &g) {
    const int P = ctx->P;
    cudaStream_t st = tmp.st;
    if (!owner && ctx->S > 1) {
        ctx->last_error = "evaluation: owner bodies are required with several suspensions";
        return MFS_ERR_INVALID_ARG;
    }
    auto device = [&](auto *user, size_t count, auto **out) -> cudaError_t {  // the pointer or a copy of host data
        if (is_device_ptr(user)) {
            *out = user;
            return cudaSuccess;
        }
        typename std::remove_const<typename std::remove_pointer<decltype(user)>::type>::type *d = nullptr;
        cudaError_t e = tmp.alloc(&d, count);
        if (e == cudaSuccess) e = cudaMemcpyAsync(d, user, sizeof(*user) * count, cudaMemcpyHostToDevice, st);
        tmp.host.push_back(nullptr);  // the caller's memory: read before the call returns, errors included
        *out = d;
        return e;
    };
    EvalGroup e;
    e.np = np;
    e.P = P;
    CK(device(points, 3 * (size_t)np, &e.points));
    if (normals) CK(device(normals, 3 * (size_t)np, &e.normals));
    if (owner) CK(device((const int *)owner, (size_t)np, &e.owner));
    e.centres = ctx->centres_d;
    if (tree) {
        e.key_of_body = ctx->ff.pos;
        e.body_of_key = ctx->ff.order;
        CK(tmp.alloc(&e.radius, P));
    }
    CK(tmp.alloc(&e.key, np));
    CK(tmp.alloc(&e.counts, (size_t)eval_chunks(np) * P));
    CK(tmp.alloc(&e.total, P));
    CK(tmp.alloc(&e.toff, P + 1));
    CK(tmp.alloc(&e.order, np));
    CK(tmp.alloc(&e.t4, np));
    CK(tmp.alloc(&e.err, 1));
    if (normals) CK(tmp.alloc(&e.n32, 3 * (size_t)np));
    if (want64) {
        CK(tmp.alloc(&e.t64, 3 * (size_t)np));
        CK(tmp.alloc(&e.tbody, np));
        if (normals) CK(tmp.alloc(&e.n64, 3 * (size_t)np));
    }
    CK(cudaMemsetAsync(e.err, 0, sizeof(int), st));
    CK(eval_group(e, st));
    g.toff.resize(P + 1);
    int bad = 0;
    CK(cudaMemcpyAsync(g.toff.data(), e.toff, sizeof(int) * (P + 1), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(&bad, e.err, sizeof(int), cudaMemcpyDeviceToHost, st));
    if (tree) {
        g.radius.resize(P);
        CK(cudaMemcpyAsync(g.radius.data(), e.radius, sizeof(double) * P, cudaMemcpyDeviceToHost, st));
    }
    CK(cudaStreamSynchronize(st));
    if (bad) {
        ctx->last_error = "evaluation: owner out of range or non-finite point or normal";
        return MFS_ERR_INVALID_ARG;
    }
    g.t4 = e.t4;
    g.n32 = e.n32;
    g.t64 = e.t64;
    g.n64 = e.n64;
    g.tbody = e.tbody;
    g.order = e.order;
    return MFS_OK;
}

namespace {
// The strengths of the representation of the last solve, [nrhs][sum_N][D] into ctx->lam_d:
// mobility (I - L) S_L^+ gamma + lambda_0 (Eq. multirep), elastance (I - L) S_L^+ gamma + alpha_0
// (Eq. erepK), resistance and capacitance S^+ gamma (Eq. reconbal).
mfs_status last_strengths(mfs_ctx *ctx, int nrhs, double *tmp, cudaStream_t st) {
    const int P = ctx->P;
    const size_t ns = (size_t)nrhs * ctx->sumN * ctx->D;
    if (ctx->last_solve >= 3) {
        DirichletScope scope(ctx);
        CKS(precond_apply_dev(ctx, ctx->keep_gamma, ctx->lam_d, 0, nrhs, st));
        return MFS_OK;
    }
    CKS(precond_apply_dev(ctx, ctx->keep_gamma, ctx->lam_d, 1, nrhs, st));
    if (ctx->last_solve == 1) {
        const size_t nb = (size_t)nrhs * P * 3;
        CK(completion_stokes(ctx->keep_lam0, ctx->keep_lam0 + nb, nrhs, P, ctx->rot64_d, ctx->G0inv_d,
                             ctx->shape_id_d, ctx->src_local64_d, ctx->src_off_d, ctx->sumN, tmp, st));
    } else {
        CK(completion_laplace(ctx->keep_lam0, nrhs, P, ctx->src_off_d, ctx->sumN, tmp, st));
    }
    add_kernel<<<(unsigned)std::min<size_t>((ns + 255) / 256, 4096), 256, 0, st>>>(ctx->lam_d, tmp, ns);
    CK(cudaGetLastError());
    return MFS_OK;
}
}  // namespace

// Sums at evaluation points (grouped by tree position) through the treecode (farfield = 1): the upward
// step on the strengths in lam_d (a forward pair-sum entry), the proxy and equivalent records in the
// layout of `variant` (a pair sum for mfs_evaluate, the stress entry for mfs_evaluate_stress), one-off
// interaction lists for the points (each owner's radius that of its farthest point), and the launch of
// `variant` with the grouped normals as target weights (the stress; null otherwise); results land in out
// [nrhs][np][dout] in the caller's order, scaled by `scale`.
static mfs_status ff_points(mfs_ctx *ctx, int variant, const Grouped &gr, int np, int nrhs, int dout, double scale,
                            double *out, Scratch &tmp) {
    auto &F = ctx->ff;
    cudaStream_t st = tmp.st;
    const int P = ctx->P, D = ctx->D, nodes = F.nodes;
    int vc = 0;
    const PairVariant *vv = pair_variants(&vc);
    const int fv = fp32_variant(ctx, D, nrhs);
    CKS(ff_upward(ctx, F, fv, ctx->lam_d, nrhs, st));
    const int layout = vv[variant].packed, REC = pair_record_floats(D, nrhs, layout);
    if (REC > F.rec_floats) {
        ctx->last_error = "far field: record layout larger than its buffer";
        return MFS_ERR_INVALID_ARG;
    }
    CK(pack_sources(D, nrhs, layout, F.src_pos, F.rec_pt, ctx->lam_d, F.nsrc, F.nrec, F.rec, st));
    CK(pack_sources(D, nrhs, layout, F.eq_pos, F.eq_pt, F.mu, nodes * FF_NE, nodes * FF_NE,
                    F.rec + (size_t)F.nrec * REC, st));
    std::vector<double> rad(P);  // by body
    for (int q = 0; q < P; ++q) rad[F.tree.order[q]] = gr.radius[q];
    std::vector<long long> seg_blocks;
    std::vector<int> seg_recs;
    ff_segments(F, seg_blocks, seg_recs);
    std::vector<int> cuts(ctx->body_off.begin(), ctx->body_off.end()), tb;
    const std::vector<int> suspension_of = suspension_of_bodies(ctx);
    FFListPlan lp;
    CKS(build_plan_lists(
        ctx, variant, 1, gr.toff, 0, cuts, seg_blocks, seg_recs,
        [&](int g0, int g1, std::vector<int> &segs) {
            tb.clear();
            for (int q = g0; q <= g1; ++q) tb.push_back(F.tree.order[q]);
            ff_interaction_list(F.tree, F.tree.roots[suspension_of[tb[0]]], tb, ctx->centres.data(), rad.data(),
                                ctx->opt.farfield_separation, 0, segs);
        },
        lp.p, &lp.seg, &lp.cum, lp.pairs, &tmp));
    PairGeom g = ff_geom(F, lp);
    g.tgt = gr.t4;
    g.ntargets = np;
    g.tgt_w = gr.n32;
    PairWork we = work_of(lp.p);
    we.tperm = gr.order;
    CKS(ff_launch(ctx, variant, g, we, st));
    CK(pair_epilogue(dout, nrhs, we, nullptr, 0.0, scale, out, np, st));
    return MFS_OK;
}

extern "C" {

mfs_status mfs_evaluate(mfs_ctx *ctx, const double *points, const int32_t *owner, int32_t npoints, double *out,
                        int32_t nrhs, void *stream) {
    if (!ctx || (npoints > 0 && (!points || !out)) || npoints < 0 || nrhs < 1) {
        if (ctx) ctx->last_error = "mfs_evaluate: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->last_solve == 0 || ctx->last_nrhs != nrhs) {
        ctx->last_error = "mfs_evaluate needs a preceding solve with the same nrhs";
        return MFS_ERR_INVALID_ARG;
    }
    if (npoints == 0) return MFS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const int D = ctx->D, np = npoints;
    Scratch tmp(ctx, st);
    Grouped gr;
    const bool fp64 = ctx->opt.precision == 1;
    CKS(group_points(ctx, points, nullptr, owner, np, ctx->ff.ready, fp64, tmp, gr));
    Staged oo;
    CKS(stage_out_alloc(ctx, oo, out, (size_t)nrhs * np * D, st));
    double *tmp_d = nullptr;
    CK(tmp.alloc(&tmp_d, (size_t)nrhs * ctx->sumN * D));
    CKS(last_strengths(ctx, nrhs, tmp_d, st));
    const double scale = kernel_scale(ctx);
    if (fp64) {  // FP64 direct sums
        double *raw_d = nullptr, *sorted_d = nullptr;
        const int S = fp64_chunks(ctx, np);
        CK(tmp.alloc(&raw_d, (size_t)S * nrhs * np * D));
        CK(tmp.alloc(&sorted_d, (size_t)nrhs * np * D));
        CK(pair_sum_fp64(D, nrhs, S, gr.t64, gr.tbody, np, ctx->src_local4_d, ctx->sumN, ctx->susp_src_begin_d,
                         ctx->susp_src_end_d, ctx->src_off_d, ctx->centres_d, ctx->lam_d, 1, raw_d, st));
        const size_t n = (size_t)nrhs * np * D;
        combine_raw_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(raw_d, nullptr, 0.0, scale, sorted_d, n, S);
        CK(cudaGetLastError());
        unsort_kernel<<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, st>>>(sorted_d, gr.order, np, D,
                                                                                          nrhs, oo.d);
        CK(cudaGetLastError());
    } else {  // the FP32 pair kernel on the new targets, all pairs of the owner's suspension
        const int variant = fp32_variant(ctx, D, nrhs);
        if (variant < 0) {
            ctx->last_error = "no pair-kernel variant for this nrhs";
            return MFS_ERR_INVALID_ARG;
        }
        if (ctx->ff.ready) {  // through the treecode
            CKS(ff_points(ctx, variant, gr, np, nrhs, D, scale, oo.d, tmp));
        } else {
            int vc = 0;
            const PairVariant *vv = pair_variants(&vc);
            PairPlan plan;
            CKS(build_plan_for(ctx, variant, 1, gr.toff, ctx->blk_off, np, plan, &tmp));
            CK(pack_sources(D, nrhs, vv[variant].packed, ctx->src_pos_d, ctx->rec_pt_d, ctx->lam_d, ctx->sumN,
                            ctx->nrec, ctx->rec_d, st));
            PairGeom g = geom_of(ctx);
            g.tgt = gr.t4;
            g.ntargets = np;
            PairWork w = work_of(plan);
            w.tperm = gr.order;  // the epilogue writes in the caller's order
            if (w.total_units > 0) CK(pair_launch(variant, g, w, ctx->err_d, st));
            CK(pair_epilogue(D, nrhs, w, nullptr, 0.0, scale, oo.d, np, st));
        }
    }
    CKS(stage_out_finish(ctx, oo, st));
    return check_device_error(ctx, st);
}

}  // extern "C"

extern "C" {

mfs_status mfs_evaluate_stress(mfs_ctx *ctx, const double *points, const double *normals, const int32_t *owner,
                               int32_t npoints, double *pressure, double *traction, int32_t nrhs, void *stream) {
    if (!ctx || npoints < 0 || nrhs < 1 || (npoints > 0 && (!points || (!pressure && !traction))) ||
        (traction && !normals)) {
        if (ctx) ctx->last_error = "mfs_evaluate_stress: invalid argument";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->kind != MFS_STOKES) {
        ctx->last_error = "mfs_evaluate_stress needs a Stokes context";
        return MFS_ERR_INVALID_ARG;
    }
    if (ctx->last_solve == 0 || ctx->last_nrhs != nrhs) {
        ctx->last_error = "mfs_evaluate_stress needs a preceding solve with the same nrhs";
        return MFS_ERR_INVALID_ARG;
    }
    if (npoints == 0) return MFS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const int P = ctx->P, np = npoints;
    Scratch tmp(ctx, st);
    Grouped gr;
    const bool fp64 = ctx->opt.precision == 1;
    CKS(group_points(ctx, points, traction ? normals : nullptr, owner, np, ctx->ff.ready, fp64, tmp, gr));
    Staged po, to;
    if (pressure) CKS(stage_out_alloc(ctx, po, pressure, (size_t)nrhs * np, st));
    if (traction) CKS(stage_out_alloc(ctx, to, traction, (size_t)nrhs * np * 3, st));
    double *tmp_d = nullptr;
    CK(tmp.alloc(&tmp_d, (size_t)nrhs * ctx->sumN * 3));
    CKS(last_strengths(ctx, nrhs, tmp_d, st));
    if (fp64) {
        // per body: the body range of its suspension
        std::vector<int> sb0(P), sb1(P);
        for (int s = 0; s < ctx->S; ++s)
            for (int k = ctx->body_off[s]; k < ctx->body_off[s + 1]; ++k) {
                sb0[k] = ctx->body_off[s];
                sb1[k] = ctx->body_off[s + 1];
            }
        int *sb0_d = nullptr, *sb1_d = nullptr;
        double *ps_d = nullptr, *ts_d = nullptr;
        CK(tmp.alloc(&sb0_d, P));
        CK(tmp.alloc(&sb1_d, P));
        if (pressure) CK(tmp.alloc(&ps_d, (size_t)nrhs * np));
        if (traction) CK(tmp.alloc(&ts_d, (size_t)nrhs * np * 3));
        CK(tmp.upload(sb0_d, std::move(sb0)));
        CK(tmp.upload(sb1_d, std::move(sb1)));
        CK(stress_f64(nrhs, gr.t64, gr.tbody, gr.n64, np, ctx->src_local64_d, ctx->src_off_d, ctx->sumN, ctx->lam_d,
                      sb0_d, sb1_d, ctx->centres_d, ps_d, ts_d, st));
        const size_t n = (size_t)nrhs * np;
        if (pressure)
            unsort_kernel<<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, st>>>(ps_d, gr.order, np, 1,
                                                                                              nrhs, po.d);
        if (traction)
            unsort_kernel<<<(unsigned)std::min<size_t>((3 * n + 255) / 256, 4096), 256, 0, st>>>(ts_d, gr.order, np,
                                                                                                  3, nrhs, to.d);
        CK(cudaGetLastError());
    } else {  // the stress entry of the pair kernel (p, T per rhs), directly or through the treecode
        const int sv = stress_variant(nrhs);
        if (sv < 0) {
            ctx->last_error = "no stress kernel for this nrhs";
            return MFS_ERR_INVALID_ARG;
        }
        double *o4_d = nullptr;
        CK(tmp.alloc(&o4_d, (size_t)nrhs * np * 4));
        const double scale = 1.0 / (4.0 * MFS_PI);
        if (ctx->ff.ready) {
            CKS(ff_points(ctx, sv, gr, np, nrhs, 4, scale, o4_d, tmp));
        } else {
            PairPlan plan;
            CKS(build_plan_for(ctx, sv, 1, gr.toff, ctx->blk_off, np, plan, &tmp));
            int vc = 0;
            CK(pack_sources(3, nrhs, pair_variants(&vc)[sv].packed, ctx->src_pos_d, ctx->rec_pt_d, ctx->lam_d,
                            ctx->sumN, ctx->nrec, ctx->rec_d, st));
            PairGeom g = geom_of(ctx);
            g.tgt = gr.t4;
            g.ntargets = np;
            g.tgt_w = gr.n32;
            PairWork w = work_of(plan);
            w.tperm = gr.order;
            if (w.total_units > 0) CK(pair_launch(sv, g, w, ctx->err_d, st));
            CK(pair_epilogue(4, nrhs, w, nullptr, 0.0, scale, o4_d, np, st));
        }
        const size_t n = (size_t)nrhs * np;
        split_stress_kernel<<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, st>>>(
            o4_d, n, pressure ? po.d : nullptr, traction ? to.d : nullptr);
        CK(cudaGetLastError());
    }
    if (pressure) CKS(stage_out_finish(ctx, po, st));
    if (traction) CKS(stage_out_finish(ctx, to, st));
    return check_device_error(ctx, st);
}

}  // extern "C"
