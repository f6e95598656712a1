// Shared definitions of libmfs (internal; not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

#define MFS_PI 3.14159265358979323846

// Device error flags (bit mask written with atomicOr by kernels that give up).
#define MFS_DEVERR_TIMEOUT 1
#define MFS_DEVERR_BADARG 2

// ---------------------------------------------------------------------------
// Pair-sum work decomposition.
//
// Targets (collocation points) are numbered globally, bodies contiguous, the
// bodies of one suspension contiguous.  A tile is a range of at most
// `tile_targets` consecutive targets of one suspension spanning at most
// MFS_MAX_TILE_BODIES bodies.  Its work is the sequence of source "units"
// (blocks of MFS_BS consecutive source records of one body) of every body of
// its suspension, except the tile's own body when the tile lies inside one
// body and self pairs are excluded.  The units of all tiles are concatenated
// into one global sequence of `total_units`, cut into G equal shares, one per
// persistent CTA (a stream-K split), so that every CTA does the same work.
// ---------------------------------------------------------------------------
#define MFS_BS 32
#define MFS_MAX_TILE_BODIES 32

struct PairTile {
    int t0, t1;          // targets [t0, t1)
    int kb0, nb;         // target bodies kb0 .. kb0+nb-1
    int skip;            // source body left out entirely, or -1
    int B0, B1;          // source bodies of the suspension [B0, B1)
    long long u0, u1;    // global unit range of this tile
    int gA, gB;          // first and last CTA whose share meets this tile
    int slotA = 0;       // the slot CTA gA wrote the tile's sum to: 0 when its share starts in the tile, 1 when
                         // it ends there (every later CTA's share starts in the tile: slot 0)
    int L0, L1;          // L0 >= 0: the tile's sources are the segments of interaction-list entries
                         // [L0, L1) (PairGeom::lst_*) instead of the bodies [B0, B1)
};

// Compensated pair sums split body-local coordinates and centre differences at multiples of
// 1/MFS_XGRID: the "high" parts of a target and a source then differ by an exactly representable
// FP32 number, and its square is exact while it is shorter than 32 (11 significant bits).
#define MFS_XGRID 64.0

struct PairGeom {
    const float4 *tgt;         // [ntargets] body-local rotated target (x,y,z), w = body id (int bits)
    const float *src;          // [sum_Npad][REC] packed source records
    const int *src_off;        // [P+1] record offset of each body (padded to a multiple of 4)
    const long long *blk_off;  // [P+1] global block offset of each body (blocks of MFS_BS records)
    const double *centres;     // [P][3]
    int ntargets;
    const float *tgt_w = nullptr;  // gradient kernel only: target strengths w, FP32 [nrhs][ntargets][3]
    // compensated kernels only: body-local targets split as x = hi + lo, hi a multiple of 1/MFS_XGRID
    const float4 *tgt_hi = nullptr, *tgt_lo = nullptr;  // [ntargets] (x, y, z, unused)
    // interaction lists (tiles with L0 >= 0): entry e names source segment lst_seg[e], whose records
    // are [seg_rec0[s], seg_rec1[s]) (blocks of MFS_BS), and starts at global unit lst_cum[e]
    // (lst_cum has one entry more than lst_seg: the units of the last tile end at its last value)
    const int *lst_seg = nullptr;
    const long long *lst_cum = nullptr;
    const int *seg_rec0 = nullptr, *seg_rec1 = nullptr;
};

struct PairWork {
    const PairTile *tiles;
    int ntiles;
    long long total_units;
    int G;                     // persistent CTAs
    double *partial;           // [G][2][tile_targets][C]
    double *direct;            // [ntargets][C]
    int tile_targets;
    int include_self;          // 1: self pairs included (right-hand side u_0)
    double *src_grad = nullptr;  // gradient kernel only: per source body sums, FP64 [P][3] (atomic adds)
    const int *tperm = nullptr;  // epilogue: target t's value goes to (and its base is read at) tperm[t]
    int max_share = 1;           // epilogue: the most CTAs that share one tile
    // epilogue: linear field per body, [nrhs][nfar][4][D] (constant, d/dx, d/dy, d/dz), that of the tile's body
    // kb0 added to its sums at the targets far_tgt (about the body's centre)
    const double *far = nullptr;
    const float4 *far_tgt = nullptr;
    int nfar = 0;
};

// ---------------------------------------------------------------------------
// Inline PTX: mbarrier + 1-D bulk copy (TMA engine), with bounded waits.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile(
        "{\n\t.reg .b64 st;\n\t"
        "mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_u32(bar)),
        "r"(bytes)
        : "memory");
}

// Returns true when phase `parity` of the barrier has completed.
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up after `limit` polls (each try_wait itself suspends for a
// hardware-defined interval), records MFS_DEVERR_TIMEOUT and returns false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity, int *err, long long limit) {
    for (long long it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    if (err) atomicOr(err, MFS_DEVERR_TIMEOUT);
    return false;
}

// Bulk copy global -> shared, completion signalled on `bar` (bytes % 16 == 0, both addresses 16-B aligned).
__device__ __forceinline__ void bulk_g2s(void *dst_smem, const void *src_gmem, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst_smem)),
        "l"(src_gmem), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Error-free transformation a + b = s + e (Knuth's TwoSum, 6 flops).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// 1/sqrt(x) in FP64: the hardware's FP64 rsqrt estimate y0 and one third-order Householder step,
// y = y0 (1 + h/2 + 3 h^2/8) with h = 1 - x y0^2: five FP64 instructions instead of a square root and a
// division.  With y0 good to 2^-20, h is at most 2^-19 and the series' remainder 5 h^3/16 below 2^-58; the
// rounding of x y0 adds 2^-54 and the last FMA 2^-53, a relative error below 1.51 x 2^-53 in all
// (test_gpu_rsqrt64.py holds it to that over the whole exponent range, which bears out the estimate's bound
// too; CUDA's own rsqrt, good to one ulp, is as fast to 1 %: FP64 matvec of 24 spheres 4.53 against 4.58 ms).
// Outside the normal range (zero, subnormal, infinite, negative, NaN; an integer test) the plain expression
// is taken.
__device__ __forceinline__ double rsqrt64(double x) {
    if ((unsigned)__double2hiint(x) - 0x00100000u >= 0x7fe00000u) return 1.0 / sqrt(x);
    double y0;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(x));
    const double h = fma(-x * y0, y0, 1.0);
    return fma(y0 * h, fma(0.375, h, 0.5), y0);
}
