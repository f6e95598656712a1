// Device-resident FP64 GMRES (Algorithm 1 SOLVE uses GMRES; zero initial guess, no restart
// within the basis capacity).  The vector of all lanes is one array; lane l (one right-hand
// side of one suspension) owns entries [seg_off[l], seg_off[l+1]) and has its own Arnoldi
// process, Hessenberg matrix and Givens rotations, so independent problems iterate together
// and stop separately (converged lanes are masked).  Orthogonalisation is classical
// Gram-Schmidt applied twice (CGS2); every reduction is deterministic (fixed block partials).
//
// Work is cut into blocks of one lane each (GmresDev::blk_*, sized on the host so that all blocks have
// about the same length whatever the lanes' sizes; with a fixed number of blocks per lane, suspensions
// of 2 to 64 bodies left most SMs waiting for the longest lane).  What bounds the step is latency and
// the FP64 pipe, not bandwidth: an iteration was ten launches, each a chain of dependent loads, so it is
// four here (dot, update and dot, update, finish), and one for short lanes (gm_arnoldi_cluster_kernel).  A
// warp's FP64 instruction holds its scheduler's FP64 pipe for 64 clocks however many of its lanes are
// active, so scalar FP64 work (norms, rotations, the tails of reductions) is done by one warp and handed
// on through shared memory, and no warp runs FP64 instructions on elements or columns that do not exist.
#include <algorithm>

#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"

namespace mfs {

#define GM_THREADS 512
#define GM_WARPS (GM_THREADS / 32)
#define GM_CLUSTER 16  // blocks per cluster of the short-lane form
#define GM_CHUNK 1024  // and the entries each of them holds

// Block-wide dots: out[i] = sum over e in [0, len) of V[i n + e] w[e], i = 0 .. cols - 1, in a fixed
// order.  A warp takes a group of four columns on a part of the elements (w is read once for the four;
// with few columns the elements are cut into parts, of at least 128 elements each); the lanes' partials
// go to shared memory and are added there, eight lanes to a column: a shuffle tree per warp and column
// would cost as many FP64 instructions as the dots themselves.  sh: 4 * GM_THREADS doubles.
__device__ __forceinline__ void block_dots(const double *V, long long n, const double *w, int len, int cols,
                                           double *sh, double *out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ng = (cols + 3) / 4;
    for (int g0 = 0; g0 < ng; g0 += GM_WARPS) {
        const int groups = min(ng - g0, GM_WARPS);
        const int parts = max(1, min(min(GM_WARPS / groups, 8), (len + 127) / 128));
        const int g = warp / parts, p = warp % parts;
        if (g < groups) {
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            const int c0 = 4 * (g0 + g), nc = min(4, cols - c0);
            const int e1 = (int)((long long)len * (p + 1) / parts);
            const double *Vc = V + (size_t)c0 * n;
            for (int eb = (int)((long long)len * p / parts); eb < e1; eb += 128) {
                const int e = eb + lane;
                double we[4], v[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) we[u] = e + 32 * u < e1 ? w[e + 32 * u] : 0.0;
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        v[c][u] = (c < nc && e + 32 * u < e1) ? Vc[(size_t)c * n + e + 32 * u] : 0.0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (eb + 32 * u < e1)
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (c < nc) acc[c] = fma(v[c][u], we[u], acc[c]);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) sh[(c * GM_WARPS + warp) * 32 + lane] = acc[c];
        }
        __syncthreads();
        // column 4 g + c: the `parts` warps of group g, 32 values each; 8 lanes add 4 parts values apiece
        const int q = threadIdx.x / 8;  // 4 groups <= 64 columns = GM_THREADS / 8
        if ((q & ~3) < 4 * groups) {    // whole warps: four columns each
            const int gg = q / 4, c = q % 4, s8 = threadIdx.x & 7;
            double r = 0.0;
            for (int pp = 0; pp < parts; ++pp) {
                const double *x = sh + (c * GM_WARPS + gg * parts + pp) * 32 + s8;
                r += (x[0] + x[8]) + (x[16] + x[24]);
            }
            for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
            const int col = 4 * (g0 + gg) + c;
            if (s8 == 0 && col < cols) out[col] = r;
        }
        __syncthreads();
    }
}

// w[e] -= sum_{i < cols} h[i] V[i n + e] over e in [0, len); returns the thread's sum of the new w[e]^2
// (0 unless NORM).  Four elements per thread and G columns at a time: 32 loads in flight with eight, the
// last round guarded instead of a remainder loop; each element's sum runs over the columns in order.
template <bool NORM, int G = 8>
__device__ __forceinline__ double block_update(const double *V, long long n, double *w, int len, int cols,
                                               const double *h) {
    double nrm = 0.0;
    const int lane = threadIdx.x & 31;
    for (int eb = threadIdx.x - lane; eb < len; eb += 4 * GM_THREADS) {  // the warp's first element
        const int e = eb + lane;
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        bool in[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) in[u] = e + u * GM_THREADS < len;
        for (int i = 0; i < cols; i += G) {
            double v[G][4];
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[g][u] = (in[u] && i + g < cols) ? V[(size_t)(i + g) * n + e + u * GM_THREADS] : 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (eb + u * GM_THREADS < len)
#pragma unroll
                    for (int g = 0; g < G; ++g)
                        if (i + g < cols) a[u] = fma(h[i + g], v[g][u], a[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (eb + u * GM_THREADS < len) {
                const double x = in[u] ? w[e + u * GM_THREADS] - a[u] : 0.0;
                if (in[u]) w[e + u * GM_THREADS] = x;
                if (NORM) nrm = fma(x, x, nrm);
            }
    }
    return nrm;
}

// Sum of v over the block in a fixed order, returned in lane 0 of warp 0: through shared memory, one warp
// adds (threads beyond `threads` hold zeros and are left out).  sh: GM_THREADS doubles.
__device__ __forceinline__ double block_sum(double v, int threads, double *sh) {
    __syncthreads();
    sh[threadIdx.x] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        for (int i = threadIdx.x; i < threads; i += 32) s += sh[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;
}

// (||x||, 1 / ||x||) from s = ||x||^2, (0, 0) for 0.
__device__ __forceinline__ double2 norm_and_inverse(double s) {
    if (s == 0.0) return make_double2(0.0, 0.0);
    const double inv = rsqrt64(s);
    return make_double2(isfinite(s) ? s * inv : sqrt(s), inv);
}

// The Givens update of column j for lane l, by one warp: hc[0 .. j] the column's entries, hn the norm of
// the new Krylov vector, cs, sn the earlier rotations (all in shared memory; hc and cs are overwritten).
// The rotations chain through one value, carry_{i+1} = -sn_i carry_i + cs_i h_{i+1}: the lanes form
// cs_i h_{i+1} first, one lane walks the chain with a single FMA a step, the lanes finish the entries.
__device__ void givens_lane(const GmresDev &gd, int l, int j, double *hc, double *cs_, const double *sn_,
                            double h_next) {
    const int m = gd.m, lane = threadIdx.x & 31;
    double *H = gd.H + (size_t)l * (m + 1) * m;  // H[i][jj] at i*m + jj
    double *cs = gd.cs + (size_t)l * m, *sn = gd.sn + (size_t)l * m, *g = gd.g + (size_t)l * (m + 1);
    // per step i < j: t = cs_i h_{i+1} and s = sn_i h_{i+1}; H_i = cs_i carry_i + s, carry_{i+1} = t - sn_i carry_i
    for (int i0 = 0; i0 < j; i0 += 32) {
        const int i = i0 + lane;
        const bool in = i < j;
        const double c1 = in ? hc[i + 1] : 0.0, ci = in ? cs_[i] : 0.0, si = in ? sn_[i] : 0.0;
        const double first = hc[i0];  // carry_{i0}
        __syncwarp();
        const double t = ci * c1;
        double carry = first, mine = first;  // carry_i of this lane's step
        const int n = min(32, j - i0);
        for (int k = 0; k < n; ++k) {  // every lane walks the same chain; lane k keeps its value
            if (lane == k) mine = carry;
            carry = fma(-__shfl_sync(0xffffffffu, si, k), carry, __shfl_sync(0xffffffffu, t, k));
        }
        if (in) H[(size_t)i * m + j] = fma(ci, mine, si * c1);
        if (lane == 0) hc[i0 + n] = carry;
        __syncwarp();
    }
    if (lane != 0) return;
    const double a = hc[j], c = h_next;
    const double r2 = fma(a, a, c * c);
    double den, cj, sj;
    if ((unsigned)__double2hiint(r2) - 0x06000000u < 0x72000000u) {  // r2 well inside the normal range
        const double ri = rsqrt64(r2);
        den = r2 * ri;
        cj = a * ri;
        sj = c * ri;
    } else {
        den = hypot(a, c);
        cj = den > 0.0 ? a / den : 1.0;
        sj = den > 0.0 ? c / den : 0.0;
    }
    cs[j] = cj;
    sn[j] = sj;
    H[j * m + j] = den;
    const double gj = g[j], gn = -sj * gj;
    g[j + 1] = gn;
    g[j] = cj * gj;
    gd.iters[l] = j + 1;
    const double res = fabs(gn) * gd.ibeta[l];
    gd.resid[l] = res;
    int keep = 1;
    if (!isfinite(res) || !isfinite(den)) {
        gd.status[l] = 2;  // breakdown
        keep = 0;
    } else if (res <= gd.tol || h_next == 0.0 || j + 1 >= m) {
        keep = 0;
    }
    gd.active[l] = keep;
}

// Called by one block (all threads): done from the lanes' flags, then j += 1 unless done or the basis is
// full; with a graph conditional handle sets it to whether another iteration follows.
__device__ void advance_step(const GmresDev &gd, int j, cudaGraphConditionalHandle cond, int cond_valid) {
    int any = 0;
    for (int l = threadIdx.x; l < gd.L; l += blockDim.x) any |= *(volatile int *)&gd.active[l];
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) {
        *gd.done = any ? 0 : 1;
        const int more = any && (j + 1 < gd.m);
        if (more) *gd.jcur = j + 1;
        if (cond_valid) cudaGraphSetConditional(cond, more ? 1u : 0u);
    }
}

// True in every thread of the block that arrives last of `total` (whose predecessors' writes it sees).
__device__ __forceinline__ bool last_to_arrive(const GmresDev &gd, unsigned total) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(gd.arrive, total - 1) == total - 1;  // wraps to 0 for the next use
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// part[b][i] = sum over block b's chunk of V[i][e] * w[e], i = 0..j
__global__ void __launch_bounds__(GM_THREADS) gm_dot_kernel(GmresDev gd, const double *w) {
    const int b = blockIdx.x, l = gd.blk_lane[b];
    if (!gd.active[l]) return;
    __shared__ double sh[4 * GM_THREADS];
    const long long e0 = gd.blk_off[b];
    block_dots(gd.V + e0, gd.n, w + e0, (int)(gd.blk_off[b + 1] - e0), *gd.jcur + 1, sh,
               gd.part + (size_t)b * (gd.m + 1));
}

// h = the lane's dots (its blocks' partials added in order, eight threads to a column); hbuf = or += h;
// w -= V h; then, in the first pass, the second pass's dots of the block's chunk (its V is still near),
// in the second pass the block's share of ||w||^2.
// With more blocks than SMs, four columns at a time and two blocks an SM (64 registers), so that one
// block's FP64 work covers the other's loads and barriers; with at most one block an SM, eight columns at
// a time (112 registers).  1024 lanes of 4320 entries, mean over 14 steps of the first and second pass:
// 109 and 74 us, with one block an SM 165 and 121 (the FP64 pipe alone: 108 and 61).
template <int PASS, int G>
__global__ void __launch_bounds__(GM_THREADS, G == 8 ? 1 : 2) gm_update_kernel(GmresDev gd, double *w) {
    const int b = blockIdx.x, l = gd.blk_lane[b];
    if (!gd.active[l]) return;
    const int cols = *gd.jcur + 1;
    __shared__ double h[1024];
    __shared__ double red[PASS ? GM_THREADS : 4 * GM_THREADS];
    const double *part = gd.part + (PASS ? (size_t)gd.nblk * (gd.m + 1) : 0);
    const int b0 = gd.lane_blk[l], nb = gd.lane_blk[l + 1] - b0;
    const size_t ld = gd.m + 1;
    for (int q0 = 0; q0 < cols; q0 += GM_THREADS / 8) {
        const int q = q0 + threadIdx.x / 8, s8 = threadIdx.x & 7;
        if ((q & ~3) >= cols) break;  // whole warps: four columns each
        double r = 0.0;
        if (q < cols) {
            const double *p = part + (size_t)b0 * ld + q;
            int i = s8;
            for (; i + 24 < nb; i += 32) {
                const double x0 = p[(size_t)i * ld], x1 = p[(size_t)(i + 8) * ld], x2 = p[(size_t)(i + 16) * ld],
                             x3 = p[(size_t)(i + 24) * ld];
                r += (x0 + x1) + (x2 + x3);
            }
            for (; i < nb; i += 8) r += p[(size_t)i * ld];
        }
        for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        if (q < cols && s8 == 0) {
            h[q] = r;
            if (b == b0) {
                double *hb = gd.hbuf + (size_t)l * ld + q;
                *hb = PASS ? *hb + r : r;
            }
        }
    }
    __syncthreads();
    const long long e0 = gd.blk_off[b];
    const double s = block_update<PASS == 1, G>(gd.V + e0, gd.n, w + e0, (int)(gd.blk_off[b + 1] - e0), cols, h);
    if (PASS == 0) {
        __syncthreads();
        block_dots(gd.V + e0, gd.n, w + e0, (int)(gd.blk_off[b + 1] - e0), cols, red,
                   gd.part + (size_t)(gd.nblk + b) * ld);
    } else {
        const double t = block_sum(s, GM_THREADS, red);
        if (threadIdx.x == 0) gd.normp[b] = t;
    }
}

// normp[b] = block b's share of ||x||^2 (all lanes)
__global__ void __launch_bounds__(GM_THREADS) gm_norm_kernel(GmresDev gd, const double *x) {
    const int b = blockIdx.x;
    __shared__ double red[GM_THREADS];
    const long long e0 = gd.blk_off[b], e1 = gd.blk_off[b + 1];
    double s = 0.0;
    for (long long e = e0 + threadIdx.x; e < e1; e += GM_THREADS) s = fma(x[e], x[e], s);
    s = block_sum(s, GM_THREADS, red);
    if (threadIdx.x == 0) gd.normp[b] = s;
}

// The lane's norm and its inverse from its blocks' shares, the same in every block of the lane.
__device__ __forceinline__ double2 lane_norm(const GmresDev &gd, int l) {
    __shared__ double2 nrm;
    if (threadIdx.x < 32) {
        double s = 0.0;
        for (int i = gd.lane_blk[l] + threadIdx.x; i < gd.lane_blk[l + 1]; i += 32) s += gd.normp[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) nrm = norm_and_inverse(s);
    }
    __syncthreads();
    return nrm;
}

// The start: v_0 = b / ||b|| (also to vin, the fixed input of the next matvec), the lanes' states,
// j = 0, done = (no lane active).
__global__ void __launch_bounds__(GM_THREADS) gm_start_kernel(GmresDev gd, const double *x, double *vin) {
    const int b = blockIdx.x, l = gd.blk_lane[b];
    const double2 ni = lane_norm(gd, l);
    const double nrm = ni.x, inv = ni.y;
    for (long long e = gd.blk_off[b] + threadIdx.x; e < gd.blk_off[b + 1]; e += GM_THREADS) {
        const double v = x[e] * inv;
        gd.V[e] = v;
        vin[e] = v;
    }
    if (b == gd.lane_blk[l] && threadIdx.x == 0) {
        gd.ibeta[l] = inv;
        gd.g[(size_t)l * (gd.m + 1)] = nrm;
        gd.active[l] = (nrm > 0.0 && isfinite(nrm)) ? 1 : 0;
        gd.iters[l] = 0;
        gd.resid[l] = (nrm > 0.0) ? 1.0 : 0.0;
        gd.status[l] = isfinite(nrm) ? 0 : 2;
    }
    if (last_to_arrive(gd, gridDim.x)) {
        int any = 0;
        for (int k = threadIdx.x; k < gd.L; k += blockDim.x) any |= *(volatile int *)&gd.active[k];
        any = __syncthreads_or(any);
        if (threadIdx.x == 0) {
            *gd.done = any ? 0 : 1;
            *gd.jcur = 0;
        }
    }
}

// v_{j+1} = w / ||w|| to the basis and to vin; the first block of each lane updates its Hessenberg column;
// with `advance` the last block to finish moves to the next column.
__global__ void __launch_bounds__(GM_THREADS) gm_finish_kernel(GmresDev gd, const double *w, double *vin, int advance) {
    const int b = blockIdx.x, l = gd.blk_lane[b], j = *gd.jcur;
    __shared__ double hs[3][1024];
    // one read for the block: the lane's first block may clear the flag meanwhile
    const int active = __syncthreads_or(threadIdx.x == 0 ? gd.active[l] : 0);
    if (active) {
        const double2 ni = lane_norm(gd, l);
        const double nrm = ni.x, inv = ni.y;
        const bool first = b == gd.lane_blk[l];
        if (first) {  // the loads of the serial update ahead of it
            for (int i = threadIdx.x; i <= j; i += GM_THREADS) {
                hs[0][i] = gd.hbuf[(size_t)l * (gd.m + 1) + i];
                hs[1][i] = gd.cs[(size_t)l * gd.m + i];
                hs[2][i] = gd.sn[(size_t)l * gd.m + i];
            }
        }
        double *v = gd.V + (size_t)(j + 1) * gd.n;
        for (long long e = gd.blk_off[b] + threadIdx.x; e < gd.blk_off[b + 1]; e += GM_THREADS) {
            const double x = w[e] * inv;
            v[e] = x;
            vin[e] = x;
        }
        __syncthreads();
        // a block of the lane that starts after its flag was cleared here skips its share of v_{j+1}, which
        // a stopped lane does not use
        if (first && threadIdx.x < 32) givens_lane(gd, l, j, hs[0], hs[1], hs[2], nrm);
    }
    if (advance && last_to_arrive(gd, gridDim.x)) advance_step(gd, j, cudaGraphConditionalHandle(), 0);
}

// j += 1 or stop, and the while node's condition (a graph iteration's last kernel; one block)
__global__ void gm_advance_kernel(GmresDev gd, cudaGraphConditionalHandle cond, int cond_valid) {
    advance_step(gd, *gd.jcur, cond, cond_valid);
}

// The whole Arnoldi step of one short lane by one cluster of GM_CLUSTER blocks: w stays in shared memory,
// the dots and the norm are exchanged through distributed shared memory, and the launches of the
// long-lane form (each at least a launch and a chain of dependent loads, about 5 us) become one.  For
// lanes of at most GM_CLUSTER * GM_CHUNK entries: beyond that the FP64 pipes of 16 SMs take longer than
// the launches saved (at j = 15, 16384 entries: 4 us a pass); and for few of them (gmres_prepare).
// Whole solves with this file's kernels against the ten-launch form, when they came in: two conductors (1200
// entries) 692 -> 445 us, six spheres (4320) 1372 -> 942 us; four launches: 40 spheroids (119 640 entries, 76
// columns) 48.1 -> 43.2 ms, 48 uneven lanes 130.7 -> 126.9 ms, solve and gradients of 100 spheres 26.1 -> 25.5.
__global__ void __launch_bounds__(GM_THREADS) gm_arnoldi_cluster_kernel(GmresDev gd, const double *w, double *vin,
                                                                        int advance) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int l = blockIdx.y, rank = blockIdx.x, j = *gd.jcur, cols = j + 1, m1 = gd.m + 1;
    extern __shared__ double dyn[];
    double *sh = dyn, *wb = sh + 4 * GM_THREADS, *pa = wb + GM_CHUNK, *pb = pa + m1, *h = pb + m1, *hc = h + m1,
           *cs = hc + m1, *sn = cs + m1;
    __shared__ double pn;
    __shared__ double2 ni;
    if (gd.active[l]) {
        const long long s0 = gd.blk_off[gd.lane_blk[l]], s1 = gd.blk_off[gd.lane_blk[l + 1]];
        const long long e0 = s0 + (s1 - s0) * rank / GM_CLUSTER;
        const int len = (int)(s0 + (s1 - s0) * (rank + 1) / GM_CLUSTER - e0);
        const double *V = gd.V + e0;
        for (int e = threadIdx.x; e < len; e += GM_THREADS) wb[e] = w[e0 + e];
        if (rank == 0)
            for (int i = threadIdx.x; i < j; i += GM_THREADS) {
                cs[i] = gd.cs[(size_t)l * gd.m + i];
                sn[i] = gd.sn[(size_t)l * gd.m + i];
            }
        __syncthreads();
        block_dots(V, gd.n, wb, len, cols, sh, pa);
        cl.sync();
        for (int i = threadIdx.x; i < cols; i += GM_THREADS) {
            double s = 0.0;
            for (int r = 0; r < GM_CLUSTER; ++r) s += cl.map_shared_rank(pa, r)[i];
            h[i] = hc[i] = s;
        }
        __syncthreads();
        block_update<false>(V, gd.n, wb, len, cols, h);
        __syncthreads();
        block_dots(V, gd.n, wb, len, cols, sh, pb);
        cl.sync();
        for (int i = threadIdx.x; i < cols; i += GM_THREADS) {
            double s = 0.0;
            for (int r = 0; r < GM_CLUSTER; ++r) s += cl.map_shared_rank(pb, r)[i];
            h[i] = s;
            hc[i] += s;
        }
        __syncthreads();
        const double t = block_sum(block_update<true>(V, gd.n, wb, len, cols, h), min(GM_THREADS, (len + 31) / 32 * 32), sh);
        if (threadIdx.x == 0) pn = t;
        cl.sync();
        if (threadIdx.x < 32) {
            double s = threadIdx.x < GM_CLUSTER ? *cl.map_shared_rank(&pn, threadIdx.x) : 0.0;
            for (int o = GM_CLUSTER / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (threadIdx.x == 0) ni = norm_and_inverse(s);
        }
        __syncthreads();
        const double nrm = ni.x, inv = ni.y;
        double *v = gd.V + (size_t)(j + 1) * gd.n + e0;
        for (int e = threadIdx.x; e < len; e += GM_THREADS) {
            const double x = wb[e] * inv;
            v[e] = x;
            vin[e0 + e] = x;
        }
        if (rank == 0 && threadIdx.x < 32) givens_lane(gd, l, j, hc, cs, sn, nrm);
        cl.sync();  // no block leaves while another reads its shared memory
    }
    if (advance && rank == 0 && last_to_arrive(gd, gd.L)) advance_step(gd, j, cudaGraphConditionalHandle(), 0);
}

// x = sum_{i<k_l} y_l[i] V[i] with H_l y = g_l (upper triangular, k_l columns): every block solves its
// lane's triangle itself (one warp, the triangle in shared memory, column by column with the diagonal's
// reciprocals taken beforehand; one thread walking it in global memory took 250 us at 76 columns), then
// combines its chunk with 32 loads in flight per thread.
#define GM_TRI 144  // columns whose triangle fits the block's shared memory (83 KB)
__global__ void __launch_bounds__(GM_THREADS) gm_solution_kernel(GmresDev gd, double *x) {
    extern __shared__ double tri[];  // row i of the triangle (columns i .. k - 1) packed by column: c (c + 1) / 2 + i
    __shared__ double y[1024], dinv[1024];
    const int b = blockIdx.x, l = gd.blk_lane[b], k = gd.iters[l], m = gd.m;
    const double *H = gd.H + (size_t)l * (m + 1) * m;
    const bool packed = k <= GM_TRI;
    for (int i = threadIdx.x; i < k; i += GM_THREADS) {
        const double d = H[(size_t)i * m + i];
        dinv[i] = d != 0.0 ? 1.0 / d : 0.0;
        y[i] = gd.g[(size_t)l * (m + 1) + i];
    }
    if (packed)
        for (int i = threadIdx.x >> 5; i < k; i += GM_WARPS)
            for (int c = i + (threadIdx.x & 31); c < k; c += 32) tri[c * (c + 1) / 2 + i] = H[(size_t)i * m + c];
    __syncthreads();
    if (threadIdx.x < 32)
        for (int c = k - 1; c >= 0; --c) {
            const double yc = y[c] * dinv[c];
            __syncwarp();
            if (threadIdx.x == 0) y[c] = yc;
            for (int i = threadIdx.x; i < c; i += 32)
                y[i] = fma(-(packed ? tri[c * (c + 1) / 2 + i] : H[(size_t)i * m + c]), yc, y[i]);
            __syncwarp();
        }
    __syncthreads();
    const long long e0 = gd.blk_off[b];
    const int len = (int)(gd.blk_off[b + 1] - e0);
    const double *V = gd.V + e0;
    for (int e = threadIdx.x; e < len; e += 4 * GM_THREADS) {
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        bool in[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) in[u] = e + u * GM_THREADS < len;
        for (int i = 0; i < k; i += 8) {
            double v[8][4];
#pragma unroll
            for (int g = 0; g < 8; ++g)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[g][u] = (in[u] && i + g < k) ? V[(size_t)(i + g) * gd.n + e + u * GM_THREADS] : 0.0;
#pragma unroll
            for (int g = 0; g < 8; ++g)
                if (i + g < k)
#pragma unroll
                    for (int u = 0; u < 4; ++u) a[u] = fma(y[i + g], v[g][u], a[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (in[u]) x[e0 + e + u * GM_THREADS] = a[u];
    }
}

bool gmres_plan_blocks(const std::vector<long long> &seg, int sm_count, std::vector<int> &blk_lane,
                       std::vector<long long> &blk_off, std::vector<int> &lane_blk) {
    const int L = (int)seg.size() - 1;
    long long longest = 0;
    for (int l = 0; l < L; ++l) longest = std::max(longest, seg[l + 1] - seg[l]);
    auto blocks = [&](long long chunk) {
        long long t = 0;
        for (int l = 0; l < L; ++l) t += std::max<long long>(1, (seg[l + 1] - seg[l] + chunk - 1) / chunk);
        return t;
    };
    // the shortest chunk (in steps of 256, at least 2048) whose blocks fill whole waves: one wave, or two
    // blocks per lane on average when the lanes alone are more than the SMs
    const long long want = L <= sm_count / 2 ? sm_count : (2LL * L + sm_count - 1) / sm_count * sm_count;
    long long lo = 8, hi = std::max<long long>(9, (longest + 255) / 256);
    while (lo < hi) {
        const long long mid = (lo + hi) / 2;
        if (blocks(256 * mid) <= want) hi = mid; else lo = mid + 1;
    }
    const long long chunk = 256 * lo;
    blk_lane.clear();
    blk_off.assign(1, seg[0]);
    lane_blk.assign(1, 0);
    for (int l = 0; l < L; ++l) {
        const long long len = seg[l + 1] - seg[l], nb = std::max<long long>(1, (len + chunk - 1) / chunk);
        for (long long i = 0; i < nb; ++i) {
            blk_lane.push_back(l);
            blk_off.push_back(seg[l] + len * (i + 1) / nb);
        }
        lane_blk.push_back((int)blk_lane.size());
    }
    return longest <= (long long)GM_CLUSTER * GM_CHUNK;
}

static size_t cluster_smem(const GmresDev &gd) { return sizeof(double) * (4 * GM_THREADS + GM_CHUNK + 6 * (size_t)(gd.m + 1)); }
static size_t solution_smem(const GmresDev &gd) {
    const size_t k = std::min(gd.m, GM_TRI);
    return sizeof(double) * (k * (k + 1) / 2);
}

cudaError_t gmres_prepare(GmresDev &gd) {
    cudaError_t e = cudaFuncSetAttribute(gm_solution_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(sizeof(double) * GM_TRI * (GM_TRI + 1) / 2));
    if (e != cudaSuccess || !gd.clusters) return e;
    e = cudaFuncSetAttribute(gm_arnoldi_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(double) * (4 * GM_THREADS + GM_CHUNK + 6 * 1024)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gm_arnoldi_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    // The lanes must fit the clusters that the device holds at once (fewer than eight on 152 SMs), twice over at most: a
    // cluster takes the 16 SMs of a GPC, so lanes beyond that queue, where the long-lane form's blocks share
    // all SMs.  Time of an iteration, one launch / four, lanes of 4320 entries: 1 lane 67 / 83 us, 8 lanes
    // 115 / 126, 12 lanes 128 / 136, 16 lanes 138 / 139, 24 lanes 167 / 153, 64 lanes 257 / 211, 256 lanes
    // 674 / 422; of 16 338 entries: 1 lane 104 / 121, 8 lanes 220 / 223, 12 lanes 271 / 275, 16 lanes
    // 328 / 319, 64 lanes 940 / 890; of 1800: 8 lanes 222 / 238, 16 lanes 267 / 267, 64 lanes 400 / 315.
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = GM_CLUSTER;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(GM_CLUSTER, gd.L);
    cfg.blockDim = dim3(GM_THREADS);
    cfg.dynamicSmemBytes = cluster_smem(gd);
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gm_arnoldi_cluster_kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    if (gd.L > 2 * n) gd.clusters = 0;
    return cudaSuccess;
}

cudaError_t gmres_init(GmresDev &gd, const double *b, double *vin, cudaStream_t st) {
    gm_norm_kernel<<<gd.nblk, GM_THREADS, 0, st>>>(gd, b);
    gm_start_kernel<<<gd.nblk, GM_THREADS, 0, st>>>(gd, b, vin);
    return cudaGetLastError();
}

int gmres_arnoldi_launches(const GmresDev &gd) { return gd.clusters ? 1 : 4; }

cudaError_t gmres_arnoldi(GmresDev &gd, double *w, double *vin, int advance, cudaStream_t st) {
    if (gd.clusters) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = GM_CLUSTER;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(GM_CLUSTER, gd.L);
        cfg.blockDim = dim3(GM_THREADS);
        cfg.dynamicSmemBytes = cluster_smem(gd);
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, gm_arnoldi_cluster_kernel, gd, (const double *)w, vin, advance);
    }
    gm_dot_kernel<<<gd.nblk, GM_THREADS, 0, st>>>(gd, w);  // CGS2
    if (gd.nblk > gd.sms) {
        gm_update_kernel<0, 4><<<gd.nblk, GM_THREADS, 0, st>>>(gd, w);
        gm_update_kernel<1, 4><<<gd.nblk, GM_THREADS, 0, st>>>(gd, w);
    } else {
        gm_update_kernel<0, 8><<<gd.nblk, GM_THREADS, 0, st>>>(gd, w);
        gm_update_kernel<1, 8><<<gd.nblk, GM_THREADS, 0, st>>>(gd, w);
    }
    gm_finish_kernel<<<gd.nblk, GM_THREADS, 0, st>>>(gd, w, vin, advance);
    return cudaGetLastError();
}

cudaError_t gmres_advance(GmresDev &gd, cudaGraphConditionalHandle cond, cudaStream_t st) {
    gm_advance_kernel<<<1, 256, 0, st>>>(gd, cond, 1);
    return cudaGetLastError();
}

cudaError_t gmres_solution(GmresDev &gd, double *x, cudaStream_t st) {
    gm_solution_kernel<<<gd.nblk, GM_THREADS, solution_smem(gd), st>>>(gd, x);
    return cudaGetLastError();
}

}  // namespace mfs
