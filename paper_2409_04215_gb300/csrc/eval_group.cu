// Evaluation points grouped by body on the device (mfs_evaluate, mfs_evaluate_stress): the owner of each
// point (given, or the nearest body centre), a stable counting sort by the owner's key, and the points
// relative to their owner's centre in the layouts of the pair kernels.
//
// Latency-bound: a few launches over the points and one copy of the bodies' offsets back to the host.
// The points are cut into chunks; each chunk counts its points per key, a scan turns the counts into
// positions, and one warp per chunk places its points in order (so equal keys keep the caller's order
// and a call's result does not depend on timing).  On the host the same grouping took 6.5 ms for
// 100 003 points without owners and 60 bodies, and 1 ms for 72 000 points with owners: the velocity call
// took 9.78 ms and takes 1.38 ms, pressure and traction took 2.61 ms and take 1.23 ms (60 spheres, N = 300;
// the pair kernels' share is about 1 ms of either).
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace mfs {

#define EVAL_THREADS 256

// chunks of 256 points (the placing warp's 8 dependent rounds), longer ones beyond 1024 chunks
int eval_chunks(int np) { return std::max(1, std::min(1024, (np + 255) / 256)); }

__device__ __forceinline__ int chunk_begin(int np, int nchunks, int c) {
    return (int)((long long)np * c / nchunks);
}
__device__ __forceinline__ int chunk_of(int np, int nchunks, int i) {
    int c = (int)((long long)i * nchunks / np);
    while (chunk_begin(np, nchunks, c + 1) <= i) ++c;
    while (chunk_begin(np, nchunks, c) > i) --c;
    return c;
}

// key[i] of every point, counts[chunk][key]; err |= MFS_DEVERR_BADARG for an owner outside [0, P) or a
// non-finite coordinate (such a point gets key 0).  Without owners the nearest centre is taken, the
// first of equals.
__global__ void __launch_bounds__(EVAL_THREADS) eval_key_kernel(const double *pts, const double *nrm, const int *owner,
                                                                int np, const double *centres, int P,
                                                                const int *key_of_body, int nchunks, int *key,
                                                                int *counts, int *err) {
    __shared__ double sc[EVAL_THREADS][3];
    const int i = blockIdx.x * EVAL_THREADS + threadIdx.x;
    const bool in = i < np;
    double x[3] = {0.0, 0.0, 0.0};
    bool ok = true;
    if (in)
        for (int a = 0; a < 3; ++a) {
            x[a] = pts[3 * (size_t)i + a];
            ok = ok && isfinite(x[a]) && (!nrm || isfinite(nrm[3 * (size_t)i + a]));
        }
    int b = 0;
    if (owner) {
        if (in) b = owner[i];
        ok = ok && b >= 0 && b < P;
    } else {
        double best = 1e300;
        for (int k0 = 0; k0 < P; k0 += EVAL_THREADS) {
            const int n = min(EVAL_THREADS, P - k0);
            __syncthreads();
            if ((int)threadIdx.x < n)
                for (int a = 0; a < 3; ++a) sc[threadIdx.x][a] = centres[3 * (size_t)(k0 + threadIdx.x) + a];
            __syncthreads();
            for (int k = 0; k < n; ++k) {
                double d2 = 0.0;
                for (int a = 0; a < 3; ++a) {
                    const double d = x[a] - sc[k][a];
                    d2 += d * d;
                }
                if (d2 < best) {
                    best = d2;
                    b = k0 + k;
                }
            }
        }
    }
    if (!in) return;
    if (!ok) {
        atomicOr(err, MFS_DEVERR_BADARG);
        b = 0;
    }
    const int q = key_of_body ? key_of_body[b] : b;
    key[i] = q;
    atomicAdd(&counts[(size_t)chunk_of(np, nchunks, i) * P + q], 1);
}

// counts[c][q] -> points of key q in the chunks before c; total[q]
__global__ void eval_chunk_scan_kernel(int *counts, int nchunks, int P, int *total) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= P) return;
    int run = 0;
    for (int c0 = 0; c0 < nchunks; c0 += 32) {  // 32 loads in flight
        int v[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = c0 + u < nchunks ? counts[(size_t)(c0 + u) * P + q] : 0;
#pragma unroll
        for (int u = 0; u < 32; ++u)
            if (c0 + u < nchunks) {
                counts[(size_t)(c0 + u) * P + q] = run;
                run += v[u];
            }
    }
    total[q] = run;
}

// toff[0 .. P]: exclusive scan of total (one block)
__global__ void __launch_bounds__(1024) eval_offsets_kernel(const int *total, int P, int *toff) {
    __shared__ int sh[1024];
    const int t = threadIdx.x;
    const int q0 = (int)((long long)P * t / 1024), q1 = (int)((long long)P * (t + 1) / 1024);
    int sum = 0;
    for (int q = q0; q < q1; ++q) sum += total[q];
    sh[t] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const int v = t >= o ? sh[t - o] : 0;
        __syncthreads();
        sh[t] += v;
        __syncthreads();
    }
    int run = sh[t] - sum;
    for (int q = q0; q < q1; ++q) {
        toff[q] = run;
        run += total[q];
    }
    if (t == 1023) toff[P] = sh[1023];
}

// One warp per chunk, 32 points at a time in order: position = toff[key] + earlier points of the key.
__global__ void eval_place_kernel(const double *pts, const double *nrm, const int *key, int np,
                                  const int *body_of_key, const double *centres, int P, int nchunks, int *counts,
                                  const int *toff, int *order, float4 *t4, float *n32, double *t64, double *n64,
                                  int *tbody, unsigned long long *radius) {
    const int c = blockIdx.x, lane = threadIdx.x;
    const int i0 = chunk_begin(np, nchunks, c), i1 = chunk_begin(np, nchunks, c + 1);
    int *run = counts + (size_t)c * P;
    for (int ib = i0; ib < i1; ib += 32) {
        const int i = ib + lane;
        const bool in = i < i1;
        const int q = in ? key[i] : -1;
        const unsigned same = __match_any_sync(0xffffffffu, q);
        const int before = __popc(same & ((1u << lane) - 1u));
        int base = 0;
        if (in && before == 0) {
            base = run[q];
            run[q] = base + __popc(same);
        }
        base = __shfl_sync(0xffffffffu, base, __ffs(same) - 1);
        if (in) {
            const int j = toff[q] + base + before;
            const int b = body_of_key ? body_of_key[q] : q;
            double x[3], r2 = 0.0;
            for (int a = 0; a < 3; ++a) {
                x[a] = pts[3 * (size_t)i + a] - centres[3 * (size_t)b + a];
                r2 += x[a] * x[a];
            }
            order[j] = i;
            t4[j] = make_float4((float)x[0], (float)x[1], (float)x[2], __int_as_float(q));
            if (t64)
                for (int a = 0; a < 3; ++a) t64[3 * (size_t)j + a] = x[a];
            if (tbody) tbody[j] = q;
            if (nrm)
                for (int a = 0; a < 3; ++a) {
                    const double v = nrm[3 * (size_t)i + a];
                    n32[3 * (size_t)j + a] = (float)v;
                    if (n64) n64[3 * (size_t)j + a] = v;
                }
            // non-negative doubles order as their bits
            if (radius) atomicMax(&radius[q], (unsigned long long)__double_as_longlong(sqrt(r2)));
        }
        __syncwarp();
    }
}

cudaError_t eval_group(const EvalGroup &e, cudaStream_t st) {
    const int nch = eval_chunks(e.np);
    cudaError_t rc = cudaMemsetAsync(e.counts, 0, sizeof(int) * (size_t)nch * e.P, st);
    if (rc == cudaSuccess && e.radius) rc = cudaMemsetAsync(e.radius, 0, sizeof(unsigned long long) * e.P, st);
    if (rc != cudaSuccess) return rc;
    eval_key_kernel<<<(e.np + EVAL_THREADS - 1) / EVAL_THREADS, EVAL_THREADS, 0, st>>>(
        e.points, e.normals, e.owner, e.np, e.centres, e.P, e.key_of_body, nch, e.key, e.counts, e.err);
    eval_chunk_scan_kernel<<<(e.P + 127) / 128, 128, 0, st>>>(e.counts, nch, e.P, e.total);
    eval_offsets_kernel<<<1, 1024, 0, st>>>(e.total, e.P, e.toff);
    eval_place_kernel<<<nch, 32, 0, st>>>(e.points, e.normals, e.key, e.np, e.body_of_key, e.centres, e.P, nch,
                                          e.counts, e.toff, e.order, e.t4, e.n32, e.t64, e.n64, e.tbody, e.radius);
    return cudaGetLastError();
}

}  // namespace mfs
