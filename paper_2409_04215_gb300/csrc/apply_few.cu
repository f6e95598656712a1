// The one-body apply for few columns (bodies of one shape times right-hand sides, at most FC_MAX), and
// the scatter that ends every one-body apply.
//
// The tensor-core GEMM (tc_gemm.cu) needs 16 columns to fill its smallest tile, splits K into partial
// sums and needs a reduction kernel after each product: about 13 us a product for six columns however
// small the factor (barrier and TMEM set-up, the TMA -> cut -> MMA -> TMEM chain, the extra launch), which
// was 40 % of an iteration on a handful of bodies.  Here warps walk the factor's rows directly:
//   out[c][row] = sum_k F[row][k] g[c][k],  F and g as FP32 (hi, lo) pairs,
// every product split exactly by an FMA, accumulated by TwoSum (about 2^-45 relative, against 2^-33
// products and FP32 accumulation runs on the tensor cores).  Bound by the factor's bytes (8 per element,
// from L2 between iterations) until eleven FP32 operations per element and column outweigh them.
// Six spheres (M = 240, N = 120), whole solve of 13 iterations: 942 -> 872 us with the apply, the scatter that
// also packs and the spread epilogue (817 us with today's Arnoldi step); velocities 7e-8 from the FP64
// solution instead of 1.2e-6.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace mfs {

// (hi, lo) += (h, l), renormalised.
__device__ __forceinline__ void fc_add(float &hi, float &lo, float h, float l) {
    float s, e;
    two_sum(hi, h, s, e);
    e = __fadd_rn(__fadd_rn(lo, l), e);
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}

// (hi, lo) += (fh + fl)(gh + gl)
__device__ __forceinline__ void fc_fma(float &hi, float &lo, float fh, float fl, float gh, float gl) {
    const float p = __fmul_rn(fh, gh);
    float e = __fmaf_rn(fh, gh, -p);
    e = __fmaf_rn(fh, gl, e);
    e = __fmaf_rn(fl, gh, e);
    float s, t;
    two_sum(hi, p, s, t);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(t, e));
}

// wpr warps per row (1, 2 or 4) share its K range; 4 warps per block.
template <int NC>
__global__ void __launch_bounds__(128) fc_apply_kernel(int rows, int ldk, const float *__restrict__ F, size_t pstride,
                                                       const float2 *__restrict__ G, float2 *__restrict__ out, int ldo,
                                                       int wpr) {
    __shared__ float2 part[4][NC];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * (4 / wpr) + warp / wpr, sub = warp % wpr;
    float hi[NC], lo[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) hi[c] = lo[c] = 0.f;
    if (row < rows) {
        const float4 *fh = reinterpret_cast<const float4 *>(F + (size_t)row * ldk);
        const float4 *fl = reinterpret_cast<const float4 *>(F + pstride + (size_t)row * ldk);
#pragma unroll 2
        for (int i = 32 * sub + lane; i < ldk / 4; i += 32 * wpr) {
            const float4 h = fh[i], l = fl[i];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float4 *g = reinterpret_cast<const float4 *>(G + (size_t)c * ldk) + 2 * i;
                const float4 g0 = g[0], g1 = g[1];
                fc_fma(hi[c], lo[c], h.x, l.x, g0.x, g0.y);
                fc_fma(hi[c], lo[c], h.y, l.y, g0.z, g0.w);
                fc_fma(hi[c], lo[c], h.z, l.z, g1.x, g1.y);
                fc_fma(hi[c], lo[c], h.w, l.w, g1.z, g1.w);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
        for (int o = 16; o > 0; o >>= 1) {
            const float h = __shfl_xor_sync(0xffffffffu, hi[c], o), l = __shfl_xor_sync(0xffffffffu, lo[c], o);
            fc_add(hi[c], lo[c], h, l);
        }
    if (lane == 0)
#pragma unroll
        for (int c = 0; c < NC; ++c) part[warp][c] = make_float2(hi[c], lo[c]);
    __syncthreads();
    if (sub == 0 && lane < NC && row < rows) {
        float h = part[warp][lane].x, l = part[warp][lane].y;
        for (int w = 1; w < wpr; ++w) fc_add(h, l, part[warp + w][lane].x, part[warp + w][lane].y);
        out[(size_t)lane * ldo + row] = make_float2(h, l);
    }
}

cudaError_t fc_apply(int ncols, int rows, int ldk, const float *F, size_t pstride, const float2 *G, float2 *out, int ldo,
                     cudaStream_t st) {
    // warps per row so that even a small factor gives every SM a few warps
    const int wpr = rows <= 1024 ? 4 : (rows <= 4096 ? 2 : 1);
    const int grid = (rows * wpr + 3) / 4;
#define FC(N_)                                                                                \
    if (ncols == N_) {                                                                        \
        fc_apply_kernel<N_><<<grid, 128, 0, st>>>(rows, ldk, F, pstride, G, out, ldo, wpr);   \
        return cudaGetLastError();                                                            \
    }
    FC(1) FC(2) FC(3) FC(4) FC(5) FC(6) FC(7) FC(8)
#undef FC
    return cudaErrorInvalidValue;
}

// Gather and rotate into the body frame (as gather_rotate), written as FP32 (hi, lo) pairs [col][ld].
__global__ void gather_rotate_hl_kernel(int D, const double *gamma, int sum_MD, const int *col_body, const int *col_rhs,
                                        const int *body_off, const double *rot, int M, float2 *out, int ld) {
    const int col = blockIdx.y, p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= M) return;
    const int k = col_body[col], h = col_rhs[col];
    const double *gk = gamma + (size_t)h * sum_MD + (size_t)body_off[k] * D;
    float2 *o = out + (size_t)col * ld;
    auto put = [&](int i, double v) {
        const float f = (float)v;
        o[i] = make_float2(f, (float)(v - (double)f));
    };
    if (D == 1) {
        put(p, gk[p]);
    } else {
        const double *R = rot + 9 * k;  // row-major R; (R^T g)_a = sum_b R[b][a] g_b
        const double g0 = gk[3 * p], g1 = gk[3 * p + 1], g2 = gk[3 * p + 2];
#pragma unroll
        for (int a = 0; a < 3; ++a) put(3 * p + a, R[a] * g0 + R[3 + a] * g1 + R[6 + a] * g2);
    }
}

cudaError_t gather_rotate_hl(int D, const double *gamma, int sum_MD, const int *col_body, const int *col_rhs,
                             const int *body_off, const double *rot, int ncols, int dM, float2 *out, int ld,
                             cudaStream_t st) {
    const int M = dM / D;
    gather_rotate_hl_kernel<<<dim3((M + 63) / 64, ncols), 64, 0, st>>>(D, gamma, sum_MD, col_body, col_rhs, body_off, rot,
                                                                      M, out, ld);
    return cudaGetLastError();
}

// The end of a one-body apply, one thread per point and column: the column's values (FP64, or (hi, lo)
// chunk partials added here in double-float), rotated to the global frame, out = base + R v (base may be
// null); with `rec` also the pair kernel's source records of the point (position, strengths, zero
// padding records), which otherwise take two more launches and another pass over the strengths.
template <int D>
__global__ void scatter_rotate_kernel(ScatterArgs a) {
    const int col = blockIdx.y, p = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = a.dN / D, Np = a.rec ? (N + 3) / 4 * 4 : N;
    if (p >= Np) return;
    const int k = a.col_body[col], h = a.col_rhs[col];
    double x[D];
#pragma unroll
    for (int c = 0; c < D; ++c) x[c] = 0.0;
    if (p < N) {
        double v[D];
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const size_t i = (size_t)col * a.dN + D * p + c;
            if (a.P) {
                float hi = 0.f, lo = 0.f;
                for (int z = 0; z < a.S; ++z) {
                    const float2 q = a.P[(size_t)z * a.ncols * a.dN + i];
                    fc_add(hi, lo, q.x, q.y);
                }
                v[c] = (double)hi + (double)lo;
            } else {
                v[c] = a.L64[i];
            }
        }
        const size_t o = ((size_t)h * a.sum_N + a.body_off[k] + p) * D;
        if constexpr (D == 3) {
            const double *R = a.rot64 + 9 * k;
#pragma unroll
            for (int c = 0; c < 3; ++c) x[c] = R[3 * c] * v[0] + R[3 * c + 1] * v[1] + R[3 * c + 2] * v[2];
        } else {
            x[0] = v[0];
        }
#pragma unroll
        for (int c = 0; c < D; ++c) a.out[o + c] = a.base ? a.base[o + c] + x[c] : x[c];
    }
    if (!a.rec) return;
    const int dup = a.packed ? 2 : 1;
    float *r = a.rec + (size_t)(a.rec_off[k] + p) * a.rec_floats;
#pragma unroll
    for (int c = 0; c < D; ++c)
        for (int d = 0; d < dup; ++d) r[dup * (3 + D * h + c) + d] = (float)x[c];
    if (h == 0) {
        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p < N) y = a.src_pos[a.body_off[k] + p];
        for (int d = 0; d < dup; ++d) {
            r[d] = y.x;
            r[dup + d] = y.y;
            r[2 * dup + d] = y.z;
        }
        for (int c = dup * (3 + D * a.nrhs); c < a.rec_floats; ++c) r[c] = 0.f;
    }
}

cudaError_t scatter_rotate(int D, const ScatterArgs &a, cudaStream_t st) {
    if (a.ncols == 0) return cudaSuccess;
    const int N = a.dN / D, Np = a.rec ? (N + 3) / 4 * 4 : N;
    const dim3 grid((Np + 63) / 64, a.ncols);
    if (D == 3)
        scatter_rotate_kernel<3><<<grid, 64, 0, st>>>(a);
    else
        scatter_rotate_kernel<1><<<grid, 64, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace mfs
