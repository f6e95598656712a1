// Far-field acceleration of the pair sums (host side): the tree over the bodies and the interaction
// lists of an equivalent-source treecode.
//
// The paper accelerates its pair sums with a fast multipole method on the CPU (Sec. 4: FMM3D, more
// than 90 % of its time).  Here the far field is represented the kernel-independent way, with the
// MFS's own device: every node of a tree over the bodies (each body, and each group of bodies) gets
// FF_NE equivalent point sources on a sphere of radius r_e around its centre whose field reproduces
// that of the node's proxy sources outside it.  The equivalent strengths are the least-squares fit
// of the sources' field on FF_NC check points at radius FF_CHECK * r_e (the "upward" step, run on the
// device), and a target at least kappa * r_e from a node's centre (kappa = farfield_separation, 3 by
// default) sees the node through them; further off through fewer points (lower orders, kernels.h), and
// where it pays through a local expansion: sources around each body that reproduce, at its targets, the
// field of all nodes well away from it.
// Targets nearer than that see the node's children, down to the bodies' own proxy points.  Both the
// fit's right-hand side and the final sums are ordinary pair sums over interaction lists, so the
// device work is the pair kernel plus a few FP64 matrix products per apply.
//
// This file builds, on the host: the tree (8-ary, by median splits of the body centres in x, then y,
// then z), the nodes' centres and radii, and the interaction list of a set of target bodies.
#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

#include "kernels.h"

namespace mfs {

namespace {

struct Builder {
    const double *centres;
    const double *rsrc;
    std::vector<FFNode> &nodes;
    std::vector<int> &order;

    int leaf(int b) {
        FFNode n;
        for (int a = 0; a < 3; ++a) n.c[a] = centres[3 * b + a];
        n.rs = rsrc[b];
        n.body = b;
        n.first = (int)order.size();
        n.count = 1;
        order.push_back(b);
        nodes.push_back(n);
        return (int)nodes.size() - 1;
    }

    // Split ids into two halves (sizes differing by at most one) by the coordinate `axis`.
    static void halve(std::vector<int> &ids, int axis, const double *centres, std::vector<int> &lo,
                      std::vector<int> &hi) {
        std::sort(ids.begin(), ids.end(), [&](int a, int b) {
            const double xa = centres[3 * a + axis], xb = centres[3 * b + axis];
            return xa < xb || (xa == xb && a < b);
        });
        const size_t h = ids.size() / 2;
        lo.assign(ids.begin(), ids.begin() + h);
        hi.assign(ids.begin() + h, ids.end());
    }

    int build(std::vector<int> ids) {
        if (ids.size() == 1) return leaf(ids[0]);
        const int me = (int)nodes.size();
        nodes.push_back(FFNode());
        std::vector<std::vector<int>> groups;
        if (ids.size() <= 8) {
            for (int b : ids) groups.push_back({b});
        } else {
            std::vector<int> x0, x1;
            halve(ids, 0, centres, x0, x1);
            for (auto *gx : {&x0, &x1}) {
                std::vector<int> y0, y1;
                halve(*gx, 1, centres, y0, y1);
                for (auto *gy : {&y0, &y1}) {
                    std::vector<int> z0, z1;
                    halve(*gy, 2, centres, z0, z1);
                    if (!z0.empty()) groups.push_back(z0);
                    if (!z1.empty()) groups.push_back(z1);
                }
            }
        }
        const int first = (int)order.size();
        std::vector<int> kids;
        for (auto &g : groups) kids.push_back(build(g));
        FFNode n;
        n.body = -1;
        n.first = first;
        n.count = (int)order.size() - first;
        n.nchild = (int)kids.size();
        for (int i = 0; i < n.nchild; ++i) n.child[i] = kids[i];
        // centre: middle of the bounding box of the descendant bodies' centres; radius of its sources
        double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
        for (int q = n.first; q < n.first + n.count; ++q)
            for (int a = 0; a < 3; ++a) {
                lo[a] = std::min(lo[a], centres[3 * order[q] + a]);
                hi[a] = std::max(hi[a], centres[3 * order[q] + a]);
            }
        for (int a = 0; a < 3; ++a) n.c[a] = 0.5 * (lo[a] + hi[a]);
        double rs = 0.0;
        for (int q = n.first; q < n.first + n.count; ++q) {
            const int b = order[q];
            double d2 = 0.0;
            for (int a = 0; a < 3; ++a) d2 += (centres[3 * b + a] - n.c[a]) * (centres[3 * b + a] - n.c[a]);
            rs = std::max(rs, std::sqrt(d2) + rsrc[b]);
        }
        n.rs = rs;
        nodes[me] = n;
        return me;
    }
};

}  // namespace

void ff_build_tree(int P, const double *centres, const double *rsrc, int S, const int *body_off, FFTree &t) {
    t.nodes.clear();
    t.order.clear();
    t.roots.clear();
    t.nodes.reserve(2 * (size_t)P);
    t.order.reserve(P);
    Builder bld{centres, rsrc, t.nodes, t.order};
    for (int s = 0; s < S; ++s) {
        std::vector<int> ids(body_off[s + 1] - body_off[s]);
        std::iota(ids.begin(), ids.end(), body_off[s]);
        t.roots.push_back(bld.build(ids));
    }
    t.pos.assign(P, 0);
    for (int q = 0; q < P; ++q) t.pos[t.order[q]] = q;
    for (auto &n : t.nodes) n.re = n.rs / FF_SRC_RATIO;
}

void ff_interaction_list(const FFTree &t, int root, const std::vector<int> &tbodies, const double *centres,
                         const double *rtgt, double kappa, int self_skip, std::vector<int> &segs) {
    const int P = (int)t.order.size();
    std::vector<int> stack{root};
    while (!stack.empty()) {
        const int ni = stack.back();
        stack.pop_back();
        const FFNode &n = t.nodes[ni];
        // far: every target point of the set is at least kappa r_e from the node's centre
        bool far = true;
        for (int b : tbodies) {
            double d2 = 0.0;
            for (int a = 0; a < 3; ++a) d2 += (centres[3 * b + a] - n.c[a]) * (centres[3 * b + a] - n.c[a]);
            if (std::sqrt(d2) - rtgt[b] < kappa * n.re) {
                far = false;
                break;
            }
        }
        if (far) {
            segs.push_back(P + ni);
        } else if (n.body >= 0) {
            if (!(self_skip && tbodies.size() == 1 && tbodies[0] == n.body)) segs.push_back(t.pos[n.body]);
        } else {
            for (int i = n.nchild - 1; i >= 0; --i) stack.push_back(n.child[i]);
        }
    }
}

int ff_order(double ratio, double kappa0) {
    const double f = std::max(1.0, kappa0 / FF_ORD_KAPPA[0]);
    if (!(ratio >= kappa0)) return -1;
    int o = 0;
    while (o + 1 < FF_NORD && ratio >= f * FF_ORD_KAPPA[o + 1]) ++o;
    return o;
}

static double distance_to(const FFNode &n, const double *c) {
    double d2 = 0.0;
    for (int a = 0; a < 3; ++a) d2 += (c[a] - n.c[a]) * (c[a] - n.c[a]);
    return std::sqrt(d2);
}

void ff_ordered_list(const FFTree &t, int root, const std::vector<int> &tbodies, const double *centres,
                     const double *rtgt, double kappa0, int self_skip, std::vector<int> &segs) {
    const int P = (int)t.order.size(), nodes = (int)t.nodes.size();
    std::vector<int> stack{root};
    while (!stack.empty()) {
        const int ni = stack.back();
        stack.pop_back();
        const FFNode &n = t.nodes[ni];
        double near = 1e300;  // the nearest target point to the node's centre, at least
        for (int b : tbodies) near = std::min(near, distance_to(n, centres + 3 * b) - rtgt[b]);
        const int o = ff_order(near / n.re, kappa0);
        if (o >= 0) {
            segs.push_back(P + o * nodes + ni);
        } else if (n.body >= 0) {
            if (!(self_skip && tbodies.size() == 1 && tbodies[0] == n.body)) segs.push_back(t.pos[n.body]);
        } else {
            for (int i = n.nchild - 1; i >= 0; --i) stack.push_back(n.child[i]);
        }
    }
}

void ff_cell_lists(const FFTree &t, int root, const std::vector<int> &tbodies, const double *centres,
                   const double *rtgt, double kappa0, double targets_per_body, std::vector<int> &local,
                   std::vector<std::vector<int>> &direct) {
    const int P = (int)t.order.size(), nodes = (int)t.nodes.size(), nt = (int)tbodies.size();
    const double gap = FF_LOC_GAP * std::max(1.0, kappa0 / FF_ORD_KAPPA[0]);
    local.clear();
    direct.assign(nt, {});
    double points = 0.0;  // equivalent points in `local`
    std::vector<int> stack{root};
    while (!stack.empty()) {
        const int ni = stack.back();
        stack.pop_back();
        const FFNode &n = t.nodes[ni];
        bool all = true;
        double near = 1e300;
        for (int b : tbodies) {
            const double d = distance_to(n, centres + 3 * b);
            near = std::min(near, d - FF_LOC_CHECK * rtgt[b]);  // its check points
            all = all && d - n.re >= gap * rtgt[b];
            if (!all) break;
        }
        const int o = all ? ff_order(near / n.re, kappa0) : -1;
        if (o >= 0) {
            local.push_back(P + o * nodes + ni);
            points += FF_ORD_N[o];
        } else if (n.body < 0) {
            for (int i = n.nchild - 1; i >= 0; --i) stack.push_back(n.child[i]);
        } else {
            for (int i = 0; i < nt; ++i) {  // one source body: each target body by its own distance
                if (tbodies[i] == n.body) continue;
                const double ratio = (distance_to(n, centres + 3 * tbodies[i]) - rtgt[tbodies[i]]) / n.re;
                const int oi = ff_order(ratio, kappa0);
                direct[i].push_back(oi >= 0 ? P + oi * nodes + ni : t.pos[n.body]);
            }
        }
    }
    if (local.empty()) return;
    const bool pays = points * targets_per_body >
                      points * FF_LOC_NC + targets_per_body * FF_LOC_N + FF_LOC_FIT_PAIRS;
    for (int i = 0; i < nt; ++i) {
        if (pays) direct[i].push_back(P + FF_NORD * nodes + t.pos[tbodies[i]]);
        else direct[i].insert(direct[i].end(), local.begin(), local.end());
    }
    if (!pays) local.clear();
}

// One block per body (tree position) and right-hand side, one thread per check point.  The constant is the
// mean over the points; the gradient 3 / (n R^2) sum (u - mean) x, as the points spread evenly over the
// sphere of radius R, made free of divergence for a velocity (the sources' field is).  It need not be the
// best fit (its sums are FP32): whatever is taken out here is added at the targets, both in FP64, and the
// local sources carry the rest.  Bound by FP64 operations (2 per clock per SM).
template <int D>
__global__ void __launch_bounds__(FF_LOC_NC)
ff_take_linear_kernel(double *u, const float4 *chk, const double *radius, int bodies, double *far) {
    constexpr int W = FF_LOC_NC / 32;
    __shared__ double mean_w[W][D];
    __shared__ float grad_w[W][3 * D];
    const int q = blockIdx.x % bodies, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *mine = u + ((size_t)blockIdx.x * FF_LOC_NC + threadIdx.x) * D;
    const float4 p = chk[(size_t)q * FF_LOC_NC + threadIdx.x];
    const float x[3] = {p.x, p.y, p.z};
    double v[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        double s = v[d] = mine[d];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) mean_w[warp][d] = s;
    }
    __syncthreads();
#pragma unroll
    for (int d = 0; d < D; ++d) {
        double mean = 0.0;
        for (int w = 0; w < W; ++w) mean += mean_w[w][d];
        mean *= 1.0 / FF_LOC_NC;
        v[d] -= mean;
        if (threadIdx.x == 0) far[(size_t)blockIdx.x * 4 * D + d] = mean;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float s = (float)v[d] * x[a];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) grad_w[warp][a * D + d] = s;
        }
    }
    __syncthreads();
    const double R = FF_LOC_CHECK * radius[q], f = 3.0 / (FF_LOC_NC * R * R);
    float g[3 * D];
#pragma unroll
    for (int c = 0; c < 3 * D; ++c) {
        g[c] = 0.f;
        for (int w = 0; w < W; ++w) g[c] += grad_w[w][c];
        g[c] = (float)(f * g[c]);
    }
    if constexpr (D == 3) {
        const float third = (g[0] + g[4] + g[8]) / 3.f;
        g[0] -= third;
        g[4] -= third;
        g[8] -= third;
    }
#pragma unroll
    for (int d = 0; d < D; ++d)
        mine[d] = v[d] - ((double)x[0] * g[d] + (double)x[1] * g[D + d] + (double)x[2] * g[2 * D + d]);
#pragma unroll
    for (int c = 0; c < 3 * D; ++c)
        if (threadIdx.x == c) far[((size_t)blockIdx.x * 4 + 1) * D + c] = g[c];
}

cudaError_t ff_take_linear(int D, double *u, const float4 *chk, const double *radius, int bodies, int nrhs, double *far,
                           cudaStream_t st) {
    const unsigned n = (unsigned)bodies * nrhs;
    if (n == 0) return cudaSuccess;
    if (D == 3)
        ff_take_linear_kernel<3><<<n, FF_LOC_NC, 0, st>>>(u, chk, radius, bodies, far);
    else
        ff_take_linear_kernel<1><<<n, FF_LOC_NC, 0, st>>>(u, chk, radius, bodies, far);
    return cudaGetLastError();
}

__global__ void ff_scale_kernel(double *mu, const double *re, int nodes, int per_node, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        mu[i] *= re[(i / per_node) % nodes];
}

cudaError_t ff_scale(double *mu, const double *re, int nodes, int per_node, int nrhs, cudaStream_t st) {
    const size_t n = (size_t)nrhs * nodes * per_node;
    if (n == 0) return cudaSuccess;
    ff_scale_kernel<<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, st>>>(mu, re, nodes, per_node, n);
    return cudaGetLastError();
}

}  // namespace mfs
