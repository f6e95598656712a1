"""The treecode's lower orders and local expansions (farfield.cu), on the CPU.

* The cell and body lists (a C++ driver on the library's own code): every target body sees every other
  body of its suspension exactly once, through its cell's local nodes or its own list; each node's
  order obeys its distance rule, each local node the gap to every body of the cell.
* The representation in NumPy: the chain 196 -> 128 -> 96 -> 64 of equivalent sources and the local
  sources reproduce a white-noise source cloud's field at the distances where the lists use them,
  within three times the errors that the parameters were chosen for (three random draws differ by
  less than a factor of two).
"""

import os
import subprocess

import numpy as np
import pytest

from test_farfield_fit import fibonacci, kernel_matrix

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_04215_gb300", "csrc")
ORD_N, ORD_NC, ORD_CHECK, ORD_KAPPA = (196, 128, 96, 64), (256, 192, 160, 128), (2.6, 4.0, 5.0, 8.0), (3.0, 4.0, 5.0, 8.0)
ORD_TRUNC, LOC_TRUNC = (1e-12, 1e-12, 1e-12, 1e-8), 1e-8
LOC_N, LOC_NC, LOC_CHECK, LOC_EQ, LOC_GAP = 96, 128, 1.1, 6.0, 5.0

DRIVER = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "kernels.h"
using namespace mfs;
int main(int argc, char **argv) {
    FILE *f = std::fopen(argv[1], "r");
    int P, S, cell; double kappa, tpb;
    if (std::fscanf(f, "%d %d %lf %d %lf", &P, &S, &kappa, &cell, &tpb) != 5) return 1;
    std::vector<int> off(S + 1);
    for (auto &o : off) if (std::fscanf(f, "%d", &o) != 1) return 1;
    std::vector<double> c(3 * P), rs(P), rt(P);
    for (int k = 0; k < P; ++k)
        if (std::fscanf(f, "%lf %lf %lf %lf %lf", &c[3 * k], &c[3 * k + 1], &c[3 * k + 2], &rs[k], &rt[k]) != 5)
            return 1;
    FFTree t;
    ff_build_tree(P, c.data(), rs.data(), S, off.data(), t);
    std::printf("order");
    for (int b : t.order) std::printf(" %d", b);
    std::printf("\n");
    for (size_t i = 0; i < t.nodes.size(); ++i)
        std::printf("node %.17g %.17g %.17g %.17g %d %d\n", t.nodes[i].c[0], t.nodes[i].c[1], t.nodes[i].c[2],
                    t.nodes[i].re, t.nodes[i].first, t.nodes[i].count);
    auto put = [](const char *what, int id, const std::vector<int> &v) {
        std::printf("%s %d", what, id);
        for (int g : v) std::printf(" %d", g);
        std::printf("\n");
    };
    std::vector<int> tb, local;
    std::vector<std::vector<int>> direct;
    for (int s = 0; s < S; ++s)
        for (int q0 = off[s]; q0 < off[s + 1]; q0 += cell) {
            tb.assign(t.order.begin() + q0, t.order.begin() + std::min(q0 + cell, off[s + 1]));
            ff_cell_lists(t, t.roots[s], tb, c.data(), rt.data(), kappa, tpb, local, direct);
            for (size_t i = 0; i < tb.size(); ++i) {
                put("local", tb[i], local);
                put("direct", tb[i], direct[i]);
                std::vector<int> segs;
                ff_ordered_list(t, t.roots[s], std::vector<int>{tb[i]}, c.data(), rt.data(), kappa, 1, segs);
                put("ordered", tb[i], segs);
            }
        }
    return 0;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("ffo")
    (d / "driver.cu").write_text(DRIVER)
    exe = d / "ff_orders"
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    str(d / "driver.cu"), os.path.join(CSRC, "farfield.cu"), "-o", str(exe)], check=True)
    return exe, d


@pytest.mark.parametrize("case", ["cluster", "suspensions"])
@pytest.mark.parametrize("kappa,cell,tpb", [(3.0, 5, 1000.0), (2.5, 2, 1000.0), (4.5, 4, 1000.0), (3.0, 5, 40.0)])
def test_cell_lists_cover_every_body_once(probe, case, kappa, cell, tpb):
    from mfs_inputs import make_workload

    exe, d = probe
    if case == "cluster":
        wl = make_workload("ellipsoidT5000_mobility", count=700, n_v=12)
    else:
        wl = make_workload("batched256_mobility", num_suspensions=7, p_lo=1, p_hi=70, m=60, n=30, seed=12)
    off = wl.body_offsets
    rs = [np.linalg.norm(wl.shapes[i].proxy, axis=1).max() for i in wl.shape_id]
    rt = [np.linalg.norm(wl.shapes[i].colloc, axis=1).max() for i in wl.shape_id]
    with open(d / "in.txt", "w") as f:
        f.write(f"{wl.num_bodies} {len(off) - 1} {kappa!r} {cell} {tpb!r}\n" + " ".join(str(int(o)) for o in off) + "\n")
        for c, a, b in zip(wl.centres, rs, rt):
            f.write(" ".join(repr(float(v)) for v in (*c, a, b)) + "\n")
    lines = subprocess.run([str(exe), str(d / "in.txt")], capture_output=True, text=True, check=True).stdout.splitlines()
    order = [int(x) for x in lines[0].split()[1:]]
    nodes, lists = [], {"local": {}, "direct": {}, "ordered": {}}
    for line in lines[1:]:
        w = line.split()
        if w[0] == "node":
            nodes.append((np.array([float(x) for x in w[1:4]]), float(w[4]), int(w[5]), int(w[6])))
        else:
            lists[w[0]][int(w[1])] = [int(x) for x in w[2:]]
    P, n = wl.num_bodies, len(nodes)
    pos = {b: q for q, b in enumerate(order)}
    scale = max(1.0, kappa / 3.0)

    def bodies(g, t, reach):  # descendants of a segment, its distance rule checked at `reach`
        if g < P:
            return [order[g]]
        o, nd = divmod(g - P, n)
        c, re, first, count = nodes[nd]
        ratio = (np.linalg.norm(wl.centres[t] - c) - reach) / re
        assert o < 4 and ratio >= (kappa if o == 0 else scale * ORD_KAPPA[o]) * (1 - 1e-12)
        return order[first:first + count]

    used = 0
    for s in range(len(off) - 1):
        for t in range(off[s], off[s + 1]):
            want = [b for b in range(off[s], off[s + 1]) if b != t]
            seen, own = [], P + 4 * n + pos[t]
            for g in lists["local"][t]:
                seen += bodies(g, t, LOC_CHECK * rt[t])
                c, re = nodes[(g - P) % n][:2]
                assert np.linalg.norm(wl.centres[t] - c) - re >= LOC_GAP * scale * rt[t] * (1 - 1e-12)
            assert lists["direct"][t].count(own) == (1 if lists["local"][t] else 0)
            used += bool(lists["local"][t])
            for g in lists["direct"][t]:
                if g != own:
                    seen += bodies(g, t, rt[t])
            assert sorted(seen) == want
            assert sorted(b for g in lists["ordered"][t] for b in bodies(g, t, rt[t])) == want
    if case == "cluster":  # many bodies: local expansions with many targets a body, none with few
        assert (used > 0) == (tpb > 100.0)


def _pinv(A, trunc=1e-12):
    U, s, Vt = np.linalg.svd(A, full_matrices=False)
    k = s > trunc * s[0]
    return (Vt[k].T / s[k]) @ U[:, k].T


def _rotated(rng, n):
    return fibonacci(n) @ np.linalg.qr(rng.standard_normal((3, 3)))[0]


@pytest.mark.parametrize("d", [1, 3])
def test_lower_orders_reproduce_the_field(d):
    rng = np.random.default_rng(4)
    src, lam = 0.83 * _rotated(rng, 300), rng.standard_normal((300 * d, 2))
    e = [fibonacci(k) for k in ORD_N]
    mu = _pinv(kernel_matrix(CHECK0 := ORD_CHECK[0] * fibonacci(ORD_NC[0]), e[0], d)) @ \
        (kernel_matrix(CHECK0, src, d) @ lam)
    for o, bound in ((1, 1.8e-7), (2, 1.5e-7), (3, 1e-7)):
        c = ORD_CHECK[o] * fibonacci(ORD_NC[o])
        mu = _pinv(kernel_matrix(c, e[o], d), ORD_TRUNC[o]) @ (kernel_matrix(c, e[o - 1], d) @ mu)
        x = ORD_KAPPA[o] * _rotated(rng, 300)
        ref = kernel_matrix(x, src, d) @ lam
        assert np.linalg.norm(kernel_matrix(x, e[o], d) @ mu - ref) <= bound * np.linalg.norm(ref)


@pytest.mark.parametrize("d", [1, 3])
def test_local_sources_reproduce_the_field(d):
    rng = np.random.default_rng(5)
    loc, chk = LOC_EQ * fibonacci(LOC_N), LOC_CHECK * fibonacci(LOC_NC)
    match, x = _pinv(kernel_matrix(chk, loc, d), LOC_TRUNC), _rotated(rng, 400)
    for gap, bound in ((LOC_GAP, 5e-7), (LOC_GAP + 1.0, 1e-7), (2 * LOC_GAP, 3e-8)):
        src = fibonacci(100) + np.array([1.0 + gap, 0, 0]) @ np.linalg.qr(rng.standard_normal((3, 3)))[0]
        lam = rng.standard_normal((100 * d, 4))
        ref = kernel_matrix(x, src, d) @ lam
        got = kernel_matrix(x, loc, d) @ (match @ (kernel_matrix(chk, src, d) @ lam))
        assert np.linalg.norm(got - ref) <= bound * np.linalg.norm(ref)
