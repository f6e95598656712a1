"""What a program does with this framework, as cases that can be timed and checked.

Every case goes through the public entry points of ``paper_2409_04215_gb300`` on bodies of the kinds
the repository's workloads use (unit spheres, prolate spheroids, triaxial ellipsoids, suspensions of
uneven size).  A case's ``dtype`` is the program's own: "f32" stands for a simulation or a training
loop whose state and results are FP32 tensors (the entry points take them as they are; the default
path sums its pairs in FP32), "f64" for one that works in FP64.  Every output goes back to that type.

``op``: matvec, mobility, elastance, resistance, vjp (forward and backward of the differentiable
mobility), field (velocity of the last solve at points in the fluid), stress (pressure and traction
of the last solve at surface points).
"""

from __future__ import annotations

import math

import numpy as np
import torch

from mfs_inputs.workloads import batched_suspensions, ellipsoid_cluster, sphere_suspension, spheroid_cluster
from paper_2409_04215_gb300 import MFS, mobility

DEV = "cuda"


def _case(name, op, bodies, shape, count, m, n, **kw):
    c = {"op": op, "bodies": bodies, "shape": shape, "count": count, "m": m, "n": n, "nrhs": 1, "precision": 0,
         "farfield": 0, "points": 0, "dtype": "f32"}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # Two conductors, the smallest problem there is: capacitance extraction, one pair at a time.
        _case("elastance_pair", "elastance", "laplace", "sphere", 2, 600, 300, dtype="f64"),
        # A handful of spheres: one velocity evaluation of a time stepper or of a Monte-Carlo move.
        _case("mobility_few", "mobility", "stokes", "sphere", 6, 240, 120),
        # One application of the operator inside a caller's own Krylov method, 100 spheres.
        _case("matvec_100", "matvec", "stokes", "sphere", 100, 1200, 600),
        # The whole solve of the same suspension: rigid-body velocities from forces and torques.
        _case("mobility_100", "mobility", "stokes", "sphere", 100, 1200, 600),
        # Many independent suspensions of uneven size, two shapes, four right-hand sides at once.
        _case("mobility_batched", "mobility", "stokes", "mixed", 12, 600, 300, nrhs=4),
        # A training step: velocities, then gradients for the positions, the forces and the torques.
        _case("vjp_100", "vjp", "stokes", "sphere", 100, 400, 200),
        # Rotated spheroids moved rigidly: drag forces and torques, sizes that are no multiple of a tile.
        _case("resistance_40", "resistance", "stokes", "spheroid", 40, 997, 501),
        # A large cluster through the treecode, one application of the operator.
        _case("treecode_2000", "matvec", "stokes", "ellipsoid", 2000, 0, 34, farfield=1),
        # A slice through the flow of a solved suspension: velocities at points between the bodies.
        _case("field_slice", "field", "stokes", "sphere", 60, 600, 300, points=100003),
        # Surface pressure and traction of a solved suspension.
        _case("stress_surface", "stress", "stokes", "sphere", 60, 600, 300, points=72000),
        # The FP64 path, which a program takes to check its results or for tight tolerances.
        _case("matvec_fp64", "matvec", "stokes", "sphere", 24, 600, 300, precision=1, dtype="f64"),
        # The compensated path: FP32 arithmetic with results near FP64 accuracy.
        _case("matvec_compensated", "matvec", "stokes", "sphere", 60, 600, 300, precision=3, dtype="f64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)) - 0.5 / hi)))


def draw(rng):
    """One more program of the same kinds: each op over its range of body counts, point counts (odd ones
    among them), shapes, right-hand sides and precisions."""
    op = rng.choice(["elastance", "mobility", "mobility", "matvec", "matvec", "batched", "vjp", "resistance", "treecode",
                     "field", "stress"])
    n = _log(rng, 100, 600)
    m = int(n * rng.uniform(1.6, 2.2))
    shape = rng.choice(["sphere", "spheroid"])
    if op == "elastance":
        return _case("", "elastance", "laplace", shape, _log(rng, 2, 100), m, n, dtype=rng.choice(["f32", "f64"]))
    if op == "matvec":
        prec = rng.choice([0, 0, 1, 2, 3])
        top = 100 if prec in (0, 2) else 24 if prec == 1 else 60
        return _case("", "matvec", rng.choice(["stokes", "stokes", "laplace"]), shape, _log(rng, 2, top), m, n,
                     nrhs=rng.choice([1, 1, 2, 3, 4]), precision=prec, dtype="f64" if prec in (1, 3) else "f32")
    if op == "batched":
        return _case("", "mobility", "stokes", "mixed", _log(rng, 2, 12), min(m, 600), min(n, 300),
                     nrhs=rng.choice([1, 2, 4]))
    if op == "treecode":
        return _case("", "matvec", "stokes", "ellipsoid", _log(rng, 150, 2000), 0, rng.randrange(14, 35), farfield=1)
    if op in ("field", "stress"):
        return _case("", op, "stokes", shape, _log(rng, 2, 60), min(m, 600), min(n, 300),
                     points=_log(rng, 500, 100000), farfield=rng.choice([0, 0, 1]))
    if op == "vjp":
        return _case("", "vjp", "stokes", shape, _log(rng, 2, 100), min(m, 400), min(n, 200),
                     nrhs=rng.choice([1, 1, 2]))
    return _case("", op, "stokes", shape, _log(rng, 2, 60), m, n)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _workload(case, seed):
    count, m, n, nrhs = case["count"], case["m"], case["n"], case["nrhs"]
    if case["shape"] == "ellipsoid":
        wl = ellipsoid_cluster(count=count, n_v=n, seed=seed)
    elif case["shape"] == "spheroid":
        wl = spheroid_cluster(count=count, m=m, n=n, seed=seed)
    elif case["shape"] == "mixed":
        # body counts of a batch of simulations: uneven, the same for every seed (positions are not)
        wl = batched_suspensions(num_suspensions=count, p_lo=2, p_hi=64, m=m, n=n, nrhs=nrhs, seed=1000 + count)
        moved = np.random.default_rng(seed)
        jitter = 0.02 * moved.uniform(-1.0, 1.0, wl.centres.shape)  # within half the 0.1 minimum gap
        wl.centres = wl.centres + jitter
    else:
        wl = sphere_suspension(count=count, m=m, n=n, volume_fraction=0.1, seed=seed)
    wl.kind = case["bodies"]
    return wl


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _randn(g, *shape, dtype):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64).to(dtype)


def _points(case, wl, seed):
    """field: points of a slice plane through the suspension that lie outside the bodies; stress: random
    points on the unit spheres (or on the spheroids' surfaces) with normals and owners."""
    rng = np.random.default_rng(seed + 77)
    np_, cen = case["points"], wl.centres
    if case["op"] == "field":
        lo, hi = cen.min(0) - 2.0, cen.max(0) + 2.0
        out = np.zeros((0, 3))
        reach = wl.shapes[0].bounding_radius
        while len(out) < np_:
            p = rng.uniform(lo, hi, (np_, 3))
            p[:, 2] = 0.5 * (lo[2] + hi[2]) + 0.05 * rng.standard_normal(np_)
            t = torch.tensor(p, device=DEV)
            d = torch.cdist(t, torch.tensor(cen, device=DEV)).amin(1)
            out = np.concatenate([out, p[(d > reach).cpu().numpy()]])
        return out[:np_], None, None
    owner = rng.integers(0, len(cen), np_).astype(np.int32)
    a, b, c = wl.shapes[0].semi_axes
    u = rng.standard_normal((np_, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    x, nrm = u * [a, b, c], u / [a, b, c]
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    if wl.quats is not None:
        R = _rotations(wl.quats)[owner]
        x, nrm = np.einsum("kij,kj->ki", R, x), np.einsum("kij,kj->ki", R, nrm)
    return cen[owner] + x, nrm, owner


def _rotations(q):
    q = q / np.linalg.norm(q, axis=1, keepdims=True)
    w, x, y, z = q.T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _inputs(case, wl, seed):
    dt, P, nrhs = _dtype(case), wl.num_bodies, case["nrhs"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    inp = {}
    if case["op"] == "matvec":  # a Krylov vector: a smooth field on the surfaces and a little roughness
        d = 3 if case["bodies"] == "stokes" else 1
        R = np.tile(np.eye(3), (P, 1, 1)) if wl.quats is None else _rotations(wl.quats)
        x = torch.tensor(np.concatenate([wl.shapes[s].colloc @ R[k].T + wl.centres[k]
                                         for k, s in enumerate(wl.shape_id)]), device=DEV)
        # plane waves; vector ones are transverse, as a flow has no net flux through a body's surface
        k, phase, a = (_randn(g, nrhs, 3, dtype=x.dtype) for _ in range(3))
        a = torch.linalg.cross(k, a) if d == 3 else a[:, :1]
        rough = 1e-6 * _randn(g, nrhs, len(x), d, dtype=x.dtype)
        inp["gamma"] = (torch.sin(x @ k.T + 3.0 * phase[:, 0]).T[:, :, None] * a[:, None, :] + rough).to(dt)
    elif case["op"] == "elastance":
        inp["q"] = _randn(g, nrhs, P, dtype=dt)
    else:
        inp["f"], inp["t"] = _randn(g, nrhs, P, 3, dtype=dt), _randn(g, nrhs, P, 3, dtype=dt)
    if case["op"] == "vjp":
        inp["c"] = torch.tensor(wl.centres, device=DEV).to(dt)
        inp["gu"], inp["gw"] = _randn(g, nrhs, P, 3, dtype=dt), _randn(g, nrhs, P, 3, dtype=dt)
    if case["points"]:
        p, nrm, own = _points(case, wl, seed)
        inp["points"] = torch.tensor(p, device=DEV).to(dt)
        inp["normals"] = None if nrm is None else torch.tensor(nrm, device=DEV).to(dt)
        inp["owner"] = None if own is None else torch.tensor(own, device=DEV)
    return inp


def prepare(case, seed):
    wl = _workload(case, seed)
    ctx = MFS.from_workload(wl, precision=case["precision"], farfield=case["farfield"], max_rhs=case["nrhs"])
    inp = _inputs(case, wl, seed)
    if case["op"] in ("field", "stress"):  # the program has solved; it now looks at the flow
        ctx.solve_mobility(inp["f"], inp["t"])
    if case["op"] == "resistance":  # the handle's bare-block factors, built once
        ctx.dirichlet_apply(torch.zeros((1, ctx.sum_M, 3), dtype=torch.float64, device=DEV))
    if case["op"] == "vjp":
        for k in ("c", "f", "t"):
            inp[k].requires_grad_(True)
    return {"case": dict(case), "ctx": ctx, **inp}


def run(state):
    case, ctx = state["case"], state["ctx"]
    op, dt = case["op"], _dtype(case)
    if op == "matvec":
        return ctx.matvec(state["gamma"]).to(dt)
    if op == "elastance":
        return ctx.solve_elastance(state["q"])[0].to(dt)
    if op == "mobility":
        u, w, _ = ctx.solve_mobility(state["f"], state["t"])
        return u.to(dt), w.to(dt)
    if op == "resistance":
        f, t, _ = ctx.solve_resistance(state["f"], state["t"])
        return f.to(dt), t.to(dt)
    if op == "vjp":
        u, w = mobility(ctx, state["c"], state["f"], state["t"])
        u, w = u.to(dt), w.to(dt)
        gc, gf, gt = torch.autograd.grad((u, w), (state["c"], state["f"], state["t"]), (state["gu"], state["gw"]))
        return u.detach(), w.detach(), gc, gf, gt
    if op == "field":
        return ctx.evaluate(state["points"], state["owner"], nrhs=case["nrhs"]).to(dt)
    p, t = ctx.evaluate_stress(state["points"], state["normals"], state["owner"], nrhs=case["nrhs"])
    return p.to(dt), t.to(dt)


# ---------------------------------------------------------------------------
# Work that a pass cannot do without
# ---------------------------------------------------------------------------
_ITERS = {"matvec": 1, "elastance": 13, "mobility": 22, "resistance": 40, "vjp": 50, "field": 0, "stress": 0}


def _counts(case):
    """Bodies per suspension, and points per body."""
    if case["shape"] == "mixed":
        off = batched_suspensions(num_suspensions=case["count"], p_lo=2, p_hi=64, m=8, n=4, nrhs=1,
                                  seed=1000 + case["count"]).body_offsets
        per = np.diff(off)
    else:
        per = np.array([case["count"]])
    if case["shape"] == "ellipsoid":  # N_v rings: the paper's totals
        nv = case["n"]
        mv = 1.15 * nv
        return per, int(17 + 3.9 * mv + 0.44 * mv * mv), int(17 + 3.9 * nv + 0.44 * nv * nv)
    return per, case["m"], case["n"]


def _pairs(case):
    per, m, n = _counts(case)
    if case["points"]:
        return float(case["points"]) * case["count"] * n
    direct = float((per * (per - 1)).sum()) * m * n
    if case["farfield"]:  # the bodies around each body, the rest through about 200 points a body
        direct = min(direct, float(per.sum()) * (26.0 * m * n + 200.0 * (m + n)))
    return direct


def work(case):
    per, m, n = _counts(case)
    d, nrhs = (3 if case["bodies"] == "stokes" else 1), case["nrhs"]
    P, its = float(per.sum()), _ITERS[case["op"]]
    item = 8 if case["dtype"] == "f64" else 4
    if case["points"]:
        per_pair = 22.0 if case["op"] == "stress" else 28.0
        moved = case["points"] * (3 + (4 if case["op"] == "stress" else 3)) * item
        return {"bytes": float(moved + P * (m + n) * 12), "flops": _pairs(case) * per_pair}
    per_pair = 10.0 + 18.0 * nrhs if d == 3 else 9.0 + 2.0 * nrhs
    applies = max(its, 1)
    apply_flops = 2.0 * P * nrhs * (d * m * d * n + d * n * d * n)
    factor = 4.0 * (d * m * d * n + d * n * d * n) * (2 if case["shape"] == "mixed" else 1)
    vectors = P * m * d * nrhs * (item if case["op"] == "matvec" else 8) * 2
    return {"bytes": applies * (factor + vectors + P * (m + n) * 12.0),
            "flops": applies * (_pairs(case) * per_pair + apply_flops)}


# ---------------------------------------------------------------------------
# The same results in FP64 by plain torch: dense one-body factors (QR), direct sums, GMRES
# ---------------------------------------------------------------------------
class _Plain:
    def __init__(self, wl, centres, bare=False, mu=1.0):
        f = dict(dtype=torch.float64, device=DEV)
        self.d = 3 if wl.kind == "stokes" else 1
        self.mu, self.P = mu, wl.num_bodies
        self.cen = centres
        R = np.tile(np.eye(3), (self.P, 1, 1)) if wl.quats is None else _rotations(wl.quats)
        self.R = torch.tensor(R, **f)
        mk, nk = wl.counts()
        self.to, self.so = np.concatenate([[0], np.cumsum(mk)]), np.concatenate([[0], np.cumsum(nk)])
        self.sid, self.off = wl.shape_id, wl.body_offsets
        self.xl = torch.cat([torch.tensor(wl.shapes[s].colloc, **f) @ self.R[k].T for k, s in enumerate(self.sid)])
        self.yl = torch.cat([torch.tensor(wl.shapes[s].proxy, **f) @ self.R[k].T for k, s in enumerate(self.sid)])
        body = lambda off: torch.repeat_interleave(torch.arange(self.P, device=DEV),  # noqa: E731
                                                   torch.tensor(np.diff(off), device=DEV))
        self.tb, self.sb = body(self.to), body(self.so)
        self.x, self.y = self.xl + self.cen[self.tb], self.yl + self.cen[self.sb]
        self.fac = {}
        for s in sorted(set(int(v) for v in self.sid)):
            X, Y = torch.tensor(wl.shapes[s].colloc, **f), torch.tensor(wl.shapes[s].proxy, **f)
            S, L = self._block(X, Y), None
            if not bare and self.d == 3:
                KN, KM = self._k(Y), self._k(X)
                G = torch.linalg.inv(KN.T @ KN)
                L = (KN, G)
                S = S - ((S @ KN) @ G) @ KN.T + KM @ KN.T
            elif not bare:
                L = "mean"
                S = S - S.mean(1, keepdim=True) + 1.0 / len(Y)
            Q, Rr = torch.linalg.qr(S)
            self.fac[s] = (Q, Rr, L)

    @staticmethod
    def _k(p):
        K = torch.zeros((len(p), 3, 6), dtype=p.dtype, device=p.device)
        K[:, 0, 0] = K[:, 1, 1] = K[:, 2, 2] = 1.0
        K[:, 0, 4], K[:, 0, 5] = p[:, 2], -p[:, 1]
        K[:, 1, 3], K[:, 1, 5] = -p[:, 2], p[:, 0]
        K[:, 2, 3], K[:, 2, 4] = p[:, 1], -p[:, 0]
        return K.reshape(-1, 6)

    def _block(self, X, Y):
        r = X[:, None, :] - Y[None, :, :]
        ri = 1.0 / r.norm(dim=2)
        if self.d == 1:
            return ri / (4 * math.pi)
        G = ri[..., None, None] * torch.eye(3, dtype=X.dtype, device=X.device) + \
            r[..., :, None] * r[..., None, :] * (ri ** 3)[..., None, None]
        return G.permute(0, 2, 1, 3).reshape(3 * len(X), 3 * len(Y)) / (8 * math.pi * self.mu)

    def _frame(self, v, k, back):
        return v if self.d == 1 else (v @ self.R[k].T if back else v @ self.R[k])

    def _project(self, lam, L):
        if L is None:
            return lam
        if L == "mean":
            return lam - lam.mean(0, keepdim=True)
        return lam - L[0] @ (L[1] @ (L[0].T @ lam))

    def _columns(self, v, off, ks):
        return torch.stack([self._frame(v[off[k]:off[k + 1]], k, False).reshape(-1) for k in ks], 1)

    def _spread(self, cols, off, ks, out):
        for i, k in enumerate(ks):
            out[off[k]:off[k + 1]] = self._frame(cols[:, i].reshape(-1, self.d), k, True)

    def apply(self, g, project):
        """S^+ g per body, [sum_M, d] -> [sum_N, d], with the projection (I - L) when asked for."""
        out = torch.zeros((int(self.so[-1]), self.d), dtype=torch.float64, device=DEV)
        for s, (Q, R, L) in self.fac.items():
            ks = [k for k in range(self.P) if self.sid[k] == s]
            lam = torch.linalg.solve_triangular(R, Q.T @ self._columns(g, self.to, ks), upper=True)
            self._spread(self._project(lam, L) if project else lam, self.so, ks, out)
        return out

    def apply_t(self, z, project):
        """The transpose of apply, [sum_N, d] -> [sum_M, d]."""
        out = torch.zeros((int(self.to[-1]), self.d), dtype=torch.float64, device=DEV)
        for s, (Q, R, L) in self.fac.items():
            ks = [k for k in range(self.P) if self.sid[k] == s]
            c = self._columns(z, self.so, ks)
            c = self._project(c, L) if project else c  # I - L is symmetric
            self._spread(Q @ torch.linalg.solve_triangular(R.T, c, upper=False), self.to, ks, out)
        return out

    def _pieces(self, toff, soff):
        """(target range, source range, bodies) over all suspensions, about 2e7 pairs each."""
        for b0, b1 in zip(self.off[:-1], self.off[1:]):
            t0, t1, s0, s1 = int(toff[b0]), int(toff[b1]), int(soff[b0]), int(soff[b1])
            step = max(1, int(2e7) // (s1 - s0))
            for a in range(t0, t1, step):
                yield a, min(a + step, t1), s0, s1

    def pair(self, lam, include_self, swap=False, points=None, pbody=None):
        """sum_j G(x_i - y_j) lam_j over the suspension's sources off the target's body (or all)."""
        x, y, tb, sb, toff, soff = ((self.y, self.x, self.sb, self.tb, self.so, self.to) if swap else
                                    (self.x, self.y, self.tb, self.sb, self.to, self.so))
        if points is not None:
            step = max(1, int(2e7) // len(y))
            pieces = [(a, min(a + step, len(points)), 0, len(y)) for a in range(0, len(points), step)]
            x = points
        else:
            pieces = self._pieces(toff, soff)
        u = torch.zeros((len(x), self.d), dtype=torch.float64, device=DEV)
        for a, b, s0, s1 in pieces:
            dx, dy, dz = (x[a:b, i, None] - y[None, s0:s1, i] for i in range(3))
            ri = torch.rsqrt(dx * dx + dy * dy + dz * dz)
            if not include_self:
                ri = ri * (tb[a:b, None] != sb[None, s0:s1])
            l = lam[s0:s1]
            if self.d == 1:
                u[a:b] = ri @ l / (4 * math.pi)
                continue
            s = (dx * l[:, 0] + dy * l[:, 1] + dz * l[:, 2]) * ri ** 3
            u[a:b] = (ri @ l + torch.stack([(s * dx).sum(1), (s * dy).sum(1), (s * dz).sum(1)], 1)) / \
                (8 * math.pi * self.mu)
        return u

    def matvec(self, g):
        return g + self.pair(self.apply(g, True), False)

    def matvec_t(self, w):
        return w + self.apply_t(self.pair(w, False, swap=True), True)

    def gmres(self, op, b, tol=1e-11, most=120):
        V, H = [b.reshape(-1) / b.norm()], np.zeros((most + 1, most))
        for j in range(most):
            w = op(V[j].reshape(b.shape)).reshape(-1)
            for _ in range(2):
                for i, v in enumerate(V):
                    h = float(v @ w)
                    H[i, j] += h
                    w = w - h * v
            H[j + 1, j] = float(w.norm())
            V.append(w / H[j + 1, j])
            e = np.zeros(j + 2)
            e[0] = float(b.norm())
            yv, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
            if np.linalg.norm(H[:j + 2, :j + 1] @ yv - e) <= tol * e[0]:
                break
        return sum(c * v for c, v in zip(yv.tolist(), V)).reshape(b.shape)

    def expand(self, f, t, unit=False):
        """K_N (K_N^T K_N)^-1 [f; t] per body (or K_N [f; t])."""
        out = torch.zeros((int(self.so[-1]), 3), dtype=torch.float64, device=DEV)
        for k in range(self.P):
            K = self._k(self.yl[self.so[k]:self.so[k + 1]])
            v = torch.cat([f[k], t[k]])
            v = v if unit else torch.linalg.solve(K.T @ K, v)
            out[self.so[k]:self.so[k + 1]] = (K @ v).reshape(-1, 3)
        return out

    def gather(self, lam):
        """K_N^T lam per body: (P, 3) and (P, 3)."""
        f = torch.zeros((self.P, 3), dtype=torch.float64, device=DEV).index_add_(0, self.sb, lam)
        t = torch.zeros_like(f).index_add_(0, self.sb, torch.linalg.cross(self.yl, lam))
        return f, t

    def mobility(self, f, t):
        lam0 = self.expand(f, t)
        gam = self.gmres(self.matvec, -self.pair(lam0, True))
        u, w = self.gather(self.apply(gam, False))
        return -u, -w, gam, self.apply(gam, True) + lam0

    def vjp(self, beta, gu, gw):
        """Gradients of (gu, u) + (gw, w) for the centres, the forces and the torques; beta: total strengths."""
        w = self.gmres(self.matvec_t, -self.apply_t(self.expand(gu, gw, unit=True), False))
        gc = torch.zeros((self.P, 3), dtype=torch.float64, device=DEV)
        for a, b, s0, s1 in self._pieces(self.to, self.so):
            d = [self.x[a:b, i, None] - self.y[None, s0:s1, i] for i in range(3)]
            ri = torch.rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
            ri = ri * (self.tb[a:b, None] != self.sb[None, s0:s1])
            wi, m = w[a:b], beta[s0:s1]
            wm = wi @ m.T
            wr = sum(wi[:, i, None] * d[i] for i in range(3))
            rm = sum(m[None, :, i] * d[i] for i in range(3))
            q, ri3 = -(wm + 3.0 * wr * rm * ri * ri), ri ** 3
            for i in range(3):
                g = (d[i] * q + wi[:, i, None] * rm + m[None, :, i] * wr) * ri3 / (8 * math.pi * self.mu)
                gc[:, i].index_add_(0, self.tb[a:b], -g.sum(1))
                gc[:, i].index_add_(0, self.sb[s0:s1], g.sum(0))
        zf, zt = self.gather(self.pair(w, True, swap=True))
        gf, gt = torch.zeros_like(gc), torch.zeros_like(gc)
        for k in range(self.P):
            K = self._k(self.yl[self.so[k]:self.so[k + 1]])
            v = -torch.linalg.solve(K.T @ K, torch.cat([zf[k], zt[k]]))
            gf[k], gt[k] = v[:3], v[3:]
        return gc, gf, gt


def exact(case, seed):
    its = max(_ITERS[case["op"]], 25 if case["op"] in ("field", "stress") else 1)
    per, m, n = _counts(case)
    direct = float((per ** 2).sum()) * m * n
    if direct * its * case["nrhs"] + _pairs(case) > 5e10 or (case["op"] == "matvec" and direct > 1e10):
        return None
    wl = _workload(case, seed)
    inp = _inputs(case, wl, seed)
    cen = torch.tensor(wl.centres, dtype=torch.float64, device=DEV) if case["op"] != "vjp" else inp["c"].double()
    p = _Plain(wl, cen, bare=case["op"] == "resistance")
    every = lambda f: [torch.stack(v) for v in zip(*[f(h) for h in range(case["nrhs"])])]  # noqa: E731
    if case["op"] == "matvec":
        y = torch.stack([p.matvec(g) for g in inp["gamma"].double()])
        return y
    if case["op"] == "elastance":
        q, out = inp["q"].double(), []
        count = torch.tensor(np.diff(p.so), device=DEV)
        for h in range(case["nrhs"]):
            gam = p.gmres(p.matvec, -p.pair((q[h] / count)[p.sb][:, None], True))
            a = p.apply(gam, False)[:, 0]
            out.append(-torch.zeros_like(q[h]).index_add_(0, p.sb, a) / count)
        return torch.stack(out)
    f, t = inp["f"].double(), inp["t"].double()
    if case["op"] == "resistance":
        def drag(h):
            b = f[h][p.tb] + torch.linalg.cross(t[h][p.tb], p.xl)
            return p.gather(p.apply(p.gmres(p.matvec, b), False))
        return tuple(every(drag))
    if case["op"] == "mobility":
        return tuple(every(lambda h: p.mobility(f[h], t[h])[:2]))
    if case["op"] == "vjp":
        def both(h):
            u, w, _, beta = p.mobility(f[h], t[h])
            return (u, w) + p.vjp(beta, inp["gu"][h].double(), inp["gw"][h].double())
        u, w, gc, gf, gt = every(both)
        return u, w, gc.sum(0), gf, gt
    beta = torch.stack([p.mobility(f[h], t[h])[3] for h in range(case["nrhs"])])
    pts = inp["points"].double()
    if case["op"] == "field":
        return torch.stack([p.pair(b, True, points=pts) for b in beta])
    nrm, pres, trac = inp["normals"].double(), [], []
    for b in beta:
        pr, tr = torch.zeros(len(pts), dtype=torch.float64, device=DEV), torch.zeros_like(pts)
        step = max(1, int(2e7) // len(p.y))
        for a in range(0, len(pts), step):
            e = min(a + step, len(pts))
            d = [pts[a:e, i, None] - p.y[None, :, i] for i in range(3)]
            ri = torch.rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
            rl = sum(d[i] * b[None, :, i] for i in range(3)) * ri ** 3
            pr[a:e] = rl.sum(1) / (4 * math.pi)
            s = rl * sum(d[i] * nrm[a:e, i, None] for i in range(3)) * ri * ri
            tr[a:e] = torch.stack([(s * d[i]).sum(1) for i in range(3)], 1) * (-3.0 / (4 * math.pi))
        pres.append(pr)
        trac.append(tr)
    return torch.stack(pres), torch.stack(trac)
