"""The work that users of this framework have it do, as measurable cases.

Every case goes through the public Python entry points (``dmn.DMN.update``,
``update_host``, the ``torch.autograd`` bindings, the finite-element operator and
its CG solver) with inputs of the kind these paths meet: trees of the paper's
depth with fiber and J2 matrix, points in the middle of a load path (a converged
plastic state and the next strain increment), orientation frames all over the
sphere, sizes from one element's Gauss points to a large mesh.

``exact`` restates the method in plain torch (FP64): level-by-level evaluation and
condensation of the laminate tree, Newton's method to well below the library's
criterion, gradients by the implicit function theorem with torch's autograd, an
assembled-by-element CG for the FE solve.  The same code makes the states that
the load paths start from, so that inputs do not depend on the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2103_08253_gb300 import autograd as ag
from paper_2103_08253_gb300 import dmn, fe
from paper_2103_08253_gb300 import workloads as W

F64 = torch.float64
R2 = math.sqrt(2.0)
POOL = 512          # distinct material states per case; the points of a case draw from them
FOREST = (5, 6, 7, 8)
MATRICES = {"linear": W.MATRIX, "explin": W.MATRIX_EXPLIN}
ELASTIC_MATRIX = W.Phase(kind=0, E=3000.0, nu=0.35)


# --------------------------------------------------------------------------------------------
# Cases

def _update(name, n, **kw):
    c = dict(name=name, kind="update", K=8, M=3, n=n, precision="f64", matrix="linear", tree="full", load="ramp",
             line_search=False)
    c.update(kw)
    return c


def listed():
    return [
        # one hexahedron's eight Gauss points: the material routine called element by element
        _update("update-f64-element", 8),
        # a small mesh or a sub-domain's batch, ragged size
        _update("update-f64-small", 4099),
        # a structural model's batch in the headline form: depth 8, FP64, one macro increment
        _update("update-f64-large", 200003),
        # a trained network (a third of the leaf weights zero) with the paper's polyamide law
        _update("update-f64-trained", 20001, tree="trained", matrix="explin"),
        # points of four depths in one call, half of them cycling through plasticity and half in the
        # elastic range, with the line search that FE computations switch on
        _update("update-f64-forest", 30011, tree="forest", load="cyclic", line_search=True),
        # the mixed form (FP64 stress and tangent from a final sweep), small and large
        _update("update-mixed-small", 4099, precision="mixed"),
        _update("update-mixed-large", 100003, precision="mixed"),
        # the mixed form for solvers that round the tangent to FP32 anyway
        _update("update-f32tangent-large", 262144, precision="mixed-f32-tangent"),
        # an FE code that holds its arrays in host memory
        _update("host-f64", 12289, kind="host"),
        # offline training, plastic samples: stresses of one increment, gradients in p, q, w and strain
        dict(name="grad-stress", kind="grad", K=8, n=4096, precision="mixed-f32-tangent", tree="full", line_search=True),
        # offline training, stiffness samples: effective stiffnesses and their gradients
        dict(name="grad-stiffness", kind="stiffness", K=8, n=4096, precision="mixed", tree="full"),
        # the FE side of one macro Newton iteration: strains, forces, diagonal, linear solve
        dict(name="fe-solve", kind="fe", n_t=24, n_r=24, n_z=4, f32=True, rtol=1e-6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["update"] * 6 + ["host", "grad", "stiffness", "fe"])
    if kind == "fe":
        f32 = rng.random() < 0.5
        return dict(kind="fe", n_t=2 * _log_int(rng, 2, 16), n_r=_log_int(rng, 3, 40), n_z=_log_int(rng, 1, 6),
                    f32=f32, rtol=1e-6 if f32 else 1e-8)
    K = rng.choice([4, 5, 6, 7, 8, 8, 8])
    tree = rng.choice(["full", "full", "trained"])
    if kind in ("grad", "stiffness"):
        return dict(kind=kind, K=K, n=_log_int(rng, 16, 8192), tree=tree, line_search=kind == "grad",
                    precision=rng.choice(["f64", "mixed-f32-tangent"] if kind == "grad" else ["f64", "mixed"]))
    if kind == "update" and rng.random() < 0.15:
        tree = "forest"
    most = {"host": 20000}.get(kind, 200000)
    line_search = rng.random() < 0.25
    return dict(kind=kind, K=8 if tree == "forest" else K, M=3 if tree != "full" else rng.choice([3, 3, 4, 6]),
                n=_log_int(rng, 1, most // 4 if line_search else most),
                precision=rng.choice(["f64", "f64", "f64", "mixed", "mixed-f32-tangent"]),
                matrix=rng.choice(["linear", "linear", "explin"]), tree=tree,
                load=rng.choice(["ramp", "ramp", "cyclic"]) if line_search else "ramp", line_search=line_search)


# --------------------------------------------------------------------------------------------
# The method in plain torch

def _rotation(Q):
    """Mandel rotation R [n, 6, 6] of frames Q [n, 9]: sigma_global = R sigma_local."""
    Q = Q.reshape(-1, 3, 3)
    i, j = [0, 1, 2, 1, 0, 0], [0, 1, 2, 2, 2, 1]
    w = torch.tensor([1.0, 1.0, 1.0, R2, R2, R2], dtype=F64, device=Q.device)
    A = Q[:, i][:, :, i] * Q[:, j][:, :, j] + Q[:, i][:, :, j] * Q[:, j][:, :, i]
    return A * (0.5 * w[:, None] * w[None, :])


def _shape(lam, M):
    l1, l2 = lam[:, 0], lam[:, 1]
    a, b, c = l1 - l2, 3.0 * (1.0 - l1 - l2), 2.0 * l1 + 4.0 * l2 - 2.0
    if M == 3:
        return torch.stack([a, b, c], 1)
    if M == 4:
        t = a * b * c
        return torch.stack([a - 9 * t, b - 9 * t, c - 9 * t, 27 * t], 1)
    return torch.stack([a * (2 * a - 1), b * (2 * b - 1), c * (2 * c - 1), 4 * a * b, 4 * a * c, 4 * b * c], 1)


def _N(v):
    """N(n) [..., 6, 3] with N(n) a = sym(a (x) n) in Mandel form."""
    x, y, z = v.unbind(-1)
    o = torch.zeros_like(x)
    s = 1.0 / R2
    return torch.stack([x, o, o, o, y, o, o, o, z, o, s * z, s * y, s * z, o, s * x, s * y, s * x, o],
                       -1).reshape(*v.shape[:-1], 6, 3)


def _mv(A, x):
    return (A @ x.unsqueeze(-1)).squeeze(-1)


def _law(ph, e, z):
    """Phase law: stress, tangent (lambda, mu, c, m: lam 1(x)1 + 2 mu I - c m(x)m) and the new state."""
    K, G = ph.E / (3 * (1 - 2 * ph.nu)), ph.E / (2 * (1 + ph.nu))
    one = torch.tensor([1.0, 1.0, 1.0, 0.0, 0.0, 0.0], dtype=F64, device=e.device)
    tr = e[..., :3].sum(-1)
    if ph.kind == 0:
        lam = torch.full_like(tr, K - 2 * G / 3)
        return 2 * G * e + (lam * tr)[..., None] * one, (lam, torch.full_like(tr, G), None, None), z
    ep = torch.stack([z[..., 1], z[..., 2], -z[..., 1] - z[..., 2], z[..., 3], z[..., 4], z[..., 5]], -1)
    xi = e - (tr / 3)[..., None] * one - ep
    nx = xi.norm(dim=-1).clamp_min(1e-150)
    ds = ph.sigma_inf - ph.sigma0 if ph.kind == 2 else 0.0
    rate = (ph.k0 - ph.H) / ds if ph.kind == 2 else 0.0
    s23 = math.sqrt(2.0 / 3.0)

    def sy(a):
        return ph.sigma0 + ph.H * a + (ds * -torch.expm1(-rate * a) if ds else 0.0)

    def slope(a):
        return ph.H + (rate * ds * torch.exp(-rate * a) if ds else torch.zeros_like(a))

    f = 2 * G * nx - s23 * sy(z[..., 0])
    plastic = f > 0
    dg = torch.zeros_like(f)
    for _ in range(25 if ds else 1):
        a = z[..., 0] + s23 * dg
        dg = dg + (2 * G * nx - 2 * G * dg - s23 * sy(a)) / (2 * G + slope(a) * (2.0 / 3.0))
    dg = torch.where(plastic, dg, torch.zeros_like(dg))
    a1 = z[..., 0] + s23 * dg
    k2 = dg / nx
    mu = G * (1 - k2)
    c = torch.where(plastic, 2 * G * (1 / (1 + slope(a1) / (3 * G)) - k2), torch.zeros_like(k2))
    sig = (2 * mu)[..., None] * xi + (K * tr)[..., None] * one
    dp = k2[..., None] * xi
    zn = torch.cat([a1[..., None], z[..., 1:3] + dp[..., :2], z[..., 3:] + dp[..., 3:]], -1)
    return sig, (K - 2 * mu / 3, mu, c, xi / nx[..., None]), zn


def _leaf_tangent(D):
    lam, mu, c, m = D
    one = torch.tensor([1.0, 1.0, 1.0, 0.0, 0.0, 0.0], dtype=F64, device=mu.device)
    C = lam[..., None, None] * (one[:, None] * one) + (2 * mu)[..., None, None] * torch.eye(6, dtype=F64, device=mu.device)
    return C if c is None else C - c[..., None, None] * (m[..., :, None] * m[..., None, :])


def _inv3(A):
    a, b, c = A[..., 0, 0], A[..., 0, 1], A[..., 0, 2]
    d, e, f = A[..., 1, 1], A[..., 1, 2], A[..., 2, 2]
    i00, i01, i02 = d * f - e * e, c * e - b * f, b * e - c * d
    i11, i12, i22 = a * f - c * c, b * c - a * e, a * d - b * b
    det = a * i00 + b * i01 + c * i02
    return torch.stack([i00, i01, i02, i01, i11, i12, i02, i12, i22], -1).reshape(A.shape) / det[..., None, None]


class _Net:
    """A DMN in heap order (root first).  Leaves of weight zero keep their place with fraction zero and
    take no part; `kept` marks the laminates that carry a jump, `slots` the leaves that carry a state."""

    def __init__(self, tree, dev, p=None, q=None, w=None):
        K = self.K = tree.K
        self.M, self.phases = tree.M, tree.phases
        self.N, self.L = (1 << K) - 1, 1 << K
        t = lambda x: torch.as_tensor(np.asarray(x), dtype=F64, device=dev)  # noqa: E731
        # paper order: level K first, the root last
        self.paper = torch.tensor([(1 << K) - (1 << k) + i for k in range(1, K + 1) for i in range(1 << (k - 1))],
                                  device=dev)
        p, q, w = (t(x) if y is None else y for x, y in ((tree.p, p), (tree.q, q), (tree.w, w)))
        self.p, self.q = p[self.paper], q[self.paper]
        levels = [w / w.sum()]
        for _ in range(K):
            levels.insert(0, levels[0].reshape(-1, 2).sum(1))
        self.wl = levels[-1]
        self.W = torch.cat(levels[:-1])
        left = torch.cat([x[0::2] for x in levels[1:]])
        safe = torch.where(self.W > 0, self.W, torch.ones_like(self.W))
        self.c1 = torch.where(self.W > 0, left / safe, torch.full_like(safe, 0.5))
        right = torch.cat([x[1::2] for x in levels[1:]])
        self.kept = (left > 0) & (right > 0)
        self.c2 = torch.where(self.kept, 1 - self.c1, (right > 0).to(F64))
        alive = self.wl > 0
        inel = torch.tensor([ph.kind != 0 for ph in self.phases], device=dev).repeat(self.L // 2)
        self.slots = (alive & inel).nonzero().flatten()
        order = torch.argsort(self.paper)          # heap positions in the paper's order
        self.jumps = order[self.kept[order]]
        self.S = 6 * len(self.slots) + 3 * len(self.jumps)
        self.n_lam = max(1, len(self.jumps))

    def normals(self, lam):
        phi = _shape(lam, self.M)
        al, be = phi @ self.p.T, phi @ self.q.T
        return torch.stack([al.sin() * be.cos(), al.sin() * be.sin(), al.cos()], -1)

    def unpack(self, state):
        """state [S, n] -> leaf states [n, L, 6], jumps [n, N, 3]."""
        n = state.shape[1]
        z = torch.zeros((n, self.L, 6), dtype=F64, device=state.device)
        a = torch.zeros((n, self.N, 3), dtype=F64, device=state.device)
        nz = 6 * len(self.slots)
        z[:, self.slots] = state[:nz].T.reshape(n, -1, 6)
        a[:, self.jumps] = state[nz:].T.reshape(n, -1, 3)
        return z, a

    def pack(self, z, a):
        n = z.shape[0]
        return torch.cat([z[:, self.slots].reshape(n, -1), a[:, self.jumps].reshape(n, -1)], 1).T.contiguous()

    def level(self, k):
        return slice((1 << k) - 1, (2 << k) - 1)

    def strains(self, Nm, E, a):
        """Strains of the leaves [n, L, 6] for macro strain E [n, 6] and jumps a [n, N, 3]."""
        e = E[:, None]
        for k in range(self.K):
            s = self.level(k)
            Na = _mv(Nm[:, s], a[:, s])
            e = torch.stack([e - self.c2[s, None] * Na, e + self.c1[s, None] * Na], 2).reshape(len(E), -1, 6)
        return e

    def leaves(self, e, z):
        """Stresses, tangents and new states of all leaves."""
        r = [_law(ph, e[:, f::2], z[:, f::2]) for f, ph in enumerate(self.phases)]
        mix = lambda x, y: torch.stack([x, y], 2).flatten(1, 2)  # noqa: E731
        return mix(r[0][0], r[1][0]), (r[0][1], r[1][1]), mix(r[0][2], r[1][2])

    def average(self, Nm, x):
        """Weighted averages of leaf values x [n, L, 6] up the tree: the root's, and every laminate's
        A^T W x [n, N, 3]."""
        R = []
        for k in range(self.K - 1, -1, -1):
            s = self.level(k)
            xl, xr = x[:, 0::2], x[:, 1::2]
            sc = (self.W * self.c1 * self.c2)[s, None]
            R.insert(0, sc * _mv(Nm[:, s].transpose(-1, -2), xr - xl))
            x = self.c1[s, None] * xl + self.c2[s, None] * xr
        return x[:, 0], torch.cat(R, 1)

    def condense(self, Nm, C, s=None):
        """Leaf tangents C [n, L, 6, 6] (and stresses s) to the root's; with s also g, H of every
        laminate, da = g + H d_eps."""
        g, H = [], []
        for k in range(self.K - 1, -1, -1):
            q = self.level(k)
            c1, c2 = self.c1[q, None, None], self.c2[q, None, None]
            c12 = c1 * c2
            CL, CR, n = C[:, 0::2], C[:, 1::2], Nm[:, q]
            B = (CR - CL) @ n
            Kn = n.transpose(-1, -2) @ ((c2 * CL + c1 * CR) @ n)
            Hk = -_inv3(Kn) @ B.transpose(-1, -2)
            C = c1 * CL + c2 * CR + c12 * (B @ Hk)
            if s is not None:
                sl, sr = s[:, 0::2], s[:, 1::2]
                gk = -_mv(_inv3(Kn), _mv(n.transpose(-1, -2), sr - sl))
                s = c1[..., 0] * sl + c2[..., 0] * sr + c12[..., 0] * _mv(B, gk)
                H.insert(0, Hk * self.kept[q, None, None])
                g.insert(0, gk * self.kept[q, None])
        return C[:, 0], (None if s is None else torch.cat(g, 1)), (None if s is None else torch.cat(H, 1))

    def descend(self, Nm, g, H, dE):
        """da [n, N, 3] of the affine map da = g + H d_eps for the macro perturbation dE [n, 6]."""
        de, da = dE[:, None], []
        for k in range(self.K):
            s = self.level(k)
            d = _mv(H[:, s], de) + (0.0 if g is None else g[:, s])
            Nd = _mv(Nm[:, s], d)
            de = torch.stack([de - self.c2[s, None] * Nd, de + self.c1[s, None] * Nd], 2).reshape(len(dE), -1, 6)
            da.append(d)
        return torch.cat(da, 1)

    def solve(self, lam, E, z, a, tol=3e-15, most=60):
        """Newton's method with backtracking: (stress, tangent, new leaf states, jumps, H) in the local frame."""
        Nm = _N(self.normals(lam))
        n = len(E)
        step = torch.ones(n, dtype=F64, device=E.device)
        best = torch.full((n,), math.inf, dtype=F64, device=E.device)
        halved = torch.zeros(n, dtype=torch.int64, device=E.device)
        kept, da, x = None, torch.zeros_like(a), a
        for it in range(most):
            sig, D, zn = self.leaves(self.strains(Nm, E, x), z)
            C = torch.stack([_leaf_tangent(D[0]), _leaf_tangent(D[1])], 2).flatten(1, 2)
            sb, R = self.average(Nm, sig)
            Cb, g, H = self.condense(Nm, C, sig)
            rn = R.flatten(1).norm(dim=1) / (self.n_lam * sb.norm(dim=1)).clamp_min(1e-300)
            now = (sb, Cb, zn, x, H, g)
            better = rn < best
            if kept is None:
                kept, better = now, torch.ones_like(better)
            else:
                kept = tuple(torch.where(better.reshape(-1, *[1] * (u.dim() - 1)), u, v) for u, v in zip(now, kept))
            best = torch.where(better, rn, best)
            halved = torch.where(better, 0, halved + 1)
            step = torch.where(better, 1.0, 0.5 * step)
            if bool(((best <= tol) | (halved > 6)).all()):
                break
            da = self.descend(Nm, kept[5], kept[4], torch.zeros_like(E))
            x = kept[3] + step[:, None, None] * da
        return kept[:5]


def _chunks(n, K):
    size = max(256, (1 << 19) >> K)
    return [slice(i, min(n, i + size)) for i in range(0, n, size)]


# --------------------------------------------------------------------------------------------
# Inputs

def _tree(case, seed, K=None):
    K = case["K"] if K is None else K
    phases = (W.FIBER, MATRICES[case.get("matrix", "linear")])
    if case["kind"] == "stiffness":
        phases = (W.FIBER, ELASTIC_MATRIX)
    if case["tree"] == "trained":
        # which weights are zero is the depth's own (it sets the state's size); the rest is the seed's
        t = W.tree_d10_fit(K, seed=seed, phases=phases)
        t.w = np.where(W.tree_with_zero_weights(K, seed=K, zero_fraction=0.3).w > 0.0, t.w, 0.0)
        return t
    M = case.get("M", 3)
    return W.tree_d10_fit(K, seed=seed, phases=phases) if M == 3 else W.tree_nodal_angles(K, M, seed=seed, phases=phases)


def _trees(case, seed):
    if case["tree"] == "forest":
        return [_tree(case, seed + 31 * k, K) for k, K in enumerate(FOREST)]
    return [_tree(case, seed)]


def _haar(n, gen, dev):
    x = torch.randn((n, 4), generator=gen, dtype=F64, device=dev)
    a, b, c, d = (x / x.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - a * d), 2 * (b * d + a * c),
                        2 * (b * c + a * d), 1 - 2 * (b * b + d * d), 2 * (c * d - a * b),
                        2 * (b * d - a * c), 2 * (c * d + a * b), 1 - 2 * (b * b + c * c)], 1)


def _pool(net, seed, load, dev, count):
    """`count` material states on their load paths: orientation eigenvalues, local macro strain,
    converged state [S, count] and the direction of the next increment (one regular step long)."""
    _, lam, _ = W.orientation_field(count, seed=seed)
    lam = torch.from_numpy(lam).to(dev)
    rng = np.random.default_rng(seed + 1)
    if load == "cyclic":      # triangle wave of +-2 %: some way up the first leg
        d = torch.from_numpy(W.random6_path_final(count, 0.02, seed=seed + 2)).to(dev)
        peak = torch.from_numpy(rng.uniform(0.3, 1.0, (count, 1))).to(dev)
        turn = torch.from_numpy(rng.choice([-1.0, -1.0, 1.0], (count, 1))).to(dev)   # two of three on the way back
        legs, step = [0.5 * peak * d, peak * d], 0.08 * turn * d
    else:                     # proportional ramp to 3 % in 50 increments, after increments 2 to 10
        d = torch.from_numpy(W.random6_path_final(count, 0.03, seed=seed + 2)).to(dev)
        at = torch.from_numpy(rng.integers(2, 11, (count, 1)) / 50.0).to(dev)
        legs, step = [0.5 * at * d, at * d], d / 50.0
    z = torch.zeros((count, net.L, 6), dtype=F64, device=dev)
    a = torch.zeros((count, net.N, 3), dtype=F64, device=dev)
    for E in legs:
        _, _, z, a, _ = net.solve(lam, E, z, a, tol=1e-13)
    return lam, legs[-1], net.pack(z, a), step


def _points(case, seed, dev):
    """n points in the middle of their load paths: dict of the arrays an update takes."""
    n = case["n"]
    gen = torch.Generator(device=dev)
    gen.manual_seed(1000003 * (seed % 1000003) + 17)
    trees = _trees(case, seed)
    nets = [_Net(t, dev) for t in trees]
    S = max(net.S for net in nets)
    Q = _haar(n, gen, dev)
    R = _rotation(Q)
    scale = 0.75 + 0.5 * torch.rand((n, 1), generator=gen, dtype=F64, device=dev)
    lam = torch.empty((n, 2), dtype=F64, device=dev)
    E, dE = (torch.empty((n, 6), dtype=F64, device=dev) for _ in range(2))
    state = torch.zeros((S, n), dtype=F64, device=dev)
    tid = torch.zeros(n, dtype=torch.int32, device=dev)
    if len(nets) > 1:
        tid = torch.randint(0, len(nets), (n,), generator=gen, device=dev).to(torch.int32)
    for k, net in enumerate(nets):
        at = (tid == k).nonzero().flatten()
        if not len(at):
            continue
        count = min(POOL, n)
        lp, Ep, sp, dp = _pool(net, seed + 101 * k, case.get("load", "ramp"), dev, count)
        pick = torch.randint(0, count, (len(at),), generator=gen, device=dev)
        lam[at], E[at], dE[at] = lp[pick], Ep[pick], dp[pick] * scale[at]
        if len(nets) == 1:
            torch.index_select(sp, 1, pick, out=state)
        else:
            state[: net.S, at] = sp[:, pick]
        if len(nets) > 1:     # every other point of a forest stays in the elastic range, from the virgin state
            el = torch.rand(len(at), generator=gen, dtype=F64, device=dev) < 0.5
            state[:, at[el]] = 0.0
            E[at[el]] = 0.0
            dE[at[el]] *= 0.05
    E, dE = _mv(R, E), _mv(R, dE)
    return dict(trees=trees, nets=nets, lam=lam, Q=Q, E_n=E, dE=dE, state_in=state,
                tid=tid if len(nets) > 1 else None, R=R)


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _handle(case, trees):
    return dmn.DMN(trees if len(trees) > 1 else trees[0], precision=case["precision"],
                   line_search=case.get("line_search", False))


def _fe_inputs(case, seed, dev):
    mesh = W.plate_with_hole_mesh(case["n_t"], case["n_r"], case["n_z"])
    rng = np.random.default_rng(seed)
    n_el = mesh.conn.shape[0]
    # tangents of a depth-3 network at plastic states, in the frames of the plate's orientation field
    net = _Net(W.tree_d10_fit(3, seed=seed), dev)
    lam, E, st, step = _pool(net, seed, "ramp", dev, 256)
    z, a = net.unpack(st)
    C = net.solve(lam, E + step, z, a, tol=1e-13)[1]
    A2 = W.plate_orientation_field(mesh.centroid, mesh.R, mesh.H, mesh.T, seed=seed)
    A = np.stack([A2[:, [0, 5, 4]], A2[:, [5, 1, 3]], A2[:, [4, 3, 2]]], 1)
    Q = torch.from_numpy(np.ascontiguousarray(np.linalg.eigh(A)[1][:, :, ::-1].reshape(n_el, 9))).to(dev)
    R = _rotation(Q).repeat_interleave(8, 0)
    pick = torch.from_numpy(rng.integers(0, 256, n_el)).to(dev).repeat_interleave(8)
    C = R @ C[pick] @ R.transpose(1, 2)
    C = (0.5 * (C + C.transpose(1, 2))).contiguous()
    free = torch.from_numpy((~mesh.fixed).astype(np.float64)).to(dev)
    # displacement of the loaded plate (uniform strain plus seeded ripples)
    x = torch.from_numpy(mesh.xyz).to(dev)
    k = torch.from_numpy(rng.uniform(0.5, 3.0, (3, 3)) * math.pi / mesh.H).to(dev)
    u = 0.3 * torch.from_numpy(mesh.affine).to(dev).reshape(-1, 3) + 0.01 * torch.sin(x @ k)
    return mesh, C, free, u.reshape(-1).contiguous()


def prepare(case, seed):
    dev = _dev()
    kind = case["kind"]
    if kind == "fe":
        mesh, C, free, u = _fe_inputs(case, seed, dev)
        m = fe.Hex8Mesh(mesh.xyz, mesh.conn)
        vec = lambda: torch.empty(m.n_dofs, dtype=F64, device=dev)  # noqa: E731
        gp6 = torch.empty((m.n_gp, 6), dtype=F64, device=dev)
        return dict(kind=kind, m=m, C=C, free=free, u=u, E=gp6, f=vec(), diag=vec(), x=vec(), rtol=case["rtol"],
                    f32=case["f32"])
    if kind == "stiffness":
        tree = _tree(case, seed)
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        _, lam, Q = W.orientation_field(case["n"], seed=seed + 1)
        t = lambda x: torch.as_tensor(x, dtype=F64, device=dev)  # noqa: E731
        G = torch.randn((case["n"], 6, 6), generator=gen, dtype=F64, device=dev)
        return dict(kind=kind, m=_handle(case, [tree]), lam=t(lam), Q=t(Q), G=G + G.transpose(1, 2),
                    params=[t(x).requires_grad_() for x in (tree.p, tree.q, tree.w)])
    s = _points(case, seed, dev)
    s["kind"], s["m"] = kind, _handle(case, s["trees"])
    del s["R"], s["nets"]
    if kind == "grad":
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        s["g"] = torch.randn((case["n"], 6), generator=gen, dtype=F64, device=dev)
        t = s["trees"][0]
        s["params"] = [torch.as_tensor(x, dtype=F64, device=dev).requires_grad_() for x in (t.p, t.q, t.w)]
        s["dE"].requires_grad_()
        return s
    if kind == "host":
        for k in ("lam", "Q", "E_n", "dE", "state_in", "tid"):
            s[k] = None if s[k] is None else s[k].cpu().pin_memory()
        s["out"] = s["m"].alloc_host_outputs(case["n"])
        return s
    s["out"] = s["m"].alloc_outputs(case["n"], dev)
    s["out"]["state_out"].zero_()     # fields past a shallower tree's own are not written
    return s


def run(state):
    s = state
    if s["kind"] == "update":
        return s["m"].update(s["lam"], s["Q"], s["E_n"], s["dE"], s["state_in"], out=s["out"], tree_id=s["tid"])
    if s["kind"] == "host":
        return s["m"].update_host(s["lam"], s["Q"], s["E_n"], s["dE"], s["state_in"], out=s["out"], tree_id=s["tid"])
    if s["kind"] == "grad":
        sig, st, status = ag.dmn_stress(s["m"], s["lam"], s["Q"], s["E_n"], s["dE"], s["state_in"], *s["params"])
        g = torch.autograd.grad((sig * s["g"]).sum(), [*s["params"], s["dE"]])
        return dict(stress=sig.detach(), state=st, status=status, p=g[0], q=g[1], w=g[2], E=g[3])
    if s["kind"] == "stiffness":
        C = ag.dmn_stiffness(s["m"], s["lam"], s["Q"], *s["params"])
        g = torch.autograd.grad((C * s["G"]).sum(), s["params"])
        return dict(C=C.detach(), p=g[0], q=g[1], w=g[2])
    m = s["m"]
    m.strain(s["u"], s["E"])
    sig = torch.bmm(s["C"], s["E"].unsqueeze(2)).squeeze(2)
    m.internal_force(sig, s["f"])
    m.tangent_diagonal(s["C"], s["diag"])
    it, res = m.pcg(s["C"], s["free"], s["diag"], s["f"], s["x"], rtol=s["rtol"], f32=s["f32"])
    return dict(strain=s["E"], force=s["f"], diag=s["diag"], x=s["x"], iterations=it)


# --------------------------------------------------------------------------------------------
# Work and exact results

def _counts(case):
    """(laminates, inelastic leaves, state fields) of a case's tree, averaged over a forest."""
    Ks = FOREST if case["tree"] == "forest" else (case["K"],)
    part = 0.7 if case["tree"] == "trained" else 1.0
    N = sum(part * (2 ** K - 1) for K in Ks) / len(Ks)
    nz = sum(part * 2 ** (K - 1) for K in Ks) / len(Ks)
    return N, nz, 6 * nz + 3 * N


def work(case):
    if case["kind"] == "fe":
        n_el = 4 * case["n_t"] * case["n_r"] * case["n_z"]
        n_dof = 3 * 4 * case["n_t"] * (case["n_r"] + 1) * (case["n_z"] + 1)
        iters = 4 * (case["n_t"] + case["n_r"]) * (1.0 if case["rtol"] > 1e-7 else 1.4)
        # inputs and outputs once; flops: two products with B and one with C per Gauss point and CG iteration
        return dict(bytes=8.0 * (8 * n_el * (36 + 25 + 6) + 6 * n_dof), flops=8.0 * n_el * (144 + 72 + 144) * iters)
    N, nz, S = _counts(dict(case, tree=case.get("tree", "full")))
    n = case["n"]
    per_pass = N * (83 + 0.5 * 678 + 0.5 * 474) + nz * 81
    if case["kind"] == "stiffness":
        return dict(bytes=8.0 * n * (11 + 36 + 36), flops=n * (per_pass + 3 * 680 * N))
    passes = 3.0 if case.get("load") == "cyclic" else 4.7
    flops = n * per_pass * passes
    if case["kind"] == "grad":
        return dict(bytes=8.0 * n * (2 + 9 + 12 + 2 * S + 6 + 6 + 6), flops=flops + n * (per_pass + 500 * N))
    return dict(bytes=8.0 * n * (2 + 9 + 12 + 2 * S + 42 + 1), flops=flops)


def _exact_update(case, seed, dev):
    s = _points(case, seed, dev)
    n, R = case["n"], s["R"]
    sig = torch.empty((n, 6), dtype=F64, device=dev)
    tan = torch.empty((n, 6, 6), dtype=F64, device=dev)
    out = torch.zeros_like(s["state_in"])
    for k, net in enumerate(s["nets"]):
        at = torch.arange(n, device=dev) if s["tid"] is None else (s["tid"] == k).nonzero().flatten()
        for c in _chunks(len(at), net.K):
            i = at[c]
            z, a = net.unpack(s["state_in"][: net.S, i])
            E = _mv(R[i].transpose(1, 2), s["E_n"][i] + s["dE"][i])
            sb, C, zn, a, _ = net.solve(s["lam"][i], E, z, a)
            sig[i], tan[i] = _mv(R[i], sb), R[i] @ C @ R[i].transpose(1, 2)
            out[: net.S, i] = net.pack(zn, a)
    return dict(state_out=out, stress=sig, tangent=tan, iters=None, status=None), s


def _exact_grad(case, seed, dev):
    o, s = _exact_update(case, seed, dev)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    G = torch.randn((case["n"], 6), generator=gen, dtype=F64, device=dev)
    t = s["trees"][0]
    par = [torch.as_tensor(x, dtype=F64, device=dev).requires_grad_() for x in (t.p, t.q, t.w)]
    total = [torch.zeros_like(x) for x in par]
    base = s["nets"][0]
    for c in _chunks(case["n"], base.K):
        Rt = s["R"][c].transpose(1, 2)
        E, g = _mv(Rt, s["E_n"][c] + s["dE"][c]), _mv(Rt, G[c])
        z, _ = base.unpack(s["state_in"][:, c])
        _, a = base.unpack(o["state_out"][:, c])
        with torch.no_grad():      # the jumps' response to a macro perturbation g, at the solution
            Nm = _N(base.normals(s["lam"][c]))
            st, D, _ = base.leaves(base.strains(Nm, E, a), z)
            C = torch.stack([_leaf_tangent(D[0]), _leaf_tangent(D[1])], 2).flatten(1, 2)
            H = base.condense(Nm, C, st)[2]
            mu = base.descend(Nm, None, H, g)
        net = _Net(t, dev, *par)
        Nm = _N(net.normals(s["lam"][c]))
        sb, R = net.average(Nm, net.leaves(net.strains(Nm, E, a), z)[0])
        for x, y in zip(total, torch.autograd.grad((g * sb).sum() + (mu * R).sum(), par)):
            x += y
    w = torch.where(par[2].detach() > 0, total[2], torch.zeros_like(total[2]))
    return dict(stress=o["stress"], state=o["state_out"], status=None, p=total[0], q=total[1], w=w,
                E=_mv(o["tangent"], G))


def _exact_stiffness(case, seed, dev):
    tree = _tree(case, seed)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    _, lam, Q = W.orientation_field(case["n"], seed=seed + 1)
    lam, Q = torch.from_numpy(lam).to(dev), torch.from_numpy(Q).to(dev)
    G = torch.randn((case["n"], 6, 6), generator=gen, dtype=F64, device=dev)
    G = G + G.transpose(1, 2)
    par = [torch.as_tensor(x, dtype=F64, device=dev).requires_grad_() for x in (tree.p, tree.q, tree.w)]
    total = [torch.zeros_like(x) for x in par]
    C = torch.empty((case["n"], 6, 6), dtype=F64, device=dev)
    for c in _chunks(case["n"], case["K"]):
        net = _Net(tree, dev, *par)
        R = _rotation(Q[c])
        z = torch.zeros((len(lam[c]), net.L, 6), dtype=F64, device=dev)
        D = net.leaves(z, z)[1]
        Ct = torch.stack([_leaf_tangent(D[0]), _leaf_tangent(D[1])], 2).flatten(1, 2)
        Cg = R @ net.condense(_N(net.normals(lam[c])), Ct)[0] @ R.transpose(1, 2)
        C[c] = Cg.detach()
        for x, y in zip(total, torch.autograd.grad((Cg * G[c]).sum(), par)):
            x += y
    w = torch.where(par[2].detach() > 0, total[2], torch.zeros_like(total[2]))
    return dict(C=C, p=total[0], q=total[1], w=w)


def _exact_fe(case, seed, dev):
    mesh, C, free, u = _fe_inputs(case, seed, dev)
    xyz, conn = torch.from_numpy(mesh.xyz).to(dev), torch.from_numpy(mesh.conn.astype(np.int64)).to(dev)
    XI = torch.tensor([[-1, -1, -1], [1, -1, -1], [1, 1, -1], [-1, 1, -1], [-1, -1, 1], [1, -1, 1], [1, 1, 1],
                       [-1, 1, 1]], dtype=F64, device=dev)
    g = torch.arange(8, device=dev)
    pt = torch.stack([(g & 1) * 2 - 1, (g >> 1 & 1) * 2 - 1, (g >> 2 & 1) * 2 - 1], 1).to(F64) / math.sqrt(3.0)
    fac = 1.0 + XI[None] * pt[:, None]                                   # [gp, node, 3]
    dn = 0.125 * torch.stack([XI[:, 0] * fac[..., 1] * fac[..., 2], XI[:, 1] * fac[..., 0] * fac[..., 2],
                              XI[:, 2] * fac[..., 0] * fac[..., 1]], -1)
    J = torch.einsum("eai,gak->egik", xyz[conn], dn)
    det = torch.linalg.det(J)
    gr = torch.einsum("gak,egki->egai", dn, torch.linalg.inv(J))         # [e, gp, node, 3]
    B = _N(gr).permute(0, 1, 3, 2, 4).reshape(len(conn), 8, 6, 24)       # Mandel strain of the element's dofs
    Cg = C.reshape(len(conn), 8, 6, 6)
    Ke = torch.einsum("egIa,egIb->eab", B, (Cg @ B) * det[..., None, None])
    dof = (3 * conn[:, :, None] + torch.arange(3, device=dev)).reshape(len(conn), 24)
    nd = 3 * len(xyz)

    def gather(fe_):
        return torch.zeros(nd, dtype=F64, device=dev).index_add_(0, dof.flatten(), fe_.flatten())

    eps = torch.einsum("egIa,ea->egI", B, u[dof])
    f = gather(torch.einsum("egIa,egI->ea", B, _mv(Cg, eps) * det[..., None]))
    diag = gather(torch.diagonal(Ke, dim1=1, dim2=2))
    b = free * f
    x, r = torch.zeros_like(b), b.clone()
    z = r / diag * free
    p, rz = z.clone(), (r @ z)
    for k in range(4000):
        Kp = free * gather(_mv(Ke, p[dof]))
        al = rz / (p @ Kp)
        x, r = x + al * p, r - al * Kp
        z = r / diag * free
        new = r @ z
        p, rz = z + (new / rz) * p, new
        if k % 50 == 49 and float(r.norm() / b.norm()) < 1e-13:
            break
    return dict(strain=eps.reshape(-1, 6), force=f, diag=diag, x=x, iterations=None)


def exact(case, seed):
    dev = _dev()
    if case["kind"] == "fe":
        return _exact_fe(case, seed, dev)
    if case["kind"] == "grad":
        return _exact_grad(case, seed, dev)
    if case["kind"] == "stiffness":
        return _exact_stiffness(case, seed, dev)
    return _exact_update(case, seed, dev)[0]
