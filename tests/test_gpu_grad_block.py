"""The adjoints in the CTA organisation (csrc/dmn_grad.cu) against the oracle's exact gradient, at the depths and
sizes where it can go wrong: 3 .. 8 (128 down to 4 points per CTA), one point, a CTA's points and one more, whole
and compressed trees, one and two inelastic phases, both seeds in a call."""
import numpy as np
import pytest
import torch

import oracle
from paper_2103_08253_gb300 import dmn, workloads as W
from test_gpu_parity import d

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
ELASTIC = W.Phase(kind=0, E=3000.0, nu=0.35)


def check(tree, grads, points, tol=1e-9):
    """g_p, g_q, g_w against the sum of the oracle's gradients of `points` (argument tuples of gradient_ift and a
    tangent seed): every entry up to depth 6, along two random directions above."""
    got = [x.cpu().numpy() for x in grads]
    if tree.K <= 6:
        want = [0.0, 0.0, 0.0]
        for a, G in points:
            o = oracle.gradient_ift(tree, *a, G_glob=G)
            want = [x + np.asarray(o[k]) for x, k in zip(want, ("p", "q", "w"))]
        want[2] = np.where(np.asarray(tree.w) > 0, want[2], 0.0)
        for x, y in zip(got, want):
            assert np.abs(x.reshape(y.shape) - y).max() <= tol * np.abs(y).max()
        return
    rng = np.random.default_rng(5)
    dirs = [(rng.standard_normal(tree.p.shape), rng.standard_normal(tree.q.shape),
             rng.standard_normal(tree.w.shape) * tree.w) for _ in range(2)]
    want = sum(np.asarray(oracle.gradient_ift(tree, *a, directions=dirs, G_glob=G)) for a, G in points)
    have = np.array([sum((x.reshape(y.shape) * y).sum() for x, y in zip(got, dd)) for dd in dirs])
    assert np.abs(have - want).max() <= tol * np.abs(want).max(), (have, want)


@pytest.mark.parametrize("K,n,kind", [(3, 129, "full"), (3, 1, "both"), (4, 3, "compressed"), (6, 17, "explin"),
                                      (7, 9, "compressed"), (8, 5, "full")])
def test_stress_seed(K, n, kind):
    phases = {"both": (W.MATRIX_EXPLIN, W.MATRIX), "explin": (W.FIBER, W.MATRIX_EXPLIN)}.get(kind, (W.FIBER, W.MATRIX))
    make = W.tree_with_zero_weights if kind == "compressed" else W.tree_d10_fit
    tree = make(K, seed=800 + K, phases=phases)
    _, lam, Q = W.orientation_field(n, seed=801)
    E = W.random6_path_final(n, 0.006, seed=802)
    m = dmn.DMN(tree, tol=1e-15)
    st = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
    z = torch.zeros((n, 6), dtype=torch.float64, device=DEV)
    out = m.update(d(lam), d(Q), z, d(E), st)
    assert (out["status"] == 0).all()
    seeded = sorted({0, n // 2, n - 1})            # the oracle's exact gradient is slow: a few points carry a seed
    g = np.zeros((n, 6))
    g[seeded] = np.random.default_rng(803).standard_normal((len(seeded), 6))
    gp, gq, gw, gE = m.grad(d(lam), d(Q), z, d(E), st, out["state_out"], d(g))
    so, s0 = out["state_out"].cpu().numpy(), np.zeros((m.state_size, n))
    check(tree, (gp, gq, gw), [((lam[i], Q[i], E[i], oracle.jumps(tree, so, i), oracle.leaf_states(tree, s0, i), g[i]),
                                None) for i in seeded])
    want = np.einsum("nji,nj->ni", out["tangent"].cpu().numpy(), g)
    assert np.abs(gE.cpu().numpy() - want).max() <= 1e-10 * np.abs(want).max()


@pytest.mark.parametrize("K,n,kind", [(3, 130, "full"), (5, 33, "compressed"), (7, 1, "full"), (8, 5, "compressed")])
def test_tangent_seed(K, n, kind):
    make = W.tree_with_zero_weights if kind == "compressed" else W.tree_d10_fit
    tree = make(K, seed=820 + K, phases=(W.FIBER, ELASTIC))
    _, lam, Q = W.orientation_field(n, seed=821)
    m = dmn.DMN(tree)
    seeded = sorted({0, n - 1})
    G = np.zeros((n, 6, 6))
    G[seeded] = np.random.default_rng(822).standard_normal((len(seeded), 6, 6))
    gp, gq, gw, _ = m.grad(d(lam), d(Q), None, None, None, None, None, g_tangent=d(G))
    a0 = np.zeros(m.state_size)
    check(tree, (gp, gq, gw), [((lam[i], Q[i], np.zeros(6), a0, np.zeros((1 << K, 7)), np.zeros(6)), G[i])
                               for i in seeded])


def test_both_seeds_and_chunks_add_up():
    """More points than a chunk (65536) and both seeds: the sum of the separate calls."""
    K, n = 3, 65536 + 77
    tree = W.tree_d10_fit(K, seed=840, phases=(W.FIBER, ELASTIC))
    _, lam, Q = W.orientation_field(n, seed=841)
    E = d(W.random6_path_final(n, 0.01, seed=842))
    m = dmn.DMN(tree)
    st = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
    z = torch.zeros_like(E)
    so = m.update(d(lam), d(Q), z, E, st)["state_out"]
    rng = np.random.default_rng(843)
    g, G = d(rng.standard_normal((n, 6))), d(rng.standard_normal((n, 6, 6)))
    a = m.grad(d(lam), d(Q), z, E, st, so, g)
    b = m.grad(d(lam), d(Q), None, None, None, None, None, g_tangent=G)
    c = m.grad(d(lam), d(Q), z, E, st, so, g, g_tangent=G)
    for x, y, both in zip(a[:3], b[:3], c[:3]):
        assert (x + y - both).abs().max() <= 1e-12 * both.abs().max()
    assert torch.equal(a[3], c[3])
