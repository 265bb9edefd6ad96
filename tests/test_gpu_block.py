"""The FP64 form's CTA organisation (csrc/dmn_block.cu): FP32 condensation with FP64 refinement of every
Newton step.  Its iterates must be those of the all-FP64 iteration, so stress, tangent, state and iteration
counts are compared with the oracle at the FP64 form's tolerances, at every depth the organisation takes
(3 .. 8: 256 down to 8 points per CTA), around the sizes where a CTA's slots run out, on compressed trees,
with one and two inelastic phases, with the line search, with several trees in a call; and points whose FP32
solve cannot contract must come out of the all-FP64 kernels."""
import copy

import numpy as np
import pytest
import torch

from paper_2103_08253_gb300 import dmn, workloads as W
from test_gpu_parity import d, rel

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def path(m, trees, lam, Q, Ef, steps, n_steps, tid=None, line_search=False):
    """Every increment of a proportional path against the oracle; returns the worst errors."""
    import oracle
    n = len(lam)
    st = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
    of = [np.arange(n) if tid is None else np.nonzero(tid == k)[0] for k in range(len(trees))]
    so = [np.zeros((m.tree_state_sizes[k], len(of[k]))) for k in range(len(trees))]
    worst = dict(stress=0.0, tangent=0.0, state=0.0, iters=0, bad=0)
    for s in range(1, steps + 1):
        En, dE = W.proportional_increment(Ef, s, n_steps)
        out = m.update(d(lam), d(Q), d(En), d(dE), st, tree_id=None if tid is None else d(tid))
        st = out["state_out"].clone()
        o = {k: v.cpu().numpy() for k, v in out.items()}
        for k, tree in enumerate(trees):
            i = of[k]
            so[k], sig, C, it, stat, gap = oracle.update(tree, lam[i], Q[i], En[i], dE[i], so[k], line_search=line_search)
            ok = (stat == 0) & (o["status"][i] == 0)
            worst["bad"] += int((stat != o["status"][i]).sum())   # a path may have points that need the line search
            worst["iters"] += int((o["iters"][i] != it)[ok].sum())
            worst["stress"] = max(worst["stress"], rel(o["stress"][i][ok], sig[ok]).max())
            clear = ok & (gap > 1e-9)
            worst["tangent"] = max(worst["tangent"], rel(o["tangent"][i][clear], C[clear]).max())
            a, b = o["state_out"][: so[k].shape[0]][:, i], so[k]
            scale = np.maximum(np.abs(b).max(axis=1, keepdims=True), 1e-5 * np.abs(b).max())
            worst["state"] = max(worst["state"], (np.abs(a - b)[:, ok] / scale).max())
            st[: so[k].shape[0], d(i)] = d(b)     # both sides go on from the oracle's state
    return worst


def inputs(n, seed, eps=0.03):
    _, lam, Q = W.orientation_field(n, seed=seed)
    return lam, Q, W.random6_path_final(n, eps, seed=seed + 1)


@pytest.mark.parametrize("K,n,kind", [(3, 257, "full"), (3, 1, "both"), (4, 129, "both"), (5, 63, "explin"),
                                      (6, 33, "compressed"), (7, 17, "both"), (7, 200, "compressed"),
                                      (8, 1, "full"), (8, 9, "compressed"), (8, 40, "explin")])
def test_iterates_are_the_oracles(K, n, kind):
    phases = {"both": (W.MATRIX_EXPLIN, W.MATRIX), "explin": (W.FIBER, W.MATRIX_EXPLIN)}.get(kind, (W.FIBER, W.MATRIX))
    make = W.tree_with_zero_weights if kind == "compressed" else W.tree_d10_fit
    tree = make(K, seed=700 + K, phases=phases)
    m = dmn.DMN(tree)
    w = path(m, [tree], *inputs(n, 710 + n), 6, 20)
    assert w["bad"] == 0 and w["iters"] == 0, w
    assert w["stress"] <= 1e-10 and w["tangent"] <= 1e-10 and w["state"] <= 1e-9, w


def test_more_points_than_the_ctas_hold():
    """Slots refill as their points converge; a point's result does not depend on the batch, bit for bit."""
    n_sm = torch.cuda.get_device_properties(DEV).multi_processor_count
    K, n = 8, 2 * 8 * 2 * n_sm + 3
    tree = W.tree_d10_fit(K, seed=720)
    lam, Q, Ef = inputs(n, 721)
    m = dmn.DMN(tree)
    z = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
    whole = m.update(d(lam), d(Q), torch.zeros_like(d(Ef)), d(Ef * 0.2), z)
    cut = n // 3
    part = m.update(d(lam[cut:]), d(Q[cut:]), torch.zeros_like(d(Ef[cut:])), d(Ef[cut:] * 0.2), z[:, cut:].contiguous())
    for k in ("stress", "tangent", "iters", "status"):
        assert torch.equal(whole[k][cut:], part[k]), k
    assert torch.equal(whole["state_out"][:, cut:], part["state_out"])


def test_several_trees_with_the_line_search_and_an_unknown_tree():
    trees = [W.tree_d10_fit(K, seed=730 + K) for K in (3, 8, 5)]
    n = 301
    lam, Q, Ef = inputs(n, 740, eps=0.05)
    tid = (np.arange(n) * 7 % 3).astype(np.int32)
    m = dmn.DMN(trees, line_search=True)
    w = path(m, trees, lam, Q, Ef, 3, 6, tid=tid, line_search=True)
    assert w["bad"] == 0 and w["iters"] == 0 and w["stress"] <= 1e-10 and w["tangent"] <= 1e-10, w
    tid[11] = 3
    out = m.update(d(lam), d(Q), torch.zeros_like(d(Ef)), d(Ef * 0.1),
                   torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV), tree_id=d(tid))
    stat = out["status"].cpu().numpy()
    assert stat[11] == dmn.STATUS_BAD_TREE and (np.delete(stat, 11) == 0).all()
    assert torch.isnan(out["stress"][11]).all() and torch.isnan(out["tangent"][11]).all()


@pytest.mark.parametrize("n", [5, 3000])
def test_points_the_fp32_solve_cannot_take_go_to_the_fp64_kernels(n):
    """Moduli whose 3x3 determinants overflow FP32 (1e9 times MPa), a point with a non-finite strain and a
    correction limit that no point meets: the all-FP64 results and statuses."""
    K = 6
    tree = W.tree_d10_fit(K, seed=750)
    big = copy.deepcopy(tree)
    big.phases = tuple(W.Phase(p.kind, 1e9 * p.E, p.nu, 1e9 * p.sigma0, 1e9 * p.H) for p in tree.phases)
    lam, Q, Ef = inputs(n, 751)
    E = Ef * 0.2
    E[2, 3] = np.nan
    outs = []
    for t in (tree, big):
        m = dmn.DMN(t)
        outs.append(m.update(d(lam), d(Q), torch.zeros_like(d(E)), d(E),
                             torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)))
    a, b = ({k: v.cpu().numpy() for k, v in o.items()} for o in outs)
    assert a["status"][2] == b["status"][2] == dmn.STATUS_NONFINITE
    ok = np.arange(n) != 2
    np.testing.assert_array_equal(a["status"], b["status"])
    ok &= a["status"] == 0          # a few points of so large a step need the line search
    assert ok.mean() > 0.79
    np.testing.assert_array_equal(a["iters"][ok], b["iters"][ok])
    assert np.isnan(b["stress"][2]).all() and np.isnan(b["state_out"][:, 2]).all()
    assert rel(1e-9 * b["stress"][ok], a["stress"][ok]).max() <= 1e-10
    assert rel(1e-9 * b["tangent"][ok], a["tangent"][ok]).max() <= 1e-10
    m = dmn.DMN(tree, max_iter=1)
    o = m.update(d(lam), d(Q), torch.zeros_like(d(E)), d(E), torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV))
    stat, it = o["status"].cpu().numpy(), o["iters"].cpu().numpy()
    assert (stat[ok] == dmn.STATUS_MAXITER).all() and (it[ok] == 1).all()


@pytest.mark.parametrize("K,n", [(3, 9), (5, 37), (7, 21), (8, 41)])
def test_a_small_calls_smaller_ctas_give_the_same_bits(K, n):
    """At most as many 256-thread CTAs as SMs: CTAs of 128 threads.  The same points at the head of a larger call
    run in CTAs of 256."""
    n_sm = torch.cuda.get_device_properties(DEV).multi_processor_count
    big = n_sm * (256 >> (K - 3)) + 1
    tree = W.tree_d10_fit(K, seed=760 + K, phases=(W.FIBER, W.MATRIX_EXPLIN))
    lam, Q, Ef = inputs(big, 761)
    m = dmn.DMN(tree)
    outs = []
    for k in (big, n):
        z = torch.zeros((m.state_size, k), dtype=torch.float64, device=DEV)
        outs.append(m.update(d(lam[:k]), d(Q[:k]), torch.zeros_like(d(Ef[:k])), d(Ef[:k] * 0.2), z))
    for k in ("stress", "tangent", "iters", "status"):
        assert torch.equal(outs[0][k][:n], outs[1][k]), k
    assert torch.equal(outs[0]["state_out"][:, :n], outs[1]["state_out"])


def test_iteration_counts_on_large_steps():
    """Increments whose last Newton step is large (it ends in a fixed set of plastic leaves, so that no quadratic
    term follows): what the FP32 solves leave of the linear residual must not show in the criterion."""
    import oracle
    n = 400
    lam, Q, Ef = inputs(n, 770, eps=0.02)
    for K in (5, 6, 8):
        tree = W.tree_d10_fit(K, seed=300 + K)
        m = dmn.DMN(tree)
        for scale in (0.0005, 0.25):
            st = np.zeros((m.state_size, n))
            _, sig, C, it, stat, gap = oracle.update(tree, lam, Q, np.zeros_like(Ef), scale * Ef, st)
            o = m.update(d(lam), d(Q), torch.zeros_like(d(Ef)), d(scale * Ef), d(st))
            ok = (stat == 0) & (o["status"].cpu().numpy() == 0)
            assert (stat != o["status"].cpu().numpy()).sum() == 0
            np.testing.assert_array_equal(o["iters"].cpu().numpy()[ok], it[ok])
            assert rel(o["stress"].cpu().numpy()[ok], sig[ok]).max() <= 1e-10
