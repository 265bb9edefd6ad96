"""Points that k_newton_block hands back to the all-FP64 kernels (here: all points of trees whose moduli are beyond
FP32's reach), through every form of the list: 32 or 8 lanes per point by its length, lanes as asked for, one thread
per point, with the line search, on compressed trees, with several trees, from a small and from a large call."""
import copy

import numpy as np
import pytest
import torch

import oracle
from paper_2103_08253_gb300 import dmn, workloads as W
from test_gpu_block import inputs
from test_gpu_parity import d, rel

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def beyond_fp32(tree):
    big = copy.deepcopy(tree)
    big.phases = tuple(W.Phase(p.kind, 1e9 * p.E, p.nu, 1e9 * p.sigma0, 1e9 * p.H) for p in tree.phases)
    return big


# every: one point in `every` belongs to a tree that is handed back; n: 3000 points pass the 32 lanes' limit
@pytest.mark.parametrize("depths,kind,n,every,opts", [
    ((5, 4, 5), "full", 601, 7, {}), ((5, 4, 5), "full", 601, 7, dict(line_search=True)),
    ((6, 3, 5), "compressed", 400, 5, {}), ((6, 3, 5), "compressed", 400, 5, dict(line_search=True)),
    ((4, 3, 3), "full", 3000, 1, {}), ((4, 3, 4), "compressed", 3000, 1, dict(line_search=True)),
    ((5, 4, 5), "full", 601, 7, dict(warp_per_point=-1)), ((5, 4, 5), "compressed", 601, 7, dict(warp_lanes=16)),
    ((3, 3, 3), "full", 200000, 5000, {}), ((3, 3, 3), "compressed", 200000, 5000, dict(warp_per_point=-1))])
def test_points_handed_back_get_the_oracles_results(depths, kind, n, every, opts):
    make = W.tree_with_zero_weights if kind == "compressed" else W.tree_d10_fit
    trees = [make(K, seed=840 + K + 10 * k) for k, K in enumerate(depths)]
    trees[1:] = [beyond_fp32(t) for t in trees[1:]]
    pool = min(n, 1000)
    lam, Q, Ef = inputs(pool, 841, eps=0.02)
    E = Ef * 0.15
    at = np.arange(n) % pool
    tid = np.where(np.arange(n) % every == 0, 1 + np.arange(n) // every % 2, 0).astype(np.int32)
    if every > pool:
        at[tid > 0] = np.arange((tid > 0).sum())       # the handed-back points of a large call are all different
    m = dmn.DMN(trees, **opts)
    out = m.update(d(lam[at]), d(Q[at]), torch.zeros((n, 6), dtype=torch.float64, device=DEV), d(E[at]),
                   torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV), tree_id=d(tid))
    o = {k: v.cpu().numpy() for k, v in out.items()}
    for k, tree in enumerate(trees):
        i = np.nonzero(tid == k)[0][:pool]
        if not len(i):
            continue
        st, sig, C, it, stat, gap = oracle.update(tree, lam[at[i]], Q[at[i]], np.zeros((len(i), 6)), E[at[i]],
                                                  np.zeros((m.tree_state_sizes[k], len(i))),
                                                  line_search=bool(opts.get("line_search")))
        np.testing.assert_array_equal(o["status"][i], stat)
        ok = stat == 0
        assert ok.mean() > 0.8
        assert np.abs(o["iters"][i] - it)[ok].max() <= 1
        assert rel(o["stress"][i][ok], sig[ok]).max() <= 1e-10, k
        clear = ok & (gap > 1e-9)
        assert rel(o["tangent"][i][clear], C[clear]).max() <= 1e-10, k
        a = o["state_out"][: len(st)][:, i]
        scale = np.maximum(np.abs(st).max(axis=1, keepdims=True), 1e-5 * np.abs(st).max())
        assert (np.abs(a - st)[:, ok] / scale).max() <= 1e-9, k
    m.close()


def test_host_calls_allocate_their_work_space_once():
    """The FP64 form's handles hold no thread-per-point scratch; the second work set, which the first call from host
    arrays makes, is still made only once."""
    n = 500
    tree = W.tree_d10_fit(7, seed=860)
    lam, Q, Ef = (torch.from_numpy(x) for x in inputs(n, 861))
    m = dmn.DMN(tree)
    st = torch.zeros((m.state_size, n), dtype=torch.float64)
    free = []
    for _ in range(3):
        m.update_host(lam, Q, torch.zeros_like(Ef), Ef * 0.1, st, chunk=200)
        free.append(torch.cuda.mem_get_info()[0])
    assert free[1] == free[0] and free[2] == free[0]
    m.close()
