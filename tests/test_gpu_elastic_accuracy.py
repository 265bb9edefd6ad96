"""Elastic points of the FP64 form: one linear Newton step, after which nothing hides what the FP32 solves left of it.
Their results must be as close to the exact ones as the all-FP64 solve's (a few roundings), not merely within the
stopping criterion."""
import numpy as np
import pytest
import torch

import oracle
from paper_2103_08253_gb300 import dmn, workloads as W
from test_gpu_block import inputs
from test_gpu_parity import d, rel

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("K,kind,opts", [(3, "full", {}), (5, "both", dict(line_search=True)), (6, "compressed", {}),
                                         (8, "explin", {}), (8, "full", dict(line_search=True)),
                                         (6, "explin", dict(max_iter=1)), (6, "full", dict(tol=1e-6))])
def test_elastic_points_are_as_accurate_as_the_fp64_solves(K, kind, opts):
    phases = {"both": (W.MATRIX_EXPLIN, W.MATRIX), "explin": (W.FIBER, W.MATRIX_EXPLIN)}.get(kind, (W.FIBER, W.MATRIX))
    make = W.tree_with_zero_weights if kind == "compressed" else W.tree_d10_fit
    tree = make(K, seed=900 + K, phases=phases)
    n = 90
    lam, Q, Ef = inputs(n, 901, eps=0.0002)
    m = dmn.DMN(tree, **opts)
    assert m.cta_threads(n) > 0
    z, st = np.zeros_like(Ef), np.zeros((m.state_size, n))
    so, sig, C, it, stat, gap = oracle.update(tree, lam, Q, z, Ef, st, tol=1e-15)
    o = {k: v.cpu().numpy() for k, v in m.update(d(lam), d(Q), d(z), d(Ef), d(st)).items()}
    el = it == 1          # elastic: a linear problem
    assert el.mean() > 0.8 and (stat[el] == 0).all()
    assert (o["status"][el] == 0).all() and (o["iters"][el] == 1).all()
    # 2^-53 per operation, some 20 operations from a leaf to the root: 2e-15, and an order to spare; the refined step
    # alone leaves 1e-13 of the stress and 1e-12 of the jumps
    assert rel(o["stress"][el], sig[el]).max() <= 2e-14
    assert np.abs(o["state_out"] - so)[:, el].max() <= 1e-13 * np.abs(so[:, el]).max()
    m.close()
