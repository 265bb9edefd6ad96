"""Small calls spread a point's normals and leaf states over several threads (point_split): the same
operations on the same values as one thread per point, so the results agree to the contraction of
multiply-adds, at every depth, on compressed trees, with one and with two inelastic phases."""
import numpy as np
import pytest
import torch

from paper_2103_08253_gb300 import dmn, workloads as W
from test_gpu_parity import d

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("K,kind", [(1, "full"), (2, "full"), (3, "both"), (4, "compressed"), (6, "full"),
                                    (7, "compressed")])
def test_a_small_call_gives_the_states_of_the_same_points_in_a_large_one(K, kind):
    phases = (W.MATRIX_EXPLIN, W.MATRIX) if kind == "both" else (W.FIBER, W.MATRIX)
    make = W.tree_with_zero_weights if kind == "compressed" else W.tree_d10_fit
    tree = make(K, seed=600 + K, phases=phases)
    n_sm = torch.cuda.get_device_properties(DEV).multi_processor_count
    n = 1024 * n_sm + 1                  # one thread per point
    _, lam, Q = W.orientation_field(n, seed=601)
    E = W.random6_path_final(n, 0.02, seed=602)
    m = dmn.DMN(tree, warp_per_point=-1)
    a = [d(lam), d(Q), torch.zeros((n, 6), dtype=torch.float64, device=DEV), d(E)]
    big = m.update(*a, torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV))
    for k in (1, 33, 2500, 70001):       # 32, 32, 32 and 2 threads per point
        out = m.update(*(x[:k] for x in a), torch.zeros((m.state_size, k), dtype=torch.float64, device=DEV))
        assert torch.equal(out["iters"], big["iters"][:k]) and torch.equal(out["status"], big["status"][:k])
        for key, x, y in (("state_out", out["state_out"], big["state_out"][:, :k]),
                          ("stress", out["stress"], big["stress"][:k]), ("tangent", out["tangent"], big["tangent"][:k])):
            # 2^-53 per operation, at most 20 operations on a path of 8 laminates, an order to spare
            assert (x - y).abs().max() <= 1e-13 * y.abs().max(), (k, key)
    assert (big["status"] == 0).double().mean() > 0.9   # a few points of so large a step need the line search
    m.close()
