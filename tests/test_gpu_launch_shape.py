"""The launch shape of the mixed forms' thread kernels (32-thread CTAs, as many per SM as the call's points can
use): a point's result does not depend on it, bit for bit, around the sizes where the number of CTAs changes."""
import pytest
import torch

from paper_2103_08253_gb300 import dmn, workloads as W
from test_gpu_block import inputs
from test_gpu_parity import d

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("prec,compressed", [("mixed", False), ("mixed-f32-tangent", True)])
@pytest.mark.parametrize("rows,extra", [(0, 1), (1, 1), (11, 0), (16, 0), (16, 1), (32, 0), (32, 1)])
def test_results_do_not_depend_on_the_shape(prec, compressed, rows, extra):
    n = rows * 32 * torch.cuda.get_device_properties(DEV).multi_processor_count + extra
    make = W.tree_with_zero_weights if compressed else W.tree_d10_fit
    tree = make(3, seed=800)
    lam, Q, Ef = (d(x) for x in inputs(n, 801))
    outs = []
    for shape in ({}, dict(block=128, ctas_per_sm=4, stage_ctas_per_sm=4)):
        m = dmn.DMN(tree, precision=prec, warp_per_point=-1, **shape)
        st = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
        outs.append(m.update(lam, Q, torch.zeros_like(Ef), Ef * 0.2, st))
    for k, v in outs[0].items():
        assert torch.equal(v, outs[1][k]), k


@pytest.mark.parametrize("compressed", [False, True])
def test_the_mixed_sweep_above_and_below_its_size_limit(compressed):
    """4096 points per SM run the CTA organisation's sweep, one more the fused final kernel: the same jumps and
    leaf states bit for bit, stress and tangent to the rounding of two FP64 condensations of depth 3."""
    n = 4096 * torch.cuda.get_device_properties(DEV).multi_processor_count + 1
    tree = (W.tree_with_zero_weights if compressed else W.tree_d10_fit)(3, seed=810)
    lam, Q, Ef = (d(x) for x in inputs(1024, 811))
    lam, Q, dE = (x.repeat(n // 1024 + 1, 1)[:n].contiguous() for x in (lam, Q, Ef * 0.2))
    m = dmn.DMN(tree, precision="mixed")
    outs = []
    for k in (n - 1, n):
        st = torch.zeros((m.state_size, k), dtype=torch.float64, device=DEV)
        o = m.update(lam[:k], Q[:k], torch.zeros_like(dE[:k]), dE[:k], st)
        outs.append({key: (v[:, :1024] if key == "state_out" else v[:1024]).clone() for key, v in o.items()})
    for key in ("state_out", "iters", "status"):
        assert torch.equal(outs[0][key], outs[1][key]), key
    for key in ("stress", "tangent"):
        a, b = (o[key].reshape(1024, -1) for o in outs)
        assert ((a - b).norm(dim=1) <= 1e-12 * b.norm(dim=1)).all(), key
