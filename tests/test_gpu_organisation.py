"""Which organisation a handle's calls run: the options that name one get it."""
import pytest
import torch

from paper_2103_08253_gb300 import dmn, workloads as W
from test_gpu_block import inputs
from test_gpu_parity import d

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("lanes,kind", [(32, "full"), (16, "compressed"), (8, "full")])
def test_lanes_asked_for_run_the_all_fp64_warp_kernel(lanes, kind):
    """warp_per_point = 1 with warp_lanes given: the warp kernel.  A handle with the first stage never runs the CTA
    organisation, and no stage in the warp organisation, so it gives that kernel's results: bit for bit the same."""
    n = 300
    tree = (W.tree_with_zero_weights if kind == "compressed" else W.tree_d10_fit)(6, seed=870)
    lam, Q, Ef = (d(x) for x in inputs(n, 871))
    outs = []
    for opts in (dict(), dict(first_stage=True)):
        m = dmn.DMN(tree, warp_per_point=1, warp_lanes=lanes, **opts)
        assert m.lanes_per_point(n) == lanes
        st = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
        outs.append(m.update(lam, Q, torch.zeros_like(Ef), Ef * 0.2, st))
        m.close()
    for k, v in outs[0].items():
        assert torch.equal(v, outs[1][k]), k
