"""A point's results depend on that point alone, bit for bit: in small calls a point's leaf states are written by
several threads, in large ones by one, and a call from host arrays runs in chunks of any size.  Around the sizes
where the number of threads per point changes, in the forms whose leaf states that kernel writes."""
import pytest
import torch

from paper_2103_08253_gb300 import dmn, workloads as W
from test_gpu_block import inputs
from test_gpu_parity import d

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("prec,opts", [("mixed", {}), ("mixed-f32-tangent", {}), ("f64", dict(predictor=True)),
                                       ("f64", dict(first_stage=True))])
@pytest.mark.parametrize("K,kind", [(2, "full"), (3, "full"), (5, "explin"), (5, "compressed")])
def test_states_do_not_depend_on_the_size_of_the_call(prec, opts, K, kind):
    n_sm = torch.cuda.get_device_properties(DEV).multi_processor_count
    n = 512 * n_sm + 2001                # one thread per point; 32 for the host call's last chunk if taken alone
    make = W.tree_with_zero_weights if kind == "compressed" else W.tree_d10_fit
    tree = make(K, seed=820 + K, phases=(W.FIBER, W.MATRIX_EXPLIN if kind == "explin" else W.MATRIX))
    m = dmn.DMN(tree, precision=prec, warp_per_point=-1, **opts)   # one organisation at every size
    lam, Q, Ef = (d(x) for x in inputs(n, 821))
    a = [lam, Q, torch.zeros_like(Ef), Ef * 0.1]
    st = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
    whole = m.update(*a, st)
    for k in (1, 33, 32 * n_sm, 512 * n_sm):
        part = m.update(*(x[:k] for x in a), st[:, :k].contiguous())
        for key, v in part.items():
            w = whole[key][:, :k] if key == "state_out" else whole[key][:k]
            assert torch.equal(v, w), (k, key)
    assert (whole["iters"] > 1).any()      # plastic states among them
    host = m.update_host(*(x.cpu() for x in a), st.cpu(), chunk=512 * n_sm)
    for key, v in host.items():
        assert torch.equal(v.reshape(whole[key].shape), whole[key].cpu()), key
    m.close()
