"""Which organisation a handle's calls run: the options that name one get it, the query reports it, and the launch
shape's tuner does not time shapes that it does not take."""
import pytest
import torch

from paper_2103_08253_gb300 import autotune, dmn, workloads as W
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


@pytest.mark.parametrize("K,opts,want", [(8, {}, 32), (4, dict(warp_per_point=-1, line_search=True), 2), (2, {}, 0),
                                         (8, dict(first_stage=True), 0), (8, dict(predictor=True), 0),
                                         (8, dict(precision="mixed"), 0), (6, dict(warp_per_point=1), 8),
                                         (6, dict(warp_per_point=1, warp_lanes=8), 0)])
def test_the_query_reports_the_cta_organisation(K, opts, want):
    m = dmn.DMN(W.tree_d10_fit(K, seed=872), **opts)
    assert m.cta_threads(1000) == want
    m.close()
    m = dmn.DMN([W.tree_d10_fit(3, seed=873), W.tree_d10_fit(K, seed=874)], **opts)
    assert m.cta_threads(1 << 20) == want
    with pytest.raises(ValueError):
        m.cta_threads(-1)
    m.close()


def test_the_tuner_times_a_kernel_without_a_launch_shape_once(tmp_path, monkeypatch):
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "autotune.json"))
    n = 3000
    tree = W.tree_d10_fit(4, seed=875)
    lam, Q, Ef = (d(x) for x in inputs(n, 876))
    st = torch.zeros((W.state_size(4), n), dtype=torch.float64, device=DEV)
    made = []
    real = dmn.DMN
    monkeypatch.setattr(dmn, "DMN", lambda *a, **k: made.append(k) or real(*a, **k))
    for stage, handles in ((None, 1), (True, 3)):
        made.clear()
        res = autotune.tune(tree, "f64", lam, Q, torch.zeros_like(Ef), Ef * 0.1, st, reps=1, first_stage=stage,
                            candidates=((128, 2), (64, 4), (32, 8)))
        assert len(made) == handles and len(res["table"]) == 3 and res["used"] == (stage is True)
        if not res["used"]:
            assert (res["block"], res["ctas_per_sm"]) == (128, 2)


@pytest.mark.parametrize("apart,fused", [(480, 512), (520, 630)])
def test_the_mixed_sweeps_two_organisations_agree(apart, fused):
    """Points per SM on both sides of the rule that chooses the mixed form's sweep at depth 8 (the last 128 points per
    SM nearly full): the same states and counts bit for bit, stress and tangent to the rounding of two FP64
    condensations."""
    n_sm = torch.cuda.get_device_properties(DEV).multi_processor_count
    sizes, k = (apart * n_sm, fused * n_sm), 512
    tree = W.tree_d10_fit(8, seed=880)
    lam, Q, Ef = (d(x) for x in inputs(512, 881))
    lam, Q, dE = (x.repeat(max(sizes) // 512 + 1, 1) for x in (lam, Q, Ef * 0.1))
    m = dmn.DMN(tree, precision="mixed", warp_per_point=-1)
    outs = []
    for n in sizes:
        st = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
        o = m.update(lam[:n].contiguous(), Q[:n].contiguous(), torch.zeros_like(dE[:n]), dE[:n].contiguous(), st)
        outs.append({key: (v[:, :k] if key == "state_out" else v[:k]).clone() for key, v in o.items()})
        del o, st
    for key in ("state_out", "iters", "status"):
        assert torch.equal(outs[0][key], outs[1][key]), key
    for key in ("stress", "tangent"):
        a, b = (o[key].reshape(k, -1) for o in outs)
        assert ((a - b).norm(dim=1) <= 1e-12 * b.norm(dim=1)).all(), key
    m.close()


@pytest.mark.parametrize("K,explin,opts,small,larger", [(3, False, {}, 0, 1), (3, True, {}, 0, 1), (4, True, {}, 0, 2),
                                                        (4, False, {}, 2, 2), (5, True, {}, 4, 4),
                                                        (3, True, dict(warp_per_point=-1), 1, 1),
                                                        (3, False, dict(line_search=True), 0, 1),
                                                        # first_stage = 1 turns the warp organisation's default off
                                                        (3, True, dict(line_search=True, first_stage=True), 1, 1)])
def test_one_elements_points_at_shallow_depth(K, explin, opts, small, larger):
    """Up to 8 points the warp organisation at depth 3, and 4 with an exponential-linear phase: the results of the
    same points in a call of 9, to rounding."""
    tree = W.tree_d10_fit(K, seed=890 + K, phases=(W.FIBER, W.MATRIX_EXPLIN if explin else W.MATRIX))
    lam, Q, Ef = (d(x) for x in inputs(9, 891))
    m = dmn.DMN(tree, **opts)
    assert m.cta_threads(8) == small and m.cta_threads(9) == larger
    outs = []
    for n in (9, 8, 1):
        st = torch.zeros((m.state_size, n), dtype=torch.float64, device=DEV)
        outs.append(m.update(lam[:n], Q[:n], torch.zeros_like(Ef[:n]), Ef[:n] * 0.1, st))
    for o, n in zip(outs[1:], (8, 1)):
        assert torch.equal(o["status"], outs[0]["status"][:n]) and torch.equal(o["iters"], outs[0]["iters"][:n])
        for key in ("stress", "tangent", "state_out"):
            a, b = o[key], outs[0][key][:, :n] if key == "state_out" else outs[0][key][:n]
            assert (a - b).norm() <= 1e-10 * b.norm(), key
    m.close()
