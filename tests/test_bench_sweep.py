"""Host-side arithmetic of the benchmark for the CTA organisation: the flops that k_sweep_block executes, and the rules
that name the kernels a call runs."""
import numpy as np

import bench


def test_sweep_flops_count_the_shortest_condensation():
    # 255 x 39 + 127 x 499 + 128 x 391 + 128 x 13 + 128 x (68 + 12) + 1150
    full = 255 * 39 + 127 * 499 + 128 * 391 + 128 * 13 + 128 * 80 + 1150
    assert bench.sweep_flops(8, 3, True) == 3 * full and full == 136420
    assert bench.sweep_flops(8, 1, False) == full - 128 * 12
    # two flops per FMA: no more than twice the 88 k FP64 instructions that a point takes, and less than the old form
    assert full <= 2 * 88000 and full < bench.final_flops(8, 1, True)
    w = np.zeros(8)
    w[[0, 1, 3, 6]] = 1.0        # leaf pair (0, 1) and leaf 3 under one laminate, with leaf 6 under the root
    c = bench.tree_counts(w)
    assert (c["N"], c["pairs"], c["inner"], c["single"]) == (3, 1, 2, 2)
    assert bench.sweep_flops(3, 1, True, w) == (3 * 39 + 2 * 499 + 391 + 2 * 84 + c["el"] * 13 + c["j2"] * 80 + 1150)


def test_rooflines_of_the_cta_organisation():
    n, steps = 4096, 10
    r = {"iters_sum": 3.5 * n * steps, "kms": {"newton": 2.0 * steps, "final": 0.9 * steps}, "block": 32, "n_sm": 152}
    line = bench.roofline_f64(r, n, steps)
    f = line["final_kernel"]
    assert line["kernel"] == "k_newton_block" and f["kernel"] == "k_sweep_block"
    assert abs(f["achieved"] - n * 136420 / 0.9e-3 / 1e9) <= 1e-9 * f["achieved"]
    m = bench.roofline_mixed(dict(r, block=0), n, steps)["final_kernel"]
    state = 255 * 39 + 128 * 68
    assert m["kernel"] == "k_sweep_block, k_final"
    assert abs(m["achieved"] - n * (136420 - 128 * 12 + state) / 0.9e-3 / 1e9) <= 1e-9 * m["achieved"]
    m = bench.roofline_mixed(dict(r, block=0), 1 << 20, steps)["final_kernel"]
    assert m["kernel"] == "k_final<sweep>"


def test_kernel_rules(monkeypatch):
    monkeypatch.setattr(bench, "n_sm", lambda: 152)
    assert bench.cta_size(8, 32) == 128 and bench.cta_size(152 * 8, 32) == 128 and bench.cta_size(152 * 8 + 1, 32) == 256
    for n, apart in ((1, True), (3 * 19456, True), (4 * 19456, False), (4 * 19456 + 1, True), (75000, True),
                     (75700, False), (200003, True), (4096 * 152 + 1, False), (1 << 20, False)):
        assert bench.sweep_apart(n, 152) == apart, n
