"""Each form of advancing a network, by name: two kernels per step in a shape
that a caller sets, one launch of the persistent kernel per window in the
default shape.  The launch counts say which form ran; results are the oracle's."""
import pytest

import workloads as W
from parity import assert_same, gpu_results, oracle_results

pytestmark = pytest.mark.gpu


def _launches(nets):
    return sum(g.stats()["kernel_launches"] for g in nets)


def _check(oracle_mod, nets, params, steps):
    for i, (g, p) in enumerate(zip(nets, params)):
        o = oracle_mod.OracleNet(p, 17 + i)
        o.run(steps)
        assert_same(gpu_results(g), oracle_results(o), steps)
        g.close()


@pytest.mark.parametrize("shape", [{"update_block": 128}, {"deliver_lanes": 8, "deliver_warps": 4, "overlap": 0}])
@pytest.mark.parametrize("n_delay,min_delay", [(254, 1), (33, 1), (1, 1), (20, 1), (254, 254), (120, 33), (20, 10), (7, 4)])
def test_two_kernels(oracle_mod, n_delay, min_delay, shape):
    """Delays on both sides of the 32 and 256 steps that a warp's prefix spans,
    exchange periods, windows and calls that start at any step of a period."""
    import paper_1902_08410_gb300 as snn
    nets, params = [], []
    for i in range(2):
        p = W.base_params(3, 2, 0.6, "AW", record_format=i)
        p.update(n_delay=n_delay, min_delay=min_delay)
        params.append(p)
        nets.append(snn.Network(p, 17 + i))
        nets[i].launch = dict(shape, window_steps=61)
    for n in (3, 390, 97, 200):
        before = _launches(nets)
        for g in nets:
            g.run(n)
        assert _launches(nets) - before >= 2 * n
    before = _launches(nets)
    snn.run_concurrent(nets, 70)
    assert _launches(nets) - before >= 2 * 70
    _check(oracle_mod, nets, params, 760)


@pytest.mark.parametrize("grids", [((40, 40),), ((28, 28), (29, 27))])
def test_one_drive_per_neuron(oracle_mod, grids):
    """More than 1.8M neurons in a launch: the external drive is kept for one step only."""
    import paper_1902_08410_gb300 as snn
    nets, params = [], []
    for i, (gx, gy) in enumerate(grids):
        p = W.base_params(gx, gy, 1.0, "AW", record_format=1 - i)
        p.update(out_degree=9, V_th=[10.0] * 3, V_r=[0.0] * 3)   # active with few synapses
        params.append(p)
        nets.append(snn.Network(p, 17 + i))
        nets[i].launch = {"window_steps": 9}
    before = _launches(nets)
    for n in (4, 20, 6):
        snn.run_batch(nets, n)
    assert _launches(nets) - before == 5
    _check(oracle_mod, nets, params, 30)


@pytest.mark.parametrize("min_delay", [1, 6])
@pytest.mark.parametrize("fused_block,fused_items_per_sm", [(128, 1), (256, 1), (128, 3), (512, 32)])
def test_threads_of_path_1(oracle_mod, fused_block, fused_items_per_sm, min_delay):
    import paper_1902_08410_gb300 as snn
    p = dict(W.base_params(3, 2, 0.6, "AW"), min_delay=min_delay)
    g = snn.Network(p, 17)
    g.launch = {"path": 1, "fused_block": fused_block, "fused_items_per_sm": fused_items_per_sm, "window_steps": 50}
    before = _launches([g])
    for n in (7, 200, 93):
        g.run(n)
    assert _launches([g]) - before == 1 + 4 + 2
    _check(oracle_mod, [g], [p], 300)
