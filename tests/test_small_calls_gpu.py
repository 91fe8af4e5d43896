"""Calls of a few steps, read after each: the raster entries that come with the
recording block (windows of up to 16 steps, 64 entries), those that are fetched
after it, and the state on both sides of the single-copy limit (64 KiB)."""
import pytest

import workloads as W
from parity import assert_same, gpu_results

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gx,gy,nu", [(2, 2, 4.5), (2, 2, 14.0), (3, 2, 4.5)])
def test_short_windows(oracle_mod, gx, gy, nu):
    import paper_1902_08410_gb300 as snn
    p = W.base_params(gx, gy, 0.4, "AW")
    p["nu_ext"] = [nu] * 3
    calls = [100, 1, 1, 2, 15, 16, 17, 1, 60, 16, 1]
    total = sum(calls)
    g = snn.Network(p, 5)
    for n in calls:
        g.run(n)
    assert_same(gpu_results(g), oracle_mod.simulate(p, 5, total), total, f"{gx}x{gy} nu {nu}")
    g.close()
    # two networks whose windows end at different steps, on the batch path
    nets = [snn.Network(p, 5 + i) for i in range(2)]
    snn.run_batch(nets, [total, total - 130])
    for n in (16, 17, 97):
        snn.run_batch(nets, [0, n])
    for i, g in enumerate(nets):
        assert_same(gpu_results(g), oracle_mod.simulate(p, 5 + i, total), total, f"{gx}x{gy} nu {nu} net {i}")
        g.close()
