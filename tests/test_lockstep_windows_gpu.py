"""Networks of unequal lengths in one launch per window, over several windows
and calls: those that stop first, or do not advance at all, leave the others'
exchange periods where they are."""
import pytest

import workloads as W
from parity import assert_same, gpu_results, oracle_results

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window", [12, 64])
@pytest.mark.parametrize("min_delay,calls", [(10, [(105, 700, 333), (0, 41, 7), (50, 9, 320)]),
                                             (3, [(10, 0, 200), (65, 130, 1)]), (1, [(10, 0, 200), (65, 130, 1)])])
@pytest.mark.parametrize("run", ["run_batch", "run_concurrent"])
def test_unequal_lengths(oracle_mod, min_delay, calls, window, run):
    import paper_1902_08410_gb300 as snn
    nets, params = [], []
    for i, (gx, gy) in enumerate(((1, 1), (3, 2), (2, 1))):
        p = W.base_params(gx, gy, 0.7, "AW", record_format=i % 2)
        p["min_delay"] = min_delay
        params.append(p)
        nets.append(snn.Network(p, 90 + i))
        nets[i].launch = {"window_steps": window}
    for steps in calls:
        getattr(snn, run)(nets, steps)
    for i, g in enumerate(nets):
        n = sum(c[i] for c in calls)
        o = oracle_mod.OracleNet(params[i], 90 + i)
        o.run(n)
        assert_same(gpu_results(g), oracle_results(o), n)
        g.close()


def test_server_with_exchange_periods():
    """Served networks of one smallest delay that end at any step."""
    import numpy as np
    import paper_1902_08410_gb300 as snn
    from paper_1902_08410_gb300.serve import Server
    p = dict(W.base_params(2, 2, 0.7, "AW"), min_delay=10)
    lengths = [1205, 3300, 2777, 600]
    srv = Server(memory_budget=8 << 30, chunk_steps=2500, realtime=False)
    for i, n in enumerate(lengths):
        srv.submit(p, 20 + i, n)
    out = srv.run()["results"]
    for i, n in enumerate(lengths):
        g = snn.Network(p, 20 + i)
        g.run(n)
        st, ids = g.spikes()
        assert len(st) and np.array_equal(out[i].spike_steps, st) and np.array_equal(out[i].spike_ids, ids)
        assert np.array_equal(out[i].rates, g.rates())
        g.close()


def test_networks_beyond_one_launch(oracle_mod):
    """Two networks too large for the persistent kernel and a small one, all on
    one stream: the large ones advance side by side on streams of their own."""
    import paper_1902_08410_gb300 as snn
    nets, params = [], []
    for i, (gx, gy) in enumerate(((44, 44), (2, 2), (45, 43))):
        p = W.base_params(gx, gy, 1.0, "AW", record_format=i % 2)
        p.update(out_degree=9, V_th=[10.0] * 3, V_r=[0.0] * 3)   # active with few synapses
        params.append(p)
        nets.append(snn.Network(p, 70 + i))
        nets[i].launch = {"window_steps": 8}
    for run, steps in (("run_batch", (19, 21, 10)), ("run_concurrent", (7, 3, 12))):
        getattr(snn, run)(nets, steps)
    for i, (g, n) in enumerate(zip(nets, (26, 24, 22))):
        o = oracle_mod.OracleNet(params[i], 70 + i)
        o.run(n)
        assert_same(gpu_results(g), oracle_results(o), n)
        g.close()


@pytest.mark.parametrize("grids,n_delay,min_delay,volley,calls", [
    (((4, 4), (5, 4), (4, 4)), 254, 254, False, [(600, 333, 0), (45, 1300, 777)]),
    (((8, 8), (8, 9)), 120, 100, False, [(150, 130), (7, 95)]),
    (((16, 16), (16, 15)), 33, 30, True, [(22, 35), (41, 9)])])
def test_part_of_an_exchange_period(oracle_mod, grids, n_delay, min_delay, volley, calls):
    """Sets whose networks do not fit a launch with the drives of a whole
    exchange period: the grid meets within the period too.  Networks that stop
    at any step, in the second call networks of different phases, and more live
    spikes than the lists hold."""
    import paper_1902_08410_gb300 as snn
    nets, params = [], []
    for i, (gx, gy) in enumerate(grids):
        p = W.base_params(gx, gy, 1.0, "AW", record_format=i % 2)
        p.update(out_degree=9 if volley else 40, n_delay=n_delay, min_delay=min_delay)
        p.update(V_th=[1.0] * 3 if volley else [10.0] * 3, V_r=[0.0] * 3)
        if volley:
            p["tau_arp"] = [0.3, 0.2, 0.1]
        params.append(p)
        nets.append(snn.Network(p, 30 + i))
    for j, steps in enumerate(calls):
        before = sum(g.stats()["kernel_launches"] for g in nets)
        snn.run_batch(nets, steps)
        if j == 0:   # in one phase: a launch per window, not per step
            assert sum(g.stats()["kernel_launches"] for g in nets) - before <= 4
    for i, g in enumerate(nets):
        n = sum(c[i] for c in calls)
        o = oracle_mod.OracleNet(params[i], 30 + i)
        o.run(n)
        assert_same(gpu_results(g), oracle_results(o), n)
        g.close()
