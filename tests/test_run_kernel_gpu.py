"""The persistent kernel at the edges of its bookkeeping, against the oracle.

test_parity_gpu.py runs it at one-step and 254-step delays, exchange periods,
single modules and runs split at every phase; here are the paths those sizes do
not reach.  Integer results must match bit for bit (see parity.py).
"""
import pytest

import workloads as W
from parity import assert_same, gpu_results, oracle_results

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def snn():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1902_08410_gb300 as snn
    snn.build()
    return snn


def _check(oracle_mod, net, p, seed, steps):
    o = oracle_mod.OracleNet(p, seed)
    o.run(steps)
    assert_same(gpu_results(net), oracle_results(o), steps)


@pytest.mark.parametrize("n_delay,min_delay,split", [(6, 1, (7, 3, 14)), (9, 4, (6, 11, 7))])
def test_live_lists_overflow(snn, oracle_mod, n_delay, min_delay, split):
    """A volley of every neuron of a grid near the kernel's largest: more live
    spikes than a block holds, within windows (spilled to the global lists) and
    at their starts (lists not taken over).  Few synapses keep the oracle fast."""
    side = 32 if min_delay == 1 else 16
    p = W.base_params(side, side, 1.0, "AW", record_format=W.REC_I16)
    p.update(out_degree=9, n_delay=n_delay, min_delay=min_delay, V_th=[1.0] * 3, V_r=[0.0] * 3,
             tau_arp=[0.3, 0.2, 0.1])
    g = snn.Network(p, 5)
    for n in split:
        g.run(n)
    _check(oracle_mod, g, p, 5, sum(split))
    g.close()


@pytest.mark.parametrize("delays", [((20, 1), (3, 1), (33, 1), (20, 1)), ((20, 10), (12, 10), (20, 10), (7, 1)),
                                    ((5, 5), (5, 2), (9, 2), (1, 1))])
def test_lockstep_sets(snn, oracle_mod, delays):
    """Networks of unequal delays, sizes and lengths in one call: those that
    stop before the others keep their live spikes, sets of different smallest
    delays or phases take turns."""
    grids = [(1, 1), (3, 2), (1, 4), (2, 2)]
    steps = [[40, 7, 90, 33], [5, 64, 13, 50]]
    nets, params = [], []
    for i, ((gx, gy), (nd, kmin)) in enumerate(zip(grids, delays)):
        p = W.base_params(gx, gy, 0.7, "AW" if i % 2 else "SWA", record_format=i % 2)
        p["n_delay"], p["min_delay"] = nd, kmin
        params.append(p)
        nets.append(snn.Network(p, 60 + i))
    snn.run_batch(nets, steps[0])
    snn.run_concurrent(nets, steps[1])
    for i, (g, p) in enumerate(zip(nets, params)):
        _check(oracle_mod, g, p, 60 + i, steps[0][i] + steps[1][i])
        g.close()


def test_forms_continue_each_other(snn, oracle_mod):
    """Windows of the persistent kernel and of the two-kernel path in turn."""
    p = W.base_params(3, 2, 0.6, "AW")
    g = snn.Network(p, 8)
    two = {"update_block": 128}
    for i, n in enumerate((1, 9, 2, 30, 21, 4, 40, 3)):
        g.launch = two if i % 2 else {"update_block": 256}
        g.run(n)
    _check(oracle_mod, g, p, 8, 110)
    g.close()
