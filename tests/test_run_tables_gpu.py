"""Networks in one launch of the persistent kernel: few, whose descriptors are
copied to shared memory, and so many that they are read from global memory."""
import pytest

import workloads as W
from parity import assert_same, gpu_results, oracle_results

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_nets,min_delay", [(2, 1), (3, 5), (320, 1), (320, 5)])
def test_descriptor_tables(oracle_mod, n_nets, min_delay):
    import paper_1902_08410_gb300 as snn
    p = W.base_params(1, 1, 1.0, "AW")
    p.update(out_degree=40, min_delay=min_delay)
    nets = []
    for i in range(n_nets):
        nets.append(snn.Network(dict(p, record_format=i % 2), 300 + i))
    for n in (45, 32):
        snn.run_batch(nets, [n + (i % 3 if n == 32 else 0) for i in range(n_nets)])
    for i in sorted({0, 1, n_nets // 2, n_nets - 1}):
        o = oracle_mod.OracleNet(dict(p, record_format=i % 2), 300 + i)
        o.run(77 + i % 3)
        assert_same(gpu_results(nets[i]), oracle_results(o), 77 + i % 3)
    for g in nets:
        g.close()
