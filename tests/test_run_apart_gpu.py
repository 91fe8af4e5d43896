"""Two large networks through snn_run_concurrent in the default launch shape:
apart on their own streams in calls of two windows or more, in one launch in
shorter ones and when they share a stream; the shape that a caller reads stays the default one."""
import pytest

import workloads as W
from parity import assert_same, gpu_results, oracle_results

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grids,streams", [(((20, 20), (25, 16)), 2), (((20, 20), (25, 16)), 1),
                                           (((20, 20), (19, 21)), 2)])   # 399 modules: below the line
def test_two_large_networks(oracle_mod, grids, streams):
    import torch
    import paper_1902_08410_gb300 as snn
    nets, params = [], []
    st = [torch.cuda.Stream() for _ in range(streams)]
    for i, (gx, gy) in enumerate(grids):
        p = W.base_params(gx, gy, 1.0, "AW", record_format=i)
        p.update(out_degree=9, V_th=[10.0] * 3, V_r=[0.0] * 3)   # active with few synapses
        params.append(p)
        nets.append(snn.Network(p, 80 + i, stream=st[i % streams].cuda_stream))
        nets[i].launch = {"window_steps": 12}
    shape = nets[0].launch
    apart = streams == 2 and all(gx * gy >= 400 for gx, gy in grids)
    for n, two_kernels in ((24, apart), (23, False), (31, apart)):
        before = sum(g.stats()["kernel_launches"] for g in nets)
        snn.run_concurrent(nets, n)
        launches = sum(g.stats()["kernel_launches"] for g in nets) - before
        assert (launches >= 4 * n) == two_kernels
        assert nets[0].launch == shape
    for i, g in enumerate(nets):
        o = oracle_mod.OracleNet(params[i], 80 + i)
        o.run(78)
        assert_same(gpu_results(g), oracle_results(o), 78)
        g.close()
