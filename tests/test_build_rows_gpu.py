"""Construction at the edges of its bucket sort, every row against the oracle.

Rows are integers (keys) and values rounded once (weights): they match bit for
bit.  Ranges of one delay and of 254, out-degrees around a warp's 32 and 128
draws, thresholds all inside one module or spread over many, ties (few targets,
one delay), and the split of a module's rows over blocks.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,lam,p_local,out_degree,n_delay,min_delay,fmt", [
    ((1, 1), 1.0, 0.8, 1125, 1, 1, W.REC_F32),      # one module, one delay: many equal keys
    ((2, 1), 0.3, 1.0, 127, 254, 1, W.REC_I16),     # nothing leaves the module; two buckets per delay
    ((5, 3), 4.0, 0.0, 129, 40, 39, W.REC_F32),     # everything leaves it, two delays
    ((1, 9), 0.05, -1.0, 33, 20, 1, W.REC_I16),     # thresholds of far modules coincide
    ((7, 6), 50.0, -1.0, 1, 3, 2, W.REC_F32),       # one synapse, flat kernel
])
def test_every_row_of_a_module(oracle_mod, grid, lam, p_local, out_degree, n_delay, min_delay, fmt):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1902_08410_gb300 as snn
    snn.build()
    p = W.base_params(*grid, lam, record_format=fmt, p_local=p_local)
    p.update(out_degree=out_degree, n_delay=n_delay, min_delay=min_delay)
    g, o = snn.Network(p, 77), oracle_mod.OracleNet(p, 77)
    G = grid[0] * grid[1]
    first = (G // 2) * W.K
    for s in np.unique(np.concatenate([np.arange(first, first + W.K), [0, g.N - 1]])):
        gk, gw = g.row(int(s))
        ok, ow = o.row(int(s))
        assert np.array_equal(gk, ok), s
        if fmt == W.REC_I16:
            ow = np.clip(np.rint(ow * np.float32(1024.0)), -32768, 32767).astype(np.float32) / np.float32(1024.0)
        assert np.array_equal(gw, ow), s
    # the delay groups that delivery reads: a run over the longest delay
    g.run(n_delay + 30)
    o.run(n_delay + 30)
    (gs, gi), (os_, oi) = g.spikes(), o.raster()
    assert np.array_equal(gs, os_) and np.array_equal(gi, oi)
    g.close()
