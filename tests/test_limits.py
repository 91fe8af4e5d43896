"""Limits of the parameters, on the host (no GPU)."""
import pytest

import workloads as W


def test_out_degree_limit():
    """2048 synapses per neuron are accepted, one more is beyond the limit."""
    import paper_1902_08410_gb300 as snn
    snn.build()
    p = W.base_params(1, 1, 1.0)
    assert snn.footprint(dict(p, out_degree=2048)) > 1250 * 2048 * 8
    with pytest.raises(snn.SnnError) as ei:
        snn.footprint(dict(p, out_degree=2049))
    assert ei.value.code == -6
