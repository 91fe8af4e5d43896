"""Algorithmic bytes that bench.py charges (no GPU)."""
import bench


def test_persistent_kernel_is_not_charged_for_state_it_keeps():
    """Two kernels per step move V, c (4 bytes each way), the refractory counter
    (1) and the input (read and cleared, 4 each); the persistent kernel only the input."""
    assert bench.neuron_bytes("concurrent") == 2 * (4 + 4 + 1) + 2 * 4
    assert bench.neuron_bytes("batch") == 2 * 4
