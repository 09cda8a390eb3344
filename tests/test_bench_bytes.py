"""The operator's algorithmic bytes that bench.py divides by the time of a forward pass."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench


def test_fused_layers_count_their_own_traffic():
    B, n, C, M = 64, 255, 32, 24
    field, T, modes = 4.0 * B * C * n * n, 4.0 * B * C * M * n, 4.0 * B * C * M * M
    one = bench._sno_forward_bytes(B, n, C, M, 1)
    # a single layer writes and reads no activation: u three times in, u_hat out
    assert one == 4.0 * B * 4 * n * n + 4 * T + 4 * modes
    # each further layer: h out and in once
    for L in range(2, 5):
        assert bench._sno_forward_bytes(B, n, C, M, L) - bench._sno_forward_bytes(B, n, C, M, L - 1) == 2 * field + 4 * T + 4 * modes
    # the workload of 4 layers measured 1.37 ms: no more than the measured copy bandwidth
    assert bench._sno_forward_bytes(B, n, C, M, 4) / 1.37e-3 < 6704.5e9


def test_other_sizes_count_the_unfused_passes():
    B, n, C, M, L = 2, 63, 8, 6, 3
    field, T, modes = 4.0 * B * C * n * n, 4.0 * B * C * M * n, 4.0 * B * C * M * M
    assert bench._sno_forward_bytes(B, n, C, M, L) == 4.0 * B * 3 * n * n + 2 * field + L * (5 * field + 4 * T + 4 * modes)
