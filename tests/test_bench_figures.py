"""Constants behind bench.py's derived figures."""
import os
import sys

from oracle import mlp_ref as M


def test_operations_per_scored_row():
    """Two per weight of the network; its 64 + 64 + 1 biases add none."""
    sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    import bench
    assert bench.MLP_FLOPS_PER_ROW == 2 * (M.NPAR - 64 - 64 - 1)
