"""The bench's byte model follows the kernels that run."""
import os
import sys
import types

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_automatic_choice_counts_the_bytes_of_its_configuration():
    """kernel = 0 runs as configuration 24 (x every fourth iteration: 74 B per node and system); 18, 22 and
    the boxes as their own iterations per update say."""
    sys.path.insert(0, ROOT)
    import bench

    def b(kernel):
        return bench.algorithmic_bytes(types.SimpleNamespace(kernel=kernel))

    assert b(0) == b(2 + bench.CHUNK_DEFAULT) == b(2 + 24) == 74.0
    assert (b(1), b(2 + 9), b(2 + 18), b(2 + 22)) == (80.0, 80.0, 80.0, 76.0)
