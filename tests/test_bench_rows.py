"""What the benchmark counts as bytes of the rows, and which sources a capture of a
prune kernel belongs to."""
import numpy as np

import bench


def test_row_codes_of_the_workloads_and_the_sources_of_their_captures():
    # the bytes of the rooflines: integer rows are read as bytes, real ones as bytes and,
    # where those leave it open, as floats; a capture of the coded prune is of its own file
    g = np.random.default_rng(1)
    ints = [g.integers(0, 256, (50, 128)).astype(np.float32) for _ in range(2)]
    real = [g.standard_normal((50, 96)).astype(np.float32)]
    assert bench.row_codes(ints, 128, bench.L2_METRIC) == "exact"
    assert bench.row_codes(ints, 128, bench.IP_METRIC) == "filter"
    assert bench.row_codes([ints[0], ints[1] + 300.0], 128, bench.L2_METRIC) == "filter"
    assert bench.row_codes(real, 96, bench.L2_METRIC) == "filter"
    assert bench.row_codes([r[:, :32] for r in real], 32, bench.L2_METRIC) == "none"
    assert any(f.endswith("prune_code.cu") for f in bench.prune_sources(4))
    assert any(f.endswith("prune.cu") for f in bench.prune_sources(3))
