"""The DRAM traffic that the bench reports beside its rooflines is taken where the working set exceeds L2 by far:
no column moves less than it must (12 M bytes for a half-sweep, 24 M for each kernel of the defect; a launch
may leave the last percent of what it writes in L2), and re-reads stay below a fifth."""
import pytest

import bench


@pytest.mark.parametrize("kind,bytes_per_level", [("smooth", 12), ("defect", 48)])
def test_traffic_is_not_below_the_algorithmic_bytes(kind, bytes_per_level):
    M, per_column = bench.TRAFFIC_PER_COLUMN[kind]
    assert 0.99 * bytes_per_level * M <= per_column <= 1.2 * bytes_per_level * M
