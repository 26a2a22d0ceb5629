"""The autotuner tries every family of solver kernels that cfg.tile_kernel selects."""
from paper_2503_16028_gb300 import batch


def test_every_tile_kernel_is_a_candidate():
    assert sorted(c.get("tile_kernel", 0) for c in batch.DEFAULT_CANDIDATES if not c or "tile_kernel" in c) == [0, 1, 2, 3, 4]
