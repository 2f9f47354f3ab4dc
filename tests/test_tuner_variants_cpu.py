"""The batched sweep times each kernel and march once."""
from paper_1204_4779_gb300 import tuner


def test_batch_variants_are_distinct_kernels():
    # FP32 row tiles (tile_y = 1) run the same strips whatever their width
    runs = [("strip" if tile[1] == 1 else tile, march) for tile, march in tuner.BATCH_VARIANTS]
    assert len(set(runs)) == len(runs)
    assert ("strip", 0) in runs
