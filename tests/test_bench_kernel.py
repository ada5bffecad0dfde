"""bench.py names the kernel that ran (no GPU): the one whose launches an ncu launch list is searched for."""
import pytest

import bench

TUNE = {"block_min_deg": 0, "merge_ratio": 0}


@pytest.mark.parametrize("variant,tune,caches,name", [
    ("persistent", TUNE, 0, "k_persistent_smp"), ("persistent", TUNE, 3, "k_persistent"),
    ("persistent", dict(TUNE, merge_ratio=10), 0, "k_persistent"),
    ("persistent", dict(TUNE, block_min_deg=1024), 3, "k_persistent_blk"),
    ("binned", TUNE, 0, "k_binned_step"), ("plain", TUNE, 3, "k_plain_step"),
])
def test_kernel_of_a_run(variant, tune, caches, name):
    assert bench.sampler_kernel(variant, tune, caches) == name
