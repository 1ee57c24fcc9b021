"""DRAM bytes per pair of the default M = 256 kernel against the data it must move (on the CPU)."""
import json
import os

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_traffic_of_the_m256_kernel_is_close_to_the_algorithmic_bytes():
    """The 16-bit particle fragments once (64 B per k-step and row, shared by the references), 8 B of row
    maxima per pair; the margins are those of the other kernels' entries."""
    entry = json.load(open(os.path.join(ROOT, "profiles", "traffic.json")))["cc_hybrid256_kernel"]
    steps = 3 + 16 * 13  # f = 0, then 8 warps x 2 parities x {3, 2, 2, 2, 1, 1, 1, 1}
    needed = steps * 64 / 100 + 8  # K = 100
    assert 0.97 * needed <= entry["bytes_per_unit"] <= 1.2 * needed
    # the kernel reads as many k-steps as the rings need: none is padding for rings 1..35
    rings = bench.ring_table(1, 35, 1)
    assert steps == sum(-(-sum(1 for _, n in rings if n // 2 >= f) // 16) for f in range(129))
