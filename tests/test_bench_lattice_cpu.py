"""CPU checks of what bench.py says about a lattice solve of the 3D grid: the kernel's own byte model, no split into the
list solver's phases, and DRAM traffic only from a profile of that kernel at these sources."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

STATS = dict(scans_discharge=1000, scans_discharge_residual=700, pushes=100, visits_discharge=50, scans_bfs=400, visits_bfs=30,
             global_relabels=2, discharge_ms=2.0, relabel_ms=1.0, rounds=7, bfs_levels=5, rounds_by_size=[0, 0, 0, 0])


def roofline(stats, traffic_of=lambda kernel: None):
    return bench.grid_roofline([stats], 10, 40, (16, 9, 8), 2.0, 100.0, "measured", traffic_of)


def test_lattice_solves_have_a_byte_model_of_their_own():
    r = roofline(STATS)
    cells = 2 * 2 * 1 * 512
    assert r["kernel"] == "mf::lattice3_kernel" and r["bound"] == "latency" and r["phases"] is None
    assert r["model_bytes_per_launch"] == 22528 * 7 + 4608 * 5 + 45 * cells * 2 + 45 * cells + 24 * 40 + 8 * 10
    assert r["achieved"] == pytest.approx(r["model_bytes_per_launch"] / 2.0e6)
    r = roofline(dict(STATS, rounds_by_size=[7, 0, 0, 0]))
    assert r["kernel"] == "mf::solve_kernel" and r["bound"] == "hbm" and r["phases"]
    assert r["model_bytes_per_launch"] == bench.model_bytes(STATS, 10, 40)


def test_traffic_comes_from_a_profile_of_the_kernel_that_ran():
    asked = []
    r = roofline(STATS, lambda kernel: asked.append(kernel) or 4e6)
    assert asked == ["mf::lattice3_kernel"] and r["traffic"] == 4e6 and r["traffic_GBps"] == pytest.approx(2.0)
    assert {"mf_lattice3.cu", "mf_lattice.cuh", "mf_tile_queue.cuh"} <= set(bench.KERNEL_SOURCES["mf::lattice3_kernel"])
    for kernel in bench.KERNEL_SOURCES:  # a stored profile counts only at the sources it was taken at
        p = os.path.join(ROOT, "profiles", kernel.split("::")[1] + "_grid3d_256x256x128.json")
        rec = json.load(open(p)) if os.path.exists(p) else {}
        same = rec.get("kernel_source_sha256_16") == bench.kernel_source_hash(kernel)
        assert bench.stored_traffic(kernel) == (rec["dram_bytes_per_launch"] if same else None)
