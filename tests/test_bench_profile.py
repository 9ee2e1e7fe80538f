"""The phase kernel's committed counters (profiles/) reach the bench line only while every
source file that its code comes from is the one they were taken on."""
import os
import shutil

import pytest

import bench

FIELDS = {"dram_bytes_per_launch", "l2_bytes_per_launch", "l2_throughput_pct"}


@pytest.fixture
def tree(tmp_path):
    """A copy of the sources with counters that belong to them."""
    csrc = tmp_path / "paper_1705_10087_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for name in bench.PHASE_SOURCES:
        shutil.copy(os.path.join(bench.ROOT, "paper_1705_10087_gb300", "csrc", name), csrc)
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / f"phase_kernel_{bench.WORKLOAD}.md").write_text(
        f"kernel_source_sha256_16: {bench.phase_sources_hash(str(tmp_path))}\n"
        "dram_bytes_per_launch: 1e6\nl2_bytes_per_launch: 2e6\nl2_throughput_pct: 3.5\n")
    return tmp_path


def test_counters_of_unchanged_sources_are_used(tree):
    assert set(bench.phase_profile(str(tree))) == FIELDS


@pytest.mark.parametrize("name", ["phase_reg_impl.cuh", "phase_rank.cuh", "packed.cuh",
                                  "csc_internal.cuh", "kernel_phase_reg.cu"])
def test_a_change_in_any_source_drops_them(tree, name):
    with open(tree / "paper_1705_10087_gb300" / "csrc" / name, "a") as f:
        f.write("// changed\n")
    assert bench.phase_profile(str(tree)) == {}
