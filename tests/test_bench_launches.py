"""bench.py against the library's step sources: the hash that guards the recorded
DRAM traffic covers every unit and the launch order, and the launch count is
that of slab_plan and run_slabs (no GPU)."""
import os
import re
import subprocess

import pytest

import bench
from paper_1503_03337_gb300 import build as pkg_build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_hash_covers_every_step_unit_and_the_launch_order(tmp_path, monkeypatch):
    """A changed byte in any of them changes the hash."""
    names = [f for f in os.listdir(pkg_build.CSRC) if re.fullmatch(r"lbm_step\w*\.cuh?", f)]
    assert len(names) >= 20
    csrc = tmp_path / "paper_1503_03337_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for f in os.listdir(pkg_build.CSRC):
        (csrc / f).write_bytes(open(os.path.join(pkg_build.CSRC, f), "rb").read())
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    base = bench.kernel_source_hash()
    for f in names + ["lbm_internal.h", "lbm_kernels.cuh"]:
        whole = (csrc / f).read_bytes()
        (csrc / f).write_bytes(whole + b"\n")
        assert bench.kernel_source_hash() != base, f
        (csrc / f).write_bytes(whole)
    assert bench.kernel_source_hash() == base


@pytest.mark.parametrize("l2", (50 << 20, 132644864, 256 << 20))
def test_launch_count_is_the_librarys(tmp_path_factory, l2):
    exe = str(tmp_path_factory.mktemp("launches") / "launch_rules")
    subprocess.run([pkg_build.nvcc(), "-std=c++20", "-O1", "--expt-relaxed-constexpr",
                    os.path.join(HERE, "launch_rules.cu"), "-o", exe], check=True)
    cases = [(Q, n, updates) for Q in (14, 18, 26) for n in (33, 100, 128, 160, 208, 224, 256, 320, 400)
             for updates in (1, 3, 7, 100, 1000)]
    out = subprocess.run([exe], check=True, capture_output=True, text=True, input="\n".join(
        "count %d %d %d %d 1 %d %d" % (Q, n, n, n, updates, l2) for Q, n, updates in cases)).stdout
    assert [bench.step_launches(Q, "f32", n, updates, l2) for Q, n, updates in cases] == \
        [int(line) for line in out.split()]
