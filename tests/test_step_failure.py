"""A step launch that fails: what run_slabs reports of the steps before it (CPU,
every launch of a run failing in turn), and the handle's counter after it."""
import os
import subprocess

import numpy as np
import pytest

from paper_1503_03337_gb300 import build as pkg_build, lbm

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("failure") / "step_failure")
    subprocess.run([pkg_build.nvcc(), "-std=c++20", "-O1", os.path.join(HERE, "step_failure.cu"),
                    "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("periodic", (0, 1))
@pytest.mark.parametrize("nz,slabs,depth,count", [(64, 1, 1, 9), (128, 3, 16, 40), (97, 7, 6, 15),
                                                  (40, 2, 11, 25)])
def test_progress_reported(harness, nz, slabs, depth, count, periodic):
    """Torn exactly where planes are at different steps; otherwise the steps
    that every plane has taken."""
    out = subprocess.run([harness] + [str(v) for v in (nz, periodic, slabs, depth, count)],
                         check=True, capture_output=True, text=True).stdout
    lines = [tuple(map(int, line.split())) for line in out.splitlines()]
    assert len(lines) > count
    for steps, torn, least, most, error in lines:
        assert torn == (least != most)
        assert steps == least if not torn else steps <= least
    assert lines[-1] == (count, 0, count, count, 0)
    assert all(line[4] != 0 for line in lines[:-1])
    assert slabs == 1 or any(line[1] for line in lines)


@pytest.mark.gpu
def test_counter_names_the_last_queued_step():
    """2 x 70000 cells: odd steps run in linear order; the pair kernel of the
    even ones goes by rows, and with one row a block the runtime refuses its
    grid (y above 65535).  The odd step before it counts, and stepping on
    with a valid block ends where an undisturbed run ends."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    pkg_build.build()
    stream = torch.cuda.current_stream().cuda_stream
    rng = np.random.default_rng(6)
    u, p = rng.uniform(-0.02, 0.02, (3, 1, 70000, 2)), rng.uniform(-0.01, 0.01, (1, 70000, 2))
    got = []
    for fail in (True, False):
        h = lbm.lbm_create(18, 2, 70000, 1, "f32", stream)
        try:
            lbm.lbm_set_geometry(h, (lbm.LBM_PERIODIC,) * 6)
            lbm.lbm_set_params(h, nu=0.05)
            lbm.lbm_init_equilibrium(h, u, p, 0)
            lbm.lbm_step(h, 1)
            if fail:
                lbm.lbm_set_launch(h, 32, 1, 2)
                with pytest.raises(lbm.LBMError) as ei:
                    lbm.lbm_step(h, 3)
                assert ei.value.code == lbm.LBM_ECUDA
                assert lbm.lbm_get_step(h) == 2
                lbm.lbm_set_launch(h, 128, 1, 1)
            lbm.lbm_step(h, 5 - lbm.lbm_get_step(h))
            got.append(lbm.read_populations(h, 18, 2, 70000, 1))
        finally:
            lbm.lbm_destroy(h)
    np.testing.assert_array_equal(got[0], got[1])
