"""Launch rules of single-domain steps (csrc/lbm_step.cu): the default block of
boxes with 64-bit population offsets and what the autotuner times (CPU), and
steps of a wide box whose rows are not whole warps."""
import os
import subprocess

import numpy as np
import pytest

from paper_1503_03337_gb300 import build as pkg_build, lbm

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("rules") / "launch_rules")
    subprocess.run([pkg_build.nvcc(), "-std=c++20", "-O1", "--expt-relaxed-constexpr",
                    os.path.join(HERE, "launch_rules.cu"), "-o", exe], check=True)

    def ask(text):
        out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return ask


@pytest.mark.parametrize("Q,nx,ny,nz,storage", [
    (18, 33, 70000, 52, "f16"), (14, 47, 100001, 33, "f32"), (26, 31, 70001, 40, "bf16"),
    (18, 1000, 400, 300, "f32"), (14, 129, 65535, 20, "f16"), (18, 63, 70000, 30, "f32")])
def test_wide_boxes_keep_the_row_block(harness, Q, nx, ny, nz, storage):
    """Boxes with Q*N >= 2^31 step by rows (k_step with 64-bit offsets), one
    block row per `by` rows of the box: the row block, whose grid fits the y
    limit wherever it did before linear order."""
    assert Q * nx * ny * nz >= 2 ** 31
    (bx, by, linear), = harness("block %d %d %d %d %d" % (Q, nx, ny, nz, lbm.STORAGE_NAMES[storage]))
    assert not linear
    assert bx == min(128, max(32, 1 << (nx - 1).bit_length())) and bx * by == 256
    assert -(-ny // by) <= 65535


def test_autotuner_times_what_steps_run(harness):
    """A choice is shared only by boxes that run the same kernels in the same
    order; two cells a thread are timed only where a step uses them; boxes
    with extrapolation faces step in whole sweeps, and slabs are timed in
    whole rounds with as many even as odd steps."""
    L2 = 135 << 20
    cases = [(18, 128, 128, 128, 1) + rest for rest in ((0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1))]
    cases += [(18, 64, 64, 64, 2, 0, 0, 0), (18, 64, 64, 64, 2, 1, 0, 0), (14, 280, 280, 64, 1, 0, 0, 0)]
    got = harness("\n".join("tune %d %d %d %d %d %d %d %d 8 %d" % (c + (L2,)) for c in cases))
    plans, steps, pairs, keys = ([g[:2] for g in got], [g[2] for g in got], [g[3] for g in got],
                                 [g[4:] for g in got])
    assert len(set(keys)) == len(keys)
    assert plans[0][0] > 1 and plans[1][0] > 1 and plans[2][0] > 1
    assert plans[3] == plans[4] == plans[5] == (1, 1)
    for (slabs, depth), n in zip(plans, steps):
        assert n >= 8 and n % 2 == 0 and (slabs == 1 or n % depth == 0)
    assert plans[6][0] > 1 and plans[6][1] % 2 == 1
    assert [p > 0 for p in pairs] == [True, False, True, True, True, False, True]


def test_only_fp32_storage_is_swept_in_slabs(harness):
    """The kernels of the other storage types ignore a launch's first plane."""
    L2 = 135 << 20
    got = harness("\n".join("tune %d %d %d 128 %d 0 %d 0 8 %d" % (Q, n, n, storage, per, L2)
                            for storage in (lbm.LBM_STORAGE_F64, lbm.LBM_STORAGE_F16,
                                            lbm.LBM_STORAGE_BF16)
                            for Q in (14, 18, 26) for n in (64, 100, 128, 256) for per in (0, 1)))
    assert all(g[:2] == (1, 1) for g in got) and len(got) == 72


@pytest.mark.gpu
@pytest.mark.parametrize("Q,nx,ny,nz", [(18, 33, 70000, 52), (14, 500, 560, 550)])
def test_wide_box_with_ragged_rows(Q, nx, ny, nz):
    """Such a box, periodic in x and y and started from a field of period 11 or
    10 in x and 8 in y, equals its tiles bit for bit (FP16, an odd step count,
    walls and a moving lid on z)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    pkg_build.build()
    mx, my = (11 if nx % 11 == 0 else 10), 8
    assert Q * nx * ny * nz >= 2 ** 31 and nx % 32 and nx % mx == 0 and ny % my == 0
    gen = torch.Generator(device="cuda").manual_seed(Q)
    us = (torch.rand((3, nz, my, mx), generator=gen, device="cuda", dtype=torch.float64) - 0.5) * 0.04
    ps = (torch.rand((nz, my, mx), generator=gen, device="cuda", dtype=torch.float64) - 0.5) * 0.02
    uw = np.zeros((6, 3))
    uw[5] = (0.05, 0.01, 0.0)
    rep = (1, ny // my, nx // mx)
    got = []
    for shape, u, p in (((nx, ny, nz), us.repeat((1,) + rep).contiguous(), ps.repeat(rep).contiguous()),
                        ((mx, my, nz), us, ps)):
        h = lbm.lbm_create(Q, *shape, "f16", torch.cuda.current_stream().cuda_stream)
        try:
            lbm.lbm_set_geometry(h, (lbm.LBM_PERIODIC,) * 4 + (lbm.LBM_WALL, lbm.LBM_MOVING_WALL), uw)
            lbm.lbm_set_params(h, nu=0.02, force=(1e-5, -2e-5, 0.0))
            lbm.lbm_init_equilibrium(h, u, p, 1)
            lbm.lbm_step(h, 3)
            out = torch.empty((3,) + shape[::-1], dtype=torch.float32, device="cuda")
            lbm.lbm_read_fields(h, lbm.LBM_FIELD_U, out, lbm.LBM_DTYPE_F32, 1)
            got.append(out)
        finally:
            lbm.lbm_destroy(h)
        del u, p
    tiled = got[1].repeat((1,) + rep)
    assert bool(torch.isfinite(got[0]).all()) and float(got[0].abs().max()) > 0.01
    assert torch.equal(got[0], tiled)
