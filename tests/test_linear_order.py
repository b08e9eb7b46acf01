"""Steps whose cells run in linear order (k_step_line): the multiplication that
divides cell numbers (CPU), the same bits as the batched path's rows, and
boxes with solid nodes against FP64 storage."""
import os
import subprocess

import numpy as np
import pytest

from paper_1503_03337_gb300 import build as pkg_build, inputs, lbm

HERE = os.path.dirname(os.path.abspath(__file__))
P, W, L, SY = 0, 1, 2, 3


def test_fast_div(tmp_path):
    exe = str(tmp_path / "fast_div")
    subprocess.run([pkg_build.nvcc(), "-std=c++20", "-O1", os.path.join(HERE, "fast_div.cu"),
                    "-o", exe], check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout == "0\n"


def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    pkg_build.build()
    return torch


def state(torch, Q, shape, seed):
    c = inputs.Case("box", Q, *shape, (P,) * 6, np.zeros((6, 3)), nu=0.05)
    return [torch.from_numpy(np.ascontiguousarray(v)).cuda()
            for v in inputs.random_state(c, seed=seed, u_scale=0.01, p_scale=0.001)]


@pytest.mark.gpu
@pytest.mark.parametrize("Q", (14, 18))
@pytest.mark.parametrize("storage,sr", (("f32", 0), ("f16", 1)))
@pytest.mark.parametrize("shape,faces", [((47, 47, 47), (W, W, W, L, W, W)),
                                         ((33, 64, 50), (P, P, W, W, P, P)),
                                         ((95, 40, 27), (W, W, W, L, W, SY)),
                                         ((2, 300, 170), (P, P, W, W, W, W)),
                                         ((129, 131, 79), (W, W, W, W, P, P))])
def test_same_bits_as_batched_rows(Q, storage, sr, shape, faces):
    """Walls, a moving lid, periodic axes and a symmetry plane, an odd number
    of steps with a force: the populations of a batched domain."""
    torch = gpu()
    stream = torch.cuda.current_stream().cuda_stream
    uw = np.zeros((6, 3))
    uw[3, 0] = 0.05
    u, p = state(torch, Q, shape, 3)
    F = (1e-5, 0.0, 2e-5)
    h = lbm.lbm_create(Q, *shape, storage, stream)
    b = lbm.lbm_batch_create(1, 0, stream)
    try:
        lbm.lbm_set_geometry(h, faces, uw)
        lbm.lbm_set_params(h, nu=0.05, force=F, rounding=sr)
        lbm.lbm_init_equilibrium(h, u, p)
        lbm.lbm_step(h, 21)
        slot = lbm.lbm_batch_add(b, Q, *shape, storage, faces, uw, nu=0.05, force=F, rounding=sr)
        lbm.lbm_batch_init_equilibrium(b, slot, u, p)
        lbm.lbm_batch_step(b, 21, 50)
        got = [torch.empty(Q * p.numel(), dtype=torch.float32, device="cuda") for _ in range(2)]
        lbm.lbm_read_fields(h, lbm.LBM_FIELD_POPULATIONS, got[0], lbm.LBM_DTYPE_F32)
        lbm.lbm_batch_read_fields(b, slot, lbm.LBM_FIELD_POPULATIONS, got[1], lbm.LBM_DTYPE_F32)
        assert bool(torch.isfinite(got[0]).all())
        assert torch.equal(got[0], got[1])
    finally:
        lbm.lbm_destroy(h)
        lbm.lbm_batch_destroy(b)


@pytest.mark.gpu
@pytest.mark.parametrize("Q", (14, 18, 26))
@pytest.mark.parametrize("shape,faces", [((1, 40, 40), (P,) * 6), ((40, 1, 40), (P,) * 6),
                                         ((64, 30, 20), (W, W, W, L, P, P)),
                                         ((61, 30, 20), (P, P, W, W, W, SY)),
                                         ((47, 47, 47), (P,) * 6)])
def test_solids_match_fp64_storage(Q, shape, faces):
    """21 FP32 steps with random solid nodes against FP64 storage.  A step
    rounds a population by at most some 64 units of 2^-24 of the largest, and
    steps do not amplify: 21 * 64 * 2^-24 of it; a wrong slot is off by it."""
    torch = gpu()
    stream = torch.cuda.current_stream().cuda_stream
    uw = np.zeros((6, 3))
    uw[3, 0] = 0.05
    u, p = state(torch, Q, shape, 4)
    solid = (np.random.default_rng(5).random(shape[::-1]) < 0.2).astype(np.uint8)
    got = []
    for storage in ("f32", "f64"):
        h = lbm.lbm_create(Q, *shape, storage, stream)
        try:
            lbm.lbm_set_geometry(h, faces, uw)
            lbm.lbm_set_params(h, nu=0.05)
            lbm.lbm_set_solid(h, solid)
            lbm.lbm_init_equilibrium(h, u, p)
            lbm.lbm_step(h, 21)
            out = torch.empty(Q * solid.size, dtype=torch.float64, device="cuda")
            lbm.lbm_read_fields(h, lbm.LBM_FIELD_POPULATIONS, out)
            got.append(out)
        finally:
            lbm.lbm_destroy(h)
    top = float(got[1].abs().max())
    assert 0 < top < 1
    assert float((got[0] - got[1]).abs().max()) <= 21 * 64 * 2.0 ** -24 * top
