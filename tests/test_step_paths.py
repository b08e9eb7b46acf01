"""Step paths that are chosen by size: linear order, two cells a thread on top of
it and of slabs, slabs and FP64 storage with 64-bit population offsets.  A box
periodic along an axis and started from a field of a period that divides it
keeps the period, so it equals the box of one period bit for bit (one cell per
thread, or pairs in both), except where the compiler fuses multiplies and adds
differently in the two kernels."""
import numpy as np
import pytest

from paper_1503_03337_gb300 import build as pkg_build, inputs, lbm

pytestmark = pytest.mark.gpu
P, W, L, SY = lbm.LBM_PERIODIC, lbm.LBM_WALL, lbm.LBM_MOVING_WALL, lbm.LBM_SYMMETRY


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    pkg_build.build()
    return torch


def run_box(torch, Q, shape, storage, faces, edge, u, p, steps, launch=None):
    """Populations after `steps` steps, as FP32 on the device."""
    uw = np.zeros((6, 3))
    uw[5] = (0.05, 0.01, 0.0)
    h = lbm.lbm_create(Q, *shape, storage, torch.cuda.current_stream().cuda_stream)
    try:
        lbm.lbm_set_geometry(h, faces, uw, edge)
        lbm.lbm_set_params(h, nu=0.02, force=(1e-5, -2e-5, 0.0))
        if launch:
            lbm.lbm_set_launch(h, *launch)
        lbm.lbm_init_equilibrium(h, u, p, 1)
        lbm.lbm_step(h, steps)
        out = torch.empty((Q,) + shape[::-1], dtype=torch.float32, device="cuda")
        lbm.lbm_read_fields(h, lbm.LBM_FIELD_POPULATIONS, out, lbm.LBM_DTYPE_F32, 1)
        return out
    finally:
        lbm.lbm_destroy(h)


def check_tiles(torch, Q, shape, tile, storage, faces, steps, edge=None, launch=None, bound=0.0):
    rep = tuple(a // b for a, b in zip(shape, tile))[::-1]
    assert all(a % b == 0 for a, b in zip(shape, tile))
    gen = torch.Generator(device="cuda").manual_seed(Q)
    u = (torch.rand((3,) + tile[::-1], generator=gen, device="cuda", dtype=torch.float64) - 0.5) * 0.04
    p = (torch.rand(tile[::-1], generator=gen, device="cuda", dtype=torch.float64) - 0.5) * 0.02
    small = run_box(torch, Q, tile, storage, faces, edge, u, p, steps, launch)
    big = run_box(torch, Q, shape, storage, faces, edge, u.repeat((1,) + rep).contiguous(),
                  p.repeat(rep).contiguous(), steps, launch)
    top = float(small.abs().max())
    assert bool(torch.isfinite(small).all()) and top > 0.001
    small = small.view((Q, 1, tile[2], 1, tile[1], 1, tile[0]))
    big = big.view((Q, rep[0], tile[2], rep[1], tile[1], rep[2], tile[0]))
    if bound == 0.0:
        assert bool((big == small).all())
    else:
        assert float((big - small).abs().max()) <= bound * top


@pytest.mark.parametrize("Q", (14, 18, 26))
@pytest.mark.parametrize("storage", ("f32", "f16", "bf16"))
@pytest.mark.parametrize("faces,edge", [((W, SY, P, P, W, L), {5: (0, 0.3, 0.7)}),
                                        ((P, P, P, P, SY, L), None)])
@pytest.mark.parametrize("launch", (None, (32, 4, 2)))
def test_linear_order_equals_rows(torch, Q, storage, faces, edge, launch):
    """98 x 96 x 12 cells in linear order against 98 x 8 x 12 by rows: walls, a
    symmetry plane and a lid with an edge profile, or periodic rows.  The two
    odd kernels of D3Q26 FP32 fuse differently (one value in a thousand off by
    one unit a step): either rounds a population by at most some 64 units of
    2^-24 of the largest a step, and steps do not amplify; a wrong slot is off
    by it."""
    bound = 7 * 2 * 64 * 2.0 ** -24 if (Q, storage) == (26, "f32") else 0.0
    check_tiles(torch, Q, (98, 96, 12), (98, 8, 12), storage, faces, 7, edge, launch, bound)


@pytest.mark.parametrize("Q", (14, 18))
def test_bf16_stochastic_linear_order(torch, Q):
    """Random bits go by cell number: linear order against a batched domain."""
    shape, faces = (47, 50, 47), (W, W, W, W, W, L)
    uw = np.zeros((6, 3))
    uw[5] = (0.05, 0.01, 0.0)
    c = inputs.Case("box", Q, *shape, (P,) * 6, np.zeros((6, 3)), nu=0.05)
    u, p = (torch.from_numpy(np.ascontiguousarray(v)).cuda()
            for v in inputs.random_state(c, seed=3, u_scale=0.01, p_scale=0.001))
    stream = torch.cuda.current_stream().cuda_stream
    h = lbm.lbm_create(Q, *shape, "bf16", stream)
    b = lbm.lbm_batch_create(1, 0, stream)
    try:
        lbm.lbm_set_geometry(h, faces, uw)
        lbm.lbm_set_params(h, nu=0.05, rounding=1)
        lbm.lbm_init_equilibrium(h, u, p)
        lbm.lbm_step(h, 21)
        slot = lbm.lbm_batch_add(b, Q, *shape, "bf16", faces, uw, nu=0.05, rounding=1)
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


@pytest.mark.parametrize("Q", (14, 18))
def test_pairs_in_slabs(torch, Q):
    """41 steps in one call (slabs) against single steps (whole sweeps), two
    cells a thread on the even ones."""
    shape = (128, 130, 110)
    L2 = torch.cuda.get_device_properties(0).L2_cache_size
    assert Q * 4 * shape[0] * shape[1] * shape[2] > 0.65 * L2
    c = inputs.Case("box", Q, *shape, (P,) * 6, np.zeros((6, 3)), nu=0.05)
    u, p = (np.ascontiguousarray(v)
            for v in inputs.random_state(c, seed=8, u_scale=0.01, p_scale=0.001))
    got = []
    for calls in ((41,), (1,) * 41):
        h = lbm.lbm_create(Q, *shape, "f32", torch.cuda.current_stream().cuda_stream)
        try:
            lbm.lbm_set_geometry(h, (W, W, P, P, P, P))
            lbm.lbm_set_params(h, nu=0.05)
            lbm.lbm_set_launch(h, 64, 1, 2)
            lbm.lbm_init_equilibrium(h, u, p, 0)
            for n in calls:
                lbm.lbm_step(h, n)
            out = torch.empty(Q * p.size, dtype=torch.float32, device="cuda")
            lbm.lbm_read_fields(h, lbm.LBM_FIELD_POPULATIONS, out, lbm.LBM_DTYPE_F32)
            got.append(out)
        finally:
            lbm.lbm_destroy(h)
    assert bool(torch.isfinite(got[0]).all())
    assert torch.equal(got[0], got[1])


@pytest.mark.parametrize("faces", [(P, P, P, P, W, L), (P,) * 6])
def test_slabs_with_64_bit_offsets(torch, faces):
    """256 x 256 x 1821 D3Q18 FP32: rounds of slabs and a remainder."""
    shape = (256, 256, 1821)
    assert 18 * shape[0] * shape[1] * shape[2] >= 2 ** 31
    check_tiles(torch, 18, shape, (8, 8, 1821), "f32", faces, 15)


def test_fp64_storage_with_64_bit_offsets(torch):
    shape = (330, 600, 603)
    assert 18 * shape[0] * shape[1] * shape[2] >= 2 ** 31
    check_tiles(torch, 18, shape, (11, 8, 603), "f64", (P, P, P, P, W, L), 3)
