"""Slabs of planes that run several steps each (csrc/lbm_internal.h): the
order of the launches keeps every plane's neighbours at most one step away
(CPU), and a box swept in slabs ends bit for bit where single steps end."""
import os
import subprocess

import numpy as np
import pytest

from paper_1503_03337_gb300 import build as pkg_build, inputs, lbm

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("slabs") / "slab_order")
    subprocess.run([pkg_build.nvcc(), "-std=c++20", "-O1", os.path.join(HERE, "slab_order.cu"),
                    "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("periodic", (0, 1))
@pytest.mark.parametrize("nz,slabs,depth", [(128, 3, 16), (128, 2, 16), (129, 5, 16), (97, 7, 6),
                                            (40, 3, 11), (61, 4, 4), (256, 30, 7)])
def test_launch_order(harness, nz, slabs, depth, periodic):
    """Plane z takes step s once, after planes z +- 1 took s - 1 and before
    either took s + 1 (the in-place update's condition), for whole rounds and
    a remainder of every length."""
    if (nz if periodic else nz - depth) // slabs <= depth:
        pytest.skip("slab_plan gives no such plan")
    for count in range(2 * depth, 3 * depth):
        out = subprocess.run([harness, str(nz), str(periodic), str(slabs), str(depth),
                              str(count)], check=True, capture_output=True, text=True).stdout
        done = [0] * nz
        for line in out.splitlines():
            s, z0, planes = map(int, line.split())
            assert 0 <= z0 < nz and 1 <= planes <= nz
            assert periodic or z0 + planes <= nz
            zs = [(z0 + k) % nz for k in range(planes)]
            for z in zs:
                assert done[z] == s
                for y in (z - 1, z + 1):
                    if periodic or 0 <= y < nz:
                        assert done[y % nz] in (s, s + 1)
            for z in zs:
                done[z] += 1
        assert done == [count] * nz


@pytest.mark.gpu
@pytest.mark.parametrize("flow,Q,shape", [("cavity", 18, (128, 128, 97)),
                                          ("cavity", 14, (160, 150, 100)),
                                          ("cavity", 26, (128, 100, 90)),
                                          ("duct", 18, (131, 131, 83)),
                                          ("porous", 18, (112, 112, 112))])
def test_slabs_same_bits(flow, Q, shape):
    """41 steps in one call (rounds of slabs and a remainder) against 41 calls
    of one step (whole sweeps): the same bits, in boxes beyond the L2 share
    that slabs start at, walls, periodic z and solid nodes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    pkg_build.build()
    nx, ny, nz = shape
    stream = torch.cuda.current_stream().cuda_stream
    if flow == "cavity":
        c = inputs.cavity(Q, nx, 400.0, ny=ny, nz=nz)
    elif flow == "duct":
        c = inputs.duct(Q, nx, nz, 0.05)
    else:
        c = inputs.porous_spheres(Q, nx)
    assert c.cells * Q * 4 > 0.65 * torch.cuda.get_device_properties(0).L2_cache_size
    c.init_u, c.init_p = inputs.random_state(c, seed=8, u_scale=0.01, p_scale=0.001)
    got = []
    for calls in ((41,), (1,) * 41):
        h = lbm.lbm_create(Q, nx, ny, nz, "f32", stream)
        try:
            lbm.lbm_set_geometry(h, c.faces, c.u_wall)
            lbm.lbm_set_params(h, nu=c.nu, force=c.force)
            if c.solid is not None:
                lbm.lbm_set_solid(h, c.solid)
            lbm.lbm_init_equilibrium(h, np.ascontiguousarray(c.init_u),
                                     np.ascontiguousarray(c.init_p), 0)
            for n in calls:
                lbm.lbm_step(h, n)
            out = torch.empty(Q * c.cells, dtype=torch.float32, device="cuda")
            lbm.lbm_read_fields(h, lbm.LBM_FIELD_POPULATIONS, out, lbm.LBM_DTYPE_F32)
            got.append(out)
        finally:
            lbm.lbm_destroy(h)
    assert bool(torch.isfinite(got[0]).all())
    assert torch.equal(got[0], got[1])


@pytest.mark.gpu
def test_batch_slabs_same_bits():
    """A batched domain alone in its L2 cluster is swept in slabs too."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    pkg_build.build()
    stream = torch.cuda.current_stream().cuda_stream
    c = inputs.pulsatile(18, 112, 112, 100, 4.0, 1e-5)
    small = inputs.cavity(18, 24, 100.0)
    b = lbm.lbm_batch_create(2, 0, stream)
    h = lbm.lbm_create(c.Q, c.nx, c.ny, c.nz, "f32", stream)
    try:
        slots = [lbm.lbm_batch_add(b, k.Q, k.nx, k.ny, k.nz, k.storage, k.faces, k.u_wall,
                                   nu=k.nu, force=k.force, force_period=k.period)
                 for k in (c, small)]
        for s in slots:
            lbm.lbm_batch_init_equilibrium(b, s)
        lbm.lbm_batch_step(b, 75, 50)
        lbm.lbm_set_geometry(h, c.faces, c.u_wall)
        lbm.lbm_set_params(h, nu=c.nu, force=c.force, force_period=c.period)
        lbm.lbm_init_equilibrium(h)
        for _ in range(75):
            lbm.lbm_step(h, 1)
        got = [torch.empty(c.Q * c.cells, dtype=torch.float32, device="cuda") for _ in range(2)]
        lbm.lbm_batch_read_fields(b, slots[0], lbm.LBM_FIELD_POPULATIONS, got[0],
                                  lbm.LBM_DTYPE_F32)
        lbm.lbm_read_fields(h, lbm.LBM_FIELD_POPULATIONS, got[1], lbm.LBM_DTYPE_F32)
        assert float(got[0].abs().max()) > 0
        assert torch.equal(got[0], got[1])
    finally:
        lbm.lbm_batch_destroy(b)
        lbm.lbm_destroy(h)
