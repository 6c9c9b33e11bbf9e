"""The automatic staging of the two-lattice step: rows only where they were measured faster than
per-thread pulls (large lattices of wide planes), pulls on narrow, flat and L2-resident ones;
and staged rows at the widths that only the automatic choice accepts (a remainder of half a
16-byte chunk of populations) hold the per-thread kernel's bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as mod
    mod.build()
    return mod


def _params(nx, ny, nz, storage, geometry=1):
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=0.9, tau_b=1.1, G=3.4, rho_H=0.03, storage=storage, geometry=geometry)
    if geometry == 1:
        p.update(sink_z0=nz - 1, sink_layers=2, wall_z0=nz // 2, wall_thickness=2)
    else:
        p.update(sphere_cx=nx / 2.0, sphere_cy=ny / 2.0, sphere_cz=nz / 2.0, R_H=0.45 * min(nx, ny, nz))
    return p


@pytest.mark.parametrize("nx,ny,nz,storage,geometry,rows", [
    (6, 6, 256, "f32", 1, False), (8, 8, 256, "f32", 1, False), (10, 10, 128, "f32", 1, False), (12, 12, 128, "f16", 1, False),
    (22, 22, 128, "f32", 1, False), (24, 24, 256, "f32", 1, False), (8, 256, 64, "f32", 1, False), (128, 4, 128, "f32", 1, False),
    (1024, 8, 512, "f32", 1, False), (64, 64, 64, "f32", 1, False), (64, 64, 64, "f16", 1, False), (40, 160, 200, "f32", 1, False),
    (128, 128, 128, "f32", 1, True), (128, 128, 128, "f32", 2, True), (40, 512, 256, "f32", 1, True), (127, 128, 128, "f32", 1, False),
    (256, 256, 256, "bf16", 1, False), (288, 288, 288, "f16", 1, True), (288, 288, 288, "f16", 2, False)])
def test_automatic_staging(sc, nx, ny, nz, storage, geometry, rows):
    lat = sc.Lattice(_params(nx, ny, nz, storage, geometry))
    assert lat.kernel_name() == ("k_step (staged rows)" if rows else "k_step (per-thread pulls)")
    lat.close()


@pytest.mark.parametrize("nx,ny,nz,storage,tile", [
    (66, 130, 100, "f32", 0), (66, 130, 100, "f32", 2), (66, 130, 100, "f32", 5), (98, 66, 131, "f32", 0), (34, 512, 241, "f32", 3),
    (132, 357, 361, "f16", 0), (132, 357, 361, "bf16", 5), (164, 320, 321, "f16s", 0)])
@pytest.mark.parametrize("geometry", [1, 2])
def test_half_chunk_widths_have_the_per_thread_bits(sc, nx, ny, nz, storage, tile, geometry):
    import torch
    if geometry == 2 and storage != "f32":
        pytest.skip("16-bit rows are not chosen with the spherical sink")
    p = _params(nx, ny, nz, storage, geometry)
    r = np.random.default_rng(nx)
    rho = [0.05 + 0.85 * r.random((nz, ny, nx), dtype=np.float32) for _ in range(2)]
    a, b = sc.Lattice(dict(p, tile=tile)), sc.Lattice(dict(p, staging="thread"))
    assert "staged rows" in a.kernel_name() and "per-thread" in b.kernel_name()
    for lat in (a, b):
        lat.init_fields_from(*rho)
    for steps in (1, 2, 5):
        for lat in (a, b):
            lat.step(steps)
        assert torch.equal(a.read_fields_device(), b.read_fields_device())
    for lat in (a, b):
        lat.close()
