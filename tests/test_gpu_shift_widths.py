"""The shifted in-place step against the per-thread two-lattice kernel, which shares none of its
staging: widths whose last tile is half a 16-byte chunk of populations, walls inside the lattice and
across the periodic seam (where a population is read at its own site), every geometry."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,storage,geometry", [
    (66, 1150, 400, "f32", "wall_sink"), (66, 1150, 400, "f32", "mid_wall"), (130, 767, 401, "f32", "sphere"),
    (68, 1150, 207, "f16", "wall_sink"), (68, 1151, 206, "bf16", "mid_wall"), (132, 767, 230, "f16s", "seam_wall"),
    (196, 577, 204, "f16", "sphere")])
def test_shifted_step_has_the_per_thread_bits(nx, ny, nz, storage, geometry):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as sc
    sc.build()
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=0.9, tau_b=1.15, G=3.5, rho_H=0.03, storage=storage, geometry=1, sink_z0=nz - 2, sink_layers=2)
    if geometry == "sphere":
        p.update(geometry=2, sphere_cx=nx / 2.0, sphere_cy=ny / 2.0, sphere_cz=nz / 2.0, R_H=0.45 * min(nx, nz))
    else:
        z0, thick = dict(wall_sink=(0, 2), mid_wall=(nz // 2, 3), seam_wall=(nz - 5, 3))[geometry]
        p.update(wall_z0=z0, wall_thickness=thick)
    a, b = sc.Lattice(dict(p, layout="aa")), sc.Lattice(dict(p, staging="thread"))
    assert "k_shift" in a.kernel_name() and "per-thread" in b.kernel_name()
    r = np.random.default_rng(nx)
    rho = [0.05 + 0.85 * r.random((nz, ny, nx), dtype=np.float32) for _ in range(2)]
    for lat in (a, b):
        lat.init_fields_from(*rho)
    for steps in (1, 2, 6):
        for lat in (a, b):
            lat.step(steps)
        assert torch.equal(a.read_fields_device(), b.read_fields_device())
    a.sync()
    a.close()
    b.close()
