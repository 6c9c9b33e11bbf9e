"""The shifted in-place step (one lattice moved a few planes through its own storage each
step, the automatic choice in place on tall lattices) reaches the two-lattice step's state bit
for bit: tile edges and remainders in x and y, the smallest heights that take it, walls and
sinks across the periodic seam, every storage type, odd and even step counts, checkpoints in
either of its two positions, and the hand-over to the persistent step."""
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


def _params(nx, ny, nz, storage, geometry):
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=0.9, tau_b=1.15, G=3.5, rho_H=0.03, storage=storage)
    if geometry == "wall_sink":  # the slab touches the seam from below, the sink from above
        p.update(geometry=1, sink_z0=nz - 2, sink_layers=2, wall_z0=0, wall_thickness=2)
    elif geometry == "seam_sink":
        p.update(geometry=1, sink_z0=nz - 1, sink_layers=3)
    elif geometry == "mid_wall":
        p.update(geometry=1, sink_z0=1, sink_layers=1, wall_z0=nz // 2, wall_thickness=3, G_rr=-1.1, G_bb=0.4)
    elif geometry == "sphere":
        p.update(geometry=2, sphere_cx=nx / 2.0, sphere_cy=ny / 2.0, sphere_cz=nz / 2.0, R_H=0.45 * min(nx, nz))
    else:
        p.update(geometry=0)
    return p


def _fields(p, seed):
    r = np.random.default_rng(seed)
    shape = (p["nz"], p["ny"], p["nx"])
    return [(0.05 + 0.85 * r.random(shape, dtype=np.float32)) for _ in range(2)]


SIZES = [  # 576 tile columns of 64 x 4 or more, 21 spare planes or more
    (64, 2301, 400, "f32", "wall_sink"),  # one tile wide, a last tile row of one site
    (68, 1150, 405, "f32", "seam_sink"),  # a ragged second tile of 4 columns
    (256, 577, 403, "f32", "sphere"),
    (72, 1152, 200, "f16", "wall_sink"),
    (200, 578, 207, "bf16", "seam_sink"),
    (136, 767, 230, "f16s", "mid_wall"),
    (512, 288, 201, "bf16", "periodic"),
    (1024, 257, 200, "f16", "sphere"),
]


@pytest.mark.parametrize("nx,ny,nz,storage,geometry", SIZES)
def test_shifted_step_has_the_two_lattice_bits(sc, nx, ny, nz, storage, geometry):
    import torch
    p = _params(nx, ny, nz, storage, geometry)
    rho = _fields(p, nx + ny)
    a, b = sc.Lattice(dict(p, layout="aa")), sc.Lattice(p)
    assert "k_shift" in a.kernel_name()
    for lat in (a, b):
        lat.init_fields_from(*rho)
    for steps in (1, 2, 7, 12):
        for lat in (a, b):
            lat.step(steps)
        assert torch.equal(a.read_fields_device(), b.read_fields_device())
        da, db = a.diagnostics(), b.diagnostics()
        assert da["status"] == 0 and abs(da["evaporated_mass"] - db["evaporated_mass"]) <= 1e-9 * nx * ny * nz
    a.close()
    b.close()


@pytest.mark.parametrize("steps", [2, 3])
def test_states_load_in_either_position(sc, steps):
    import torch
    p = _params(72, 1152, 200, "f16", "wall_sink")
    a, b = sc.Lattice(dict(p, layout="aa")), sc.Lattice(p)
    a.init_fields_from(*_fields(p, 1))
    a.step(steps)
    for lat in (a, b):
        lat.init_fields_from(*_fields(p, 2))
        lat.step(3)
    assert torch.equal(a.read_fields_device(), b.read_fields_device())
    a.close()
    b.close()


def test_bands_hand_the_lattice_to_the_persistent_step(sc):
    p = _params(512, 288, 200, "f16", "seam_sink")
    rho = _fields(p, 3)
    a, b = sc.Lattice(dict(p, layout="aa")), sc.Lattice(p)
    assert "k_shift" in a.kernel_name()
    for lat in (a, b):
        lat.init_fields_from(*rho)
        lat.step(3)
    assert a.persist_bands(2) == 2
    assert a.launch_info()["staging"] == "persistent"
    for lat in (a, b):
        lat.step(2)
        lat.sync()
    for u, v in zip(a.read_fields(), b.read_fields()):
        assert np.array_equal(u, v)
    a.close()
    b.close()


def test_low_lattices_keep_the_other_steps(sc):
    a = sc.Lattice(dict(_params(64, 2304, 300, "f32", "seam_sink"), layout="aa"))
    assert a.launch_info()["staging"] == "persistent"  # a plane of 2^17 sites or more
    a.close()
    a = sc.Lattice(dict(_params(64, 1536, 300, "f32", "seam_sink"), layout="aa"))
    assert a.launch_info()["staging"] == "thread"
    a.close()
