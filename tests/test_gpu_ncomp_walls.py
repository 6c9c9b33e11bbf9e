"""The marched N-component step with a solid slab: lattices small enough for the two-launch step are
compared with copies of themselves side by side in y, large enough for the marched one. Two
components, marched, against the two-component step."""
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


def _g(nc):
    return [[0.1 * (a + 1) if a == b else 3.0 + 0.2 * (a + b) for b in range(nc)] for a in range(nc)]


@pytest.mark.parametrize("nc,nx,ny,nz,z0,thick", [(2, 67, 37, 60, 0, 2), (3, 40, 37, 60, 58, 2), (3, 33, 45, 50, 24, 3)])
def test_copies_between_walls_evolve_like_one(sc, nc, nx, ny, nz, z0, thick):
    from paper_1701_03637_gb300.ncomp import NLattice
    copies = 4
    assert 2 * nc * 19 * 4 * nx * ny * nz < 126e6 < 2 * nc * 19 * 4 * nx * ny * nz * copies
    rho = np.random.default_rng(nx).uniform(0.1, 0.6, (nc, nz, ny, nx)).astype(np.float32)
    tau = [0.9 + 0.1 * c for c in range(nc)]
    one = NLattice(nx, ny, nz, tau, _g(nc), wall_z0=z0, wall_thickness=thick)
    many = NLattice(nx, ny * copies, nz, tau, _g(nc), wall_z0=z0, wall_thickness=thick)
    one.init_fields(rho)
    many.init_fields(np.concatenate([rho] * copies, axis=2))
    for lat in (one, many):
        lat.step(7)
    a = one.read_populations()
    b = many.read_populations().reshape(nc, 19, nz, copies, ny, nx)
    assert np.all(np.isfinite(a)) and not a[:, :, z0:z0 + thick].any()
    for k in range(copies):
        assert np.array_equal(b[:, :, :, k], a)


@pytest.mark.parametrize("wall", [0, 3])
def test_marched_two_components_are_the_two_component_step(sc, wall):
    from paper_1701_03637_gb300.ncomp import NLattice
    nx, ny, nz = 97, 83, 56
    assert 2 * 2 * 19 * 4 * nx * ny * nz > 126e6
    g = np.array([[-0.7, 3.2], [3.2, 0.35]])
    rho = np.random.default_rng(5).uniform(0.1, 0.6, (2, nz, ny, nx)).astype(np.float32)
    a = NLattice(nx, ny, nz, [0.95, 1.1], g, wall_z0=20, wall_thickness=wall)
    b = sc.Lattice(dict(nx=nx, ny=ny, nz=nz, tau_r=0.95, tau_b=1.1, G=3.2, G_rr=-0.7, G_bb=0.35, geometry=0, wall_z0=20,
                        wall_thickness=wall, staging="thread"))
    a.init_fields(rho)
    b.init_fields(rho[0], rho[1])
    a.step(9)
    b.step(9)
    assert np.array_equal(a.read_populations(), b.read_populations())
    a.close()
    b.close()
