"""The flux profile's two forms (Psi of three planes in shared memory for planes of up to 1000
sites, at every neighbour in turn above) against the definition in plain NumPy FP64 on the
state's own populations: plane sizes at the limit, one-site extents, a wall and a sink."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
     (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 5), (4, 4, 125), (3, 7, 9), (25, 40, 6), (7, 143, 5), (33, 31, 5), (40, 30, 4)])
def test_flux_profile_matches_its_definition(nx, ny, nz):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as sc
    sc.build()
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=1.0, tau_b=1.0, G=3.5, G_rr=-0.4, G_bb=0.3, rho_H=0.02, geometry=1, sink_z0=0,
             sink_layers=1, wall_z0=nz - 2, wall_thickness=1)
    lat = sc.Lattice(p)
    r = np.random.default_rng(nx + ny)
    lat.init_fields_from(*[r.uniform(0.1, 0.9, (nz, ny, nx)).astype(np.float32) for _ in range(2)])
    lat.step(3)
    f = lat.read_populations()
    got = lat.flux_profile()
    lat.close()
    rho = f.sum(1)
    solid = np.zeros(nz, bool)
    solid[nz - 2] = True
    psi = np.where(solid[:, None, None], 0.0, 1.0 - np.exp(-rho))
    a, m = np.zeros((2, 3, nz, ny, nx)), np.zeros((2, 3, nz, ny, nx))
    for i, e in enumerate(E):
        s = np.roll(psi, (-e[0], -e[1], -e[2]), (3, 2, 1))  # Psi(x + e)
        for d in range(3):
            a[:, d] += W[i] * e[d] * s
            m[:, d] += e[d] * f[:, i]
    F = [-psi[0] * (3.5 * a[1] - 0.4 * a[0]), -psi[1] * (3.5 * a[0] + 0.3 * a[1])]
    with np.errstate(divide="ignore", invalid="ignore"):
        U = (m[0] + m[1] + 0.5 * (F[0] + F[1])) / (rho[0] + rho[1])
        Ur = (m[0] + F[0] + rho[0] * (m[0] + m[1]) / (rho[0] + rho[1])) / (2 * rho[0])
        j = rho[0] * (Ur - U)
    j[:, solid] = 0.0
    j[:, 0] = 0.0
    # the kernel's weights are the FP32 ones' doubles or 1/18, 1/36: differences of 1e-7 of the force
    assert np.max(np.abs(got - j.mean((2, 3)))) < 1e-6
