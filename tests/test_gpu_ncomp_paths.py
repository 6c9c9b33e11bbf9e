"""The N-component step's two forms (two launches, a site per thread, where both buffers fit the
L2; the marched one beyond) give the same bits: a periodic lattice and four copies of it on top
of one another, large enough for the marched step, evolve alike."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc,nx,ny,nz", [(2, 67, 37, 60), (3, 40, 37, 60), (3, 33, 45, 50)])
def test_stacked_copies_evolve_like_one(nc, nx, ny, nz):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as sc
    from paper_1701_03637_gb300.ncomp import NLattice
    sc.build()
    copies = 4
    assert 2 * nc * 19 * 4 * nx * ny * nz < 126e6 < 2 * nc * 19 * 4 * nx * ny * nz * copies
    rho = np.random.default_rng(nx).uniform(0.1, 0.6, (nc, nz, ny, nx)).astype(np.float32)
    g = [[0.1 * (a + 1) if a == b else 3.0 + 0.2 * (a + b) for b in range(nc)] for a in range(nc)]
    tau = [0.9 + 0.1 * c for c in range(nc)]
    one, many = NLattice(nx, ny, nz, tau, g), NLattice(nx, ny, nz * copies, tau, g)
    one.init_fields(rho)
    many.init_fields(np.concatenate([rho] * copies, axis=1))
    for lat in (one, many):
        lat.step(7)
    a = np.asarray(one.read_populations()).reshape(nc, 19, nz, ny, nx)
    b = np.asarray(many.read_populations()).reshape(nc, 19, copies, nz, ny, nx)
    assert np.all(np.isfinite(a))
    for k in range(copies):
        assert np.array_equal(b[:, :, k], a)
