"""Single steps of lattices of one or a few sites per plane: nearly empty tiles would make the
two-lattice launch the slower one, so these calls stay with the resident launch."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 2000), (1, 2, 4000), (1, 8, 1000)])
def test_single_steps_of_narrow_columns(nx, ny, nz):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as sc
    sc.build()
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=0.9, tau_b=1.1, G=3.4, rho_H=0.03, geometry=1, sink_z0=nz - 1, sink_layers=1)
    r = np.random.default_rng(nz)
    rho = [r.uniform(0.05, 0.9, (nz, ny, nx)).astype(np.float32) for _ in range(2)]
    lats = [sc.Lattice(p), sc.Lattice(dict(p, staging="thread"))]
    took, got = [], []
    for lat in lats:
        lat.init_fields_from(*rho)
        for n in (1, 3, 1, 1, 2):
            lat.step(n)
        got.append(lat.read_populations())
        best = 1.0
        for _ in range(12):
            lat.sync()
            t = time.perf_counter()
            for _ in range(40):
                lat.step(1)
            lat.sync()
            best = min(best, time.perf_counter() - t)
        took.append(best)
        lat.close()
    assert np.array_equal(got[0], got[1])
    assert took[0] <= 0.85 * took[1]  # 0.3 to 0.75 by launch times; 1.0 when both take the same launch
