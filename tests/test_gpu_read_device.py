"""Densities read into device memory: the kernel writes the caller's arrays, in either order
and at any distance; overlapping arrays and host memory get the copies they always got."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_device_read_out_into_any_arrays():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as sc
    from paper_1701_03637_gb300._native import load
    sc.build()
    lat = sc.Lattice(dict(nx=12, ny=10, nz=9, tau_r=1.0, tau_b=1.0, G=3.5, rho_H=0.03))
    r = np.random.default_rng(1)
    lat.init_fields_from(*[r.uniform(0.1, 0.9, (9, 10, 12)).astype(np.float32) for _ in range(2)])
    lat.step(3)
    rr, rb = [torch.from_numpy(v).reshape(-1) for v in lat.read_fields()]
    n = 12 * 10 * 9
    read = load().sc_lbm_read_fields_device
    buf = torch.zeros(4 * n, device="cuda")

    def at(k):
        return C.c_void_p(buf.data_ptr() + 4 * k)

    for a, b in ((0, n), (n, 0), (3, 2 * n + 1)):  # disjoint
        assert read(lat._h, at(a), at(b)) == 0
        lat.sync()
        assert torch.equal(buf[a:a + n].cpu(), rr) and torch.equal(buf[b:b + n].cpu(), rb)
    assert read(lat._h, at(0), at(n // 2)) == 0  # overlapping: rho^b is written last
    lat.sync()
    assert torch.equal(buf[:n // 2].cpu(), rr[:n // 2]) and torch.equal(buf[n // 2:n // 2 + n].cpu(), rb)
    pinned = torch.zeros(2 * n).pin_memory()
    assert read(lat._h, C.c_void_p(pinned.data_ptr()), C.c_void_p(pinned.data_ptr() + 4 * n)) == 0
    lat.sync()
    assert torch.equal(pinned[:n], rr) and torch.equal(pinned[n:], rb)
    lat.close()
