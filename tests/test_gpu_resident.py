"""The resident step (a whole small lattice in the shared memory of one cluster) and the
staged rows reach the per-thread kernel's state bit for bit: cluster sizes 1 to 16, sites that
do not fill the last CTA, extents of 1 and 2, and the largest lattice the cluster holds; tile
edges and remainders of the staged rows; sites exactly on the spherical sink's radius."""
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


def _fields(p, seed):
    r = np.random.default_rng(seed)
    shape = (p["nz"], p["ny"], p["nx"])
    return [r.uniform(0.05, 0.9, shape).astype(np.float32) for _ in range(2)]


def _same(sc, p, kinds, steps):
    ref = None
    for kind in kinds:
        lat = sc.Lattice(dict(p, **kind))
        lat.init_fields_from(*_fields(p, p["nx"] + p["nz"]))
        got = []
        for n in steps:
            lat.step(n)
            got.append((lat.read_populations(), lat.diagnostics()))
        name = lat.kernel_name()
        lat.close()
        if ref is None:
            ref = got
            continue
        for (f, d), (f0, d0) in zip(got, ref):
            assert np.array_equal(f, f0), name
            assert d["status"] == 0 and d["step"] == d0["step"]
            assert abs(d["evaporated_mass"] - d0["evaporated_mass"]) <= 1e-9 * p["nx"] * p["ny"] * p["nz"]
    return name


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (2, 1, 2), (1, 3, 40), (5, 7, 11), (4, 4, 128), (16, 16, 8), (3, 43, 16),
                                      (16, 16, 31), (16, 16, 32), (20, 20, 21)])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "f16s"])
def test_resident_step_has_the_per_thread_bits(sc, nx, ny, nz, storage):
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=0.9, tau_b=1.1, G=3.4, rho_H=0.03, storage=storage)
    if nz >= 8:
        p.update(geometry=1, sink_z0=nz - 1, sink_layers=2, wall_z0=nz // 2, wall_thickness=2)
    name = _same(sc, p, [dict(staging="thread"), dict()], (1, 2, 5, 64))
    assert ("k_resident" in name) == (nx * ny * nz <= 8192)


@pytest.mark.parametrize("nx,ny,nz", [(4, 1, 5), (4, 5, 4), (28, 3, 6), (32, 8, 5), (36, 9, 7), (60, 4, 5), (64, 6, 9), (68, 7, 6),
                                      (128, 2, 5)])
@pytest.mark.parametrize("tile", [1, 2, 3, 4, 5])
def test_staged_rows_have_the_per_thread_bits(sc, nx, ny, nz, tile):
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=0.9, tau_b=1.1, G=3.4, rho_H=0.03, geometry=1, sink_z0=nz - 1, sink_layers=1,
             wall_z0=1, wall_thickness=1)
    _same(sc, p, [dict(staging="thread", tile=tile), dict(staging="rows", tile=tile)], (1, 2, 5))


def test_sites_on_the_sphere_are_classified_in_fp64(sc, oracle_mod):
    """Integer centre and radius: (3, 4, 0), (0, 0, 5), (3, 4, 12), ... lie exactly on spheres of
    radius 5, 13 and 25 (sinks), their neighbours just inside are not."""
    for n, R, c in ((16, 5.0, 8.0), (32, 13.0, 15.0), (56, 25.0, 27.0), (56, 25.0 + 2.0 ** -40, 27.0)):
        p = dict(nx=n, ny=n, nz=n, tau_r=1.0, tau_b=1.0, G=3.6, rho_H=0.02, geometry=2, sphere_cx=c, sphere_cy=c, sphere_cz=c,
                 R_H=R)
        init = dict(shape=1, cx=c, cy=c, cz=c, radius=0.5 * R, rho_hi=0.7, rho_lo=0.04, noise_amp=1e-4, seed=3)
        g, o = sc.Lattice(p), oracle_mod.Lattice(p)
        g.init(init)
        o.init_shape(init)
        g.step(1)
        o.step(1)
        sink_g, sink_o = g.read_fields()[0] == np.float32(0.02), np.abs(o.fields()[0] - 0.02) < 1e-12
        assert np.array_equal(sink_g, sink_o), R
        g.close()
