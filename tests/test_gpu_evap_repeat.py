"""The evaporated mass is a function of the run: repeated runs give the same bits, also where a
launch has more work items than evaporated-mass slots (chosen chunks of one plane on small tiles;
the shifted step's chunks), and any plan books the same mass to FP64 rounding."""
import pytest

pytestmark = pytest.mark.gpu


def _run(p, steps):
    import paper_1701_03637_gb300 as sc
    lat = sc.Lattice(p)
    lat.init(dict(shape=1, cx=p["nx"] / 2, cy=p["ny"] / 2, cz=p["nz"] / 2, radius=0.3 * min(p["nx"], p["ny"], p["nz"]), rho_hi=0.7,
                  rho_lo=0.04, noise_amp=1e-2, seed=5))
    lat.step(steps)
    d = lat.diagnostics()
    assert d["status"] == 0
    lat.close()
    return d["evaporated_mass"]


@pytest.mark.parametrize("nx,ny,nz,more,times_slots", [
    (64, 66, 70, dict(tile=4, zchunk=1), 2.3), (130, 95, 64, dict(tile=4, zchunk=1), 6.3), (128, 96, 80, dict(tile=4, zchunk=1, staging="rows"), 7.5),
    (130, 95, 64, dict(), 0.9), (1024, 257, 200, dict(storage="f16", layout="aa"), 1.3)])
@pytest.mark.parametrize("geometry", [1, 2])
def test_repeated_runs_book_the_same_bits(nx, ny, nz, more, times_slots, geometry):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as sc
    sc.build()
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=0.9, tau_b=1.1, G=3.4, rho_H=0.01, geometry=geometry)
    if geometry == 1:
        p.update(sink_z0=nz // 3, sink_layers=max(2, nz // 3))
    else:
        p.update(sphere_cx=nx / 2, sphere_cy=ny / 2, sphere_cz=nz / 2, R_H=0.4 * min(nx, ny, nz))
    masses = [_run(dict(p, **more), 9) for _ in range(4)]
    assert len(set(masses)) == 1 and masses[0] != 0.0
    if "layout" not in more:
        assert abs(masses[0] - _run(dict(p, staging="thread"), 9)) <= 1e-12 * max(1.0, abs(masses[0]))
