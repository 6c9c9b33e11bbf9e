"""Band requests on a lattice of the shifted in-place step: a refused one changes nothing (the step,
the state's bits, the wait limit), an accepted one keeps the wait limit and an error that is due."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LIMIT = 50_000_000  # ns
P = dict(nx=512, ny=288, nz=200, tau_r=1.0, tau_b=1.0, G=3.5, rho_H=0.03, storage="f16", geometry=1, sink_z0=199, sink_layers=2)
INIT = dict(shape=1, cx=256.0, cy=144.0, cz=100.0, radius=60.0, rho_hi=0.7, rho_lo=0.04, noise_amp=1e-3, seed=5)


@pytest.fixture()
def lat():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as sc
    sc.build()
    lat = sc.Lattice(dict(P, layout="aa"))
    assert "k_shift" in lat.kernel_name()
    lat.init(INIT)
    yield lat
    lat.close()


def _refused(lat):
    import paper_1701_03637_gb300 as sc
    for bad in (3, 512, 1024, -2):  # no divisors of nx into bands of two sites or more; no such request
        with pytest.raises(sc.ScError, match="-1"):
            lat.persist_bands(bad)


def _times_out(lat):
    import paper_1701_03637_gb300 as sc
    with pytest.raises(sc.ScError) as e:
        lat.sync()
    return e.value.code == -5  # SC_ETIMEOUT


def _noalloc_status(lat):
    import torch
    from paper_1701_03637_gb300._native import check, load
    out = torch.zeros(8, dtype=torch.float64, device="cuda")
    check(load().sc_lbm_diagnostics_noalloc(lat.handle, out.data_ptr()))
    return out[7].item()


@pytest.mark.parametrize("steps", [1, 2])
def test_refused_requests_change_nothing(lat, steps):
    import torch
    import paper_1701_03637_gb300 as sc
    ref = sc.Lattice(dict(P, staging="thread"))
    ref.init(INIT)
    for x in (lat, ref):
        x.step(steps)
    info = lat.launch_info()
    _refused(lat)
    assert "k_shift" in lat.kernel_name() and lat.persist_bands() == 0 and lat.launch_info() == info
    for x in (lat, ref):
        x.step(5)
        x.sync()
    assert torch.equal(lat.read_fields_device(), ref.read_fields_device())
    ref.close()


def test_the_wait_limit_survives(lat):
    lat.set_wait(LIMIT, 0)
    _refused(lat)
    lat.step(2)
    assert _times_out(lat) and _noalloc_status(lat) == -5
    assert lat.persist_bands(2) == 2 and lat.launch_info()["staging"] == "persistent"
    # the error of the shifted step stays until a state is loaded, the limit and the hook for good
    assert _times_out(lat) and _noalloc_status(lat) == -5 and lat.diagnostics()["status"] == -5
    lat.init(INIT)
    lat.sync()
    assert _noalloc_status(lat) == 0
    lat.step(2)
    assert _times_out(lat) and _noalloc_status(lat) == -5
