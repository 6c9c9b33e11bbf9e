"""Failure detection of the shifted in-place step without a GPU fault: the waits between tile
columns have a time limit that holds for captured and single launches alike. A test hook makes
one CTA withhold its reports, so that its neighbours' waits run out after 50 ms; the host reads
SC_ETIMEOUT, and after a state is loaded again the same lattice steps to the right bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LIMIT = 50_000_000  # ns


@pytest.fixture(scope="module")
def sc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as mod
    mod.build()
    return mod


def _lattice(sc, storage="f16", **kind):
    """The smallest planes that take the shifted step, and two random states."""
    nx, ny, nz = 72, 1152, 200
    p = dict(nx=nx, ny=ny, nz=nz, tau_r=1.0, tau_b=1.0, G=3.5, rho_H=0.03, storage=storage, geometry=1, sink_z0=nz - 1, sink_layers=2,
             wall_z0=nz // 2, wall_thickness=2)
    return sc.Lattice(dict(p, **kind))


def _state(lat, seed):
    r = np.random.default_rng(seed)
    lat.init_fields_from(*[0.05 + 0.85 * r.random(lat.shape, dtype=np.float32) for _ in range(2)])


@pytest.fixture(scope="module")
def reference(sc):
    """The state `seed 2` after 5 steps of the per-thread two-lattice kernel."""
    lat = _lattice(sc, staging="thread")
    _state(lat, 2)
    lat.step(5)
    return lat.read_fields_device()


@pytest.mark.parametrize("steps", [3, 4, 9])
@pytest.mark.parametrize("cta", [0, "last"])
def test_withheld_reports_give_etimeout_and_the_device_stays_usable(sc, reference, steps, cta):
    import torch
    lat = _lattice(sc, layout="aa")
    assert "k_shift" in lat.kernel_name()
    _state(lat, 1)
    lat.step(4)  # captures the launches with the default limit
    lat.sync()
    lat.set_wait(LIMIT, lat.launch_info()["ctas"] - 1 if cta == "last" else cta)
    lat.step(steps)
    with pytest.raises(sc.ScError) as e:
        lat.sync()
    assert e.value.code == -5  # SC_ETIMEOUT
    assert lat.diagnostics()["status"] == -5
    lat.set_wait(2_000_000_000, -1)
    _state(lat, 2)
    lat.step(5)
    lat.sync()
    assert lat.diagnostics()["status"] == 0
    assert torch.equal(lat.read_fields_device(), reference)
    lat.close()


def test_wait_policy_is_validated(sc):
    lat = _lattice(sc, layout="aa")
    ctas = lat.launch_info()["ctas"]
    for args in ((0, -1), (1000, ctas), (1000, -2)):
        with pytest.raises(sc.ScError, match="-1"):
            lat.set_wait(*args)
    lat.close()
