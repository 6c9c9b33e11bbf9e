"""After a step whose waits ran out the state is undefined: every call that hands it to the host
says so (SC_ETIMEOUT), so that no checkpoint or profile is taken from it; a state loaded behind such
a step, without a synchronisation in between, is valid. The waits run out because one CTA withholds
its reports (a test hook); no GPU fault is involved."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LIMIT = 50_000_000  # ns
SHIFTED = dict(nx=72, ny=1152, nz=200, storage="f16", layout="aa")  # the smallest planes of the shifted step
PERSISTENT = dict(nx=48, ny=48, nz=48, storage="f32", layout="aa", staging="persistent")
INIT = dict(shape=1, cx=24.0, cy=24.0, cz=24.0, radius=9.0, rho_hi=0.7, rho_lo=0.04, noise_amp=1e-4, seed=3)


@pytest.fixture(scope="module")
def sc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as mod
    mod.build()
    return mod


def _lattice(sc, kind, **more):
    p = dict(kind, tau_r=1.0, tau_b=1.0, G=3.5, rho_H=0.03, geometry=1, sink_z0=kind["nz"] - 1, sink_layers=2)
    return sc.Lattice(dict(p, **more))


@pytest.mark.parametrize("kind,word", [(SHIFTED, "shifted"), (PERSISTENT, "persistent")])
def test_reads_of_an_undefined_state_say_so(sc, kind, word):
    lat = _lattice(sc, kind)
    lat.init(INIT)
    lat.set_wait(LIMIT, 0)
    lat.step(3)
    reads = [lat.read_fields, lat.profile, lat.flux_profile]
    if word == "persistent":  # the shifted lattice's populations would be 5 GB of doubles
        reads.append(lat.read_populations)
    for read in reads:
        with pytest.raises(sc.ScError, match=word) as e:
            read()
        assert e.value.code == -5  # SC_ETIMEOUT
    lat.set_wait(2_000_000_000, -1)
    lat.init(INIT)
    lat.step(2)
    for read in reads:
        assert all(np.all(np.isfinite(a)) for a in np.atleast_1d(read()))
    lat.close()


@pytest.mark.parametrize("kind", [SHIFTED, PERSISTENT])
def test_a_state_loaded_behind_a_failing_step_is_valid(sc, kind):
    import torch
    lat, ref = _lattice(sc, kind), _lattice(sc, dict(kind, layout="two", staging="thread"))
    for x in (lat, ref):
        x.init(INIT)
        x.step(2)
        x.sync()
    lat.set_wait(LIMIT, 0)
    lat.step(3)
    lat.set_wait(2_000_000_000, -1)
    for x in (lat, ref):
        x.init(INIT)
        x.step(5)
    lat.sync()
    assert torch.equal(lat.read_fields_device(), ref.read_fields_device())
    lat.close()
    ref.close()
