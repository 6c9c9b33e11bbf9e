"""The packed form of a slab's face, as the header states it: population array k = 19 c + i's two
planes at offset k * face_bytes / 38, in the storage type, as the buffer holds them (population i
that arrives at x + e_i, at x). Faces go to aligned and unaligned device memory and to pinned host
memory alike, and come back from there."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
Q = 19


def _slab(storage, nx=6, ny=5):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1701_03637_gb300 as sc
    sc.build()
    from paper_1701_03637_gb300.slab import Slab
    return Slab(dict(nx=nx, ny=ny, nz=16, tau_r=1.0, tau_b=1.0, G=3.5, rho_H=0.03, geometry=0, storage=storage), 3, 9)


def _face(slab, side, where="device"):
    """The packed bytes (numpy uint8)."""
    import torch
    from paper_1701_03637_gb300._native import check, load
    n = slab.face_bytes if hasattr(slab, "face_bytes") else slab.send[side].numel() * slab.send[side].element_size()
    buf = torch.zeros(n + 1, dtype=torch.uint8, pin_memory=True) if where == "host" else torch.zeros(n + 1, dtype=torch.uint8, device="cuda")
    off = 1 if where == "unaligned" else 0
    check(load().sc_slab_pack(slab.handle, side, buf.data_ptr() + off))
    slab.sync()
    return buf[off:off + n].cpu().numpy()


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "f16s"])
def test_packed_arrays_are_the_documented_ones(storage):
    import paper_1701_03637_gb300 as sc
    slab = _slab(storage)
    nz, ny, nx = slab.shape
    e, w = sc.lattice_directions()
    f = np.random.default_rng(3).uniform(0.4, 0.6, (2, Q, nz, ny, nx)) * w[None, :, None, None, None]
    slab.write_populations(f)
    for side, z0 in ((0, 2), (1, nz - 4)):
        raw = _face(slab, side)
        if storage == "bf16":
            got = (np.frombuffer(raw, np.uint16).astype(np.uint32) << 16).view(np.float32)
        else:
            got = np.frombuffer(raw, dict(f32=np.float32).get(storage, np.float16)).astype(np.float32)
        got = got.reshape(2, Q, 2, ny, nx).astype(np.float64)
        wi = w[None, :, None, None, None]
        got = got * wi if storage == "f16s" else got if storage == "f32" else got + wi
        # half a unit in the last place of the stored value (offsets below w, scaled values below 1), and of FP32
        tol = {"f32": 2.0 ** -24, "f16": 2.0 ** -11 * 0.6, "bf16": 2.0 ** -8 * 0.6, "f16s": 2.0 ** -11 * 0.6}[storage] * wi + 2.0 ** -22 * wi
        for i in range(Q):
            want = np.roll(f[:, i], (-e[i][2], -e[i][1], -e[i][0]), (1, 2, 3))[:, z0:z0 + 2]
            assert np.all(np.abs(got[:, i] - want) <= tol[:, i]), (side, i)
        for where in ("unaligned", "host"):
            assert np.array_equal(_face(slab, side, where), raw)
    slab.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("where", ["device", "unaligned", "host"])
def test_unpacked_faces_are_the_packed_planes(storage, where):
    import torch
    from paper_1701_03637_gb300._native import check, load
    a, b = _slab(storage), _slab(storage)
    rng = np.random.default_rng(4)
    fa, fb = [rng.uniform(0.01, 0.05, (2, Q) + a.shape) for _ in range(2)]
    a.write_populations(fa)
    b.write_populations(fb)
    raw = _face(a, 1)
    buf = torch.zeros(raw.size + 1, dtype=torch.uint8, device="cpu" if where == "host" else "cuda", pin_memory=where == "host")
    off = 1 if where == "unaligned" else 0
    buf[off:off + raw.size] = torch.from_numpy(raw.copy()).to(buf.device)
    check(load().sc_slab_unpack(b.handle, 0, buf.data_ptr() + off))
    b.sync()
    ra, rb = a.read_populations(), b.read_populations()
    top = a.shape[0] - 4  # a's highest own planes are b's planes 0 and 1
    import paper_1701_03637_gb300 as sc
    e, _ = sc.lattice_directions()
    for i in range(Q):
        for z in (0, 1):  # arrivals at z + e_z from the unpacked planes
            assert np.array_equal(rb[:, i, z + e[i][2]] if z + e[i][2] >= 0 else rb[:, i, -1], ra[:, i, top + z + e[i][2]]), (i, z)
    a.close()
    b.close()
