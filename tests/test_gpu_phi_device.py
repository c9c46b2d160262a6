"""The potential into a caller's device array (pic_get_phi_device): the mixed store
rebuilds it there, or, where the array is not one its kernel may write (no whole
double alignment, another kind of memory), copies its own. Both give the bytes of
the host's pic_get_phi, for rows of whole vectors and others, and leave what lies
around the array alone."""
import numpy as np
import pytest

from tests._cases import bare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2606_05893_gb300 as p
    p.load_library()
    return p


@pytest.mark.parametrize("nx,ny,nz", [(8, 4, 6), (5, 3, 7), (1, 1, 2), (16, 12, 33)])
@pytest.mark.parametrize("shift", [0, 8, 4])
@pytest.mark.parametrize("mixed", [True, False])
def test_phi_into_device_array(pkg, nx, ny, nz, shift, mixed):
    import torch
    wl = bare(nx=nx, ny=ny, nz=nz, h=5e-9, phi_c=-3.0, phi_a=40.0)
    sim = pkg.Simulation(wl, precision=pkg.PIC_MIXED if mixed else pkg.PIC_FP64)
    rng = np.random.default_rng(nx * ny * nz)
    phi = rng.standard_normal((nz + 1, ny, nx)) * 5.0
    phi[0], phi[nz] = wl.phi_cathode, wl.phi_anode
    sim.set_phi(phi)
    sim.step()  # a solve: the mixed store now holds the potential in FP32 pairs alone
    n = 8 * phi.size
    got = []
    for _ in range(2):  # rebuilt in the array, then copied (the host's read below leaves an FP64 copy)
        buf = torch.full((n + 32,), 0x5A, dtype=torch.uint8, device="cuda")
        pkg.pic_get_phi_device(sim.h, 0, buf.data_ptr() + shift)
        host = buf.cpu().numpy()
        got.append(host[shift:shift + n].tobytes())
        assert (host[:shift] == 0x5A).all() and (host[shift + n:] == 0x5A).all()
        want = sim.phi()
    assert got[0] == got[1] == np.ascontiguousarray(want).tobytes()
    sim.close()


@pytest.mark.parametrize("nx,ny,nz", [(8, 4, 6), (5, 3, 7), (16, 12, 33)])
@pytest.mark.parametrize("start", ["zero", "random", "charged"])
def test_rebuild_rounds_as_fp64_additions(pkg, tmp_path, nx, ny, nz, start):
    """phi = vac + (hi + lo) bit for bit, hi and lo as a checkpoint holds them behind the rebuilt phi."""
    wl = bare(nx=nx, ny=ny, nz=nz, h=5e-9, phi_c=0.0, phi_a=float(nz), weight=1.0)  # vac(k) = k exactly
    rng = np.random.default_rng(nx + ny + nz)
    if start == "charged":
        x = rng.random((300, 3)) * np.array([nx, ny, nz]) * wl.h
        wl.preload = [(x, np.zeros_like(x)), (np.zeros((0, 3)),) * 2, (np.zeros((0, 3)),) * 2]
    sim = pkg.Simulation(wl, precision=pkg.PIC_MIXED)
    if start == "random":
        phi = rng.standard_normal((nz + 1, ny, nx)) * 5.0
        phi[0], phi[nz] = wl.phi_cathode, wl.phi_anode
        sim.set_phi(phi)
    sim.step()
    path = str(tmp_path / "a.bin")
    sim.save(path)
    raw = open(path, "rb").read()
    nnode, nu = (nz + 1) * ny * nx, (nz - 1) * ny * nx
    lo_at = len(raw) - 4 * nu
    hi_at = lo_at - 4 * nnode
    got = np.frombuffer(raw[hi_at - 8 * nnode:hi_at], np.float64).reshape(nz + 1, ny, nx)
    hi = np.frombuffer(raw[hi_at:lo_at], np.float32).reshape(nz + 1, ny, nx)
    lo = np.frombuffer(raw[lo_at:], np.float32).reshape(nz - 1, ny, nx)
    if start == "charged":
        assert np.count_nonzero(lo) > nu // 2
    want = np.arange(1, nz)[:, None, None] + (hi[1:nz].astype(np.float64) + lo.astype(np.float64))
    assert np.array_equal(got[1:nz].view(np.int64), want.view(np.int64))
    sim.close()
