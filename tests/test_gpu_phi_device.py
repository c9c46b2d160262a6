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
