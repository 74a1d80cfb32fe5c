"""More z blocks asked for than the planes fill: every block has planes (the
seismograms and gradients are the bits of one block)."""
import numpy as np
import pytest

from paper_2502_12350_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,zs", [(18, 16), (9, 12), (26, 8)])
def test_no_empty_z_blocks(nz, zs):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_12350_gb300 import build, mamute
    build.build()
    ctx = mamute.Context(0)
    w = synth.small_case(seed=nz, nx=30, ny=22, nz=nz, border=8, nt=25, density=True, n_src=1, n_rec=6)
    dev = torch.device("cuda:0")
    vel, rho = torch.from_numpy(w.vel).to(dev), torch.from_numpy(w.rho).to(dev)
    args = (mamute.grid_of(w), vel, rho, w.src_xyz, w.wavelet, w.rec_offset, w.rec_xyz)
    out = []
    for z in (1, zs):
        seis = torch.full((int(w.rec_offset[-1]), w.nt), float("nan"), device=dev)
        grad = torch.full_like(vel, float("nan"))
        tiles = (32, 8, z, 32, 8, z)
        ctx.model(*args, seis, tiles=tiles)
        ctx.gradient(*args, torch.zeros_like(seis), grad, tiles=tiles)
        out.append((seis.cpu().numpy(), grad.cpu().numpy()))
    ctx.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
