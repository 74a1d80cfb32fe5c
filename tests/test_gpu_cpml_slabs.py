"""CPML slabs at the sizes where their bookkeeping can go wrong: layers that
meet or overlap, windows not a multiple of 4 wide, layers cut into pieces,
apertures, and windows above the size where a slab launch covers every piece.
Tolerances as in the CPML parity tests: seismogram relative L2 1e-4, gradient
cosine 0.9999 and relative L2 1e-3, against the FP64 oracle."""
import numpy as np
import pytest

from paper_2502_12350_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_12350_gb300 import build, mamute
    build.build()
    c = mamute.Context(0)
    yield c
    c.close()


def _dev(x):
    return None if x is None else torch.from_numpy(np.ascontiguousarray(x, np.float32)).cuda()


@pytest.mark.parametrize("nx,ny,nz,border,fs", [
    (5, 6, 5, 9, 0),     # the slabs of every axis merge
    (9, 10, 11, 4, 0),   # gaps of 1 to 3 cells between the slabs
    (23, 17, 14, 5, 1),  # ragged rows, no layer at the surface
    (64, 61, 40, 13, 0), # a window above the small-window limit, cut slabs
])
def test_slab_edges_match_oracle(ctx, oracle, nx, ny, nz, border, fs):
    from oracle import cpml
    from paper_2502_12350_gb300 import mamute
    w = synth.small_case(seed=nx, nx=nx, ny=ny, nz=nz, border=border, nt=36, density=True, n_src=1,
                         n_rec=6)
    w.src_xyz[:, 2] = np.maximum(w.src_xyz[:, 2], 2 * w.h)
    w.rec_xyz[:, 2] = np.maximum(w.rec_xyz[:, 2], w.h)
    og = oracle.make_grid(nx, ny, nz, border, w.h, w.dt, w.nt, free_surface=fs)
    g = mamute.grid_of(w, cerjan=0.0, pml=1, free_surface=fs)
    args = (_dev(w.vel), _dev(w.rho), w.src_xyz, w.wavelet, w.rec_offset, w.rec_xyz)
    ref = cpml.model(oracle, og, w.vel, w.src_xyz, w.wavelet, w.rec_offset, w.rec_xyz, f0=w.fpeak,
                     rho=w.rho)
    seis = torch.full((int(w.rec_offset[-1]), w.nt), float("nan"), device="cuda:0")
    ctx.model(g, *args, seis)
    got = seis.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)
    dobs = (1.1 * ref).astype(np.float32)
    J, gr = cpml.gradient(oracle, og, w.vel, w.src_xyz, w.wavelet, w.rec_offset, w.rec_xyz, dobs,
                          f0=w.fpeak, rho=w.rho)
    grad = torch.full((nz, ny, nx), float("nan"), device="cuda:0")
    ctx.gradient(g, *args, _dev(dobs), grad)
    a, b = grad.cpu().numpy().astype(np.float64).ravel(), np.asarray(gr).ravel()
    assert a @ b >= 0.9999 * np.linalg.norm(a) * np.linalg.norm(b)
    assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b)
