"""CPML modelling with one slab launch per axis (windows above the size where the
pieces are spread over several), at the edges of the slabs: layers that merge,
gaps of 1 to 3 cells between them, ragged rows under a free surface, and shots in
apertures of different sizes.  Tolerance as in the CPML parity tests: seismogram
relative L2 1e-4 against the FP64 oracle."""
import numpy as np
import pytest

from paper_2502_12350_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LIMIT = 128 * 1024  # padded points


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
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).cuda()


def _below(w):
    w.src_xyz[:, 2] = np.maximum(w.src_xyz[:, 2], 2 * w.h)
    w.rec_xyz[:, 2] = np.maximum(w.rec_xyz[:, 2], w.h)
    return w


def _model(ctx, w, fs=0, **opts):
    from paper_2502_12350_gb300 import mamute
    seis = torch.full((int(w.rec_offset[-1]), w.nt), float("nan"), device="cuda:0")
    ctx.model(mamute.grid_of(w, cerjan=0.0, pml=1, free_surface=fs), _dev(w.vel), _dev(w.rho), w.src_xyz,
              w.wavelet, w.rec_offset, w.rec_xyz, seis, **opts)
    return seis.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("nx,ny,nz,border,fs", [
    (5, 6, 5, 24, 0),     # the slabs of every axis merge
    (5, 9, 6, 24, 1),     # merged, no layer at the surface
    (9, 10, 11, 22, 0),   # gaps of 1 to 3 cells between the slabs
    (23, 17, 33, 20, 1),  # ragged rows, no layer at the surface
])
def test_slab_edges_match_oracle(ctx, oracle, nx, ny, nz, border, fs):
    from oracle import cpml
    assert (nx + 2 * border) * (ny + 2 * border) * (nz + 2 * border) > LIMIT
    w = _below(synth.small_case(seed=nx + nz, nx=nx, ny=ny, nz=nz, border=border, nt=36, density=True,
                                n_src=1, n_rec=6))
    og = oracle.make_grid(nx, ny, nz, border, w.h, w.dt, w.nt, free_surface=fs)
    ref = cpml.model(oracle, og, w.vel, w.src_xyz, w.wavelet, w.rec_offset, w.rec_xyz, f0=w.fpeak, rho=w.rho)
    assert np.linalg.norm(_model(ctx, w, fs) - ref) <= 1e-4 * np.linalg.norm(ref)


def test_apertures_of_one_launch_match_the_oracle(ctx, oracle):
    """Two shots whose windows have merged and separate slabs; each shot's window
    holds all that reaches its receivers, so the oracle runs on the window's crop
    of a laterally constant model."""
    from oracle import cpml
    w = _below(synth.small_case(seed=3, nx=48, ny=40, nz=24, border=16, nt=36, density=True, n_src=2,
                                n_rec=4))
    w.vel[:], w.rho[:] = w.vel[:, :1, :1], w.rho[:, :1, :1]
    ap = np.array([(0, 7, 4, 12), (12, 47, 0, 39)], np.int32)
    for s, (x0, x1, y0, y1) in enumerate(ap):
        lo, hi = np.array([x0, y0, 2]), np.array([x1, y1, w.nz])
        rng = np.random.default_rng(s)
        w.src_xyz[s] = rng.integers(lo, hi) * np.float32(w.h)
        w.rec_xyz[4 * s:4 * s + 4] = rng.integers(lo, hi, (4, 3)) * np.float32(w.h)
    got = _model(ctx, w, aperture=ap)
    for s, (x0, x1, y0, y1) in enumerate(ap):
        og = oracle.make_grid(int(x1 - x0), int(y1 - y0), w.nz, w.border, w.h, w.dt, w.nt)
        shift = np.array([x0, y0, 0], np.float32) * np.float32(w.h)
        ref = cpml.model(oracle, og, np.ascontiguousarray(w.vel[:, y0:y1, x0:x1]),
                         (w.src_xyz[s:s + 1] - shift).astype(np.float32), w.wavelet,
                         np.array([0, 4], np.int32), (w.rec_xyz[4 * s:4 * s + 4] - shift).astype(np.float32),
                         f0=w.fpeak, rho=np.ascontiguousarray(w.rho[:, y0:y1, x0:x1]))
        assert np.linalg.norm(got[4 * s:4 * s + 4] - ref) <= 1e-4 * np.linalg.norm(ref)
