"""Calls on one context that differ only in what the captured time loop holds
by value: the plane of a free surface, the receivers' form (nodes or off-grid
points with as many columns) with streamed seismograms, and the rows and planes
of a two-level launch.  Each call gives, bit for bit, the seismograms of the
same call with its launches issued directly."""
import numpy as np
import pytest

from paper_2502_12350_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_12350_gb300 import build, mamute
    build.build()
    c = mamute.Context(0)
    yield c
    c.close()


def _case(nx=40, ny=38, nz=24, border=8, nt=40, n_rec=8):
    w = synth.small_case(seed=5, nx=nx, ny=ny, nz=nz, border=border, nt=nt, density=True, n_src=1,
                         n_rec=n_rec)
    w.src_xyz = np.array([[nx // 2, ny // 2, 4]], np.float32) * np.float32(w.h)
    n = int(w.rec_offset[-1])
    w.rec_xyz = np.stack([4 + np.arange(n) % (nx - 8), np.full(n, ny // 2 + 1), np.full(n, 2)],
                         axis=1).astype(np.float32) * np.float32(w.h)
    return w


def _model(ctx, w, **kw):
    from paper_2502_12350_gb300 import mamute
    opts = {k: kw.pop(k) for k in ("time_blocking", "tiles") if k in kw}
    vel, rho = torch.from_numpy(w.vel).cuda(), torch.from_numpy(w.rho).cuda()
    out = torch.full((int(w.rec_offset[-1]), w.nt), float("nan"), device="cuda:0")
    ctx.model(mamute.grid_of(w, **kw), vel, rho, w.src_xyz, w.wavelet, w.rec_offset, w.rec_xyz, out, **opts)
    return out.cpu().numpy()


@pytest.mark.parametrize("pml", [0, 1])
def test_free_surface_alternates(ctx, monkeypatch, pml):
    w = _case()
    seq = (0, 1, 0, 1)
    monkeypatch.setenv("MAMUTE_GRAPHS", "1")
    got = [_model(ctx, w, free_surface=fs, pml=pml) for fs in seq]
    monkeypatch.setenv("MAMUTE_GRAPHS", "0")
    ref = [_model(ctx, w, free_surface=fs, pml=pml) for fs in seq]
    assert not np.array_equal(ref[0], ref[1])  # the surface is felt
    for g, r in zip(got, ref):
        np.testing.assert_array_equal(g, r)


def test_receiver_forms_streamed_to_the_host(ctx, monkeypatch):
    """Eight receivers on nodes and one between eight nodes: both eight columns."""
    from paper_2502_12350_gb300 import mamute
    w = _case(n_rec=8)
    nodes = (w.rec_offset, w.rec_xyz)
    point = (np.array([0, 1], np.int32), np.array([[17.3, 18.6, 3.4]], np.float32) * np.float32(w.h))
    assert int(w.rec_offset[-1]) == 8
    grid = mamute.grid_of(w, xyz_interp=1)
    out = np.zeros((8, w.nt), np.float32)

    def run():
        res = []
        for off, xyz in (nodes, point, nodes, point):
            n = int(off[-1])
            out[:] = -7.0
            ctx.model_host(grid, w.vel, w.rho, w.src_xyz, w.wavelet, off, xyz, out[:n])
            assert (out[n:] == -7.0).all()  # nothing past the call's own rows
            res.append(out[:n].copy())
        return res

    monkeypatch.setenv("MAMUTE_GRAPHS", "1")
    got = run()
    monkeypatch.setenv("MAMUTE_GRAPHS", "0")
    for g, r in zip(got, run()):
        np.testing.assert_array_equal(g, r)


@pytest.mark.parametrize("sizes", [((48, 24), (40, 24)), ((40, 16), (40, 15))])
def test_two_level_windows(ctx, monkeypatch, sizes):
    """Rows and planes that leave the one-step plan's size as it is."""
    from paper_2502_12350_gb300 import mamute
    ws = [_case(ny=ny, nz=nz, n_rec=5) for ny, nz in sizes]
    seq = (ws[0], ws[1], ws[0])
    kw = dict(time_blocking=2, tiles=(64, 16, 2, 0, 0, 0))
    monkeypatch.setenv("MAMUTE_GRAPHS", "1")
    got = [_model(ctx, w, **kw) for w in seq]
    monkeypatch.setenv("MAMUTE_GRAPHS", "0")
    for w, g in zip(seq, got):
        np.testing.assert_array_equal(g, _model(ctx, w, **kw))
