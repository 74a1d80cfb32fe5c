"""Resampling around the tile sizes (32 outputs, 128 traces, chunks of 64
samples), for ratios from upsampling to strong decimation, and the locality of
a non-finite sample: it reaches the outputs whose band holds it and no others.
Each output is the ascending FP32 sum of its band, so it is compared with that
sum in FP64 at 1e-5 of the trace's largest output."""
import numpy as np
import pytest

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


CASES = [(1, 5, 1, 1.0), (129, 70, 31, 2.2), (127, 200, 33, 6.1), (128, 64, 200, 0.31),
         (5, 900, 40, 23.0), (260, 96, 96, 1.0)]


@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("traces,nt_in,nt_out,ratio", CASES)
def test_tiles_and_ratios(ctx, traces, nt_in, nt_out, ratio, mode, adjoint):
    from oracle import postproc
    name = {1: "nearest", 2: "sinc"}[mode]
    rng = np.random.default_rng(nt_in + nt_out)
    dt_in, dt_out = np.float32(1e-3), np.float32(1e-3 * ratio)
    n, m = (nt_out, nt_in) if adjoint else (nt_in, nt_out)
    x = rng.standard_normal((traces, n)).astype(np.float32)
    kw = dict(adjoint=True, nt_in=nt_in) if adjoint else {}
    ref = postproc.resample(x, float(dt_in), None if adjoint else nt_out, float(dt_out), name, **kw)
    y = torch.full((traces, m), float("nan"), device="cuda:0")
    ctx.resample(torch.from_numpy(x).cuda(), dt_in, nt_out, dt_out, mode, y, adjoint=adjoint)
    np.testing.assert_allclose(y.cpu().numpy(), ref, atol=1e-5 * max(np.abs(ref).max(), 1e-30))


def test_non_finite_samples_stay_in_their_bands(ctx):
    x = np.zeros((3, 400), np.float32)
    x[1, 200] = np.inf
    y = torch.full((3, 100), float("nan"), device="cuda:0")
    ctx.resample(torch.from_numpy(x).cuda(), 1e-3, 100, 4e-3, 2, y)
    y = y.cpu().numpy()
    bad = ~np.isfinite(y[1])
    lim = np.abs(np.arange(100) * 4 - 200) < 32  # |t - t_k| < 8 D
    assert not bad[~lim].any() and bad.any()
    assert np.isfinite(y[[0, 2]]).all()
