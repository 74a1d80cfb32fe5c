"""Sizes on both sides of the dispatch rules: coefficient preparation where the
border is shorter than, equal to and longer than the stencil's reach into it,
checkpointed gradients whose slots hold blocks of stored terms, convolution
volumes whose blocking differs, and resampling with a thread per output or with
tiles of outputs and traces.

Bounds: 1e-4 relative for seismograms (FP32 propagation of a few tens of steps,
the bound of the parity tests); the same bits across slot counts; 1e-5 of the
largest value for a convolution (FP32 sums of 432 products of BF16 values) and
for a resampled trace (ascending FP32 sums)."""
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


def _dev(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


@pytest.mark.parametrize("border", [0, 1, 4, 5, 6, 11])
def test_coefficients_around_the_model(ctx, border):
    from oracle import oracle
    from paper_2502_12350_gb300 import mamute
    oracle.build()
    w = synth.small_case(seed=70 + border, nx=23, ny=18, nz=15, border=border, nt=40, density=True,
                         n_src=1, n_rec=9)
    seis = torch.full((int(w.rec_offset[-1]), w.nt), float("nan"), device="cuda:0")
    ctx.model(mamute.grid_of(w), _dev(w.vel), _dev(w.rho), w.src_xyz, w.wavelet, w.rec_offset,
              w.rec_xyz, seis)
    g = oracle.make_grid(w.nx, w.ny, w.nz, w.border, w.h, w.dt, w.nt)
    ref = oracle.model(g, w.vel, w.src_xyz, w.wavelet, w.rec_offset, w.rec_xyz, rho=w.rho)
    assert np.linalg.norm(seis.cpu().numpy() - ref) <= 1e-4 * np.linalg.norm(ref)


@pytest.mark.parametrize("nt,density", [(1, False), (7, True), (24, False), (61, True)])
def test_blocks_of_terms_are_bitwise_all_terms(ctx, nt, density):
    from paper_2502_12350_gb300 import mamute
    w = synth.small_case(seed=80 + nt, nx=29, ny=22, nz=17, border=9, nt=nt, density=density,
                         n_src=2, n_rec=5)
    vel, rho = _dev(w.vel), _dev(w.rho)
    d = torch.zeros((int(w.rec_offset[-1]), nt), device="cuda:0")
    got = []
    for slots in (-1, 1, 2, 3, 5, 8, 13):
        g = torch.full_like(vel, float("nan"))
        J = ctx.gradient(mamute.grid_of(w), vel, rho, w.src_xyz, w.wavelet, w.rec_offset, w.rec_xyz,
                         d, g, n_snapshots=slots)
        got.append((J, g.cpu().numpy()))
    for J, g in got[1:]:
        assert J == got[0][0]
        np.testing.assert_array_equal(g, got[0][1])


@pytest.mark.parametrize("shape", [(1, 1, 1), (35, 2, 3), (1, 70, 63), (4, 17, 62), (33, 9, 125)])
def test_convolution_blockings(ctx, shape):
    from oracle import conv
    from paper_2502_12350_gb300 import cnn
    rng = np.random.default_rng(sum(shape))
    x = conv.bf16_round(rng.standard_normal(shape + (16,)).astype(np.float32))
    w = conv.bf16_round((0.2 * rng.standard_normal((27, 16, 16))).astype(np.float32))
    b = rng.standard_normal(16).astype(np.float32)
    net = cnn.Net(ctx, weights=([w.astype(np.float32)] * 4, [b] * 4))
    xt = _dev((np.asarray(x, np.float32).view(np.uint32) >> 16).astype(np.uint16).view(np.int16))
    y = torch.full(shape + (16,), float("nan"), device="cuda:0")
    net._check(net.lib.mamute_conv3d(ctx._h, *shape, cnn._p(xt), cnn._p(net.wf[0]), cnn._p(net.b[0]), 0,
                                     None, cnn._p(y), None))
    ref = conv.forward(np.moveaxis(x, -1, 0), cnn.to_oracle_layout(w), b)
    got = np.moveaxis(y.cpu().numpy(), -1, 0)
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("traces,nt_in,nt_out,ratio", [
    (128 * 39 + 1, 700, 160, 3.3), (128 * 49, 700, 127, 5.5), (128 * 110 - 3, 61, 40, 3.4),
    (128 * 100 - 5, 41, 200, 0.2), (128 * 24, 830, 256, 3.2), (128 * 25, 830, 250, 3.2)])
def test_resampling_tiles(ctx, traces, nt_in, nt_out, ratio, adjoint):
    from oracle import postproc
    rng = np.random.default_rng(traces)
    dt_in, dt_out = np.float32(1e-3), np.float32(1e-3 * ratio)
    n, m = (nt_out, nt_in) if adjoint else (nt_in, nt_out)
    x = rng.standard_normal((traces, n)).astype(np.float32)
    x[traces // 2, n // 2] = np.inf  # reaches the outputs of its trace whose band holds it, no others
    some = np.unique(np.r_[0, 1, traces - 1, traces // 2, rng.integers(0, traces, 8)])
    clean = x[some].copy()
    clean[~np.isfinite(clean)] = 0.0
    kw = dict(adjoint=True, nt_in=nt_in) if adjoint else {}

    def oracle(a):
        return postproc.resample(a, float(dt_in), None if adjoint else nt_out, float(dt_out), "sinc", **kw)

    ref = oracle(clean)
    y = torch.full((traces, m), float("nan"), device="cuda:0")
    ctx.resample(_dev(x), float(dt_in), nt_out, float(dt_out), 2, y, adjoint=adjoint)
    got = y.cpu().numpy()
    bad = ~np.isfinite(got)
    assert set(np.nonzero(bad.any(axis=1))[0]) <= {traces // 2}
    # 8 steps of the coarser axis on each side of the sample
    assert 0 < bad.sum() <= 16 * max(1.0, ratio if adjoint else 1.0 / ratio) + 2
    ok = np.isfinite(got[some])
    assert np.abs(np.where(ok, got[some] - ref, 0.0)).max() <= 1e-5 * np.abs(ref).max()
