"""The tiled resampling kernel (bands of 48 taps and more on 200 blocks and more of
32 outputs x 128 traces, in chunks of 32 samples) at the remainders of its tiles,
and with samples that are not finite, which take its masked second pass: each
reaches the outputs of its trace whose band holds it and no others.

Each output is the ascending FP32 sum of its band: within 1e-5 of the largest
output of the FP64 product."""
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


def _run(ctx, x, nt_in, nt_out, ratio, adjoint):
    """The kernel's result and the FP64 matrix [outputs][inputs] that it applies."""
    from oracle import postproc
    dt_in, dt_out = np.float32(1e-3), np.float32(1e-3 * ratio)
    K = postproc.resample_matrix(nt_in, float(dt_in), nt_out, float(dt_out), "sinc")
    K = K.T if adjoint else K
    y = torch.full((len(x), len(K)), float("nan"), device="cuda:0")
    ctx.resample(torch.from_numpy(x).cuda(), float(dt_in), nt_out, float(dt_out), 2, y, adjoint=adjoint)
    assert max(np.count_nonzero(K, axis=1)) >= 48
    assert -(-len(x) // 128) * -(-len(K) // 32) >= 200
    return y.cpu().numpy(), K


# (outputs, other axis, ratio, adjoint): 49 to 52 taps
FORMS = [(351, 1075, 3.06, False), (352, 1075, 3.06, False), (353, 1075, 3.06, False),
         (382, 1201, 3.2, False), (350, 1130, 0.31, True), (353, 1130, 0.31, True)]


@pytest.mark.parametrize("traces", [128 * 19 - 1, 128 * 19, 128 * 19 + 1])
@pytest.mark.parametrize("m,n,ratio,adjoint", FORMS)
def test_remainders(ctx, m, n, ratio, adjoint, traces):
    x = np.random.default_rng(m + traces).standard_normal((traces, n)).astype(np.float32)
    got, K = _run(ctx, x, *((m, n) if adjoint else (n, m)), ratio, adjoint)
    ref = x.astype(np.float64) @ K.T
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("m,n,ratio,adjoint", FORMS[2:5])
def test_non_finite_samples_stay_in_their_bands(ctx, m, n, ratio, adjoint):
    traces = 128 * 19 + 1
    x = np.random.default_rng(m).standard_normal((traces, n)).astype(np.float32)
    clean = x.copy()
    # first and last samples and traces, and both sides of a chunk of samples
    where = [(0, 0, np.nan), (127, n - 1, np.inf), (128, 31, -np.inf), (300, 32, np.nan),
             (traces - 2, n // 2, np.inf), (traces - 1, n - 1, np.nan)]
    for t, k, v in where:
        x[t, k], clean[t, k] = v, 0.0
    got, K = _run(ctx, x, *((m, n) if adjoint else (n, m)), ratio, adjoint)
    ref = clean.astype(np.float64) @ K.T
    bad = ~np.isfinite(got)
    assert set(np.nonzero(bad.any(axis=1))[0]) <= {t for t, _, _ in where}
    for t, k, _ in where:
        w = np.abs(K[:, k])
        assert bad[t][w > 1e-9 * w.max()].all()
        assert not bad[t][w == 0.0].any()
    ok = ~bad
    assert np.abs(np.where(ok, got - ref, 0.0)).max() <= 1e-5 * np.abs(ref).max()
