"""Gradient filters with lengths of a hundred cells and more, up to lengths far
beyond the model, along each axis.

Reference: the operators inverted in FP64 by their cosine transform.  Bounds, as
relative L2: up to 200 cells 9e-7, the error that dense FP32 cosine transforms
of 700 cells have on the same zero-mean noise; beyond, on noise about one, 1e-6:
sums of terms of one sign whose rounding errors (2^-24 each; along x a random
walk of at most 2 x 28 dependent steps of a lane and its scan, plus a few of the
constants, along y and z carried along) stay below 16 x 2^-24."""
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


def _reference(g, mode, cells):
    u = g.astype(np.float64)
    lam, mats = [], []
    for ax, n in enumerate(u.shape):
        k = np.arange(n)
        C = np.cos(np.pi * k[:, None] * (k[None, :] + 0.5) / n) * np.sqrt(2.0 / n)
        C[0] *= np.sqrt(0.5)
        mats.append(C)
        shape = [1, 1, 1]
        shape[ax] = n
        lam.append((4.0 * cells[2 - ax] ** 2 * np.sin(np.pi * k / (2 * n)) ** 2).reshape(shape))
        u = np.moveaxis(np.tensordot(C, u, ([1], [ax])), 0, ax)
    u = u / (1 + lam[0] + lam[1] + lam[2] if mode == 1 else (1 + lam[0]) * (1 + lam[1]) * (1 + lam[2]))
    for ax, C in enumerate(mats):
        u = np.moveaxis(np.tensordot(C.T, u, ([1], [ax])), 0, ax)
    return u


@pytest.mark.parametrize("cells", [100.0, 200.0, 1e4, 1e9, 1e14])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("mode", [1, 2])
def test_long_filters(ctx, mode, axis, cells):
    shape = [4, 4, 4]
    shape[2 - axis] = 700
    lens = [1.0, 1.0, 1.0]
    lens[axis] = cells
    far = cells > 200
    g = (np.random.default_rng(axis).standard_normal(shape) + (1.0 if far else 0.0)).astype(np.float32)
    lengths = np.array([10.0 * c for c in lens], np.float32)
    ref = _reference(g, mode, lengths.astype(np.float64) / 10.0)
    out = torch.full(shape, float("nan"), device="cuda:0")
    ctx.smooth(10.0, mode, torch.from_numpy(g).cuda(), out, lengths=lengths)
    got = out.cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    assert np.linalg.norm(got - ref) <= (1e-6 if far else 9e-7) * np.linalg.norm(ref)
