"""Gradient filters at the sizes where the solves and transforms can go wrong:
axes of one cell, odd and even lengths around the tile sizes, rows longer than
a warp's and than shared memory holds, and long filters.  Reference: the same
operators inverted in FP64.  Tolerance 1e-5 of the largest value: FP32 sums of
at most a few hundred terms of one sign-consistent kernel."""
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
    lams, mats = [], []
    for ax, n in enumerate(u.shape):
        k = np.arange(n)
        lam = 4.0 * cells[2 - ax] ** 2 * np.sin(np.pi * k / (2 * n)) ** 2
        if n > 4096:  # a spectral form would need an n x n matrix: solved below
            lams.append(None)
            mats.append(None)
            continue
        C = np.cos(np.pi * k[:, None] * (k[None, :] + 0.5) / n) * np.sqrt(2.0 / n)
        C[0] *= np.sqrt(0.5)
        u = np.moveaxis(np.tensordot(C, u, ([1], [ax])), 0, ax)
        lams.append(lam)
        mats.append(C)
    lz, ly = lams[0][:, None], lams[1][None, :]
    if lams[2] is not None:
        lx = lams[2]
        den = 1 + lz[..., None] + ly[..., None] + lx if mode == 1 else \
            (1 + lz[..., None]) * (1 + ly[..., None]) * (1 + lx)
        u = u / den
    else:
        from scipy.linalg import solve_banded
        n, mu = u.shape[2], cells[0] ** 2
        for z in range(u.shape[0]):
            for y in range(u.shape[1]):
                s = 1 + lz[z, 0] + ly[0, y] if mode == 1 else 1.0
                ab = np.zeros((3, n))
                ab[0, 1:] = ab[2, :-1] = -mu
                ab[1] = s + 2 * mu
                ab[1, 0] = ab[1, -1] = s + mu
                u[z, y] = solve_banded((1, 1), ab, u[z, y])
                if mode == 2:
                    u[z, y] /= (1 + lz[z, 0]) * (1 + ly[0, y])
    for ax in range(3):
        if mats[ax] is not None:
            u = np.moveaxis(np.tensordot(mats[ax].T, u, ([1], [ax])), 0, ax)
    return u


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("shape,cells", [
    ((1, 1, 1), (2.0, 2.0, 2.0)),
    ((1, 1, 33), (3.0, 2.0, 2.0)),
    ((1, 130, 1), (2.0, 5.0, 2.0)),
    ((129, 1, 2), (2.0, 2.0, 8.0)),
    ((7, 65, 31), (2.0, 4.0, 1.0)),
    ((63, 64, 66), (0.3, 1.5, 30.0)),
    ((3, 257, 1025), (12.0, 6.0, 2.0)),
    ((2, 3, 26000), (20.0, 2.0, 2.0)),
])
def test_filters_match_fp64(ctx, mode, shape, cells):
    rng = np.random.default_rng(sum(shape))
    g = rng.standard_normal(shape).astype(np.float32)
    ref = _reference(g, mode, cells)
    x = torch.from_numpy(g).cuda()
    out = torch.full_like(x, float("nan"))
    ctx.smooth(10.0, mode, x, out, lengths=[10.0 * c for c in cells])
    np.testing.assert_array_equal(x.cpu().numpy(), g)  # the input is left alone
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()
    ctx.smooth(10.0, mode, x, x, lengths=[10.0 * c for c in cells])
    np.testing.assert_array_equal(x.cpu().numpy(), out.cpu().numpy())
