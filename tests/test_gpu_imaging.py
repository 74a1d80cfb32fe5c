"""The all-terms gradient images up to three adjoint levels per launch: every
remainder of the step count modulo three, with and without density, gives the
bits of the checkpointed gradient, which images one level per launch, and of
the transposed Jacobian's path."""
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


@pytest.mark.parametrize("density", [False, True])
@pytest.mark.parametrize("nt", [1, 2, 3, 4, 5, 31])
def test_grouped_imaging_is_bitwise_one_level_per_launch(ctx, nt, density):
    from paper_2502_12350_gb300 import mamute
    w = synth.small_case(seed=50 + nt, nx=37, ny=26, nz=19, border=7, nt=nt, density=density,
                         n_src=2, n_rec=6)
    dev = torch.device("cuda:0")
    vel = torch.from_numpy(w.vel).to(dev)
    rho = None if w.rho is None else torch.from_numpy(w.rho).to(dev)
    d = torch.from_numpy(np.random.default_rng(nt).standard_normal(
        (int(w.rec_offset[-1]), nt)).astype(np.float32)).to(dev)
    grads = []
    for snaps in (-1, 2):
        for call in ("gradient", "adjoint"):
            g = torch.full_like(vel, float("nan"))
            getattr(ctx, call)(mamute.grid_of(w), vel, rho, w.src_xyz, w.wavelet, w.rec_offset,
                               w.rec_xyz, d, g, n_snapshots=snaps)
            grads.append(g.cpu().numpy())
    np.testing.assert_array_equal(grads[0], grads[2])
    np.testing.assert_array_equal(grads[1], grads[3])
