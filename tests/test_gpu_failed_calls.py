"""A refused call returns with nothing in flight on its stream: the host arrays
whose upload it had started may be freed or changed at once."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["model_host", "gradient_host"])
def test_refused_host_calls_wait_for_their_uploads(call):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_12350_gb300 import build, mamute
    build.build()
    stream = torch.cuda.Stream()
    ctx = mamute.Context(0, stream.cuda_stream)
    try:
        n, nt = 448, 8
        vel = torch.full((n, n, n), 2000.0).pin_memory().numpy()  # 360 MB: milliseconds of copying
        grid = mamute.make_grid(n, n, n, 8, 10.0, 1e-3, nt)
        src = np.array([[10.0 * n + 50.0, 0.0, 0.0]], np.float32)  # outside the model
        off, rec = np.array([0, 1], np.int32), np.zeros((1, 3), np.float32)
        out = np.zeros((1, nt), np.float32)
        args = (grid, vel, None, src, np.zeros(nt, np.float32), off, rec, out)
        for _ in range(2):  # the first call allocates, which may wait
            with pytest.raises(mamute.MamuteError) as e:
                if call == "model_host":
                    ctx.model_host(*args)
                else:
                    ctx.gradient_host(*args, np.zeros((n, n, n), np.float32))
            assert stream.query()
            assert e.value.code == mamute.EINVAL
    finally:
        stream.synchronize()
        ctx.close()
