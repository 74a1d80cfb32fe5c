"""The last factor of the gradient, 2 acc / (c^3 dt^2), and of the
pseudo-Hessian, acc / (c dt)^4, as one FP64 quotient rounded to FP32.

Inputs are the accumulator values whose quotient lies nearest to the middle
between two FP32 numbers, found for each velocity among all 2^23 mantissas, so
that an FP64 error of a few units in the last place shows.  The kernel and the
reference make the same IEEE operations in the same order: equal bits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHIM = r"""
#include "aux.h"
using namespace mamute;
extern "C" int vol_bytes() { return (int)sizeof(VolDesc); }
extern "C" void fill_vol(void* p, int nx) {  // one window over a row of nx cells, no border
  VolDesc V{};
  V.Nx = V.nxi = nx;
  V.Ny = V.Nz = V.nyi = V.nzi = 1;
  V.pitch = V.tpitch = (nx + 7) / 8 * 8;
  *static_cast<VolDesc*>(p) = V;
}
extern "C" int finalize(const float* acc, const void* vol, const float* vel, int nx, double dt, int kind,
                        float* out) {
  FinalizeArgs a{acc, static_cast<const VolDesc*>(vol), 1, vel, nx, 1, 1, 0, dt, kind, 0, out};
  return launch_finalize(a, 0);
}
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_12350_gb300 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("finalize")
    src, so = str(d / "shim.cu"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-I", build.CSRC, "-o", so, src, os.path.abspath(lib)], check=True)
    return ctypes.CDLL(so)


def _denominator(c, dt, kind):
    if kind == 0:
        return c * c * c * dt * dt
    A2 = c * c * dt * dt
    return A2 * A2


@pytest.mark.parametrize("kind", [0, 1])
def test_quotient_is_rounded_once(shim, kind):
    dt = float(np.float32(1.3e-3))
    mant = (np.arange(2 ** 23, 2 ** 24, dtype=np.float64) * 2.0 ** -23).astype(np.float32)
    acc, vel = [], []
    for c in np.random.default_rng(kind).uniform(1400, 4500, 24).astype(np.float32):
        q = (2.0 if kind == 0 else 1.0) * mant.astype(np.float64) / _denominator(np.float64(c), dt, kind)
        off = np.abs((q.view(np.int64) & (2 ** 29 - 1)) - 2 ** 28)  # units of the 53-bit quotient from a tie
        pick = np.argpartition(off, 40)[:40]
        acc.append(mant[pick])
        vel.append(np.full(40, c, np.float32))
    acc, vel = np.concatenate(acc), np.concatenate(vel)
    acc[::17], acc[5::17] = 0.0, -0.0  # cells that no wave has reached
    n = len(acc)
    total = 0.0 + acc.astype(np.float64)  # the sum over windows starts at zero
    want = ((2.0 if kind == 0 else 1.0) * total /
            _denominator(vel.astype(np.float64), dt, kind)).astype(np.float32)
    vol = np.zeros(shim.vol_bytes(), np.uint8)
    shim.fill_vol(ctypes.c_void_p(vol.ctypes.data), n)
    accd = torch.zeros((n + 7) // 8 * 8, device="cuda:0")
    accd[:n] = torch.from_numpy(acc).cuda()
    vd, vold = torch.from_numpy(vel).cuda(), torch.from_numpy(vol).cuda()
    out = torch.full((n,), float("nan"), device="cuda:0")
    torch.cuda.synchronize()
    assert shim.finalize(ctypes.c_void_p(accd.data_ptr()), ctypes.c_void_p(vold.data_ptr()),
                         ctypes.c_void_p(vd.data_ptr()), n, ctypes.c_double(dt), kind,
                         ctypes.c_void_p(out.data_ptr())) == 0
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy().view(np.int32), want.view(np.int32))
