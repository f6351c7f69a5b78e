"""The mode sum at mode counts around the staged chunk and the unrolled loop, and
on lattices with few nodes, a remainder of z rows, and more node pairs than a
block has threads, against the sum in FP64 on the host.  Tolerances are those
of the mode field's parity test: 1e-12 (FP64), 1e-6 (mixed) of the largest
value."""
import math
from types import SimpleNamespace

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_10761_gb300 as T  # noqa: E402

DELTA = 0.02


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_10761_gb300 import build
    build.build()
    T.load()


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("shape", [(4, 2, 4), (162, 3, 9), (1024, 2, 6)])
@pytest.mark.parametrize("nm", [1, 3, 63, 64, 66, 130])
def test_mode_sum_matches_host(prec, shape, nm):
    nx, ny, nz = shape
    lx, lz = 2 * math.pi * DELTA, math.pi * DELTA
    yf = synth.y_faces(ny, DELTA, 1.5)
    Y = synth.node_y(yf)
    rng = np.random.default_rng(nm)
    hx, hz = (nx - 1) // 2, (nz - 1) // 2
    m = SimpleNamespace(nxi=rng.integers(-hx, hx + 1, nm).astype(np.int32),
                        nzi=rng.integers(-hz, hz + 1, nm).astype(np.int32), ky=rng.uniform(-200, 200, nm),
                        amp=rng.standard_normal((nm, 3)), phase=rng.uniform(0, 2 * math.pi, nm))
    ubar, damp = rng.standard_normal(ny + 2), rng.uniform(0.5, 1, ny + 2)
    t = 1e-3
    x, z = (np.arange(nx) + 0.5) * (lx / nx), (np.arange(nz) + 0.5) * (lz / nz)
    ref = np.zeros((3, nz, ny + 2, nx))
    ref[0] += ubar[None, :, None]
    for e in range(nm):
        kx, kz = 2 * math.pi * m.nxi[e] / lx, 2 * math.pi * m.nzi[e] / lz
        w = damp[None, :, None] * np.cos(kx * (x[None, None, :] - ubar[None, :, None] * t) + m.ky[e] * Y[None, :, None]
                                         + kz * z[:, None, None] + m.phase[e])
        ref += m.amp[e][:, None, None, None] * w
    ch = T.Channel(nx, ny, nz, lx, lz, yf, T.Params(precision=prec))
    ch.set_modes(m, ubar, damp, 0.0)
    got = ch.eval_modes(t).cpu().numpy().astype(np.float64)
    ch.close()
    tol = 1e-12 if prec == T.TRIBO_FP64 else 1e-6
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
