"""Cell location of FP64 and FP32 positions on and next to cell faces, at zero,
at the smallest magnitudes and at the ends of the box: the cell a step reports
for particles at rest is the largest index whose face (i dx in FP64, the y
faces) is not above the coordinate, exactly."""
import math

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


def _near(faces, real, top):
    """Every face's neighbourhood: the face, two values on either side, tiny values, within [0, top)."""
    f = np.asarray(faces, np.float64).astype(real)
    v = [f]
    for d in (-np.inf, np.inf):
        a = np.nextafter(f, real(d))
        v += [a, np.nextafter(a, real(d))]
    v = np.concatenate(v + [np.array([0.0, np.finfo(real).tiny, 1e-30, np.nextafter(real(0), real(1))], real)])
    v = v.astype(np.float64)
    return np.unique(v[(v >= 0) & (v < top)])


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("shape", [(4, 2, 4), (54, 37, 27), (384, 256, 162), (1024, 2, 6)])
def test_cells_of_positions_on_faces(prec, shape):
    nx, ny, nz = shape
    real = np.float64 if prec == T.TRIBO_FP64 else np.float32
    lx, ly, lz = 2 * math.pi * DELTA, 2 * DELTA, math.pi * DELTA
    yf = synth.y_faces(ny, DELTA, 2.0)
    xf, zf = np.arange(nx + 1) * (lx / nx), np.arange(nz + 1) * (lz / nz)
    d = 1e-9
    x, z = _near(xf, real, real(lx)), _near(zf, real, real(lz))
    y = _near(yf, real, ly)
    y = y[(y > d) & (y < ly - d)]
    n = max(len(x), len(y), len(z))
    x, y, z = (np.resize(v, n) for v in (x, y, z))
    zero = np.zeros(n)
    params = T.Params(precision=prec, drag_law=T.TRIBO_DRAG_OFF, electrostatics=0)
    ch = T.Channel(nx, ny, nz, lx, lz, yf, params, None)
    P = T.Particles.from_numpy(dict(x=x, y=y, z=z, vx=zero, vy=zero, vz=zero, d=np.full(n, d), q=zero), prec,
                               with_cell=True)
    ch.step(P, 1e-6, 1)
    ch.sync()
    got = P.to_numpy()
    ch.close()
    assert np.array_equal(got["x"], x.astype(real)) and np.array_equal(got["y"], y.astype(real))
    at = lambda v, f: np.clip(np.searchsorted(f, v.astype(real).astype(np.float64), side="right") - 1, 0, len(f) - 2)  # noqa: E731
    ref = (at(z, zf) * ny + at(y, yf)) * nx + at(x, xf)
    assert np.array_equal(got["cell"].astype(np.int64), ref)
