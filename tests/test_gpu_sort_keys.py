"""The order in which the re-sort leaves the particles: by the lattice nodes they gather
from, x fastest, then y, then z.  Particles are put into known node cells (half a
spacing off the cells; the two halves of the lowest and of the top cell next to the
walls, and the periodic seam, among them), well away from the nodes, and no particle
moves in the step that sorts them.  Every array goes with its particle."""
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


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("nx,ny,nz,n", [(4, 2, 4, 3), (6, 3, 9, 1000), (48, 37, 12, 50_001), (16, 20, 162, 20_000)])
def test_order_is_by_gathered_nodes(prec, nx, ny, nz, n):
    lx, ly, lz = 2 * math.pi * DELTA, 2 * DELTA, math.pi * DELTA
    yf = synth.y_faces(ny, DELTA, 1.5)
    rng = np.random.default_rng(n)
    frac = lambda: rng.uniform(0.02, 0.98, n)  # noqa: E731
    i, k, j, up = rng.integers(0, nx, n), rng.integers(0, nz, n), rng.integers(0, ny, n), rng.integers(0, 2, n)
    x = np.mod((i + 0.5 + frac()) * lx / nx, lx)
    z = np.mod((k + 0.5 + frac()) * lz / nz, lz)
    y = yf[j] + 0.5 * (up + frac()) * (yf[j + 1] - yf[j])
    key = (k * ny + np.minimum(j + up, ny - 1)) * nx + i
    d = np.full(n, 1e-3 * yf[1])
    state = dict(x=x, y=y, z=z, vx=rng.standard_normal(n), vy=rng.standard_normal(n), vz=rng.standard_normal(n), d=d,
                 q=rng.standard_normal(n), id=np.arange(n, dtype=np.uint32))
    params = T.Params(precision=prec, drag_law=T.TRIBO_DRAG_OFF, electrostatics=0, sort_every=1)
    ch = T.Channel(nx, ny, nz, lx, lz, yf, params, None, max_particles=n)
    P = T.Particles.from_numpy(state, prec)
    before = {name: v.copy() for name, v in P.to_numpy().items()}
    ch.step(P, 1e-30, 1)
    ch.sync()
    got = P.to_numpy()
    ch.close()
    ids = got["id"].astype(np.int64)
    assert np.array_equal(np.sort(ids), np.arange(n))
    assert (np.diff(key[ids]) >= 0).all()
    for name, v in got.items():
        assert np.array_equal(v, before[name][ids]), name
