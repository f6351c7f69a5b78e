"""The particle re-sort on grids and positions where its key can go wrong: the
periodic ends and the half cells next to them, positions on faces and nodes, the
walls' half cells, several particles of one cell, counts around the gather's four
slots a thread.  Without forces between particles and field, a run that re-sorts
before every step has each particle's values of a run that never does, bit for bit."""
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
@pytest.mark.parametrize("shape", [(4, 2, 4), (6, 3, 9), (48, 37, 12)])
@pytest.mark.parametrize("n", [1, 7, 5001])
def test_sorted_run_equals_unsorted_by_id(prec, shape, n):
    nx, ny, nz = shape
    real = np.float64 if prec == T.TRIBO_FP64 else np.float32
    lx, ly, lz = 2 * math.pi * DELTA, 2 * DELTA, math.pi * DELTA
    yf = synth.y_faces(ny, DELTA, 2.0)
    rng = np.random.default_rng(nx + n)
    d = 1e-4 * ly

    def axis(h, cells, top):
        v = rng.random(n) * top
        v[::3] = (rng.integers(0, 2 * cells, n) * (0.5 * h))[::3]        # faces and nodes
        v[1::7] = np.nextafter(real(top), real(0))
        v = v.astype(real).astype(np.float64)
        return np.where(v >= float(real(top)), 0.0, v)

    y = d + (ly - 2 * d) * rng.random(n)
    edge = rng.integers(0, 3, n)
    y = np.where(edge == 1, 0.6 * d, np.where(edge == 2, ly - 0.6 * d, y)) if n > 1 else y
    x, z = axis(lx / nx, nx, lx), axis(lz / nz, nz, lz)
    state = dict(x=x, y=y, z=z, vx=rng.standard_normal(n), vy=0.1 * rng.standard_normal(n), vz=rng.standard_normal(n),
                 d=np.full(n, d), q=1e-15 * rng.standard_normal(n), id=np.arange(n, dtype=np.uint32))
    u = rng.standard_normal((3, nz, ny + 2, nx)).astype(real)
    runs = []
    for every in (0, 1):
        params = T.Params(precision=prec, drag_law=T.TRIBO_DRAG_STOKES, electrostatics=0, sort_every=every)
        ch = T.Channel(nx, ny, nz, lx, lz, yf, params, torch.from_numpy(u).cuda(), max_particles=n)
        P = T.Particles.from_numpy({k: v.copy() for k, v in state.items()}, prec)
        ch.step(P, 1e-5, 4)
        torch.cuda.synchronize()
        runs.append({k: v for k, v in P.to_numpy().items() if v is not None})
    order = np.argsort(runs[1]["id"])
    assert np.array_equal(runs[1]["id"][order], np.arange(n, dtype=np.uint32))
    for k, v in runs[0].items():
        if k != "cell":
            assert np.array_equal(v, runs[1][k][order]), k
