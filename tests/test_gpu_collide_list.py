"""Collisions where many pairs fall to one block: dense clusters of approaching
pairs (up to a block of particles all in pairs), counts that are
not a multiple of four, against the oracle in FP64.

The FP64 tolerance is that of the other collision parity tests, 1e-12 of each
quantity's largest magnitude."""
import math

import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("pairs,extra", [(1, 0), (3, 1), (1500, 2), (2600, 3)])
def test_every_mutual_pair_collides_once(pairs, extra):
    nx, ny, nz = 32, 20, 16
    lx, ly, lz = 2 * math.pi * DELTA, 2 * DELTA, math.pi * DELTA
    faces = synth.y_faces(ny, DELTA, 1.0)
    rng = np.random.default_rng(pairs)
    d = 2e-5
    # pair centres at least four diameters from each other's cell neighbours on average; partners
    # 0.6 diameters apart and closing
    c = np.stack([rng.uniform(0.01, 0.99, pairs) * lx, rng.uniform(0.1, 0.9, pairs) * ly, rng.uniform(0.01, 0.99, pairs) * lz])
    e = rng.standard_normal((3, pairs))
    e /= np.linalg.norm(e, axis=0)
    s = np.concatenate([c - 0.3 * d * e, c + 0.3 * d * e, rng.uniform(0.2, 0.8, (3, extra)) * np.array([[lx], [ly], [lz]])], 1)
    v = np.concatenate([0.1 * e, -0.1 * e, np.zeros((3, extra))], 1) + 0.01 * rng.standard_normal((3, 2 * pairs + extra))
    n = s.shape[1]
    order = rng.permutation(n)
    s, v = s[:, order], v[:, order]
    parts = dict(x=s[0], y=s[1], z=s[2], vx=v[0], vy=v[1], vz=v[2], d=np.full(n, d), q=rng.standard_normal(n) * 1e-15)
    dt = 1e-7
    params = T.Params(precision=T.TRIBO_FP64, drag_law=T.TRIBO_DRAG_OFF, electrostatics=0, collisions=1)
    ch = T.Channel(nx, ny, nz, lx, lz, faces, params, None, max_particles=n)
    P = T.Particles.from_numpy(parts, T.TRIBO_FP64)
    ch.step(P, dt, 2)
    ch.sync()
    got = P.to_numpy()
    ch.close()
    g = oracle.Grid(nx, nz, lx, lz, faces)
    st = oracle.State.from_arrays(*(parts[k].copy() for k in ("x", "y", "z", "vx", "vy", "vz", "q", "d")))
    op = oracle.Params(drag_law=params.drag_law, electrostatics=0, collisions=1, rho_p=params.rho_p)
    ref = oracle.run(g, op, st, np.zeros((nz, ny + 2, nx, 3)), dt, 2)
    moved = int((np.abs(ref.vx - parts["vx"]) > 1e-6).sum())
    assert moved >= 2 * (9 * pairs // 10)
    for k in ("vx", "vy", "vz", "q"):
        r = getattr(ref, k)
        assert np.abs(got[k] - r).max() <= 1e-12 * np.abs(r).max(), k
