"""Collisions of so many particles that a block of the colliding kernel looks at
several rounds of them and works its list off in between, and at the particle counts
where the kernel's block size changes: particle i and particle i + pairs collide, one
pair to a cell, so that every particle of the first rounds is in the lists.  The time
step is too short to move a particle by a unit in the last place, so velocities and
charges are those of the formulas (oracle.pp_charge, an elastic exchange along the
line of centres) at the starting positions, to the 1e-12 of each quantity's largest
magnitude of the other collision tests; every particle that has no partner keeps its
bits."""
import math

import numpy as np
import pytest

import oracle
import synth
from oracle.particles import pp_charge

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_10761_gb300 as T  # noqa: E402

DELTA = 0.02
ROUND = 4 * 512        # particles of a round of the largest block


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_10761_gb300 import build
    build.build()
    T.load()


# (particles per SM, more or fewer): the last of a block size and the first of the next, the first
# with a second round, and six rounds whose first three are full of pairs
COUNTS = [(2 * 4 * 64, 0), (2 * 4 * 64, 1), (2 * 4 * 128, 0), (2 * 4 * 128, 3), (2 * 4 * 256, 0), (2 * 4 * 256, 2),
          (6 * ROUND, 1031)]


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("per_sm,more", COUNTS)
def test_lists_of_many_rounds(prec, per_sm, more):
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    pairs = n // 2
    nx, ny, nz = 144, 64, 128
    assert n - pairs <= nx * ny * nz
    lx, lz = 2 * math.pi * DELTA, math.pi * DELTA
    faces = synth.y_faces(ny, DELTA, 1.0)
    rng = np.random.default_rng(more)
    real = np.float64 if prec == T.TRIBO_FP64 else np.float32
    d = 2e-5
    # the pair's cell; an odd particle out has a cell of its own
    cell = rng.permutation(nx * ny * nz)[:n - pairs]
    k, j, i = np.unravel_index(cell, (nz, ny, nx))
    c = np.stack([(i + 0.5) * lx / nx, 0.5 * (faces[j] + faces[j + 1]), (k + 0.5) * lz / nz])
    e = rng.standard_normal(c.shape)
    e /= np.linalg.norm(e, axis=0)
    s = np.concatenate([c + 0.3 * d * e, (c - 0.3 * d * e)[:, :pairs]], 1)
    v = np.concatenate([-0.1 * e, (0.1 * e)[:, :pairs]], 1) + 0.01 * rng.standard_normal((3, n))
    s, v = s.astype(real).astype(np.float64), v.astype(real).astype(np.float64)
    dia = (d * rng.uniform(0.9, 1.1, n)).astype(real).astype(np.float64)
    q = rng.standard_normal(n) * 1e-15
    a, b = np.arange(pairs), n - pairs + np.arange(pairs)
    parts = dict(x=s[0], y=s[1], z=s[2], vx=v[0], vy=v[1], vz=v[2], d=dia, q=q)
    params = T.Params(precision=prec, drag_law=T.TRIBO_DRAG_OFF, electrostatics=0, collisions=1)
    ch = T.Channel(nx, ny, nz, lx, lz, faces, params, None, max_particles=n)
    P = T.Particles.from_numpy(parts, prec)
    ch.step(P, 1e-30, 1)
    ch.sync()
    got = P.to_numpy()
    ch.close()
    assert all(np.array_equal(got[name].astype(np.float64), parts[name]) for name in ("x", "y", "z"))
    op = oracle.Params(rho_p=params.rho_p)
    r = s[:, a] - s[:, b]
    dist, rel = np.linalg.norm(r, axis=0), v[:, a] - v[:, b]
    hit = (dist < 0.5 * (dia[a] + dia[b])) & ((r * rel).sum(0) < 0)
    assert hit.mean() > 0.99
    a, b, r, dist, rel = a[hit], b[hit], r[:, hit], dist[hit], rel[:, hit]
    nrm = r / dist
    vn = (rel * nrm).sum(0)
    m = dia ** 3
    ref_v, ref_q = v.copy(), q.copy()
    ref_v[:, a] -= 2.0 * m[b] / (m[a] + m[b]) * vn * nrm
    ref_v[:, b] += 2.0 * m[a] / (m[a] + m[b]) * vn * nrm
    dq, _ = pp_charge(op, dia[a], dia[b], q[a], q[b], np.linalg.norm(rel, axis=0))
    ref_q[a] += dq
    ref_q[b] -= dq
    assert np.abs(got["q"] - ref_q).max() <= 1e-12 * np.abs(ref_q).max()
    # velocities are stored in the real type: half a unit in the last place more in mixed precision
    tol = 1e-12 if prec == T.TRIBO_FP64 else 2.0 ** -24 + 1e-12
    gv = np.stack([got["vx"], got["vy"], got["vz"]]).astype(np.float64)
    assert np.abs(gv - ref_v).max() <= tol * np.abs(ref_v).max()
    alone = np.setdiff1d(np.arange(n), np.concatenate([a, b]))
    assert np.array_equal(gv[:, alone], v[:, alone]) and np.array_equal(got["q"][alone], q[alone])
