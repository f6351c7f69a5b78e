"""Batch steps after a captured graph has been replayed, when the caller has since
changed what the graph holds: a particle array replaced by another (with the same
values, aligned alike or to its elements only; the old one is kept and must stay as
it was), and electrostatics switched on or off.  The particles must be those of the
same channels stepped alone, to the tolerances of the other batch tests (FP64 1e-13,
mixed 1e-6 of each quantity's largest magnitude; impact counts equal)."""
import numpy as np
import pytest

from _problems import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_10761_gb300 as T  # noqa: E402

STEPS = 8         # a graph holds two sort periods, or eight steps without sorting
ARRAYS = ("x", "y", "z", "vx", "vy", "vz", "d", "q", "q_wall", "n_imp", "id")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_10761_gb300 import build
    build.build()
    T.load()


def _channels(prec, sort, **pkw):
    """Two channels of one grid (solved together in mixed precision) and one of another."""
    real = np.float64 if prec == T.TRIBO_FP64 else np.float32
    out = []
    for nx, ny, nz, n, seed in ((16, 12, 8, 300, 1), (16, 12, 8, 701, 2), (24, 16, 12, 400, 3)):
        c, faces, lat, parts = problem(nx, ny, nz, n=n, re_tau=300.0, dplus=(0.8, 2.0), q_scale=1e-13, vy_scale=0.3,
                                       near_wall=0.1, seed=seed)
        params = T.Params(precision=prec, rho_p=c.rho_p, nu=c.nu, rho=c.rho_f, U_c=500.0, sort_every=sort, **pkw)
        ch = T.Channel(nx, ny, nz, c.lx, c.lz, faces, params,
                       torch.from_numpy(np.ascontiguousarray(lat.astype(real))).cuda(), max_particles=n)
        out.append((ch, T.Particles.from_numpy(parts, prec), c.dt))
    return [list(v) for v in zip(*out)]


def _by_id(P):
    a = P.to_numpy()
    order = np.argsort(a["id"])
    return {k: v[order].astype(np.float64) for k, v in a.items()}


def _same(prec, chans, Ps, ref_chans, ref_Ps):
    tol = 1e-13 if prec == T.TRIBO_FP64 else 1e-6
    for ch, P, rc, rP in zip(chans, Ps, ref_chans, ref_Ps):
        ch.sync()
        got, ref = _by_id(P), _by_id(rP)
        assert np.array_equal(got["id"], np.arange(P.n)) and np.array_equal(got["n_imp"], ref["n_imp"])
        assert ref["n_imp"].sum() > 0
        for k in ("x", "y", "z", "vx", "vy", "vz", "d", "q", "q_wall"):
            assert np.abs(got[k] - ref[k]).max() <= tol * max(np.abs(ref[k]).max(), 1e-40), k


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("sort", [0, 2])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("name", ARRAYS)
def test_replaced_array(prec, sort, offset, name):
    chans, Ps, dts = _channels(prec, sort)
    ref_chans, ref_Ps, _ = _channels(prec, sort)
    B = T.Batch(chans, sort_every=sort)
    B.step(Ps, dts, STEPS)
    B.sync()
    old = []
    for P in Ps:
        a = getattr(P, name)
        new = torch.empty(P.n + offset, dtype=a.dtype, device=a.device)[offset:]
        new.copy_(a)
        old.append((a, a.clone()))
        setattr(P, name, new)
    B.step(Ps, dts, STEPS)
    B.sync()
    for ch, P, dt in zip(ref_chans, ref_Ps, dts):
        ch.step(P, dt, 2 * STEPS)
    _same(prec, chans, Ps, ref_chans, ref_Ps)
    for a, was in old:
        assert torch.equal(a, was)
    B.close()


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("sort", [0, 2])
@pytest.mark.parametrize("first,which", [(0, (0, 1, 2)), (0, (1,)), (1, (0, 1, 2)), (1, (2,))])
def test_electrostatics_switched(prec, sort, first, which):
    chans, Ps, dts = _channels(prec, sort, electrostatics=first)
    ref_chans, ref_Ps, _ = _channels(prec, sort, electrostatics=first)
    B = T.Batch(chans, sort_every=sort)
    for run in range(2):
        B.step(Ps, dts, STEPS)
        B.sync()
        for ch, P, dt in zip(ref_chans, ref_Ps, dts):
            ch.step(P, dt, STEPS)
        _same(prec, chans, Ps, ref_chans, ref_Ps)
        for i in which:
            for ch in (chans[i], ref_chans[i]):
                ch.set_params(ch.params.with_(electrostatics=1 - first))
    B.close()
