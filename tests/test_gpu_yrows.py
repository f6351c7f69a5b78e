"""The y solve at its smallest heights and with pencil counts that fill the last warp
partly, where a pencil's two halves, run by two lanes, are empty or one row long and
meet at once in the row between them: every repetition of a solve gives the same bits,
which are the oracle's field to the tolerances of the other Poisson parity tests
(1e-12 FP64, 2e-6 mixed, of each output's largest magnitude)."""
import math

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_10761_gb300 as T  # noqa: E402

DELTA = 0.02
EPS = 8.854e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_10761_gb300 import build
    build.build()
    T.load()


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("nx,nz", [(4, 4), (6, 9), (64, 48), (256, 128)])
@pytest.mark.parametrize("ny", [2, 3, 4, 5, 13])
def test_low_channels_repeat_bit_for_bit(prec, nx, ny, nz):
    lx, lz = 2 * math.pi * DELTA, math.pi * DELTA
    faces = synth.y_faces(ny, DELTA, 1.5)
    rho = np.random.default_rng(nx + ny).standard_normal((nz, ny, nx)) * 1e-6 + 3e-7
    g = oracle.Grid(nx, nz, lx, lz, faces)
    phi_ref = oracle.poisson(g, rho, EPS)
    E_ref = oracle.efield(g, phi_ref)
    ch = T.Channel(nx, ny, nz, lx, lz, faces, T.Params(precision=prec, eps=EPS))
    r = torch.from_numpy(rho).cuda()
    phi, E = ch.poisson(r, want_phi=True)
    for _ in range(40):
        phi2, E2 = ch.poisson(r, want_phi=True)
        assert torch.equal(phi, phi2) and torch.equal(E, E2)
    ch.close()
    tol = 1e-12 if prec == T.TRIBO_FP64 else 2e-6
    assert np.abs(phi.cpu().numpy() - phi_ref).max() <= tol * np.abs(phi_ref).max()
    En = E.double().cpu().numpy()
    for comp in range(3):
        ref = E_ref[..., comp]
        assert np.abs(En[comp] - ref).max() <= tol * max(np.abs(ref).max(), 1e-300), comp
