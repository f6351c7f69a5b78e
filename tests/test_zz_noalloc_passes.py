"""The allocation-free Poisson solve on grids of every kind of length against the
FP64 oracle, and with a density, a potential and a field that are aligned to
their elements only: the same values as with aligned arrays.

Tolerances are those of the other Poisson parity tests: 1e-12 (FP64) and 2e-6
(mixed) of each output's largest magnitude."""
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


def _off(t, by):
    """The values of t in memory that starts `by` elements after an allocation's start."""
    flat = torch.zeros(t.numel() + by, dtype=t.dtype, device=t.device)
    flat[by:] = t.reshape(-1)
    return flat[by:].view(t.shape)


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("shape", [(4, 2, 4), (6, 3, 9), (54, 7, 27), (162, 5, 81), (256, 3, 256), (48, 201, 16),
                                   (96, 96, 36)])
def test_noalloc_matches_oracle_at_any_alignment(prec, shape):
    nx, ny, nz = shape
    lx, lz = 2 * math.pi * DELTA, math.pi * DELTA
    faces = synth.y_faces(ny, DELTA, 1.5)
    rng = np.random.default_rng(nx + ny)
    rho = rng.standard_normal((nz, ny, nx)) * 1e-6 + 3e-7
    g = oracle.Grid(nx, nz, lx, lz, faces)
    phi_ref = oracle.poisson(g, rho, EPS)
    E_ref = oracle.efield(g, phi_ref)
    real = torch.float64 if prec == T.TRIBO_FP64 else torch.float32
    tol = 1e-12 if prec == T.TRIBO_FP64 else 2e-6
    dev = dict(device="cuda")
    base = torch.from_numpy(rho).cuda()
    got = []
    for by in (0, 1, 3):
        r = _off(base, by)
        phi = _off(torch.zeros((nz, ny, nx), dtype=torch.float64, **dev), by)
        E = _off(torch.zeros((3, nz, ny + 2, nx), dtype=real, **dev), by)
        for p in (phi, None):
            T.tribo_poisson_noalloc(nx, ny, nz, lx, lz, faces, EPS, prec, r, p, E)
            torch.cuda.synchronize()
            got.append((phi.clone(), E.clone()))
        assert torch.equal(r, base)
    for phi, E in got[1:]:
        assert torch.equal(phi, got[0][0]) and torch.equal(E, got[0][1])
    phi, E = (v.cpu().numpy().astype(np.float64) for v in got[0])
    assert np.abs(phi - phi_ref).max() <= tol * np.abs(phi_ref).max()
    for comp in range(3):
        ref = E_ref[..., comp]
        assert np.abs(E[comp] - ref).max() <= tol * max(np.abs(ref).max(), 1e-300), comp
