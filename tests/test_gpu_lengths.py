"""Poisson solve of every transform length the library takes (2^a 3^b, nx and nz
up to 1024) against the FP64 oracle, in both precisions, with and without the
potential.

Tolerances are those of the other Poisson parity tests: 1e-12 (FP64) and 2e-6
(mixed, set by the FP32 transforms) of the largest magnitude of each output.
"""
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


def _lengths(lo):
    return sorted(n for n in (2 ** a * 3 ** b for a in range(11) for b in range(7)) if lo <= n <= 1024)


GRIDS = {"x": [(n, 3, 6) for n in _lengths(4) if n % 2 == 0], "z": [(6, 2 + n % 3, n) for n in _lengths(4)]}


@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
@pytest.mark.parametrize("axis", ["x", "z"])
def test_poisson_of_every_length(axis, prec):
    tol = 1e-12 if prec == T.TRIBO_FP64 else 2e-6
    rng = np.random.default_rng(3)
    lx, lz = 2 * math.pi * DELTA, math.pi * DELTA
    for nx, ny, nz in GRIDS[axis]:
        faces = synth.y_faces(ny, DELTA, 1.0)
        rho = rng.standard_normal((nz, ny, nx)) * 1e-6 + 3e-7
        phi_ref = oracle.poisson(oracle.Grid(nx, nz, lx, lz, faces), rho, 8.854e-12)
        E_ref = oracle.efield(oracle.Grid(nx, nz, lx, lz, faces), phi_ref)
        ch = T.Channel(nx, ny, nz, lx, lz, faces, T.Params(precision=prec), None)
        phi, E = ch.poisson(torch.from_numpy(rho).cuda(), want_phi=True)
        _, E2 = ch.poisson(torch.from_numpy(rho).cuda())
        ch.sync()
        assert torch.equal(E, E2), (nx, ny, nz)
        phi, E = phi.cpu().numpy(), E.cpu().numpy().astype(np.float64)
        ch.close()
        assert np.abs(phi - phi_ref).max() <= tol * np.abs(phi_ref).max(), (nx, ny, nz)
        for comp in range(3):
            ref = E_ref[..., comp]
            err = np.abs(E[comp] - ref).max() / max(np.abs(ref).max(), 1e-300)
            assert err <= tol, (nx, ny, nz, comp, err)
