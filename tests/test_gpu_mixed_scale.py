"""The mixed solve's right-hand-side factor -1 / (eps nx nz), which multiplies the whole
solution: with a permittivity that puts it midway between two FP32 numbers, the mean
factor between the solution and the oracle's, for a density that is mostly its mean (a
mode that meets no twiddle but 1), stays below half a rounding unit, 2^-25, where
rounding the factor takes a whole one, 2^-24."""
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


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("shape", [(64, 48, 64), (128, 33, 32), (48, 97, 32), (54, 40, 81)])
def test_factor_is_not_rounded(shape, sign):
    nx, ny, nz = shape
    lx, lz = 2 * math.pi * DELTA, math.pi * DELTA
    faces = synth.y_faces(ny, DELTA, 2.0)
    factor = float(np.float32(1.0 / (8.854e-12 * nx * nz)))
    factor *= 1.0 + sign * 0.98 * 0.5 * float(np.spacing(np.float32(factor))) / factor
    eps = 1.0 / (factor * nx * nz)
    rho = (1.0 + 0.2 * np.random.default_rng(nx * ny).standard_normal((nz, ny, nx))) * 1e-6
    g = oracle.Grid(nx, nz, lx, lz, faces)
    phi_ref = oracle.poisson(g, rho, eps)
    r = torch.from_numpy(rho).cuda()
    ch = T.Channel(nx, ny, nz, lx, lz, faces, T.Params(precision=T.TRIBO_MIXED, eps=eps))
    solves = [ch.poisson(r, want_phi=True)[0]]
    phi = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
    E = torch.zeros((3, nz, ny + 2, nx), dtype=torch.float32, device="cuda")
    T.tribo_poisson_noalloc(nx, ny, nz, lx, lz, faces, eps, T.TRIBO_MIXED, r, phi, E)
    torch.cuda.synchronize()
    ch.close()
    for got in solves + [phi]:
        off = ((got.cpu().numpy() - phi_ref) * phi_ref).sum() / (phi_ref * phi_ref).sum()
        assert abs(off) <= 2.0 ** -25, off
