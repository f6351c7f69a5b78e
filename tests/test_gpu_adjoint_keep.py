"""The adjoint gives the same gradients whatever its memory budget lets it keep
of the forward steps: fields and states, fields alone, or neither, with the
budget just enough and one byte short, electrostatics on and off, and a number
of steps that the checkpoint interval does not divide.

FP64: 1e-12 of each result's largest magnitude (the sums' atomics reorder);
mixed: 1e-5 (FP32 atomics of the field adjoint)."""

import numpy as np
import pytest

from _problems import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_10761_gb300 as T  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_10761_gb300 import build
    build.build()
    T.load()


@pytest.mark.parametrize("electro", [0, 1])
@pytest.mark.parametrize("prec", [T.TRIBO_FP64, T.TRIBO_MIXED])
def test_gradients_do_not_depend_on_what_is_kept(prec, electro):
    nx, ny, nz, n, steps, ckpt = 16, 12, 8, 333, 7, 3
    c, faces, lat, parts = problem(nx, ny, nz, n=n, q_scale=2e-13, vy_scale=0.4, near_wall=0.3, seed=9, dplus=(0.8, 2.5))
    R = 8 if prec == T.TRIBO_FP64 else 4
    up = lambda b: (b + 255) // 256 * 256  # noqa: E731
    fields = steps * up(3 * nz * (ny + 2) * nx * R) * electro
    states = steps * (6 * up(n * R) + up(8 * n))
    real = np.float64 if R == 8 else np.float32
    tol = 1e-12 if R == 8 else 1e-5
    ref = None
    for budget in (-1, fields + states, fields + states - 1, fields, max(fields - 1, 0), 0):
        ch = T.Channel(nx, ny, nz, c.lx, c.lz, faces,
                       T.Params(precision=prec, rho_p=c.rho_p, nu=c.nu, rho=c.rho_f, U_c=300.0, electrostatics=electro),
                       torch.from_numpy(np.ascontiguousarray(lat.astype(real))).cuda(), max_particles=n)
        T.tribo_set_adjoint_memory(ch.ctx, budget)
        out = []
        for _ in range(2):                       # the second call finds the memory of the first
            P = T.Particles.from_numpy(parts, prec)
            J, dU, dK, dd = ch.adjoint(P, 8 * c.dt, steps, ckpt)
            s = P.to_numpy()
            out.append([np.array([J]), np.array([dU]), np.array([dK]), dd.cpu().numpy(), s["x"], s["vy"], s["q"],
                        s["q_wall"], s["n_imp"]])
        ch.close()
        ref = ref or out[0]
        assert ref[8].sum() > 20
        for o in out:
            assert np.array_equal(o[8], ref[8])
            for a, b in zip(o[:8], ref[:8]):
                assert np.abs(a.astype(np.float64) - b).max() <= tol * max(np.abs(b).max(), 1e-300), budget
