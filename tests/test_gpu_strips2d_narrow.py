"""The D2Q9 strip kernels on tall grids of a few columns, whose inner columns lie next to both x faces:
FP64 against the plain per-node kernels (the same sums in other orders, each operation rounded to
1.1e-16, over six steps and their adjoint far below 1e-12 of the largest value), FP32 against the same
(about 30 roundings of 6e-8 a step: below 2e-5)."""
import numpy as np
import pytest

from paper_2506_23895_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FACES = {
    "channel": (W.INLET, W.OUTLET, W.WALL, W.WALL),
    "rotated": (W.WALL, W.WALL, W.OUTLET, W.INLET),
    "open": (W.OUTLET, W.INLET, W.OUTLET, W.INLET),
    "xper": (W.PERIODIC, W.PERIODIC, W.WALL, W.WALL),
}


@pytest.fixture(scope="module")
def L():
    from paper_2506_23895_gb300 import build as B
    B.build()
    from paper_2506_23895_gb300 import lks
    import torch
    assert torch.cuda.is_available()
    return lks


def run(L, w, init, prec, flags):
    s = L.Solver(w.problem, prec, flags=flags)
    s.set_design(np.zeros(0))
    s.set_motion(w.motion)
    s.set_initial_state(init)
    J = s.forward()
    st = s.get_state()
    s.adjoint()
    lam = s.get_adjoint_state()
    s.close()
    return J, st, lam


@pytest.mark.parametrize("nx,ny,faces", [(3, 10, "channel"), (3, 40, "open"), (3, 70, "rotated"),
                                         (3, 41, "xper"), (4, 40, "channel"), (5, 41, "open")])
def test_narrow_grids_match_plain_kernels(L, nx, ny, faces):
    w = W.small_channel2d(n_steps=6, omega=0.02, trans_amp=0.0, seed=nx + 7 * ny)
    p = w.problem
    p.n = (nx, ny, 1)
    p.L = (0, 0, 0)
    p.bc = FACES[faces] + (W.PERIODIC,) * 2
    p.bc_val = ((0.03, 0.002, 0.0, 1.0), (0.02, -0.001, 0.0, 1.01), (0.001, 0.01, 0.0, 0.99),
                (0.004, 0.02, 0.0, 1.0), (0.0, 0.0, 0.0, 1.0), (0.0, 0.0, 0.0, 1.0))
    p.obj_kind = W.OBJ_PRESSURE if (nx + ny) % 2 else W.OBJ_VELOCITY
    p.obj_dir = (0.6, 0.8, 0.0)
    p.obj_box = (0, nx - 1, 0, ny - 1, 0, 0)
    r = np.random.RandomState(nx * 100 + ny)
    init = np.zeros((4, 1, ny, nx))
    init[0] = 1.0 + 0.01 * r.randn(1, ny, nx)
    init[1:3] = 0.02 * r.randn(2, 1, ny, nx)
    Jp, sp, lp = run(L, w, init, L.FP64, L.FLAG_PLAIN_KERNELS)
    for prec, tol in ((L.FP64, 1e-12), (L.FP32, 2e-5)):
        J, st, lam = run(L, w, init, prec, 0)
        assert abs(J - Jp) <= tol * max(abs(Jp), 1e-3)
        assert np.max(np.abs(st - sp)) <= tol * np.max(np.abs(sp))
        assert np.max(np.abs(lam - lp)) <= tol * np.max(np.abs(lp))
