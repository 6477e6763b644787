"""The 3D FP32 row marches at the widths where their tiles change, against the 64-bit oracle: 28 columns a
tile in the adjoint (with the face columns in the halo of grids whose march is longer than a wave: 32 | 33,
60 | 61, 88 | 89 nodes), 30 inner columns in the forward step.  Nine FP32 steps of about 30 roundings of
6e-8 stay below 2e-5 of the largest state, four times that on the gradient."""
import numpy as np
import pytest

import oracle
from paper_2506_23895_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2506_23895_gb300 import build as B
    B.build()
    from paper_2506_23895_gb300 import lks
    import torch
    assert torch.cuda.is_available()
    return lks


def run(L, w, v, av=1):
    s = L.Solver(w.problem, L.FP32)
    s.step_variant(v)
    s.adjoint_variant(av)
    s.set_design(w.gamma)
    s.set_motion(w.motion)
    J = s.forward()
    st = s.get_state()
    g = s.adjoint()
    lam = s.get_adjoint_state()
    s.close()
    return J, st, g, lam


SMALL = [(nx, 13) for nx in (4, 5, 28, 29, 30, 31, 32, 33, 34, 56, 57, 60, 61, 62, 63, 84, 85, 88, 89)]
TALL = [(29, 900), (31, 900), (32, 900), (33, 900), (59, 500), (60, 500), (88, 400)]


@pytest.mark.parametrize("nx,nz", SMALL + TALL)
def test_widths_around_whole_tiles_match_oracle(L, nx, nz):
    w = W.small_duct3d(nx=nx, ny=14, nz=nz, LD=4, n_steps=9 if nz < 100 else 4, trans_amp=0.5, seed=nx)
    if nx < 12:   # no room for a design
        w.problem.L = (0, 0, 0)
        w.gamma = np.zeros((0,))
        w.problem.obj_kind, w.problem.obj_box, w.problem.obj_cyl_r = W.OBJ_PRESSURE, (0, nx - 1, 1, 12, 0, 5), 0.0
    Jo, go, lo = oracle.gradient(w.problem, w.gamma, w.motion, want_lam0=True)
    _, so = oracle.forward(w.problem, w.gamma, w.motion)
    for av in (0, 1):
        J, st, g, lam = run(L, w, 2, av)
        assert abs(J - Jo) <= 2e-5 * abs(Jo)
        assert np.max(np.abs(st - so)) <= 2e-5 * np.max(np.abs(so))
        assert np.linalg.norm(np.ravel(g) - np.ravel(go)) <= 8e-5 * np.linalg.norm(go)
        assert np.max(np.abs(lam - lo)) <= 8e-5 * np.max(np.abs(lo))
