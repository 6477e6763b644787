"""The 3D FP32 adjoint on axes of three and four nodes, where every node lies within two rows of both faces of the
axis: the march's stored face values, the overlapping one-sided corrections and the transposed boundary
copies, in both adjoint variants against the 64-bit oracle's lambda^0.  About 30 roundings of 6e-8 a step
and nine steps and their adjoint stay below 8e-5 of the largest value."""
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


@pytest.mark.parametrize("nx,ny,nz", [(3, 20, 9), (40, 3, 9), (31, 17, 4), (3, 3, 4), (31, 17, 3), (4, 5, 30)])
@pytest.mark.parametrize("kind", [W.OBJ_PRESSURE, W.OBJ_VELOCITY])
def test_adjoint_march_on_short_axes(L, nx, ny, nz, kind):
    w = W.small_duct3d(nx=nx, ny=ny, nz=nz, LD=5, n_steps=9, obj_kind=W.OBJ_PRESSURE)
    p = w.problem
    p.L = (0, 0, 0)
    p.obj_kind = kind
    p.obj_dir = (0.6, 0.0, 0.8)
    p.obj_box = (0, nx - 1, 1, ny - 1, 0, nz - 2)
    Jo, _, lo = oracle.gradient(p, np.zeros((0,)), w.motion, want_lam0=True)
    for v in (0, 1):
        s = L.Solver(p, L.FP32)
        assert s.kernels == ("fused3d" if nz >= 4 else "plain")
        s.adjoint_variant(v)
        s.set_design(np.zeros((0,)))
        s.set_motion(w.motion)
        J = s.forward()
        s.adjoint()
        lam = s.get_adjoint_state()
        s.close()
        assert abs(J - Jo) <= 2e-5 * max(abs(Jo), 1e-3)
        assert np.max(np.abs(lam - lo)) <= 8e-5 * np.max(np.abs(lo))
