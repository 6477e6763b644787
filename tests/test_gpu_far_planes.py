"""The 3D sensitivity gather of design planes far from the first where the z shift x_G - xi_G lies one
rounding below an integer: (zeta - xi_G) + x_G is then below the integer on near planes and rounds to it
on far ones, while the gather's z weights come from one fraction.  FP64: nine steps of about 200
roundings of 1.1e-16 stay below 1e-12; FP32: about 30 roundings of 6e-8 a step, 8e-5 on the gradient."""
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


@pytest.mark.parametrize("shift", [7.0 - 2.0 ** -48, 7.0, 7.0 + 2.0 ** -47])
def test_far_planes_match_oracle(L, shift):
    w = W.small_duct3d(nx=16, ny=15, nz=46, n_steps=9, trans_amp=0.5)
    p = w.problem
    p.L = (5, 5, 33)
    p.xi_G = (2.0, 2.0, 13.0)
    w.gamma = W.make_gamma(p.L, 1.0, 5)
    w.motion[:, 4] = 13.0 + shift
    assert np.all(w.motion[:, 4] - p.xi_G[2] == shift)   # no rounding in the shift itself
    Jo, go = oracle.gradient(p, w.gamma, w.motion)
    for prec, tj, tg in ((L.FP64, 1e-12, 1e-12), (L.FP32, 2e-5, 8e-5)):
        s = L.Solver(p, prec)
        s.set_design(w.gamma)
        s.set_motion(w.motion)
        J = s.forward()
        g = s.adjoint()
        s.close()
        assert abs(J - Jo) <= tj * abs(Jo)
        assert np.max(np.abs(g - go)) <= tg * np.max(np.abs(go))
