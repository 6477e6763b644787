"""Grids on which the default forward step takes the z-march or the row march, on either side of the rule,
against the row march: nine FP32 steps of about 30 roundings of 6e-8 stay below 2e-5 of the largest state,
four times that on the gradient."""
import numpy as np
import pytest

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


def run(L, w, v):
    s = L.Solver(w.problem, L.FP32)
    s.step_variant(v)
    s.set_design(w.gamma)
    s.set_motion(w.motion)
    J = s.forward()
    st = s.get_state()
    g = s.adjoint()
    s.close()
    return J, st, g


@pytest.mark.parametrize("n", [(64, 64, 330), (160, 90, 90), (200, 100, 70)])
def test_default_forward_step_agrees_with_the_row_march(L, n):
    w = W.small_duct3d(nx=n[0], ny=n[1], nz=n[2], LD=9, n_steps=9, trans_amp=0.5)
    J1, s1, g1 = run(L, w, 1)
    J2, s2, g2 = run(L, w, 2)
    assert abs(J1 - J2) <= 2e-5 * abs(J2)
    assert np.max(np.abs(s1 - s2)) <= 2e-5 * np.max(np.abs(s2))
    assert np.linalg.norm(g1 - g2) <= 8e-5 * np.linalg.norm(g2)
