"""A motion whose footprint leaves the grid is refused, and the one set before stays whole: the next run
gives bitwise what it gave.  The refused motion moves the design along x inside the grid (which alone
would change the footprint box) and out of it along the next axis."""
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


@pytest.mark.parametrize("make", [lambda: W.small_channel2d(nx=44, ny=26, n_steps=12),
                                  lambda: W.small_duct3d(nx=24, ny=17, nz=16, n_steps=12)])
@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("static", [False, True])
def test_refused_motion_leaves_the_one_before(L, make, prec, static):
    w = make()
    s = L.Solver(w.problem, getattr(L, prec))
    s.set_design(w.gamma)
    s.set_motion(w.motion)
    if static:
        s.set_static(np.zeros(s.state_shape[1:]))
    J, g, k = s.forward(), s.adjoint(), s.transfer(7)
    far = w.motion.copy()
    far[:, 2] += np.linspace(-4.0, 4.0, far.shape[0])
    far[6, 3] = 1.0
    with pytest.raises(L.LksError) as e:
        s.set_motion(far)
    assert e.value.status == 1
    if static:   # builds the kernels' table anew
        s.set_static(np.zeros(s.state_shape[1:]))
    J2, g2, k2 = s.forward(), s.adjoint(), s.transfer(7)
    s.close()
    assert J2 == J and np.array_equal(g2, g)
    assert np.array_equal(k2[0], k[0]) and np.array_equal(k2[1], k[1])
