"""The D2Q9 strip kernels (warps marching up 28-column strips) against the plain per-node kernels in
FP64, at the sizes where a strip can go wrong: grids of three nodes, one node more or less than a
strip or two, strips ending at n - 3 and n - 2, every strip height's remainders, periodic axes,
static solids, corners of every precedence, and runs longer than a group of transfers.

Both sides evaluate the same sums in other orders: about a hundred operations per node and step, each
rounded to 1.1e-16, over at most 70 steps of a scheme that does not amplify them, stay below 1e-12 of
the largest value."""
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


FACES = {
    "channel": (W.INLET, W.OUTLET, W.WALL, W.WALL),
    "rotated": (W.WALL, W.WALL, W.OUTLET, W.INLET),
    "open": (W.OUTLET, W.INLET, W.OUTLET, W.INLET),
    "xper": (W.PERIODIC, W.PERIODIC, W.WALL, W.WALL),
    "yper": (W.INLET, W.OUTLET, W.PERIODIC, W.PERIODIC),
    "box": (W.PERIODIC,) * 4,
}


def problem(nx, ny, faces, steps, LD):
    w = W.small_channel2d(nx=max(nx, 24), ny=max(ny, 20), LD=max(LD, 1), n_steps=steps,
                          omega=0.02, trans_amp=0.0, seed=nx + 7 * ny)
    p = w.problem
    p.n = (nx, ny, 1)
    if LD == 0:
        p.L = (0, 0, 0)
    p.bc = FACES[faces] + (W.PERIODIC,) * 2
    p.bc_val = ((0.03, 0.002, 0.0, 1.0), (0.02, -0.001, 0.0, 1.01), (0.001, 0.01, 0.0, 0.99),
                (0.004, 0.02, 0.0, 1.0), (0.0, 0.0, 0.0, 1.0), (0.0, 0.0, 0.0, 1.0))
    p.obj_kind = W.OBJ_PRESSURE if (nx + ny) % 2 else W.OBJ_VELOCITY
    p.obj_dir = (0.6, 0.8, 0.0)
    p.obj_box = (0, nx - 1, 0, ny // 2, 0, 0)
    w.motion[:, 2] = (nx - 1) / 2.0
    w.motion[:, 3] = (ny - 1) / 2.0
    r = np.random.RandomState(nx * 100 + ny)
    s = np.zeros((4, 1, ny, nx))
    s[0] = 1.0 + 0.01 * r.randn(1, ny, nx)
    s[1:3] = 0.02 * r.randn(2, 1, ny, nx)
    return w, s


def run(L, w, init, flags, ks=None):
    s = L.Solver(w.problem, L.FP64, flags=flags)
    s.set_design(w.gamma if w.problem.L[0] else np.zeros(0))
    s.set_motion(w.motion)
    if ks is not None:
        s.set_static(ks)
    s.set_initial_state(init)
    J = s.forward()
    st = s.get_state()
    g = s.adjoint()
    lam = s.get_adjoint_state()
    s.close()
    return J, st, g, lam


def close(a, b):
    return np.max(np.abs(a - b)) <= 1e-12 * max(np.max(np.abs(b)), 1e-300)


CASES = [(3, 3, "channel", 6, 0), (3, 9, "open", 6, 0), (4, 3, "rotated", 6, 0),
         (5, 4, "xper", 6, 0), (27, 7, "channel", 8, 0), (28, 20, "rotated", 8, 6),
         (29, 21, "channel", 8, 6), (30, 22, "open", 8, 6), (31, 23, "box", 8, 6),
         (32, 33, "yper", 8, 6), (57, 25, "channel", 8, 8), (58, 34, "xper", 8, 8),
         (59, 40, "open", 8, 8), (60, 37, "channel", 8, 8), (61, 64, "rotated", 8, 8),
         (86, 35, "channel", 70, 12), (113, 66, "box", 8, 16)]


@pytest.mark.parametrize("nx,ny,faces,steps,LD", CASES)
def test_strips_match_plain_kernels(L, nx, ny, faces, steps, LD):
    w, init = problem(nx, ny, faces, steps, LD)
    Jp, sp, gp, lp = run(L, w, init, L.FLAG_PLAIN_KERNELS)
    Jf, sf, gf, lf = run(L, w, init, 0)
    assert abs(Jf - Jp) <= 1e-12 * abs(Jp)
    assert close(sf, sp) and close(lf, lp)
    if LD:
        assert close(gf, gp)


def test_strips_with_static_solid_match_plain_kernels(L):
    w, init = problem(59, 41, "xper", 12, 8)
    ks = np.zeros((1, 41, 59))
    ks[0, 3:9, 20:40] = 20.0
    Jp, sp, gp, lp = run(L, w, init, L.FLAG_PLAIN_KERNELS, ks)
    Jf, sf, gf, lf = run(L, w, init, 0, ks)
    assert abs(Jf - Jp) <= 1e-12 * abs(Jp)
    assert close(sf, sp) and close(lf, lp) and close(gf, gp)


@pytest.mark.parametrize("slots", [3, 5, 9])
def test_small_snapshot_pools_give_the_full_history_gradient(L, slots):
    """Transfers of a recomputed segment are kept, or formed again in groups of any size: bitwise
    the same gradient."""
    w, init = problem(60, 45, "channel", 45, 12)
    ref = None
    for ck in (0, slots * L.state_bytes(w.problem, L.FP64)):
        s = L.Solver(w.problem, L.FP64, ckpt_bytes=ck)
        s.set_design(w.gamma)
        s.set_motion(w.motion)
        s.set_initial_state(init)
        got = (s.forward(), s.adjoint())
        s.close()
        if ref is None:
            ref = got
        else:
            assert got[0] == ref[0] and np.array_equal(got[1], ref[1])
