"""hh_solve_host against hh_solve: the staged right-hand side is read whole before anything
of the solve is written over it.

The bilinear load vector of a point reads f at its eight neighbours, so a staging buffer that
the start of a solve writes would give a right-hand side mixed of f and b.  The sizes take many
blocks; n_i = 2 and block leaves iterate on the whole grid, GMRES and n_i = 1 on the cut rows.
The two calls run the same kernels on the same numbers: equal to the bit."""
import numpy as np
import pytest

from oracle import direct
from oracle.problem import Problem
from workloads import random_complex

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = {
    # n, k, n_inner, precision, bilinear, more
    "q1_inner2_fp64": (255, 20.0, 2, "fp64", True, {}),
    "q1_inner2_mixed": (300, 20.0, 2, "mixed", True, {}),
    "q1_cut_mixed": (255, 20.0, 1, "mixed", True, {}),
    "q1_gmres": (255, 20.0, 1, "mixed", True, {"outer": "gmres"}),
    "q1_inner2_gmres": (255, 20.0, 2, "mixed", True, {"outer": "gmres"}),
    "fd_inner2": (255, 20.0, 2, "mixed", False, {}),
    "fd_block": (127, 20.0, 1, "mixed", False, {"leaf_solver": "block", "outer": "gmres"}),
}


@pytest.mark.parametrize("case", list(CASES))
def test_host_buffers_give_the_device_solution(case):
    import paper_2512_12538_gb300 as hh
    n, k, n_inner, precision, q1, more = CASES[case]
    S, tol = n + 2, 1e-11
    f, g = random_complex((S, S), 31), random_complex((4, S), 32)
    h, _ = hh.hh_setup(hh.make_params(2, n, k, 2, 2, 16, 8, n_inner, tol, 400, precision, 1,
                                      flags=hh.HH_FLAG_BILINEAR if q1 else 0, **more))
    try:
        fd, gd = torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda()
        u = torch.empty_like(fd)
        dev = hh.hh_solve(h, fd, gd, u)
        torch.cuda.synchronize()
        for _ in range(3):
            uh = np.empty_like(f)
            st = hh.hh_solve_host(h, f, g, uh)
            assert st.iters == dev.iters and st.rel_res == dev.rel_res < tol
            assert np.array_equal(uh, u.cpu().numpy())
    finally:
        hh.hh_destroy(h)
    # cond(A) times the relative residual bounds the error: 1e-6 of 1e-11 is generous here
    # (a wrong right-hand side gives an error of order one)
    want = direct.solve(Problem(2, n, k, scheme="q1" if q1 else "fd"), f, g)
    assert np.linalg.norm(uh.reshape(-1) - want) / np.linalg.norm(want) < 1e-6
