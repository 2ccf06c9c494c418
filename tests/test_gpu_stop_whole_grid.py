"""The stopping test on the device where it still runs: eigenbasis leaves with n_i = 1 and a
hierarchy that the cut-row launch does not take (six levels, r = 32 in FP64).  As in
test_gpu_device_stop.py the reference is the same solver stopped by max_iter: the run stopped
by tol takes as many steps as the first iterate below it, and returns it bit for bit, at the
start, inside and at the end of a queued chunk."""
import numpy as np
import pytest

from workloads import random_complex

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_stop_on_device_matches_stepwise_definition():
    import paper_2512_12538_gb300 as hh
    n, k, levels, rank = 254, 60.0, 6, 32
    S = n + 2
    f = torch.from_numpy(random_complex((S, S), 41)).cuda()
    g = torch.from_numpy(random_complex((4, S), 42)).cuda()

    def run(tol, max_iter):
        h, _ = hh.hh_setup(hh.make_params(2, n, k, levels, 2, rank, 0, 1, tol, max_iter, "fp64", 5))
        try:
            u = torch.empty((S, S), dtype=torch.complex128, device="cuda")
            launches = hh.hh_launch_count()
            st = hh.hh_solve(h, f, g, u, allow_noconv=True)
            torch.cuda.synchronize()
            # a step on the whole grid is one sweep and a launch a level, a round on the cut
            # rows about ten launches in all
            assert hh.hh_launch_count() - launches > 5 * max_iter or st.iters < max_iter
            assert abs(hh.hh_residual(h, f, g, u) - st.rel_res) < 1e-10 * st.rel_res
            return st, u.cpu().numpy()
        finally:
            hh.hh_destroy(h)

    # history: u_m and its residual for m = 1..K, each from a run stopped by max_iter
    K, hist = 18, {}
    for m in range(1, K + 1):
        st, u = run(1e-300, m)
        assert st.iters == m
        hist[m] = (st.rel_res, u)
    print([f"{v[0]:.3f}" for v in hist.values()])
    for m in (8, 15, 16, 17, K):
        tol = hist[m][0] * (1 + 1e-12)
        assert tol < 1.0                       # (above 1 the right-hand side itself ends the solve)
        want = next(j for j in range(1, K + 1) if hist[j][0] < tol)
        st, u = run(tol, 10 * K)
        assert st.iters == want and st.rel_res == hist[want][0]
        assert np.array_equal(u, hist[want][1])
