"""The profiler of a flexible-GMRES solve on the cut rows counts what hh.h says: one leaf
sweep, one coarse correction per level and one residual for each of its steps (and the first
residual), with their times, over several cycles."""
import pytest

from workloads import random_complex

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n,levels,restart", [("mixed", 63, 2, 40), ("mixed", 63, 2, 6), ("fp64", 63, 2, 40),
                                                        ("fp64", 63, 2, 6), ("mixed", 62, 3, 10)])
def test_gmres_steps_are_counted(precision, n, levels, restart):
    import paper_2512_12538_gb300 as hh
    S = n + 2
    f = torch.from_numpy(random_complex((S, S), 43)).cuda()
    g = torch.zeros((4, S), dtype=torch.complex128, device="cuda")
    u = torch.empty_like(f)
    h, _ = hh.hh_setup(hh.make_params(2, n, 12.0, levels, 2, 16, 4, 1, 1e-9, 400, precision, 1, outer="gmres",
                                      restart=restart))
    try:
        for _ in range(2):
            hh.hh_profile_categories(h, None)
            hh.hh_profile_enable(h, True)
            st = hh.hh_solve(h, f, g, u)
            prof = hh.hh_profile_read(h)
            assert prof["leaf_sweep"][1] == st.iters > 5
            assert prof["coarse_project"][1] == levels * st.iters
            assert prof["residual"][1] == st.iters + 1
            for c in ("leaf_sweep", "coarse_project", "residual"):
                assert 0.0 < prof[c][0] < st.t_solve_ms
            # one category alone
            hh.hh_profile_categories(h, ["coarse_project"])
            hh.hh_profile_enable(h, True)
            st = hh.hh_solve(h, f, g, u)
            prof = hh.hh_profile_read(h)
            assert prof["coarse_project"][1] == levels * st.iters
            assert all(prof[c][1] == 0 for c in hh.PROFILE_CATEGORIES if c != "coarse_project")
    finally:
        hh.hh_destroy(h)
