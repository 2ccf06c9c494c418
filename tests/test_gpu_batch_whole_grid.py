"""Batch members whose hierarchy the cut-row launch does not take (six levels, r = 32 in FP64:
4032 corrections): they are solved on the whole grid, and a member whose stationary iteration
diverges, as it does for both of them, is re-solved by GMRES like any other."""
import pytest

from workloads import random_complex

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_large_hierarchies_are_rescued_too():
    import paper_2512_12538_gb300 as hh
    tol = 1e-4
    probs = [(254, 5.0, 6, 32, 0), (63, 20.0, 2, 8, 6), (254, 60.0, 6, 32, 0)]
    hs = hh.hh_setup_batch([hh.make_params(2, n, k, L, 2, r, p, 1, tol, 300, "fp64", 1) for n, k, L, r, p in probs])
    try:
        fs = [torch.from_numpy(random_complex((n + 2, n + 2), n)).cuda() for n, *_ in probs]
        gs = [torch.zeros((4, n + 2), dtype=torch.complex128, device="cuda") for n, *_ in probs]
        us = [torch.empty_like(f) for f in fs]
        stats = hh.hh_solve_batch(hs, fs, gs, us)
        for h, f, g, u, st in zip(hs, fs, gs, us, stats):
            res = hh.hh_residual(h, f, g, u)
            print(st.iters, st.rel_res, res)
            assert res < tol and abs(st.rel_res - res) < 1e-6 * tol and 0 < st.iters < 600
    finally:
        for h in hs:
            hh.hh_destroy(h)
