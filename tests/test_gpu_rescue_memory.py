"""A batch member whose stationary iteration diverges is re-solved by GMRES, for which the
Krylov space is allocated.  Where the allocator refuses it, the call says HH_ENOMEM and the
member's statistics and iterate are those of its stationary run."""
import ctypes

import numpy as np
import pytest

from workloads import point_source_rhs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_a_refused_rescue_keeps_the_stationary_figures(precision):
    from paper_2512_12538_gb300 import _lib as hh
    state = {"left": None}

    def _alloc(nbytes, stream, ctx):
        if state["left"] is not None:
            if state["left"] == 0:
                return None
            state["left"] -= 1
        return torch.cuda.caching_allocator_alloc(int(nbytes), stream=stream or 0)

    def _free(ptr, nbytes, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    a, f = hh._ALLOC_T(_alloc), hh._FREE_T(_free)
    n = 63
    S = n + 2
    hh.hh_set_allocator(ctypes.cast(a, ctypes.c_void_p), ctypes.cast(f, ctypes.c_void_p))
    hs = []
    try:
        # the first diverges (test_gpu_batch.py), the second converges
        ks = (0.57 * 64, 20.0)
        hs = [hh.hh_setup(hh.make_params(2, n, k, 2, 2, 16, 8, 1, 1e-10, 400, precision, 1))[0] for k in ks]
        fs = [torch.from_numpy(point_source_rhs(n, 3 + i)).cuda() for i in range(2)]
        g = torch.zeros((4, S), dtype=torch.complex128, device="cuda")
        us = [torch.empty_like(f) for f in fs]
        torch.cuda.synchronize()

        def solve(allowed):
            state["left"] = allowed
            VP, st = ctypes.c_void_p * 2, (hh.hh_stats * 2)()
            for s in st:
                s.iters, s.rel_res = -1, -1.0
            r = hh.LIB.hh_solve_batch(VP(*[h.value for h in hs]), VP(*[x.data_ptr() for x in fs]),
                                      VP(g.data_ptr(), g.data_ptr()), VP(*[x.data_ptr() for x in us]), 2, None, st)
            state["left"] = None
            torch.cuda.synchronize()
            return r, [(s.iters, s.rel_res) for s in st]

        r, st = solve(1)                        # the batch's tables, and no more
        assert r == hh.HH_ENOMEM
        assert st[0][0] > 0 and st[0][1] > 1e-10 and st[1][1] < 1e-10
        # the figure is that of the iterate handed out
        assert abs(hh.hh_residual(hs[0], fs[0], g, us[0]) - st[0][1]) <= 1e-6 * st[0][1]
        r, st2 = solve(None)
        assert r == hh.HH_OK and st2[0][0] > st[0][0] and st2[0][1] < 1e-10
        assert np.isclose(hh.hh_residual(hs[0], fs[0], g, us[0]), st2[0][1], rtol=1e-3)
    finally:
        for h in hs:
            hh.hh_destroy(h)
        hh.hh_set_allocator()
