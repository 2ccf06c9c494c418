"""Every wait that hh_debug_set_wait_limit reaches runs out as HH_ETIMEOUT and leaves the
context and the handle usable: the grid barrier of the whole-grid coarse corrections (n_i = 2,
block leaves), the barriers of the cut-row steps on a grid and their exchanges on a cluster,
alone, in GMRES and for more problems than clusters run at once, and the column waits of the
coarse matrices' inverse in a set-up."""
import numpy as np
import pytest

from workloads import random_complex

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# n, levels, rank, precision, n_inner, more
CASES = {
    "grid_barrier_inner2": (45, 2, 6, "fp64", 2, {}),
    "grid_barrier_inner2_gmres": (45, 2, 6, "mixed", 2, {"outer": "gmres"}),
    "grid_barrier_block": (45, 2, 6, "fp64", 1, {"leaf_solver": "block"}),
    "cut_cluster": (63, 2, 16, "mixed", 1, {}),
    "cut_cluster_gmres": (63, 2, 16, "mixed", 1, {"outer": "gmres"}),
    "cut_grid_mixed": (62, 3, 16, "mixed", 1, {"outer": "gmres"}),
    "cut_grid_fp64": (63, 2, 16, "fp64", 1, {}),
    "cut_grid_fp64_gmres": (63, 2, 16, "fp64", 1, {"outer": "gmres"}),
}


@pytest.fixture(scope="module")
def hh():
    from paper_2512_12538_gb300 import build
    build.build()
    import paper_2512_12538_gb300 as m
    return m


@pytest.fixture
def no_wait(hh):
    def switch(on):
        hh.hh_debug_set_wait_limit(0 if on else -1)
    yield switch
    hh.hh_debug_set_wait_limit(-1)


def _timeout(hh, call):
    with pytest.raises(hh.HHError) as ei:
        call()
    assert ei.value.status == hh.HH_ETIMEOUT


@pytest.mark.parametrize("case", list(CASES))
def test_a_solve_whose_wait_runs_out(hh, no_wait, case):
    n, levels, rank, precision, n_inner, more = CASES[case]
    S = n + 2
    h, _ = hh.hh_setup(hh.make_params(2, n, 12.0, levels, 2, rank, 4, n_inner, 1e-10, 300, precision, 1, **more))
    f = torch.from_numpy(random_complex((S, S), 3)).cuda()
    g = torch.zeros((4, S), dtype=torch.complex128, device="cuda")
    u = torch.empty_like(f)
    try:
        no_wait(True)
        _timeout(hh, lambda: hh.hh_solve(h, f, g, u))
        no_wait(False)
        torch.cuda.synchronize()
        # the graphs captured meanwhile keep the limit of their capture (hh.h): a new handle
        if n_inner > 1 or "leaf_solver" in more:
            hh.hh_destroy(h)
            h, _ = hh.hh_setup(hh.make_params(2, n, 12.0, levels, 2, rank, 4, n_inner, 1e-10, 300, precision, 1,
                                              **more))
        hh.hh_solve(h, f, g, u)
        assert hh.hh_residual(h, f, g, u) < 1e-10
    finally:
        no_wait(False)
        hh.hh_destroy(h)


@pytest.mark.parametrize("rank", [8, 32])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_set_up_whose_wait_runs_out(hh, no_wait, rank, precision):
    """2 x rank rows: the cluster form of the inverse.  Its waits are the only limited ones of
    these set-ups (transforms on CUDA cores)."""
    p = hh.make_params(2, 62, 12.0, 2, 2, rank, 4, 1, 1e-10, 300, precision, 1, flags=hh.HH_FLAG_CUDA_CORE_SWEEPS)
    no_wait(True)
    _timeout(hh, lambda: hh.hh_setup(p))
    no_wait(False)
    torch.cuda.synchronize()
    h, _ = hh.hh_setup(p)
    hh.hh_destroy(h)


@pytest.mark.parametrize("count,precision", [(3, "fp64"), (24, "mixed")])
def test_a_batch_whose_wait_runs_out(hh, no_wait, count, precision):
    n = 63
    S = n + 2
    hs = hh.hh_setup_batch([hh.make_params(2, n, 20.0, 2, 2, 8, 6, 1, 1e-10, 400, precision, 1 + i)
                            for i in range(count)])
    try:
        fs = [torch.from_numpy(random_complex((S, S), 60 + i)).cuda() for i in range(count)]
        gs = [torch.zeros((4, S), dtype=torch.complex128, device="cuda")] * count
        us = [torch.empty_like(f) for f in fs]
        no_wait(True)
        _timeout(hh, lambda: hh.hh_solve_batch(hs, fs, gs, us))
        no_wait(False)
        torch.cuda.synchronize()
        hh.hh_solve_batch(hs, fs, gs, us)
        for h, f, g, u in zip(hs, fs, gs, us):
            assert hh.hh_residual(h, f, g, u) < 1e-10
    finally:
        no_wait(False)
        for h in hs:
            hh.hh_destroy(h)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_server_serves_on_after_a_wait_that_ran_out(hh, no_wait, precision):
    """The set-ups of these requests have no limited wait (ranks below the cluster inverse's,
    transforms on CUDA cores), so it is a round of the server's engine that gives up."""
    import time
    n = 63
    S = n + 2
    p = hh.make_params(2, n, 20.0, 2, 2, 7, 6, 1, 1e-10, 400, precision, 1, flags=hh.HH_FLAG_CUDA_CORE_SWEEPS)
    f = torch.from_numpy(random_complex((S, S), 90)).cuda()
    g = torch.zeros((4, S), dtype=torch.complex128, device="cuda")
    srv = hh.hh_server_create(2 << 30, 4)

    def serve():
        u = torch.empty_like(f)
        torch.cuda.synchronize()
        ticket, t0, res = hh.hh_server_submit(srv, p, f, g, u), time.time(), None
        while res is None:
            assert time.time() - t0 < 60.0
            res = hh.hh_server_poll(srv, ticket)
        return res[0]

    try:
        assert serve() == hh.HH_OK
        no_wait(True)
        assert serve() == hh.HH_ETIMEOUT
        no_wait(False)
        assert [serve() for _ in range(3)] == [hh.HH_OK] * 3
    finally:
        no_wait(False)
        hh.hh_server_destroy(srv)
