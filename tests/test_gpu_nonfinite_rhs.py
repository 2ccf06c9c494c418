"""A right-hand side that holds a NaN or an infinity is no solved problem: HH_ENOCONV, with the
last iterate u = 0, from every outer loop, a batch and the server; its residual is not finite."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (dim, n, k, levels, overlap, rank, oversample, options): the cut rows in both forms and by
# GMRES, the whole grid (n_i = 2, block leaves), one dimension
CONFIGS = {
    "cut_mixed": (2, 63, 20.0, 2, 2, 8, 6, {"precision": "mixed"}),
    "cut_fp64": (2, 63, 20.0, 2, 2, 8, 6, {}),
    "cut_gmres": (2, 63, 20.0, 2, 2, 8, 6, {"outer": "gmres"}),
    "inner2": (2, 63, 20.0, 2, 2, 8, 6, {"n_inner": 2}),
    "inner2_q1": (2, 63, 20.0, 2, 2, 8, 6, {"n_inner": 2, "flags": 8}),
    "block": (2, 63, 20.0, 2, 2, 8, 6, {"leaf_solver": "block"}),
    "block_gmres": (2, 63, 20.0, 2, 2, 8, 6, {"leaf_solver": "block", "outer": "gmres"}),
    "one_dim": (1, 200, 40.0, 2, 2, 1, 0, {}),
}
VALUES = {"nan": complex(np.nan, 0.0), "nan_imag": complex(0.0, np.nan), "inf": complex(np.inf, 0.0)}


def _inputs(dim, n, value, where="f"):
    S = n + 2
    f = torch.zeros((S, S) if dim == 2 else (S,), dtype=torch.complex128, device="cuda")
    g = torch.zeros((4, S) if dim == 2 else (2,), dtype=torch.complex128, device="cuda")
    f.view(-1)[S // 2] = 1.0
    (f if where == "f" else g).view(-1)[-1] = value
    return f, g


@pytest.mark.parametrize("where", ["f", "g"])
@pytest.mark.parametrize("value", list(VALUES))
@pytest.mark.parametrize("config", list(CONFIGS))
def test_solve_reports_no_convergence(config, value, where):
    import paper_2512_12538_gb300 as hh
    dim, n, k, levels, overlap, rank, over, opts = CONFIGS[config]
    assert hh.HH_FLAG_BILINEAR == 8
    s = hh.Solver(dim, n, k, levels, overlap, rank, over, tol=1e-10, max_iter=50, **opts)
    f, g = _inputs(dim, n, VALUES[value], where)
    u = torch.full((s.S, s.Sx), 1.0 + 1.0j, dtype=torch.complex128, device="cuda")
    with pytest.raises(hh.HHError) as ei:
        hh.hh_solve(s.handle, f, g, u)
    assert ei.value.status == hh.HH_ENOCONV
    assert (u == 0).all()
    assert not np.isfinite(hh.hh_residual(s.handle, f, g, u))
    if config in ("cut_fp64", "one_dim"):        # the 5-point operator with one k
        assert not np.isfinite(hh.hh_residual_noalloc(dim, n, k, f, g, u))
    # the handle answers the next right-hand side
    f, g = _inputs(dim, n, 0.0)
    st = hh.hh_solve(s.handle, f, g, u, allow_noconv=True)
    assert st.iters > 0 and torch.isfinite(u.abs()).all()
    s.close()


@pytest.mark.parametrize("value", list(VALUES))
def test_batch_reports_no_convergence(value):
    import paper_2512_12538_gb300 as hh
    vals = [0.0, VALUES[value], 0.0]
    hs = hh.hh_setup_batch([hh.make_params(2, 63, 20.0, 2, 2, 8, 6, 1, 1e-10, 200, "mixed", 1) for _ in vals])
    fs, gs = zip(*[_inputs(2, 63, v) for v in vals])
    us = [torch.ones_like(f) for f in fs]
    try:
        with pytest.raises(hh.HHError) as ei:
            hh.hh_solve_batch(hs, fs, gs, us)
        assert ei.value.status == hh.HH_ENOCONV
        assert (us[1] == 0).all()
        for k in (0, 2):
            assert hh.hh_residual(hs[k], fs[k], gs[k], us[k]) < 1e-10
    finally:
        for h in hs:
            hh.hh_destroy(h)


@pytest.mark.parametrize("value", list(VALUES))
def test_server_reports_no_convergence(value):
    import paper_2512_12538_gb300 as hh
    p = hh.make_params(2, 63, 20.0, 2, 2, 8, 6, 1, 1e-10, 200, "mixed", 1)
    srv = hh.hh_server_create(2 << 30, 4)
    try:
        vals = [VALUES[value], 0.0]
        fs, gs = zip(*[_inputs(2, 63, v) for v in vals])
        us = [torch.ones_like(f) for f in fs]
        torch.cuda.synchronize()
        tickets = [hh.hh_server_submit(srv, p, f, g, u) for f, g, u in zip(fs, gs, us)]
        res, t0 = [None] * 2, time.time()
        while None in res:
            assert time.time() - t0 < 60.0
            res = [r or hh.hh_server_poll(srv, t) for r, t in zip(res, tickets)]
        assert [r[0] for r in res] == [hh.HH_ENOCONV, hh.HH_OK]
    finally:
        hh.hh_server_destroy(srv)
    assert (us[0] == 0).all()
