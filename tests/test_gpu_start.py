"""A solve that its first residual ends (u = 0): no step counted, no change to u = 0.

The outer loops queue their first steps before the host has seen |b|; what they leave in
the buffers meanwhile must not show."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (dim, n, k, levels, overlap, rank, oversample, extra options)
CONFIGS = {
    "cut_mixed": (2, 63, 20.0, 2, 2, 8, 6, {}),
    "cut_fp64": (2, 63, 20.0, 2, 2, 8, 6, {"precision": "fp64"}),
    "cut_gmres": (2, 63, 20.0, 2, 2, 8, 6, {"outer": "gmres"}),
    "inner2": (2, 63, 20.0, 2, 2, 8, 6, {"n_inner": 2}),
    "block": (2, 63, 20.0, 2, 2, 8, 6, {"leaf_solver": "block"}),
    "block_gmres": (2, 63, 20.0, 2, 2, 8, 6, {"leaf_solver": "block", "outer": "gmres"}),
    "one_dim": (1, 200, 40.0, 2, 2, 1, 0, {"precision": "fp64"}),
}


def _inputs(dim, n, what):
    S = n + 2
    f = torch.zeros((S, S) if dim == 2 else (S,), dtype=torch.complex128, device="cuda")
    g = torch.zeros((4, S) if dim == 2 else (2,), dtype=torch.complex128, device="cuda")
    if what != "zero":
        f.view(-1)[S // 2] = 1.0
    if what == "inf":
        f.view(-1)[S // 3] = complex(np.inf, 0.0)
    if what == "nan":
        f.view(-1)[S // 3] = complex(np.nan, 0.0)
    return f, g


@pytest.mark.parametrize("what", ["zero", "tol", "inf", "nan"])
@pytest.mark.parametrize("config", list(CONFIGS))
def test_a_first_residual_that_ends_the_solve(config, what):
    import paper_2512_12538_gb300 as hh
    dim, n, k, levels, overlap, rank, over, opts = CONFIGS[config]
    s = hh.Solver(dim, n, k, levels, overlap, rank, over, tol=2.0 if what == "tol" else 1e-10, max_iter=50, **opts)
    f, g = _inputs(dim, n, what)
    u, st = s.solve(f, g, allow_noconv=True)
    assert st["iters"] == 0 and not u.abs().max().item() > 0.0
    if what == "inf":
        assert np.isnan(st["rel_res"])
    else:
        assert st["rel_res"] == (1.0 if what == "tol" else 0.0)
    # and the handle solves afterwards
    if what != "tol":
        f, g = _inputs(dim, n, "one")
        u, st = s.solve(f, g, allow_noconv=True)
        assert st["iters"] > 0 and torch.isfinite(u.abs()).all()
    s.close()


def test_such_problems_in_a_batch():
    import paper_2512_12538_gb300 as hh
    what = ["zero", "one", "inf", "nan", "one"]
    hs = hh.hh_setup_batch([hh.make_params(2, 63, 20.0, 2, 2, 8, 6, 1, 1e-10, 50, "mixed", 1) for _ in what])
    fs, gs = zip(*[_inputs(2, 63, w) for w in what])
    us = [torch.ones_like(f) for f in fs]
    try:
        hh.hh_solve_batch(hs, fs, gs, us)
    except hh.HHError as e:
        assert e.status == hh.HH_ENOCONV
    for w, u in zip(what, us):
        assert torch.isfinite(u.abs()).all() if w == "one" else not (u.abs() > 0).any()
    for h in hs:
        hh.hh_destroy(h)
