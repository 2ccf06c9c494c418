"""The stationary iteration on the cut rows against the oracle's iterates on every row.

A few steps are run (HH_ENOCONV at max_iter, the last iterate returned) and u_K is compared
with the oracle's u_K.  The sizes sit at the edges of the kernels' items: one column per
lane and one past it, the smallest bands, one basis column and the most, one level to five,
bands of unequal height, corrections formed by every block (up to 128 of them) or shared
out, the cluster form and the grid form.  Tolerances are those of one step (FP64 1e-8,
complex64 1e-3, test_gpu_parity.py): K steps of a contraction or near it add up no more
than K of its errors, each relative to a residual of the size of the first."""
import numpy as np
import pytest

from oracle.method import OMethod
from oracle.problem import Problem
from workloads import random_complex

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    # n, k, levels, overlap, rank, oversample, scheme
    (6, 2.0, 1, 2, 1, 0, "fd"),          # two bands of 5 rows, 8 columns
    (14, 4.0, 2, 2, 3, 2, "fd"),         # the smallest bands
    (30, 8.0, 2, 2, 4, 4, "fd"),         # 32 columns: one a lane
    (31, 8.0, 2, 4, 5, 3, "q1"),         # 33 columns
    (62, 14.0, 3, 2, 16, 6, "fd"),       # 112 corrections
    (63, 14.0, 3, 4, 17, 6, "fd"),       # 238: shared out; 17 columns
    (78, 30.0, 2, 2, 32, 16, "fd"),      # the most columns
    (101, 18.0, 4, 2, 4, 4, "q1"),       # 16 bands of unequal height
    (130, 20.0, 5, 2, 2, 2, "fd"),       # 32 bands: more leaves than a cluster's blocks
    (200, 40.0, 1, 6, 12, 4, "fd"),      # two tall bands
]


@pytest.fixture(scope="module")
def hh():
    from paper_2512_12538_gb300 import build
    build.build()
    import paper_2512_12538_gb300 as m
    return m


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"n{c[0]}L{c[2]}r{c[4]}{c[6]}")
def test_iterates_match_the_oracle(hh, case):
    n, k, levels, overlap, rank, over, scheme = case
    P = Problem(2, n, k, scheme=scheme)
    O = OMethod(P, levels, overlap, rank, over, seed=3)
    f = random_complex((P.S, P.S), 11)
    g = random_complex((4, P.S), 12)
    K = 3
    want, _, _ = O.solve(P.rhs(f, g), tol=0.0, maxit=K)
    flags = hh.HH_FLAG_BILINEAR if scheme == "q1" else 0
    for prec, tol in (("fp64", 1e-8), ("mixed", 1e-3)):
        s = hh.Solver(2, n, k, levels, overlap, rank, over, tol=1e-300, max_iter=K, precision=prec, seed=3,
                      flags=flags)
        u, st = s.solve(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda(), allow_noconv=True)
        s.close()
        assert st["iters"] == K
        err = np.linalg.norm(u.cpu().numpy().reshape(-1) - want) / np.linalg.norm(want)
        print(f"{prec}: err {err:.2e}")
        assert err < tol, prec


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"n{c[0]}L{c[2]}r{c[4]}{c[6]}")
def test_gmres_iterates_match_the_oracle(hh, case):
    """Flexible GMRES with its vectors on the cut rows: five steps at restart 3 (a full cycle
    and a cut one) are those of GMRES on the whole grid."""
    n, k, levels, overlap, rank, over, scheme = case
    P = Problem(2, n, k, scheme=scheme)
    O = OMethod(P, levels, overlap, rank, over, seed=3)
    f = random_complex((P.S, P.S), 13)
    g = random_complex((4, P.S), 14)
    K = 5
    want, steps, _ = O.solve_gmres(P.rhs(f, g), tol=0.0, restart=3, maxit=K)
    assert steps == K
    flags = hh.HH_FLAG_BILINEAR if scheme == "q1" else 0
    for prec, tol in (("fp64", 1e-8), ("mixed", 1e-3)):
        s = hh.Solver(2, n, k, levels, overlap, rank, over, tol=1e-300, max_iter=K, precision=prec, seed=3,
                      flags=flags, outer="gmres", restart=3)
        u, st = s.solve(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda(), allow_noconv=True)
        s.close()
        err = np.linalg.norm(u.cpu().numpy().reshape(-1) - want) / np.linalg.norm(want)
        print(f"{prec}: {st['iters']} steps, err {err:.2e}")
        assert st["iters"] == K and err < tol, prec


def test_a_handle_solves_alone_after_a_batch(hh):
    """The rounds of a batch leave the iterate in either of a handle's two buffers."""
    n, k = 63, 20.0
    S = n + 2
    ps = [hh.make_params(2, n, k, 2, 2, 8, 6, 1, 1e-10, 400, "mixed", 1 + i) for i in range(2)]
    hs = hh.hh_setup_batch(ps)
    try:
        fs = [torch.from_numpy(random_complex((S, S), 15 + i)).cuda() for i in range(2)]
        gs = [torch.zeros((4, S), dtype=torch.complex128, device="cuda")] * 2
        for _ in range(2):
            ub = [torch.empty_like(f) for f in fs]
            hh.hh_solve_batch(hs, fs, gs, ub)
            for h, f, g, u in zip(hs, fs, gs, ub):
                alone = torch.empty_like(f)
                hh.hh_solve(h, f, g, alone)
                assert ((alone - u).norm() / u.norm()).item() < 1e-12
    finally:
        for h in hs:
            hh.hh_destroy(h)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_a_rescued_handle_is_left_as_it_was(hh, precision):
    """GMRES on a stationary handle (a batch's diverging member, see test_gpu_batch.py)
    borrows the handle's set-up: the handle answers the next batch alike, to the bit, and
    as a handle set up for GMRES does, to the accuracy both solve to."""
    n, k = 63, 0.57 * 64
    S = n + 2
    ps = [hh.make_params(2, n, kk, 2, 2, 16, 8, 1, 1e-10, 400, precision, 1) for kk in (k, 20.0)]
    hs = hh.hh_setup_batch(ps)
    try:
        fs = [torch.from_numpy(random_complex((S, S), 25 + i)).cuda() for i in range(2)]
        gs = [torch.zeros((4, S), dtype=torch.complex128, device="cuda")] * 2
        got = []
        for _ in range(2):
            got.append([torch.empty_like(f) for f in fs])
            hh.hh_solve_batch(hs, fs, gs, got[-1])
        for a, b in zip(*got):
            assert torch.equal(a, b)
    finally:
        for h in hs:
            hh.hh_destroy(h)
    s = hh.Solver(2, n, k, 2, 2, 16, 8, tol=1e-10, max_iter=400, precision=precision, seed=1, outer="gmres", restart=40)
    u, st = s.solve(fs[0], gs[0])
    s.close()
    assert ((u - got[0][0]).norm() / u.norm()).item() < 1e-8
