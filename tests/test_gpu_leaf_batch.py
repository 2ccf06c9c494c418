"""Explicit-inverse problems of several heights set up and solved side by side from several
host threads: a kernel's shared-memory limit is its own maximum, whatever another thread's
problem needs."""
import numpy as np
import pytest

from workloads import random_complex

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# pairs of heights that share a form of the factorisation (up to 32, 64, 96, 128 rows; above)
SIZES = {"fp64": (40, 62, 126, 150, 186, 220), "mixed": (40, 62, 126, 150, 186, 220, 250, 262, 300)}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_heights_mixed_in_one_batch(precision):
    import paper_2512_12538_gb300 as hh
    ns = [n for n in SIZES[precision] for _ in range(2)]
    rng = np.random.default_rng(7)
    for _ in range(3):
        order = [ns[i] for i in rng.permutation(len(ns))]
        ps = [hh.make_params(2, n, 0.1 * (n + 1), 1, 2, 4, 2, 1, 1e-8, 60, precision, 1, "block", "gmres")
              for n in order]
        hs = hh.hh_setup_batch(ps)
        fs = [torch.from_numpy(random_complex((n + 2, n + 2), n)).cuda() for n in order]
        gs = [torch.zeros((4, n + 2), dtype=torch.complex128, device="cuda") for n in order]
        us = [torch.empty_like(f) for f in fs]
        try:
            hh.hh_solve_batch(hs, fs, gs, us)
            for h, f, g, u in zip(hs, fs, gs, us):
                assert hh.hh_residual(h, f, g, u) < 1e-8
        finally:
            for h in hs:
                hh.hh_destroy(h)
