"""The explicit-inverse leaves at the edges of their kernels, against the oracle.

The factorisation holds a leaf's block in registers in tiles of 32 rows and changes its
form at 32, 64, 96 and 128 rows; both it and the sweep run two chains of columns that
meet in the middle, so odd and even column counts and chains shorter than a group of eight
columns are taken too.  Tolerances: 1e-11 for FP64 and 5e-4 for the mixed form, the bounds of
`test_gpu_leaf_shapes.py` (larger grids and wave numbers than here); a wrong row, column
or chain gives an error of order one.
"""
import numpy as np
import pytest

from oracle.method import OMethod
from oracle.problem import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "mixed": 5e-4}


@pytest.mark.parametrize("n,precision", [
    (6, "fp64"), (7, "mixed"), (9, "fp64"),
    (60, "mixed"), (61, "fp64"), (62, "mixed"),
    (124, "fp64"), (126, "mixed"), (126, "fp64"),
    (188, "fp64"), (190, "mixed"), (190, "fp64"),
    (252, "mixed"), (254, "mixed")])
def test_block_leaves_at_tile_edges(n, precision):
    import paper_2512_12538_gb300 as hh
    k = 0.3 * (n + 1)
    P = Problem(2, n, k)
    O = OMethod(P, 1, 2, 0, 0)
    p = hh.make_params(2, n, k, 1, 2, 2, 2, 1, 1e-10, 10, precision, 1, "block")
    h, _ = hh.hh_setup(p)
    rng = np.random.default_rng(n)
    try:
        for nd in O.tree:
            if not nd.is_leaf:
                continue
            for nc in (1, 3):
                v = rng.standard_normal((nd.b, P.Sx, nc)) + 1j * rng.standard_normal((nd.b, P.Sx, nc))
                x = torch.empty((nd.b, P.Sx, nc), dtype=torch.complex128, device="cuda")
                hh.hh_leaf_solve(h, nd.id, torch.from_numpy(v).cuda(), x, nc)
                torch.cuda.synchronize()
                want = O.leaf_solve(nd.id, v)
                err = float(np.linalg.norm(x.cpu().numpy() - want) / np.linalg.norm(want))
                assert err < TOL[precision], (nd.id, nd.b, nc, err)
    finally:
        hh.hh_destroy(h)
