"""The tallest explicit-inverse bands that a set-up accepts (169 rows in complex64, 119 in
complex128) against the oracle: 142 is the last the sweep took with two right-hand sides and
144 the last with one before its row pieces were sized by need.  Tolerances as in
test_gpu_leaf_block.py; a missing or doubled row piece gives an error of order one."""
import numpy as np
import pytest

from oracle.method import OMethod
from oracle.problem import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "mixed": 5e-4}


@pytest.mark.parametrize("b,precision", [(142, "mixed"), (143, "mixed"), (144, "mixed"), (145, "mixed"),
                                         (160, "mixed"), (169, "mixed"), (118, "fp64"), (119, "fp64")])
def test_tall_block_leaves(b, precision):
    import paper_2512_12538_gb300 as hh
    n = 2 * (b - 1) - 2                     # one level, overlap 2: two bands of b rows
    k = 0.2 * (n + 1)
    P = Problem(2, n, k)
    O = OMethod(P, 1, 2, 0, 0)
    # the set-up's sketches sweep several right-hand sides
    h, _ = hh.hh_setup(hh.make_params(2, n, k, 1, 2, 4, 2, 1, 1e-10, 200, precision, 1, "block", "gmres"))
    rng = np.random.default_rng(b)
    try:
        assert hh.hh_node_info(h, 1)["rb"] - hh.hh_node_info(h, 1)["ra"] == b
        for node in (1, 2):
            for nc in (1, 2, 3):
                v = rng.standard_normal((b, P.Sx, nc)) + 1j * rng.standard_normal((b, P.Sx, nc))
                x = torch.empty((b, P.Sx, nc), dtype=torch.complex128, device="cuda")
                hh.hh_leaf_solve(h, node, torch.from_numpy(v).cuda(), x, nc)
                torch.cuda.synchronize()
                want = O.leaf_solve(node, v)
                err = float(np.linalg.norm(x.cpu().numpy() - want) / np.linalg.norm(want))
                print(b, precision, nc, f"{err:.1e}")
                assert err < TOL[precision], (node, nc, err)
        f = torch.from_numpy(rng.standard_normal((P.S, P.S)) + 0j).cuda()
        g = torch.zeros((4, P.S), dtype=torch.complex128, device="cuda")
        u = torch.empty_like(f)
        hh.hh_solve(h, f, g, u)
        assert hh.hh_residual(h, f, g, u) < 1e-10
    finally:
        hh.hh_destroy(h)
