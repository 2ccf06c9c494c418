"""Sketch blocks on both sides of the rules that choose how many CTAs orthonormalise them.

The singular values of the sketched interface maps need an orthonormal Q: both precision
forms take the same Gaussian samples, so their values agree to the complex64 form's leaf
accuracy, 5e-4 of the largest (the bound of `test_gpu_leaf_shapes.py`).  A lost row or
column of a block, or a Q that is not orthonormal, changes them by order one.  The two forms
never share a kernel here: (S_x, m) of 16384 entries and more take four CTAs in complex64;
FP64 takes one up to 200 KB and eight above."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rank,over", [
    (255, 32, 10), (407, 32, 8), (408, 32, 8), (419, 24, 7), (640, 30, 10), (1022, 8, 8)])
def test_singular_values_agree_across_forms(n, rank, over):
    import paper_2512_12538_gb300 as hh
    sig = {}
    for precision in ("mixed", "fp64"):
        h, _ = hh.hh_setup(hh.make_params(2, n, 0.2 * (n + 1), 3, 4, rank, over, 1, 1e-10, 10, precision, 7))
        try:
            for child in (1, 2, 3, 7, 14):
                V = np.empty((n + 2, rank), dtype=np.complex128)
                s = np.empty(rank + over)
                hh.hh_get_basis(h, child, V, s)
                sig[precision, child] = s[:rank].copy()
        finally:
            hh.hh_destroy(h)
    for child in (1, 2, 3, 7, 14):
        a, b = sig["mixed", child], sig["fp64", child]
        err = np.abs(a - b).max() / b.max()
        print(f"n {n} child {child}: {err:.1e}")
        assert b.max() > 0 and err < 5e-4, (child, err)
