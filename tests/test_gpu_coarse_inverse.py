"""The inverse of the coarse matrices at the edges of its kernels (16 to 64 rows on a
cluster, two rows a lane above 32; other sizes on one block).

Z = C A_c^-1 C^H reproduces the span of C: Z A Z r = Z r.  The bounds are the unit roundoff
of the form (1.1e-16; 6e-8 for the complex64 bases and inverse) times 1e6, a generous condition
number of A_c and of the basis, capped at 1e-2 for the mixed form; a wrong pivot, row or
column gives an error of order one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("rank", [4, 7, 8, 9, 15, 16, 17, 24, 31, 32])
def test_coarse_correction_is_a_projection(rank, precision):
    import paper_2512_12538_gb300 as hh
    n, k = 127, 50.0
    S = n + 2
    h, _ = hh.hh_setup(hh.make_params(2, n, k, 2, 2, rank, 4, 1, 1e-10, 10, precision, 5))
    rng = np.random.default_rng(rank)
    try:
        r = torch.from_numpy(rng.standard_normal((S, S)) + 1j * rng.standard_normal((S, S))).cuda()
        z, az, zz = torch.empty_like(r), torch.empty_like(r), torch.empty_like(r)
        hh.hh_coarse_apply(h, 0, r, z)
        hh.hh_apply_operator(h, 0, z, az, 1)
        hh.hh_coarse_apply(h, 0, az, zz)
        torch.cuda.synchronize()
        err = ((zz - z).norm() / z.norm()).item()
        print(f"rank {rank} {precision}: {err:.2e}")
        assert z.norm().item() > 0 and err < {"fp64": 1.1e-10, "mixed": 1e-2}[precision]
    finally:
        hh.hh_destroy(h)
