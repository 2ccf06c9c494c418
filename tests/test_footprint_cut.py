"""What the iteration on the cut rows adds to a handle's footprint (host only; the server
admits by it): the bases' rows at the cuts, the packed inverse of the coarse system and rows,
which the iteration reads.  What the set-up alone needs lies in storage of the whole-grid
calls, and nothing grows as the square of the number of corrections D = 2 r (2^L - 1)."""
import pytest

CASES = [(63, 2, 16, 8), (255, 2, 16, 10), (126, 4, 32, 10), (254, 5, 32, 10), (254, 6, 16, 8), (254, 6, 32, 0),
         (62, 4, 32, 0), (30, 3, 16, 8), (500, 3, 32, 10), (1023, 6, 32, 10)]


def _rows(S, levels, e=1):
    """Rows of the bands of levels 1 .. levels (owned rows and e more on each inner side)."""
    out, owned = [], [(0, S)]
    for _ in range(levels):
        owned = [x for a, b in owned for x in ((a, a + (b - a) // 2), (a + (b - a) // 2, b))]
        out.append([min(S, b + e) - max(0, a - e) for a, b in owned])
    return out


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n,L,r,p", CASES)
def test_cut_rows_add_what_they_read(n, L, r, p, precision):
    import paper_2512_12538_gb300 as hh

    def fp(n_inner):       # n_i = 2 iterates on the whole grid: the same handle without the cut rows
        return hh.hh_footprint(hh.make_params(2, n, 20.0, L, 2, r, p, n_inner, precision=precision))

    c, S, m, cuts = (8 if precision == "mixed" else 16), n + 2, r + p, 2 ** L - 1
    D = 2 * r * cuts
    packed = 4 * r * r * (L * 2 ** L - cuts)                        # M by subtree
    panels = 2 * S * r * cuts * (2 * L + 1)                         # C and A C at every cut
    groups = sum(2 ** l * (2 * L - l) for l in range(L))            # of A C alone
    keep = c * (panels + packed + 6 * cuts * S + 3 * D)
    items = c * 4 * S * (148 + 2 ** L * 8) * 8                      # rows per item of a step (generous)
    # the set-up's own: A C in FP64, the system and its inverse, one level's sketch rows
    level = max(2 ** l * (c * (6 * S * m + (24 * (L - l + 1) * r * m if l < L else 0)) + 32 * (L - l) * r * m)
                for l in range(1, L + 1))
    setup = 16 * (2 * S * r * groups + 2 * packed) + level
    rows = _rows(S, L)
    pool = c * max(m, r) * S * (sum(map(sum, rows)) + sum(map(sum, rows[:-1])))
    tables = 2 << 20
    extra = fp(1) - fp(2)
    assert extra <= keep + items + max(0, setup - pool) + tables, (extra, keep, items, setup, pool)
    if D > 1000:           # two full complex128 matrices would not fit in this
        assert extra < keep + items + max(0, setup - pool) + tables < 32 * D * D + keep
