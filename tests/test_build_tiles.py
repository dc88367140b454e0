"""Graph builds at the edges of the sort's and the de-duplication's tiles: raw
edge counts around one tile, around the size from which the sort takes larger
tiles, and tiles that are part full; 8- and 9-bit digits; many duplicates, and
every key in one digit.  Whole numbers: equal to the oracle's."""
import numpy as np
import pytest

import oracle
import paper_1606_07550_gb300 as gpr

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGE = 152 * 4096  # the largest sort on the small tiles


@pytest.mark.parametrize("n", [1, 16, 600, 300_000])  # ids of 1, 4, 10 and 19 bits
@pytest.mark.parametrize("m", [1, 33, 4096, 4097, EDGE, EDGE + 1, 90 * 8192 + 1])
@pytest.mark.parametrize("skewed", [False, True])
def test_tile_edges(n, m, skewed):
    rng = np.random.default_rng(n * 7919 + m + skewed)
    src, dst = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    if skewed:  # half of the edges into one node, a quarter out of another, and repeated
        dst[: m // 2] = n - 1
        src[m // 4: m // 2] = n // 2
    ref = oracle.build_csc(n, src, dst)
    g = gpr.graph_build(torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), n)
    cp, ri, od = g.export()
    assert g.info().m == ref.m
    np.testing.assert_array_equal(cp, ref.col_ptr)
    np.testing.assert_array_equal(ri, ref.row_idx)
    np.testing.assert_array_equal(od, ref.outdeg)
    g.free()
