"""M2M and L2L of the mixed path on levels with cells enough for a warp to apply
one map to several cells (2,048 parents, or cells): the smallest and largest
orders that do so, the first that does not, full octants (one map for all of a
warp's cells) and missing siblings (a map per cell)."""
import numpy as np
import pytest

from paper_1106_2176_gb300 import inputs

from gpu_common import rel, run_fmm

pytestmark = pytest.mark.gpu


# p = 13 and 14: the staging of M2M fits and does not; 19: the largest order
# whose L2L staging does (deep trees overflow FP32 from p = 18 on)
@pytest.mark.parametrize("P,gen,n,ncrit", [(1, "uniform", 60000, 8), (2, "plummer", 40000, 4), (6, "uniform", 60001, 8),
                                           (11, "plummer", 30000, 4), (13, "uniform", 60000, 8), (13, "plummer", 30000, 4),
                                           (14, "plummer", 30000, 4), (16, "uniform", 60000, 8), (17, "plummer", 20000, 4),
                                           (19, "uniform", 60000, 8)])
def test_expansions_within_rounding_of_fp64(P, gen, n, ncrit):
    x, q = getattr(inputs, "uniform_cube" if gen == "uniform" else "plummer")(n, 120 + P)
    q = np.abs(q)  # one sign: a cell's total charge does not cancel (p = 1 has nothing else to scale by)
    p64, g64, f64 = run_fmm(x, q, P, 0.5, ncrit, precision="fp64")
    pm, gm, fmx = run_fmm(x, q, P, 0.5, ncrit, precision="mixed")
    assert fmx.stats()["async_error"] == 0
    lev = f64.export_tree()["level"]
    assert np.bincount(lev)[2:].max() >= 8 * 2048 or gen == "plummer" and np.bincount(lev).max() >= 2048
    # M: at most 10 nested FP32 sums of 8 p^2 products, 2e-5 of a cell's largest
    # coefficient (the bound of the M2L tests on L)
    (Mx, _), (M64, _) = fmx.export_expansions(), f64.export_expansions()
    sel = lev >= 2
    sc = np.max(np.abs(M64[sel]), axis=1, keepdims=True) + 1e-300
    assert np.max(np.abs(Mx[sel] - M64[sel]) / sc) < 2e-5
    # L by its results (cell by cell the M2L's own rounding comes first): a cell
    # left out or mapped wrongly would show as 1e-3 and more; 2e-6 is the bound
    # that mixed precision keeps to FP64 throughout
    assert rel(pm, p64) < 2e-6 and rel(gm, g64) < 2e-6
    f64.close()
    fmx.close()
