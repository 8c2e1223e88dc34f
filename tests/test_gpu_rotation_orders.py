"""The rotation engine's kernel at every way its work is cut: orders of four and
of eight warps, odd sizes of a degree's maps (padded rows), trees with one and
with many ranges of vectors per tile, partly filled tiles; against the dense
engine on the same tree."""
import pytest

from paper_1106_2176_gb300 import inputs

from gpu_common import rel, run_fmm

pytestmark = pytest.mark.gpu


# FP64: both engines sum O(10^4) terms in FP64, in another order (1e-15; 1e-12 is
# the bound the engines are held to against the oracle)
@pytest.mark.parametrize("P,gen,n,ncrit", [(1, "uniform", 3000, 32), (2, "uniform", 3000, 32), (3, "plummer", 5000, 16),
                                           (7, "plummer", 5000, 16), (8, "uniform", 40000, 16), (9, "uniform", 5000, 64),
                                           (10, "plummer", 5000, 32), (11, "uniform", 3000, 32), (13, "plummer", 3000, 32),
                                           (15, "uniform", 2000, 32)])
def test_fp64_matches_dense_engine(P, gen, n, ncrit):
    x, q = getattr(inputs, "uniform_cube" if gen == "uniform" else "plummer")(n, 40 + P)
    pr, gr, f = run_fmm(x, q, P, 0.5, ncrit, precision="fp64", engine="rotation")
    pd, gd, _ = run_fmm(x, q, P, 0.5, ncrit, precision="fp64", engine="cudacore")
    assert f.stats()["async_error"] == 0
    assert rel(pr, pd) <= 1e-12 and rel(gr, gd) <= 1e-12


# FP32 rotation against the FP64 FMM of the same tree: FP32 rounding alone (sums
# of both signs), far below the mixed path's bound of 2e-6
@pytest.mark.parametrize("P,gen", [(4, "uniform"), (9, "plummer"), (12, "plummer"), (14, "uniform"), (15, "plummer")])
def test_fp32_within_rounding_of_fp64(P, gen):
    x, q = getattr(inputs, "uniform_cube" if gen == "uniform" else "plummer")(6000, 60 + P)
    pm, gm, _ = run_fmm(x, q, P, 0.5, 32, precision="mixed", engine="rotation")
    p64, g64, _ = run_fmm(x, q, P, 0.5, 32, precision="fp64", engine="rotation")
    assert rel(pm, p64) < 2e-6 and rel(gm, g64) < 2e-6
