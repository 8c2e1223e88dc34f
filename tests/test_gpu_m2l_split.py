"""Tensor-core M2L in split FP16: the rows and operators are brought into FP16's
range by powers of two, so the results must not depend on the scale of the
charges, at any order and whether a tile's vectors are cut into ranges or not;
and every order stays within FP32 rounding of the FP64 path."""
import numpy as np
import pytest

from paper_1106_2176_gb300 import inputs

from gpu_common import rel, run_fmm

pytestmark = pytest.mark.gpu

# (order, particles, leaf size): pooled tiles alone, few and many tiles (the
# ranges per tile fall from 30 to 1), 1 and 2 k-blocks, packed rows (p <= 5)
CASES = [(2, 3000, 32), (4, 16384, 64), (5, 60000, 32), (6, 1000, 64), (7, 200000, 64), (8, 30000, 32), (9, 20000, 64),
         (10, 100003, 64), (11, 20000, 64)]


@pytest.mark.parametrize("P,n,ncrit", CASES)
@pytest.mark.parametrize("gen", ["uniform_cube", "plummer"])
def test_results_scale_exactly_with_the_charges(P, n, ncrit, gen):
    x, _ = getattr(inputs, gen)(n, 90 + P)
    q = np.random.default_rng(P).uniform(-1, 1, n).astype(np.float32)
    x = x.astype(np.float32)
    p1, g1, f = run_fmm(x, q, P, 0.5, ncrit, precision="mixed", dtype=np.float32)
    assert f.stats()["m2l_engine"] == 1 and f.stats()["async_error"] == 0
    _, L1 = f.export_expansions()
    for e in (40, -40):
        # powers of two: every product and sum scales exactly (nothing is near FP32's limits)
        p2, g2, f2 = run_fmm(x, np.ldexp(q, e), P, 0.5, ncrit, precision="mixed", dtype=np.float32)
        _, L2 = f2.export_expansions()
        assert np.array_equal(L2, np.ldexp(L1, e))
        assert np.array_equal(p2, np.ldexp(p1, e)) and np.array_equal(g2, np.ldexp(g1, e))
        f2.close()
    f.close()


@pytest.mark.parametrize("P,n,ncrit", CASES)
def test_within_rounding_of_fp64(P, n, ncrit):
    n = min(n, 30000)
    x, q = inputs.uniform_cube(n, 70 + P)
    pm, gm, _ = run_fmm(x, q, P, 0.5, ncrit, precision="mixed")
    p64, g64, _ = run_fmm(x, q, P, 0.5, ncrit, precision="fp64")
    assert rel(pm, p64) < 2e-6 and rel(gm, g64) < 2e-6
