"""Levels below the last one with a dense lattice map: source lookups through
bricks of the cells of that level, and through hash tables on the levels whose
bricks would be larger than the map. Points at log-uniform distances from a
centre give a tree of 16 levels and more, with both kinds."""
import numpy as np
import pytest

import oracle
from paper_1106_2176_gb300 import inputs

from gpu_common import rel, run_fmm

pytestmark = pytest.mark.gpu

MIXED_SLACK = 2e-6


def nested(n, octaves, seed):
    r = np.random.default_rng(seed)
    d = r.normal(size=(n, 3))
    d *= (2.0 ** -r.uniform(0, octaves, n) / np.linalg.norm(d, axis=1))[:, None]
    return d + 0.1, r.uniform(-1, 1, n)


def brick_levels(level):
    """How many levels below 8 have bricks (8^(l - 8) entries per cell of level 8,
    from level 9 down while all together are no more than 8^8) and how many not."""
    top, words, k = int(np.sum(level == 8)), 0, 0
    for l in range(9, int(level.max()) + 1):
        words += top << (3 * (l - 8))
        if words > 8**8:
            break
        k += 1
    return k, max(0, int(level.max()) - 8 - k)


# nested shells: bricks on the first levels below 8, tables on the others;
# Plummer with more than 512 cells on levels 9 and 10 (tiles of one octant, several
# ranges of vectors), both in bricks
@pytest.mark.parametrize("gen,n,ncrit,depth", [("nested", 36000, 8, 12), ("nested", 20000, 4, 16), ("plummer", 200000, 8, 10)])
def test_deep_levels_against_direct_sum(gen, n, ncrit, depth):
    x, q = nested(n, {36000: 12, 20000: 17}[n], 7) if gen == "nested" else inputs.plummer(n, 47)
    t = inputs.sample_targets(n, 512, seed=47)
    pd, gd = oracle.direct(x, q, targets=t)
    p64, g64, f64 = run_fmm(x, q, 6, 0.5, ncrit, precision="fp64")
    pm, gm, fm = run_fmm(x, q, 6, 0.5, ncrit, precision="mixed")
    bricks, tables = brick_levels(fm.export_tree()["level"])
    assert bricks >= 2 and (tables >= 2 if gen == "nested" else True)
    assert fm.stats()["depth"] >= depth and fm.stats()["async_error"] == 0 and f64.stats()["async_error"] == 0
    # a lookup that misses a cell, or finds another, leaves out whole interactions (1e-2 and more)
    assert rel(p64[t], pd) < 1e-4 and rel(g64[t], gd) < 1e-4
    assert rel(pm[t], pd) <= rel(p64[t], pd) + MIXED_SLACK and rel(gm[t], gd) <= rel(g64[t], gd) + MIXED_SLACK
    f64.close()
    fm.close()
