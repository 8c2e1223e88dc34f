"""Tensor-core M2L on cells of one level whose multipoles differ by more than
FP16's range: weak charges far from strong ones that cancel. The levels on which
the weak ones' potential would lose bits are summed in FP32; mixed precision then
keeps to FP64 over the weak group alone as it does elsewhere."""
from math import factorial, log2, sqrt

import numpy as np
import pytest

from paper_1106_2176_gb300 import inputs

from gpu_common import ensure_built, rel, run_fmm, torch_cuda

pytestmark = pytest.mark.gpu


def two_groups(n, Q, spread, seed):
    """n charges U[-1, 1] in a ball of radius `spread`, and n more in a ball far
    away: squares of +Q, -Q, -Q, +Q, whose monopoles and dipoles cancel."""
    r = np.random.default_rng(seed)

    def ball(m):
        d = r.normal(size=(m, 3))
        return d * (spread * r.uniform(0, 1, m) ** (1 / 3) / np.linalg.norm(d, axis=1))[:, None]

    def on_grid(v):  # exact in FP32
        return np.round(v * 2.0**24) * 2.0**-24

    c, m = np.array([0.5, 0.25, 0.125]), n // 4
    xw, qw = on_grid(ball(n) - c), r.uniform(-1, 1, n)
    o, side = on_grid(ball(m) + c), on_grid(spread / 8)
    k = r.integers(0, 3, m)
    e1, e2 = np.eye(3)[k] * side, np.eye(3)[(k + 1) % 3] * side
    x = np.concatenate([xw, o, o + e1, o + e2, o + e1 + e2])
    q = np.concatenate([qw, np.repeat([1.0, -1.0, -1.0, 1.0], m) * Q])
    return x.astype(np.float32), q.astype(np.float32)


def exposed_levels(f, p):
    """Levels with a cell that is 2^-16 and more below the level's largest
    coefficient, its ancestors included (per cell width)."""
    a = np.array([2.0 ** (round(log2(sqrt(factorial(n + (k + 1) // 2) * factorial(n - (k + 1) // 2)))) - n)
                  for n in range(p) for k in range(2 * n + 1)])
    M, _ = f.export_expansions()
    t = f.export_tree()
    lev, par = t["level"], t["parent"]
    c = np.abs(M * a).max(axis=1)
    s = np.where(c > 0, np.floor(np.log2(np.where(c > 0, c, 1))), -200) + lev  # exponent of a / w, up to the root's
    for i in range(1, len(s)):  # parents come first
        if par[i] > 0:
            s[i] = max(s[i], s[par[i]])
    s = np.maximum(s, s[0])
    e = [np.floor(np.log2(c[lev == l].max())) for l in range(lev.max() + 1)]
    return {int(l) for l in range(2, lev.max() + 1) if np.any(s[lev == l] <= e[l] - 16 + l)}


# balls 2^-12 wide, 8,000 particles, depth 14. 2e-6: the bound that mixed keeps to
# FP64 throughout. (The seed gives strong charges that no cell face cuts above level
# 11: cut, halves of them with large dipoles leave 1e-5 of FP32 rounding in M2M in
# any engine.) Q = 2^32: rounding the strong charges' moments to FP32 leaves
# dipoles of about 2^-25 Q 2^-14 each, sqrt(4000) of them over |D|^2 = 1.3: 0.2 of a
# potential of 1.7e5, and as much again at each of the 14 levels of M2M: 2e-5.
# (Rows scaled by the level alone: 2e-5 at 2^24, 3e-4 at 2^28, 4e-3 at 2^32.)
@pytest.mark.parametrize("P", [3, 5, 6, 8, 9, 11])
@pytest.mark.parametrize("e,bound", [(24, 2e-6), (28, 2e-6), (32, 2e-5)])
def test_weak_charges_far_from_strong_ones(P, e, bound):
    n = 4000
    x, q = two_groups(n, 2.0**e, 2.0**-12, 5)
    p64, g64, f64 = run_fmm(x, q, P, 0.5, 32, precision="fp64")
    for pool in (-1, 0):  # pooled tiles, tiles of one octant
        pm, gm, f = run_fmm(x, q, P, 0.5, 32, precision="mixed", dtype=np.float32, m2l_pool=pool)
        assert f.stats()["m2l_engine"] == 1 and f.stats()["async_error"] == 0
        assert len(exposed_levels(f, P)) >= 3
        assert rel(pm[:n], p64[:n]) < bound and rel(gm[:n], g64[:n]) < bound
        assert rel(pm, p64) < 2e-6 and rel(gm, g64) < 2e-6
        f.close()
    f64.close()


# a full level whose sources otherwise come by TMA (5: 32,768 cells): tiny charges
# and eight strong ones of alternating sign; by gathers too, bit for bit, at orders
# of packed rows, one and two k-blocks
@pytest.mark.parametrize("P", [4, 8, 10])
def test_wide_levels_are_the_same_with_and_without_lattice_loads(P):
    n = 1000000
    x, q = inputs.uniform_cube(n, 33)
    corner = np.array([[i, j, k] for i in (0, 1) for j in (0, 1) for k in (0, 1)])
    x[:8] = 0.25 + corner / 16.0
    q *= 2.0**-32
    q[:8] = 1.0 - 2.0 * (corner.sum(axis=1) % 2)
    x, q = x.astype(np.float32), q.astype(np.float32)
    p1, g1, f1 = run_fmm(x, q, P, 0.5, 64, precision="mixed", dtype=np.float32, m2l_lattice=True)
    assert f1.stats()["lattice_levels"] & (1 << 5) and 5 in exposed_levels(f1, P)
    p0, g0, f0 = run_fmm(x, q, P, 0.5, 64, precision="mixed", dtype=np.float32, m2l_lattice=False)
    assert f1.stats()["async_error"] == 0 and f0.stats()["async_error"] == 0
    assert np.array_equal(p1, p0) and np.array_equal(g1, g0)
    f1.close()
    f0.close()


# a few systems, and enough of them that every block takes wide and other items in turn
@pytest.mark.parametrize("P,copies", [(6, 1), (4, 12), (8, 12), (10, 6)])
def test_batch_with_wide_systems_matches_their_own_evaluations(P, copies):
    torch = torch_cuda()
    ensure_built()
    from paper_1106_2176_gb300.batch import FMMBatch
    systems = []
    for k in range(copies):
        systems += [two_groups(4000, 2.0**28, 2.0**-12, 5 + k), inputs.uniform_cube(5000, 6 + k, dtype=np.float32),
                    inputs.plummer(20000, 7 + k, dtype=np.float32), two_groups(1000, 2.0**40, 2.0**-9, 8 + k)]
    b = FMMBatch([(torch.tensor(x, device="cuda"), torch.tensor(q, device="cuda")) for x, q in systems], p=P, theta=0.5,
                 ncrit=32, precision="mixed")
    assert [bool(exposed_levels(f, P)) for f in b.handles[:4]] == [True, False, False, True]
    ref = [(p.clone(), g.clone()) for p, g in b.evaluate_each()]
    for k in range(3):  # the later ones on the earlier ones' workspaces
        for p, g in b.out:
            p.fill_(float("nan"))
            g.fill_(float("nan"))
        b.evaluate() if k < 2 else b.replay()
        torch.cuda.synchronize()
        assert b.status()[0] == 0
        for (p, g), (pr, gr) in zip(b.out, ref):
            assert bool((p == pr).all()) and bool((g == gr).all())
    b.close()
