"""Settings that take effect at the next build (include/fmm.h) leave the tree
that is built alone: an evaluation after the setter is bitwise the one before."""
import numpy as np
import pytest

from paper_1106_2176_gb300 import inputs

from gpu_common import run_fmm, torch_cuda

pytestmark = pytest.mark.gpu


# pooled tiles walk the union of the octants' stencils, tiles of one octant less:
# the ranges of a tile's vectors must be those of the tiles that were built
@pytest.mark.parametrize("P,precision,engine", [(6, "fp64", "rotation"), (8, "fp64", "auto"), (16, "mixed", "auto"),
                                                (8, "mixed", "tensor"), (6, "fp64", "cudacore")])
@pytest.mark.parametrize("before,after", [(4096, 0), (0, 4096), (-1, 0)])
def test_pool_threshold_waits_for_the_next_build(P, precision, engine, before, after):
    torch = torch_cuda()
    x, q = inputs.uniform_cube(30000, 3)
    phi, grad, f = run_fmm(x, q, P, 0.5, 32, precision=precision, engine=engine, m2l_pool=before)
    f.set_m2l_pool(after)
    phi2, grad2 = (t.clone() for t in f.evaluate())
    f.update_charges(torch.tensor(q, device="cuda"))
    phi3, grad3 = f.evaluate()
    torch.cuda.synchronize()
    for a, b in ((phi2, grad2), (phi3, grad3)):
        assert np.array_equal(a.cpu().numpy(), phi) and np.array_equal(b.cpu().numpy(), grad)
    f.close()
