"""M2M and L2L at the orders where their blocks change shape: rows of two z-halves in two column parts (up to
p = 15, where they fill a block of 1,024 threads), in one (p = 16), less than a warp of rows (p = 2, 3), and levels
with few and with many parents."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2002_01334_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2002_01334_gb300 import build as B  # noqa: E402

B.build()
from paper_2002_01334_gb300 import lpbfmm as F  # noqa: E402

DEV = torch.device("cuda:0")


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def run(w, p, depth, prec):
    m = w["medium"]
    ctx = F.Context(m["d"], m["eps"], m["lam"], p, precision=prec, uniform_depth=depth)
    phi, fld = ctx.eval(torch.tensor(w["q"], device=DEV), torch.tensor(w["xyz"], device=DEV),
                        torch.tensor(w["layer"], dtype=torch.int32, device=DEV))
    return phi.cpu().numpy(), fld.cpu().numpy()


@pytest.mark.parametrize("p,n", [(10, 1501), (10, 60), (12, 60)])
def test_octant_passes_match_the_direct_sum(p, n):
    """FP64 on depth-4 trees against the direct sum, to the truncation's gate of 1e-6.  1,501 charges fill more
    parents than the limit up to which source types are split over blocks; 60 leave most parents one child."""
    w = inputs.workload("three_layer", n=n, seed=43)
    phi, fld = run(w, p, 4, F.FP64)
    ref = oracle.direct(oracle.Medium(**w["medium"]), w["q"], w["xyz"], w["layer"])
    assert rel(phi, ref[0]) < 1e-6 and rel(fld, ref[1]) < 1e-6, (rel(phi, ref[0]), rel(fld, ref[1]))


@pytest.mark.parametrize("p", [2, 14, 16])
def test_octant_passes_agree_in_both_precisions(p):
    """One depth-4 tree in FP32 expansions against FP64 ones: the 1e-6 gate of the mixed mode."""
    w = inputs.workload("three_layer", n=300, seed=44)
    a, b = run(w, p, 4, F.FP64), run(w, p, 4, F.MIXED)
    assert rel(b[0], a[0]) < 1e-6 and rel(b[1], a[1]) < 1e-6, (rel(b[0], a[0]), rel(b[1], a[1]))
    if p >= 14:  # truncation (below 5e-9 at p = 10, falling fourfold per order)
        ref = oracle.direct(oracle.Medium(**w["medium"]), w["q"], w["xyz"], w["layer"])
        assert rel(a[0], ref[0]) < 1e-8, rel(a[0], ref[0])
