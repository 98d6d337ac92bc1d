"""The tensor-core multipole-to-local (mixed mode) at the edges of its layouts and scalings."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2002_01334_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2002_01334_gb300 import build as B  # noqa: E402

B.build()
from paper_2002_01334_gb300 import lpbfmm as F  # noqa: E402

DEV = torch.device("cuda:0")


def rel(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("p,ws,scale", [(2, 2, 1.0), (3, 1, 1.0), (5, 2, 1e-19), (6, 2, 1e12), (7, 1, 1.0),
                                        (8, 2, 1.0), (9, 2, 1.0), (10, 1, 1.0), (10, 2, 1e-19)])
@pytest.mark.parametrize("layout", ["three_layer", "four_layer"])
def test_mixed_matches_fp64_on_the_same_trees(p, ws, scale, layout):
    """One column chunk (p = 2) to four (p = 10), odd and even column counts, both separations, sparse trees
    with absent source types, charges far from 1: mixed against FP64 FMM of the same trees, relative L2
    within the library's 1e-6 gate for the mixed mode."""
    w = inputs.workload(layout, n=2500, seed=100 + p)
    m = w["medium"]
    q = torch.tensor(w["q"] * scale, device=DEV)
    x, l = torch.tensor(w["xyz"], device=DEV), torch.tensor(w["layer"], dtype=torch.int32, device=DEV)
    out = []
    for prec in (F.FP64, F.MIXED):
        ctx = F.Context(m["d"], m["eps"], m["lam"], p, precision=prec, uniform_depth=4, separation=ws)
        out.append(ctx.eval(q, x, l, parts=3 + 4))  # the direct reaction near field left out
        assert ctx.status() == 0
    (a, fa), (b, fb) = out
    assert rel(b, a) < 1e-6 and rel(fb, fa) < 1e-6, (rel(b, a), rel(fb, fa))
