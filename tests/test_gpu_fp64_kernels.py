"""FP64 kernels at the sizes where they can go wrong: the operator-sorted multipole-to-local lists at
the smallest, odd and largest orders."""
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


def run(m, q, xyz, layer, p, parts, depth, field=True):
    ctx = F.Context(m["d"], m["eps"], m["lam"], p, uniform_depth=depth)
    phi, fld = ctx.eval(torch.tensor(q, device=DEV), torch.tensor(xyz, device=DEV),
                        torch.tensor(layer, dtype=torch.int32, device=DEV), parts=parts, field=field)
    return phi.cpu().numpy(), (fld.cpu().numpy() if field else None)


@pytest.mark.parametrize("p,parts", [(2, 1), (2, 2), (7, 3), (16, 1)])
def test_operator_sorted_m2l(p, parts):
    """Against the oracle's CPU FMM of the same trees (rounding: 1e-10), free and reaction translations into
    the same expansions included; at p = 16 against the direct sum, whose distance is the truncation,
    falling 16-fold per two orders from 6.6e-9 at p = 10 (bound 1e-10)."""
    from oracle import fmm as cfmm
    w = inputs.workload("three_layer", n=201, seed=41)
    m = w["medium"]
    md = oracle.Medium(**m)
    phi, fld = run(m, w["q"], w["xyz"], w["layer"], p, parts, 3)
    if p == 16:
        ref = oracle.direct(md, w["q"], w["xyz"], w["layer"], parts=1)
    else:
        ref = [0.0, 0.0]
        if parts & 1:
            ref = [a + b for a, b in zip(ref, cfmm.free_fmm(md, w["q"], w["xyz"], w["layer"], p, 3, 2))]
        if parts & 2:
            ref = [a + b for a, b in zip(ref, cfmm.react_fmm(md, w["q"], w["xyz"], w["layer"], p, 3, 2))]
    assert rel(phi, ref[0]) < 1e-10 and rel(fld, ref[1]) < 1e-10, (rel(phi, ref[0]), rel(fld, ref[1]))
