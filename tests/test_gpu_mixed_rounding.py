"""Rounding of the mixed mode, as the geometric mean over seeds of its relative L2 distance from the FP64 FMM of the same
trees (one seed's error is a few close pairs or one cancelling sum; the mean over 24 is known to 1.5 %)."""
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


def rounding(layout, n, p, parts, lam_scale, seeds=24, ws=2):
    """Geometric means over the seeds of |mixed - FP64| / |FP64|: potential, field."""
    ctx, e = None, []
    for s in range(500, 500 + seeds):
        w = inputs.workload(layout, n=n, seed=s)
        m = w["medium"]
        if ctx is None:
            lam = [lam_scale * v for v in m["lam"]]
            ctx = [F.Context(m["d"], m["eps"], lam, p, precision=pr, separation=ws) for pr in (F.FP64, F.MIXED)]
        q, x = (torch.tensor(np.float32(w[k]).astype(float), device=DEV) for k in ("q", "xyz"))
        l = torch.tensor(w["layer"], dtype=torch.int32, device=DEV)
        (a, fa), (b, fb) = [c.eval(q, x, l, parts=parts) for c in ctx]
        e.append([float((b - a).norm() / a.norm()), float((fb - fa).norm() / fa.norm())])
    assert ctx[1].status() == 0
    return np.exp(np.log(np.array(e)).mean(0))


@pytest.mark.parametrize("layout,n,p,phi,fld", [("four_layer", 2000, 9, 3.902e-7, 3.876e-7),
                                                ("three_layer", 3000, 10, 4.143e-7, 4.006e-7)])
def test_tensor_core_m2l(layout, n, p, phi, fld):
    """The reaction far field alone, no further off than an M2L on TF32 pairs (11 + 11 bits, 8-bit exponents) on the same
    inputs; 5 % for the mean's own spread."""
    e = rounding(layout, n, p, 2 + 4, 1.0)
    assert e[0] <= phi * 1.05 and e[1] <= fld * 1.05, e



@pytest.mark.parametrize("layout,n,phi", [("four_layer", 10000, 1.382e-7), ("three_layer", 3000, 1.451e-7),
                                          ("three_layer", 30000, 1.145e-7)])
def test_fp32_near_field_sums(layout, n, phi):
    """The free-space part under screening that leaves little but the near field, in leaves of some tens to a hundred
    charges, no further off than sums folded into the compensated totals leaf by leaf on the same inputs; 5 % for the
    mean's own spread."""
    e = rounding(layout, n, 5, 1, 60.0)
    assert e[0] <= phi * 1.05, e
