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


@pytest.mark.parametrize("n,lam,spread", [(1, 1.0, 0.1), (2, 1.0, 0.0), (33, 1.0, 0.1), (64, 1e-4, 0.1), (65, 30.0, 0.5),
                                          (129, 1.0, 0.5), (1000, 1.0, 0.5)])
def test_fp32_near_field_groups_and_chunks(n, lam, spread):
    """The FP32 near field alone (depth 2, two-box lists: every pair is near) against the FP64 sum in numpy:
    one to many target groups, chunks that span leaves and end odd, coincident charges, screening from none to strong.  The pair arithmetic is FP32 with 2^-22 special functions: relative L2 within the
    1e-6 gate, times lambda r (the exponent's relative rounding) where that is large.  The potential alone
    equals the potential with the field."""
    rng = np.random.default_rng(n)
    xyz = np.column_stack([rng.uniform(-spread, spread, n), rng.uniform(-spread, spread, n),
                           rng.uniform(-0.6 - spread, -0.6 + spread, n)])
    if n > 2:
        xyz[-1] = xyz[0]
    q = rng.uniform(0.5, 1.0, n)
    ctx = F.Context([0.0, -1.2], [1.0, 2.0, 5.0], [0.5, lam, 0.8], 4, precision=F.MIXED, uniform_depth=2)
    args = (torch.tensor(q, device=DEV), torch.tensor(xyz, device=DEV),
            torch.ones(n, dtype=torch.int32, device=DEV))
    phi, fld = (t.cpu().numpy() for t in ctx.eval(*args, parts=1))
    only, _ = ctx.eval(*args, parts=1, field=False)
    d = xyz[:, None, :] - xyz[None, :, :]
    r = np.sqrt((d * d).sum(-1))
    ri = np.divide(1.0, r, out=np.zeros_like(r), where=r > 0)
    e = q[None, :] * np.exp(-lam * r) * ri / (4 * np.pi * 2.0)
    ref_p, ref_f = e.sum(1), ((e * (1 + lam * r) * ri * ri)[:, :, None] * d).sum(1)
    if n <= 2:  # no pair at a distance
        assert np.all(phi == 0.0) and np.all(fld == 0.0)
        return
    tol = 1e-6 * max(1.0, lam * spread / 10)
    assert np.linalg.norm(phi - ref_p) <= tol * np.linalg.norm(ref_p)
    assert np.linalg.norm(fld - ref_f) <= tol * np.linalg.norm(ref_f)
    assert np.array_equal(only.cpu().numpy(), phi)
