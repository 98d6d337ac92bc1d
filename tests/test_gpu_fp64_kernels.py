"""FP64 kernels at the sizes where they can go wrong: the operator-sorted multipole-to-local lists at
the smallest, odd and largest orders, and the near field at the edges of its target groups."""
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


@pytest.mark.parametrize("n,lam", [(2, 1.0), (31, 1.0), (32, 1.0), (33, 1e-4), (67, 30.0), (257, 2500.0)])
def test_near_field_target_groups_and_screening(n, lam):
    """n charges of one leaf (all within a box of a depth-2 tree) and two coincident ones, from weak
    screening to lambda r beyond the exponent range, against the FP64 sum in numpy: 1e-13, the sum's own
    rounding; potential alone equal to the potential with the field."""
    rng = np.random.default_rng(n)
    xyz = np.column_stack([rng.uniform(-0.1, 0.1, n), rng.uniform(-0.1, 0.1, n), rng.uniform(-0.8, -0.6, n)])
    xyz[-1] = xyz[0]
    q = rng.uniform(0.5, 1.0, n)
    m = dict(d=[0.0, -1.2], eps=[1.0, 2.0, 5.0], lam=[0.5, lam, 0.8])
    layer = np.ones(n, np.int32)
    phi, fld = run(m, q, xyz, layer, 4, 1, 2)
    only, _ = run(m, q, xyz, layer, 4, 1, 2, field=False)
    d = xyz[:, None, :] - xyz[None, :, :]
    r = np.sqrt((d * d).sum(-1))
    ri = np.divide(1.0, r, out=np.zeros_like(r), where=r > 0)
    e = q[None, :] * np.exp(-lam * r) * ri / (4 * np.pi * 2.0)
    ref_p, ref_f = e.sum(1), ((e * (1 + lam * r) * ri * ri)[:, :, None] * d).sum(1)
    if n == 2:  # the two charges coincide: no interaction
        assert np.all(phi == 0.0) and np.all(fld == 0.0)
        return
    # lambda r rounds to relative 2^-53: the exponential's relative error grows with lambda r
    tol = 1e-13 * max(1.0, lam / 100.0)
    assert rel(phi, ref_p) < tol and rel(fld, ref_f) < tol, (rel(phi, ref_p), rel(fld, ref_f))
    assert np.array_equal(only, phi)
