"""Kernels at the block shapes that small trees do not reach: M2M with every source type in one block, near fields whose
leaves hold exactly the numbers of targets at which their groups and rounds change."""
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


def dev(*a):
    return [torch.tensor(v, device=DEV, dtype=torch.int32 if np.asarray(v).dtype.kind == "i" else torch.float64) for v in a]


@pytest.mark.parametrize("p", [3, 10])
def test_m2m_of_many_parents_takes_the_types_in_turn(p):
    """Image multipoles of one group where level 4 has more than 2,048 parents over all groups (counted here), so that a
    block takes a parent's source types in turn, and where that group is evaluated alone (fewer parents, a block per
    type): the same sums, in FP64 rounding, 1e-12 of each box's largest coefficient."""
    w = inputs.workload("four_layer", n=40000, seed=51)
    m = w["medium"]
    ctx = F.Context(m["d"], m["eps"], m["lam"], p, uniform_depth=5)
    K, nt = (p + 1) * (p + 2) // 2, 2 * len(m["d"])

    def image_moments(q, mask=None):
        a = dev(q, w["xyz"], w["layer"].astype(np.int32))
        if mask is None:
            ctx.eval(*a, parts=2 + 4)
        else:
            ctx.eval_groups(*a, mask=mask)
        n = [len(ctx.debug_array(1, 1, "ikeys", lev, np.uint64)) for lev in (2, 3, 4)]
        return n, [ctx.debug_array(1, 1, "Mimg", lev, np.float64).reshape(k, nt, 2 * K) for lev, k in zip((2, 3, 4), n)]

    n, M = image_moments(w["q"])
    groups = [(0, 1), (1, 1), (1, 2), (2, 1), (2, 2), (3, 2)]
    parents = sum(len(ctx.debug_array(l, a, "ikeys", 4, np.uint64)) for l, a in groups)
    assert parents > 2048, parents
    # the group (1, 1) alone: fewer parents, a block per type
    mask = [0] * (2 * len(m["eps"]))
    mask[2 * 1 + 1 - 1] = 2
    n1, M1 = image_moments(w["q"], mask)
    assert n1 == n and n[2] <= 2048
    for a, b in zip(M, M1):
        top = np.abs(b).max(axis=(1, 2), keepdims=True)
        assert np.all(np.abs(a - b) <= 1e-12 * top)
    assert np.abs(M[0]).max() > 0


def one_leaf(n, rng):
    """n charges in one octant of the middle layer's box around (0.3, 0.3, -0.9) and four anchors without charge that fix the
    extents of the tree."""
    x = np.column_stack([rng.uniform(0.2, 0.4, n), rng.uniform(0.2, 0.4, n), rng.uniform(-0.95, -0.75, n)])
    anchor = np.array([[-0.5, -0.5, -0.6], [0.5, -0.5, -0.6], [-0.5, 0.5, -0.6], [-0.5, -0.5, -0.7]])
    q = np.concatenate([rng.uniform(0.5, 1.0, n), np.zeros(4)])
    return q, np.concatenate([x, anchor])


@pytest.mark.parametrize("prec,tol", [(F.FP64, 1e-13), (F.MIXED, 1e-6)])
@pytest.mark.parametrize("n", [1, 2, 3, 16, 17, 31, 32, 33, 63, 64, 65, 128, 129, 192, 193])
def test_near_field_of_exactly_n_targets_in_a_leaf(n, prec, tol):
    """Against the FP64 sum in numpy.  Positive charges, so nothing cancels: FP64 1e-13, FP32 pair arithmetic 1e-6."""
    q, x = one_leaf(n, np.random.default_rng(n))
    lam, eps = 1.0, 2.0
    ctx = F.Context([0.0, -1.2], [1.0, eps, 5.0], [0.5, lam, 0.8], 4, precision=prec, uniform_depth=2)
    a = dev(q, x, np.ones(n + 4, np.int32))
    phi, fld = (t.cpu().numpy() for t in ctx.eval(*a, parts=1))
    keys = ctx.debug_tree(1, 1)["keys_t"]
    assert n in np.unique(keys, return_counts=True)[1].tolist()
    d = x[:, None, :] - x[None, :, :]
    r = np.sqrt((d * d).sum(-1))
    ri = np.divide(1.0, r, out=np.zeros_like(r), where=r > 0)
    e = q[None, :] * np.exp(-lam * r) * ri / (4 * np.pi * eps)
    ref_p, ref_f = e.sum(1), ((e * (1 + lam * r) * ri * ri)[:, :, None] * d).sum(1)
    s = slice(0, n)  # the anchors may be further than the near field reaches
    if n == 1:
        assert np.all(phi[s] == 0.0) and np.all(fld[s] == 0.0)
        return
    assert np.linalg.norm(phi[s] - ref_p[s]) <= tol * np.linalg.norm(ref_p[s])
    assert np.linalg.norm(fld[s] - ref_f[s]) <= tol * np.linalg.norm(ref_f[s])
    only, _ = ctx.eval(*a, parts=1, field=False)
    assert np.array_equal(only.cpu().numpy()[s], phi[s])


def test_fp64_inverse_distance_over_many_binades():
    """One charge and targets at distances 2^-500 to 0.5 on a line through it (a tenth of a binade apart), screening too weak to
    count: phi is q / (4 pi eps r).  Roundings of the FP64 pair: r^2, 1/r (one step), r, the exponential's table and polynomial, two
    products, the scale and two sums, at most 2^-53 each and 2^-52 for 1/r and the exponential: 12 * 2^-53; the field
    along the line has two more 1/r and two products: 18 * 2^-53, where the 1 / r^3 in it is a finite number."""
    k = np.arange(5001)
    r = np.exp2(-k / 10.0 - 1.0)
    x = np.column_stack([np.concatenate([[0.0], r]), np.zeros(len(r) + 1), np.full(len(r) + 1, -0.6)])
    q = np.zeros(len(x))
    q[0] = 1.0
    eps, lam = 2.0, 1e-18
    ctx = F.Context([0.0, -1.2], [1.0, eps, 5.0], [0.5, lam, 0.8], 4, uniform_depth=2)
    phi, fld = (t.cpu().numpy()[1:] for t in ctx.eval(*dev(q, x, np.ones(len(x), np.int32)), parts=1))
    L = np.longdouble
    ref = 1 / (4 * L("3.14159265358979323846264338327950288") * L(eps) * r.astype(L))
    assert np.all(np.abs(phi - ref) <= 12 * 2.0 ** -53 * ref)
    fr = ref / r.astype(L)
    ok = r > 1e-100
    assert ok.sum() > 3300 and np.all(np.abs(fld[ok, 0] - fr[ok]) <= 18 * 2.0 ** -53 * fr[ok])
