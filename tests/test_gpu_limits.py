"""Evaluations in less memory than they would like: the FP64 multipole-to-local in windows and parts, which large inputs need,
reached on small ones by lower limits."""
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


def problem(layout, n, p, depth, prec=F.FP64):
    w = inputs.workload(layout, n=n, seed=77)
    m = w["medium"]
    ctx = F.Context(m["d"], m["eps"], m["lam"], p, precision=prec, uniform_depth=depth)
    return ctx, (torch.tensor(w["q"], device=DEV), torch.tensor(w["xyz"], device=DEV),
                 torch.tensor(w["layer"], dtype=torch.int32, device=DEV))


@pytest.mark.parametrize("window,part", [(4096, 0), (4095, 0), (0, 30000), (1021, 21296)])
def test_windows_and_parts_agree_with_the_undivided_run(window, part):
    """Translations in windows of that many slots and parts of that many (a part holds whole targets, at least 21,296
    numbers; free-space and reaction jobs end up in different ones).  Only the additions of up to some thousand
    translations per target are reassociated: 1e-13."""
    p = 5
    ctx, args = problem("four_layer", 700, p, 3)
    a, fa = ctx.eval(*args, parts=3 + 4)
    base = ctx.counts()["launches"]
    ctx.debug_limits(window=window * 16 * (p + 1) * (p + 2) // 2, part=part)
    b, fb = ctx.eval(*args, parts=3 + 4)
    assert ctx.counts()["launches"] > base + 10  # several of them
    assert rel(b, a) < 1e-13 and rel(fb, fa) < 1e-13, (rel(b, a), rel(fb, fa))
    ctx.debug_limits()
    c, fc = ctx.eval(*args, parts=3 + 4)
    assert torch.equal(c, a) and torch.equal(fc, fa) and ctx.counts()["launches"] == base


def test_short_memory_halves_the_windows():
    """A work space with room for a quarter of the translations' slots beside everything else: evaluated in smaller windows, to
    rounding.  What everything else takes is measured first, by a run whose windows hold an eighth."""
    p = 4
    ctx, args = problem("three_layer", 20000, p, 4)
    a, fa = ctx.eval(*args, parts=3 + 4)
    n = ctx.counts()
    slots = (n["m2l_free"] + n["m2l_react"] // 4) * 16 * (p + 1) * (p + 2) // 2  # at least: not every type is everywhere
    ctx.close()
    ctx, args = problem("three_layer", 20000, p, 4)
    free = torch.cuda.mem_get_info()[0]
    ctx.debug_limits(window=slots // 8)
    ctx.eval(*args, parts=3 + 4)
    held = free - torch.cuda.mem_get_info()[0]
    ctx.close()
    ctx, args = problem("three_layer", 20000, p, 4)
    ctx.debug_limits(memory=held + slots // 4)
    for _ in range(2):  # the second run starts without the first one's pieces
        b, fb = ctx.eval(*args, parts=3 + 4)
        assert ctx.counts()["launches"] > n["launches"]
        assert rel(b, a) < 1e-13 and rel(fb, fa) < 1e-13, (rel(b, a), rel(fb, fa))


@pytest.mark.parametrize("prec", [F.FP64, F.MIXED])
def test_nothing_runs_on_after_an_error(prec):
    """Out of memory at every stage that a growing limit reaches: once the error is returned, the outputs are the caller's
    again (no kernel of another stream adds into them later), and the context goes on to give the same results."""
    ctx, args = problem("three_layer", 100000, 5, 0, prec)
    a, fa = ctx.eval(*args)
    ctx.close()
    phi, fld = torch.empty_like(a), torch.empty_like(fa)
    seen = 0
    for mb in range(64, 100 * 64, 64):
        ctx, args = problem("three_layer", 100000, 5, 0, prec)
        ctx.debug_limits(memory=mb << 20)
        try:
            ctx.eval(*args, out=(phi, fld))
            break
        except F.LpbfmmError as e:
            assert e.code == 7
        seen += 1
        phi.fill_(3.0)
        fld.fill_(4.0)
        torch.cuda.synchronize()
        assert bool((phi == 3.0).all()) and bool((fld == 4.0).all()), mb
        ctx.debug_limits()
        b, fb = ctx.eval(*args)
        assert rel(b, a) < 1e-13 and rel(fb, fa) < 1e-13 and ctx.status() == 0
        ctx.close()
    assert seen >= 2
