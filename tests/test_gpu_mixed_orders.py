"""The mixed mode at the orders between its multipole-to-local kernels: p = 4 and 10 on the tensor cores (two and four
chunks of columns), 11 alone in the double-buffered FP32 kernel, 12 and up in the tiled one."""
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


@pytest.mark.parametrize("p", [4, 10, 11, 12])
@pytest.mark.parametrize("layout,n", [("four_layer", 900), ("three_layer", 5000)])
def test_mixed_matches_fp64(p, layout, n):
    """Sparse boxes (most source types absent) and full ones, against the FP64 FMM of the same trees: the mixed mode's 1e-6
    gate; twice, the second time in the work space of a larger evaluation."""
    w, w2 = inputs.workload(layout, n=n, seed=31), inputs.workload(layout, n=2 * n, seed=32)
    m = w["medium"]
    out = []
    for prec in (F.FP64, F.MIXED):
        ctx = F.Context(m["d"], m["eps"], m["lam"], p, precision=prec, uniform_depth=3)
        for v in (w, w2, w):
            r = ctx.eval(torch.tensor(v["q"], device=DEV), torch.tensor(v["xyz"], device=DEV),
                         torch.tensor(v["layer"], dtype=torch.int32, device=DEV), parts=3 + 4)
            out.append(r)
        assert ctx.status() == 0
    for (a, fa), (b, fb) in zip(out[:3], out[3:]):
        assert rel(b, a) < 1e-6 and rel(fb, fa) < 1e-6, (rel(b, a), rel(fb, fa))
    assert torch.equal(out[3][0], out[5][0]) and torch.equal(out[3][1], out[5][1])
