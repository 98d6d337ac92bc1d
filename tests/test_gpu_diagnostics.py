"""Arrays copied out for inspection: what an evaluation leaves out reads as zero, whatever the work space held before."""
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


@pytest.mark.parametrize("prec,p", [(F.FP64, 5), (F.MIXED, 5), (F.MIXED, 11)])
def test_absent_rows_and_entries_are_zero(prec, p):
    T = np.float64 if prec == F.FP64 else np.float32
    ctx = None
    for n in (6000, 900):  # the larger run fills the work space that the smaller one is given
        w = inputs.workload("four_layer", n=n, seed=9)
        m = w["medium"]
        ctx = ctx or F.Context(m["d"], m["eps"], m["lam"], p, precision=prec, uniform_depth=3)
        ctx.eval(torch.tensor(w["q"], device=DEV), torch.tensor(w["xyz"], device=DEV),
                 torch.tensor(w["layer"], dtype=torch.int32, device=DEV), parts=3 + 4)
    K, KT, nt = (p + 1) * (p + 2) // 2, 2 * p + 3, 2 * len(m["d"])
    absent = 0
    for (l, a) in [(1, 1), (2, 2)]:
        tr = ctx.debug_tree(l, a)
        dense = np.where(tr["type_i"] % 2 == 0, 2 * (tr["type_i"] // 2), 2 * (tr["type_i"] // 2) - 1)
        for lev in (2, 3):
            keys = ctx.debug_array(l, a, "ikeys", lev, np.uint64)
            box = np.searchsorted(keys, tr["keys_i"] >> np.uint64(3 * (tr["depth"] - lev)))
            have = np.zeros((len(keys), nt), bool)
            have[box, dense] = True
            M = ctx.debug_array(l, a, "Mimg", lev, T).reshape(len(keys), nt, 2 * K)
            assert np.all(M[~have] == 0) and np.all(np.abs(M[have]).max(-1) > 0)
            absent += int((~have).sum())
            used = ctx.debug_array(l, a, "used", lev, np.uint8).astype(bool)
            S = ctx.debug_array(l, a, "stab", lev, np.float64).reshape(len(used), nt, KT + 1, KT + 1, 4)
            k, d = np.meshgrid(np.arange(KT + 1), np.arange(KT + 1), indexing="ij")
            out = (d > k) | ((k - d) % 2 == 0)
            assert np.all(S[:, :, out] == 0) and np.all(S[~used] == 0) and np.any(S[used] != 0)
    assert absent > 0
