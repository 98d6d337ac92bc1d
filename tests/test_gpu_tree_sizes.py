"""Trees at the sizes where the sorts and box scans change their form: arrays of at most 8,192 points sort in one
block, longer ones in tiles of 2,048; box numbering scans tiles of 2,048 points."""
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


@pytest.mark.parametrize("per_layer", [1, 683, 2048, 2049, 8192, 8193])
def test_keys_and_lists_bit_exact(per_layer):
    """Keys, order of the images and every box list against the oracle (whole numbers: equal)."""
    w = inputs.workload("three_layer", n=3 * per_layer, seed=11)
    md, m, D = oracle.Medium(**w["medium"]), w["medium"], 3
    ctx = F.Context(m["d"], m["eps"], m["lam"], 2, uniform_depth=D)
    ctx.eval(torch.tensor(w["q"], device=DEV), torch.tensor(w["xyz"], device=DEV),
             torch.tensor(w["layer"], dtype=torch.int32, device=DEV), parts=3 + 4)
    for (l, a) in [(0, 1), (1, 2)]:
        tr = ctx.debug_tree(l, a)
        root = np.array(tr["root"])
        tk, tsrc, _ = oracle.tree_keys(md, w["xyz"], w["layer"], l, a, D, root, 0)
        ik, isrc, ityp = oracle.tree_keys(md, w["xyz"], w["layer"], l, a, D, root, 1)
        o, og = np.lexsort((tsrc, tk)), np.lexsort((tr["src_t"], tr["keys_t"]))
        assert np.array_equal(tk[o], tr["keys_t"][og]) and np.array_equal(tsrc[o], tr["src_t"][og])
        assert np.all(np.diff(tr["keys_t"].astype(np.int64)) >= 0)
        dense = np.where(ityp % 2 == 0, 2 * (ityp // 2), 2 * (ityp // 2) - 1)
        o2 = np.lexsort((isrc, dense, ik))
        assert np.array_equal(ik[o2], tr["keys_i"]) and np.array_equal(isrc[o2], tr["src_i"])
        for lev in (2, 3):
            tb, sb = oracle.level_boxes(tk, D, lev), oracle.level_boxes(ik, D, lev)
            for kind in ((0, 1) if lev == D else (0,)):
                off, idx = oracle.lists(tb, sb, lev, kind, 2)
                goff, gidx = ctx.debug_lists(l, a, lev, kind, 1)
                assert np.array_equal(off, goff) and np.array_equal(idx, gidx), (l, a, lev, kind)
