"""Kernel launches as counted by phylo_kernel_launches, against what the tree
and the path ask for: whole passes in one launch, split levels, one launch per
level, pre-order levels without a contraction, tip tables and the nodes with
two tips."""
import numpy as np
import pytest

import synth
from oracle import phylo_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_04390_gb300 import build as B
    B.build()


def _levels(w):
    """Nodes by height and by depth, and their children."""
    kids, root = O.tree_children(w.parent)
    height, depth = {}, {root: 0}
    for v in O.postorder_list(w.parent):
        height[v] = 0 if not kids[v] else 1 + max(height[c] for c in kids[v])
    for v in reversed(O.postorder_list(w.parent)):
        for c in kids[v]:
            depth[c] = depth[v] + 1
    inner = range(w.n_tips, len(w.parent))
    up, down = {}, {}
    for v in inner:
        up.setdefault(height[v], []).append(v)
        down.setdefault(depth[v], []).append(v)
    return [up[h] for h in sorted(up)], [down[d] for d in sorted(down)], kids


def _launches(sizes, wide):
    """Split levels, and the runs between them."""
    n, run = 0, False
    for s in sizes:
        n += (s > wide) or not run
        run = s <= wide
    return n


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("n,S,R,C,precision,tree", [
    (8, 4, 1, 250, "fp64", "yule"), (61, 4, 4, 70, "fp32", "yule"),       # whole passes
    (300, 4, 4, 9, "fp64", "yule"), (100, 4, 4, 2500, "fp64", "yule"),    # split levels; no room
    (130, 4, 4, 40, "fp32", "yule"), (12, 20, 4, 50, "fp32", "yule"),     # by level
    (20, 61, 4, 50, "fp32", "yule"), (13, 61, 2, 40, "fp64", "balanced"),
    (96, 61, 8, 130, "fp32", "balanced"), (96, 61, 8, 130, "fp32", "caterpillar"),  # tables
    (9, 122, 2, 40, "fp32", "yule"), (2, 122, 2, 40, "fp32", "yule"),
])
def test_launches(n, S, R, C, precision, tree, use_graph):
    import paper_2303_04390_gb300 as pg
    w = synth.small_workload(n, S, R, C, seed=64, tree=tree)
    up, down, kids = _levels(w)
    ctx = pg.from_workload(w, precision, use_graph=use_graph)
    total, phases = ctx.kernel_launches()
    ctx.evaluate()
    assert ctx.kernel_launches() == (total, phases)
    n_post, n_pre = ctx.level_counts()
    ctx.close()
    if S == 4 and (precision, n) in (("fp64", 8), ("fp32", 61)):
        assert (total, phases) == (3, (1, 1, 1, 1))
        return
    if S == 4 and precision == "fp64":
        room = C < 1217  # (two blocks per SM for its 8-pattern tiles)
        want = (1, _launches([len(x) for x in up], 24) if room else 1,
                _launches([len(x) for x in down], 8) if room else 1, 1)
    elif S <= 20:
        want = (1, n_post, n_pre, 1)
    elif precision == "fp64" or (S == 61 and n * R * -(-C // 128) < 1536):
        want = (1, n_post, n_pre + 1, 1)  # the Eq. 8 ratios
    else:
        def tips(v):
            return sum(c < n for c in kids[v])
        levels = sum(any(tips(v) < 2 for v in x) for x in down)
        cherries = any(tips(v) == 2 for x in down for v in x)
        want = (2, n_post, levels + cherries + 1, 1)
    assert phases == want
    assert total == sum(want)
