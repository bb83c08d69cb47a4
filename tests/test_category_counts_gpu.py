"""FP32 with 4 states, level by level (past what one wave of blocks walks):
every category count, trees with only cherries at their deepest level and
mixed ones, gaps, partial vectors, ragged tiles, against the oracle."""
import numpy as np
import pytest

import synth
from parity import compare, oracle_eval

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_04390_gb300 import build as B
    B.build()


@pytest.mark.parametrize("R", range(1, 9))
@pytest.mark.parametrize("n,S,C,tree,partial", [
    (130, 4, 40, "yule", 0), (130, 4, 33, "balanced", 0), (121, 3, 31, "balanced", 4),
])
def test_matches_oracle(n, S, C, tree, partial, R):
    import paper_2303_04390_gb300 as pg
    from oracle import phylo_oracle as O
    n *= 4 if R < 4 else 1  # a walk holds more nodes of fewer categories
    w = synth.small_workload(n, S, R, C, seed=65, tree=tree)
    rng = np.random.default_rng(n + R)
    w.tip_states[1:][rng.random(w.tip_states[1:].shape) < 0.05] = S  # gaps
    tp = None
    ctx = pg.from_workload(w, "fp32", tip_partials=partial > 0)
    if partial:
        tp = O.tip_partial_vectors(S, w.tip_states)
        for tip in range(0, n, partial):
            tp[tip] = rng.random((C, S)) ** 3 + 0.01
            ctx.set_tip_partials(tip, tp[tip])
    logL, grad = ctx.evaluate()
    assert ctx.kernel_launches()[0] > 4  # by level, not a walk
    compare(logL, grad, oracle_eval(w, tip_partials=tp), "fp32", f"{w.name} {tree}")
    ctx.close()
