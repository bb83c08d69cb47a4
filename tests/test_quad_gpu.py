"""FP32 with 5 to 20 states on alignments large enough for four patterns per
thread: ragged tiles, every category width, few states, partial vectors and
gaps, on trees whose wide levels take that kernel and whose narrow ones do
not, and both sides of the rule, against the oracle."""
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


@pytest.mark.parametrize("n,S,R,C,tree,partial", [
    (160, 20, 4, 993, "balanced", 0),   # 32 tiles, one pattern in the last
    (160, 20, 4, 992, "balanced", 0),   # 31 tiles: one pattern per thread
    (152, 20, 4, 1024, "yule", 7),
    (110, 7, 3, 1451, "balanced", 0),
    (140, 20, 8, 519, "balanced", 5),
    (150, 11, 2, 2050, "yule", 0),
    (152, 5, 1, 4098, "balanced", 9),
])
def test_matches_oracle(n, S, R, C, tree, partial):
    import paper_2303_04390_gb300 as pg
    from oracle import phylo_oracle as O
    w = synth.small_workload(n, S, R, C, seed=97, tree=tree)
    rng = np.random.default_rng(n + C)
    w.tip_states[1:][rng.random(w.tip_states[1:].shape) < 0.03] = S
    tp = None
    ctx = pg.from_workload(w, "fp32", tip_partials=partial > 0)
    if partial:
        tp = O.tip_partial_vectors(S, w.tip_states)
        for tip in range(0, n, partial):
            tp[tip] = rng.random((C, S)) ** 3 + 0.01
            ctx.set_tip_partials(tip, tp[tip])
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w, tip_partials=tp), "fp32", f"{w.name} {tree}")
    ctx.close()
