"""The 4-state passes that run as one launch (a pattern tile walks the whole
tree): every tile shape and remainder, the largest problem that shared
memory holds and the smallest that it does not, groups of one, two and four
tiles per block, against the oracle at the parity tests' tolerances."""
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


def _with_gaps(w, seed):
    rng = np.random.default_rng(seed)
    w.tip_states[rng.random(w.tip_states.shape) < 0.1] = w.n_states
    w.tip_states[0] = np.minimum(w.tip_states[0], w.n_states - 1)  # no all-gap column
    return w


# (taxa, categories, patterns, tree)
SHAPES = [
    (2, 4, 1, "yule"), (3, 4, 7, "yule"), (5, 4, 8, "caterpillar"), (5, 4, 9, "yule"),
    (12, 1, 31, "yule"), (12, 1, 33, "balanced"), (9, 2, 17, "yule"), (9, 3, 16, "yule"),
    (9, 5, 13, "caterpillar"), (9, 8, 5, "yule"), (70, 4, 20, "balanced"),
    (56, 4, 9, "yule"), (57, 4, 9, "yule"),      # FP64: shared memory holds 56 taxa
    (111, 4, 9, "yule"), (112, 4, 9, "yule"),    # FP32: 111 taxa
    (10, 4, 1216, "yule"), (10, 4, 1217, "yule"),  # one tile per block up to 1,216 patterns
    (10, 4, 2433, "yule"),                         # four tiles per block
    (60, 4, 77, "caterpillar"),
]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,R,C,tree", SHAPES)
def test_matches_oracle(n, R, C, tree, precision):
    import paper_2303_04390_gb300 as pg
    w = _with_gaps(synth.small_workload(n, 4, R, C, seed=91, tree=tree), n + C)
    ctx = pg.from_workload(w, precision)
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w), precision, f"{w.name} {tree}")
    ctx.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [14, 80])
def test_tip_partials(n, precision):
    import paper_2303_04390_gb300 as pg
    from oracle import phylo_oracle as O
    w = synth.small_workload(n, 4, 4, 21, seed=92)
    tp = O.tip_partial_vectors(4, w.tip_states)
    rng = np.random.default_rng(n)
    ctx = pg.from_workload(w, precision, tip_partials=True)
    for tip in range(0, n, 3):
        tp[tip] = rng.random((21, 4)) ** 3 + 0.01
        ctx.set_tip_partials(tip, tp[tip])
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w, tip_partials=tp), precision, "tip partials")
