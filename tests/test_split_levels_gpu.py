"""FP64 with 4 states past what shared memory holds: wide levels split over
several blocks per tile, runs of narrow ones in one launch.  Few and many
tiles around the lines of the rule (8 patterns a tile with 4 categories; 38
tiles: a quarter of the SMs; 152: no room for a second block), trees with only
wide, only narrow and both kinds of levels, against the oracle."""
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


@pytest.mark.parametrize("n,R,C,tree", [
    (400, 4, 1, "yule"), (300, 4, 9, "balanced"), (70, 4, 9, "caterpillar"), (300, 1, 33, "yule"),
    (300, 8, 5, "yule"), (257, 2, 17, "balanced"), (120, 4, 304, "yule"), (120, 4, 305, "yule"),
    (100, 4, 1216, "balanced"), (100, 4, 1217, "balanced"),
])
def test_matches_oracle(n, R, C, tree):
    import paper_2303_04390_gb300 as pg
    w = synth.small_workload(n, 4, R, C, seed=61, tree=tree)
    rng = np.random.default_rng(n + C)
    w.tip_states[1:][rng.random(w.tip_states[1:].shape) < 0.1] = 4  # gaps
    ctx = pg.from_workload(w, "fp64")
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w), "fp64", f"{w.name} {tree}")
    log_t = torch.tensor(np.log(w.t), device="cuda", requires_grad=True)
    ll = pg.branch_loglik(log_t, ctx)
    (g,) = torch.autograd.grad(ll, log_t)
    t = torch.exp(log_t.detach())
    ctx.set_branch_lengths(t)
    logL, grad = ctx.evaluate()
    assert ll.item() == logL
    np.testing.assert_allclose(g.cpu().numpy(), grad * t.cpu().numpy(), rtol=1e-15)
    ctx.close()


def test_many_taxa_few_patterns_use_the_gpu():
    """4,096 taxa x 1 pattern: 0.33 ms; one block for the tile takes 4.1 ms."""
    import paper_2303_04390_gb300 as pg
    w = synth.small_workload(4096, 4, 4, 1, seed=62)
    ctx = pg.from_workload(w, "fp64")
    best = float("inf")
    for _ in range(10):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        ctx.evaluate_device()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    ctx.close()
    assert best < 1.5
