"""FP32 with 21 to 64 states on both sides of the line past which compact tips
get tables of their numerators (taxa x 128-pattern tiles x categories >=
1,536): below it every child has its own contraction.  Trees of cherries and
ladders, gaps, ragged tiles, tips with partial vectors, against the oracle."""
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
    (96, 21, 8, 129, "balanced", 0), (95, 21, 8, 129, "balanced", 0),
    (96, 40, 8, 256, "caterpillar", 5), (95, 40, 8, 256, "caterpillar", 5),
    (2, 61, 4, 130, "yule", 0), (3, 64, 3, 1, "yule", 2), (12, 61, 1, 128, "yule", 3),
])
def test_matches_oracle(n, S, R, C, tree, partial):
    import paper_2303_04390_gb300 as pg
    from oracle import phylo_oracle as O
    w = synth.small_workload(n, S, R, C, seed=63, tree=tree)
    rng = np.random.default_rng(n + C)
    w.tip_states[1:][rng.random(w.tip_states[1:].shape) < 0.05] = S  # gaps
    tp = None
    ctx = pg.from_workload(w, "fp32", tip_partials=partial > 0)
    if partial:
        tp = O.tip_partial_vectors(S, w.tip_states)
        for tip in range(0, n, partial):
            tp[tip] = rng.random((C, S)) ** 3 + 0.01
            ctx.set_tip_partials(tip, tp[tip])
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w, tip_partials=tp), "fp32", f"{w.name} {tree}")
    log_t = torch.tensor(np.log(w.t), device="cuda", requires_grad=True)
    ll = pg.branch_loglik(log_t, ctx)
    (g,) = torch.autograd.grad(ll, log_t)
    t = torch.exp(log_t.detach())
    ctx.set_branch_lengths(t)
    logL, grad = ctx.evaluate()
    assert ll.item() == logL
    np.testing.assert_allclose(g.cpu().numpy(), grad * t.cpu().numpy(), rtol=1e-15)
    ctx.close()
