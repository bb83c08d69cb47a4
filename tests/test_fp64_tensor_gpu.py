"""FP64 with 21 to 64 states, whose products are exact integer contractions
of base-256 digits on the tensor cores: the smallest and largest state counts,
ragged pattern tiles, odd category counts (a matrix block then holds a tip's
and an internal branch's matrices), partial vectors, gaps, long and zero
branches, deep trees, against the oracle at the FP64 tolerances."""
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


@pytest.mark.parametrize("n,S,R,C,tree,mean_t", [
    (2, 21, 1, 1, "yule", 0.1), (3, 64, 3, 127, "yule", 0.1), (6, 61, 1, 128, "yule", 0.1),
    (7, 61, 5, 129, "caterpillar", 0.1), (11, 40, 8, 20, "balanced", 0.02),
    (60, 61, 2, 9, "caterpillar", 0.5), (9, 61, 4, 33, "yule", 20.0),
    (9, 61, 4, 33, "yule", 1e-5),
])
def test_matches_oracle(n, S, R, C, tree, mean_t):
    import paper_2303_04390_gb300 as pg
    w = synth.small_workload(n, S, R, C, seed=95, mean_t=mean_t, tree=tree)
    rng = np.random.default_rng(n + C)
    w.tip_states[1:][rng.random(w.tip_states[1:].shape) < 0.05] = S  # gaps
    if n > 5:
        w.t[n] = 0.0
    ctx = pg.from_workload(w, "fp64")
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w), "fp64", f"{w.name} {tree}")
    ctx.close()


def test_partial_vectors_and_reverse_mode():
    import paper_2303_04390_gb300 as pg
    from oracle import phylo_oracle as O
    w = synth.small_workload(10, 61, 3, 140, seed=96)
    tp = O.tip_partial_vectors(61, w.tip_states)
    rng = np.random.default_rng(3)
    ctx = pg.from_workload(w, "fp64", tip_partials=True)
    for tip in (0, 4, 5, 9):
        tp[tip] = rng.random((140, 61)) ** 3 + 0.001
        ctx.set_tip_partials(tip, tp[tip])
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w, tip_partials=tp), "fp64", "partial vectors")
    log_t = torch.tensor(np.log(w.t), device="cuda", requires_grad=True)
    ll = pg.branch_loglik(log_t, ctx)
    (g,) = torch.autograd.grad(ll, log_t)
    ctx.set_branch_lengths(torch.exp(log_t.detach()))
    logL, grad = ctx.evaluate()
    assert ll.item() == logL
    np.testing.assert_allclose(g.cpu().numpy(), grad * w.t, rtol=1e-14)
