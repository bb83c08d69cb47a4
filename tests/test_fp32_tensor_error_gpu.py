"""How far the FP32 tensor-core paths are from exact.  Every operand is FP32
(u = 2^-24); an MMA's accumulation cuts off up to 2^-23 of the sum so far, and
a contraction of the six split products has 4 MMAs of each order: with the
largest product last, 4 cuts of a full-size sum (8 u) and the roundings of P,
Q, U and q; with it first, 24 cuts (48 u).  The gradient's error in the 2-norm
is held to 12 u (geometric mean over seeds)."""
import numpy as np
import pytest

import synth
from parity import oracle_eval

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_04390_gb300 import build as B
    B.build()


@pytest.mark.parametrize("S,n,C", [(61, 37, 150), (122, 24, 80)])
def test_gradient_error(S, n, C):
    import paper_2303_04390_gb300 as pg
    errs = []
    for seed in range(4):
        w = synth.small_workload(n, S, 4, C, seed=70 + seed, mean_t=0.05)
        ctx = pg.from_workload(w, "fp32")
        _, grad = ctx.evaluate()
        ctx.close()
        _, ref, _, _ = oracle_eval(w)
        errs.append(np.linalg.norm(grad - ref) / np.linalg.norm(ref))
    print(S, errs)
    assert np.exp(np.mean(np.log(errs))) <= 12 * 2.0 ** -24
