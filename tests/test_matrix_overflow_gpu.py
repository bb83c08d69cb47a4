"""Matrix entries past the range of FP32 (65 to 128 states), from a decomposition
that is exact and accepted but not of a rate matrix (a symmetric model's, one
state scaled by 2^140): the evaluation has to be refused, as its likelihood is
infinite, not answered from the states whose entries fit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_04390_gb300 import build as B
    B.build()


def _hadamard(n):
    h = np.ones((1, 1))
    while len(h) < n:
        h = np.block([[h, h], [h, -h]])
    return h


@pytest.mark.parametrize("power", [130, 140, 200])
@pytest.mark.parametrize("t", [0.03, 0.5])
def test_overflow_is_refused(power, t):
    import paper_2303_04390_gb300 as pg
    S = 128
    w = synth.small_workload(5, 4, 1, 40, seed=8)
    h = _hadamard(S)
    d = np.ones(S)
    d[3] = np.ldexp(1.0, power)
    ctx = pg.PhyloContext(5, 40, S, 1, "fp32")
    ctx.set_tree(w.parent)
    rng = np.random.default_rng(power)
    ctx.set_tip_states(rng.integers(4, S, (5, 40)).astype(np.uint8))
    ctx.set_pattern_weights(np.ones(40))
    ctx.set_eigen(d[:, None] * h, h / S / d[None, :], -np.arange(S) / 4.0, np.full(S, 1.0 / S))
    ctx.set_categories(np.ones(1), np.ones(1))
    ctx.set_branch_lengths(np.full(8, t))
    with pytest.raises(pg.PhyloError):
        ctx.evaluate()
    ctx.close()
