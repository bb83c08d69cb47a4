"""The forward and backward halves of reverse mode against a whole
evaluation, captured and launched directly."""
import ctypes

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


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("n,S,precision", [(20, 4, "fp32"), (20, 4, "fp64"), (80, 4, "fp64"),
                                           (130, 4, "fp32"), (12, 20, "fp32")])
def test_forward_and_backward_are_the_evaluation(n, S, precision, use_graph):
    """The same log P and gradient bit for bit, captured or launched directly;
    a forward runs no pre-order pass, so the last gradient stays."""
    import paper_2303_04390_gb300 as pg
    from paper_2303_04390_gb300 import _native as N
    lib = N.load()
    w = synth.small_workload(n, S, 4, 45, seed=93)
    ctx = pg.from_workload(w, precision, use_graph=use_graph)
    ctx.set_branch_lengths(2.0 * w.t)
    first = ctx.evaluate()[1]
    ctx.set_branch_lengths(w.t)
    out = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    g = torch.empty(2 * n - 2, dtype=torch.float64, device="cuda")
    gen = ctypes.c_uint64(0)
    assert lib.phylo_forward_device(ctx._ctx, ctypes.c_void_p(out.data_ptr()),
                                    ctypes.byref(gen)) == 0
    every = np.arange(2 * n - 2)
    assert ctx.gradient_branch_sum(every[3:4]) == first[3]
    for _ in range(2):  # a backward pass may be repeated
        g.fill_(float("nan"))
        assert lib.phylo_backward_device(ctx._ctx, ctypes.c_void_p(g.data_ptr()), gen) == 0
        torch.cuda.synchronize()
        got = g.cpu().numpy().copy()
    logL, grad = ctx.evaluate()
    assert out.item() == logL
    assert np.array_equal(got, grad)
    compare(logL, grad, oracle_eval(w), precision, w.name)
    ctx.close()
