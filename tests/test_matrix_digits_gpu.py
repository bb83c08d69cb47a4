"""Transition matrices from the exact digit contractions (FP32 with 65 to 128
states, FP64 with 21 to 64): the smallest and largest state counts and the
edge of the second block of eigenvalues, short, long and zero branches, and
eigenvector pairs whose free factors differ by many powers of two, against
the oracle at the usual tolerances."""
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


@pytest.mark.parametrize("n,S,R,C,mean_t", [
    (2, 65, 1, 1, 0.1), (5, 128, 3, 130, 0.1), (6, 122, 2, 17, 1e-5),
    (6, 127, 1, 40, 20.0), (9, 96, 4, 129, 0.02),
])
def test_matches_oracle(n, S, R, C, mean_t):
    import paper_2303_04390_gb300 as pg
    w = synth.small_workload(n, S, R, C, seed=31, mean_t=mean_t)
    w.tip_states[1:, ::7] = S  # gaps
    if n > 2:
        w.t[n] = 0.0
    ctx = pg.from_workload(w, "fp32")
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w), "fp32", w.name)
    ctx.close()


@pytest.mark.parametrize("S,precision", [(122, "fp32"), (61, "fp64")])
def test_free_factors_of_the_eigenvectors(S, precision):
    import paper_2303_04390_gb300 as pg
    w = synth.small_workload(6, S, 2, 40, seed=32)
    ctx = pg.from_workload(w, precision)
    # the symmetric decomposition, each pair with a factor of its own
    root = np.sqrt(w.pi)
    lam, U = np.linalg.eigh(root[:, None] * w.Q / root[None, :])
    f = np.ldexp(1.0, np.random.default_rng(5).integers(-60, 61, S))
    ctx.set_eigen(U / root[:, None] * f, (U * root[:, None]).T / f[:, None],
                  np.minimum(lam, 0.0), w.pi)
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w), precision, "scaled eigenvectors")
    ctx.close()


@pytest.mark.parametrize("S,precision", [(122, "fp32"), (61, "fp64"), (21, "fp64")])
def test_entries_above_one(S, precision):
    """A decomposition whose exponentials are positive but not stochastic:
    D Q D^-1, with entries and row sums far above 1 off the diagonal."""
    import paper_2303_04390_gb300 as pg
    w = synth.small_workload(6, S, 2, 40, seed=33, mean_t=0.5)
    ctx = pg.from_workload(w, precision)
    root = np.sqrt(w.pi)
    lam, U = np.linalg.eigh(root[:, None] * w.Q / root[None, :])
    d = np.ldexp(1.0, np.random.default_rng(6).integers(-6, 7, S))
    ctx.set_eigen(U / root[:, None] * d[:, None], (U * root[:, None]).T / d[None, :],
                  np.minimum(lam, 0.0), w.pi)
    w.Q = d[:, None] * w.Q / d[None, :]
    logL, grad = ctx.evaluate()
    compare(logL, grad, oracle_eval(w), precision, "entries above one")
    ctx.close()
