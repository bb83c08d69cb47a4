"""FP64 codons on both sides of a short internal branch that differ by one,
two and three nucleotides: the site likelihood then hangs on entries of P of
the order t, t^2 and t^3 beside a diagonal near 1.  The result may be at most
ten times as far from the oracle as plain FP64 products on the same
eigenvectors are (summed over the patterns without cancellation, since either
side's errors may cancel in a sum), plus rounding of the sums themselves."""
import numpy as np
import pytest

import synth
from oracle import phylo_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_04390_gb300 import build as B
    B.build()


# ((0, 1), (2, 3)): tips 0, 1 carry one codon, tips 2, 3 another
PARENT = np.array([4, 4, 5, 5, 6, 6, -1], dtype=np.int32)


def _codons(differ, rng, n):
    names, _ = synth.sense_codons()
    pairs = [(a, b) for a in range(61) for b in range(61)
             if sum(x != y for x, y in zip(names[a], names[b])) == differ]
    return np.array([pairs[i] for i in rng.permutation(len(pairs))[:n]])


def _eigen(Q, pi):
    root = np.sqrt(pi)
    s = root[:, None] * Q / root[None, :]
    lam, U = np.linalg.eigh((s + s.T) / 2)
    lam = np.minimum(lam, 0.0)
    lam[-1] = 0.0
    return U / root[:, None], (U * root[:, None]).T, lam


def _by_pattern(P, dP, pi, a, b):
    """log L and the six derivatives of every pattern, from the matrices of
    the tips' branches and of the internal ones (Eqs. 2, 3, 4 and 8)."""
    (Pt, Pi), (dPt, dPi) = P, dP
    p = [Pt[:, a] ** 2, Pt[:, b] ** 2]                    # [S, C]
    u = [Pi @ p[0], Pi @ p[1]]
    L = (pi[:, None] * u[0] * u[1]).sum(0)
    g = np.empty((6, len(a)))
    for x, y in ((0, b), (1, a)):
        up = pi[:, None] * u[1 - x]
        g[4 + x] = (up * (dPi @ p[x])).sum(0) / L
        own = a if x == 0 else b
        q = (Pi.T @ up) * Pt[:, own]
        g[2 * x] = g[2 * x + 1] = (q * dPt[:, own]).sum(0) / (q * Pt[:, own]).sum(0)
    return np.log(L), g


LENGTHS = [(0.05, 2e-3), (0.05, 1e-4), (1e-3, 1e-3), (0.01, 1e-6), (1e-4, 1e-4),
           (1e-6, 1e-6), (1e-8, 1e-8), (1e-290, 1e-290)]


# t^2 and t^3 past what the eigenvectors resolve are left out: at 1e-8 three
# nucleotides are all rounding noise, of either sign.
@pytest.mark.parametrize("differ,tip,internal", [
    (d, *t) for d in (1, 2, 3) for t in LENGTHS if t[0] ** d > 1e-20 or d == 1])
def test_conflicting_codons(differ, tip, internal):
    import paper_2303_04390_gb300 as pg
    rng = np.random.default_rng([17, differ])
    pi = np.maximum(rng.dirichlet(np.full(61, 5.0)), 1e-4)
    Q, pi = synth.codon_gy94(2.0, 0.3, pi / pi.sum())
    a, b = _codons(differ, rng, 24).T
    V, W, lam = _eigen(Q, pi)
    eye = np.eye(61)
    t = (tip, internal)
    fp64 = _by_pattern([eye + (V * np.expm1(lam * x)) @ W for x in t],
                       [(V * (lam * np.exp(lam * x))) @ W for x in t], pi, a, b)
    P = [O.expm_taylor(x * Q) for x in t]
    ref = _by_pattern(P, [Q @ M for M in P], pi, a, b)
    ctx = pg.PhyloContext(4, 24, 61, 1, "fp64")
    ctx.set_tree(PARENT)
    ctx.set_tip_states(np.stack([a, a, b, b]).astype(np.uint8))
    ctx.set_pattern_weights(np.ones(24))
    ctx.set_eigen(V, W, lam, pi)
    ctx.set_categories(np.ones(1), np.ones(1))
    ctx.set_branch_lengths(np.array([tip] * 4 + [internal] * 2))
    logL, grad = ctx.evaluate()
    ctx.close()
    for what, got, i in [("log P", logL, None)] + [(f"branch {x}", grad[x], x) for x in range(6)]:
        r = ref[0] if i is None else ref[1][i]
        f = fp64[0] if i is None else fp64[1][i]
        bound = 10.0 * np.abs(f - r).sum() + 1e-13 * np.abs(r).sum()
        err = abs(got - r.sum())
        print(f"{differ} nt, {tip:g} / {internal:g}, {what}: {err:.3g}, bound {bound:.3g}")
        assert err <= bound, (what, err, bound)
