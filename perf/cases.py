"""What this library is timed on: log-likelihood and branch-length gradient
evaluations through its public entry points.

The cases follow the repository's own workloads: an 8-taxon nucleotide tree
in FP64, nucleotide, amino-acid, codon and Markov-modulated codon trees in
FP32 with four Gamma categories, and the served stream's range of tree and
alignment sizes (16 to 2,048 taxa, 100 to 20,000 patterns).  A pass is one
step of the program that has the problem resident: new branch lengths in,
log-likelihood and every branch's derivative out.  It goes through one of
the three ways that step is called:

  device    branch lengths from a CUDA tensor, results to a CUDA tensor
            (a Hamiltonian sampler's leapfrog step)
  host      branch lengths from a numpy array, results to numpy (a program
            that keeps its state on the host, as served requests do)
  autograd  the differentiable log-likelihood and its backward pass (a fit
            of log branch lengths by a torch optimiser)

A program that chooses the FP32 path keeps its parameters and gradients in
FP32 (the path's own accuracy); one that chooses FP64 keeps them in FP64.
"""
import math

import numpy as np
import torch

import paper_2303_04390_gb300 as pg

DEV = "cuda"


# -- the cases ---------------------------------------------------------------

def listed():
    return [
        # The smallest call: the 8-taxon JC69 tree of 1,000 sites (about 250
        # unique patterns), one category, FP64, results read on the host.
        case("nuc-8-fp64", "host", 8, 250, 4, 1, "fp64", 0.1),
        # Small served sessions (chains of short alignments): latency counts.
        case("nuc-61-small", "device", 61, 733, 4, 4, "fp32", 0.05),
        case("aa-45-small", "host", 45, 311, 20, 4, "fp32", 0.05),
        # The nucleotide workload of the headline benchmark.
        case("nuc-1024", "device", 1024, 10000, 4, 4, "fp32", 0.002),
        # The largest served request.
        case("nuc-2048-large", "device", 2048, 20000, 4, 4, "fp32", 0.05),
        # The amino-acid workload, differentiated by autograd.
        case("aa-256", "autograd", 256, 5000, 20, 4, "fp32", 0.1),
        # Amino acids with ambiguous residues: partial vectors on some tips.
        case("aa-96-ambiguous", "device", 96, 1201, 20, 4, "fp32", 0.1, 4),
        # A single gene under a codon model, an odd size.
        case("codon-37-gene", "autograd", 37, 389, 61, 4, "fp32", 0.05),
        # The codon workload and its Markov-modulated form (122 states).
        case("codon-128", "device", 128, 2000, 61, 4, "fp32", 0.05),
        case("mmm-128", "device", 128, 2000, 122, 4, "fp32", 0.05),
        # FP64 where a program wants it: nucleotides by autograd, and codons.
        case("nuc-256-fp64", "autograd", 256, 3001, 4, 4, "fp64", 0.02),
        case("codon-61-fp64", "device", 61, 601, 61, 4, "fp64", 0.05),
    ]


def case(name, way, tips, patterns, states, cats, precision, mean_t, partial_every=0):
    """partial_every = m > 0: every m-th tip carries partial vectors."""
    return {"name": name, "way": way, "tips": tips, "patterns": patterns, "states": states,
            "cats": cats, "precision": precision, "mean_t": mean_t,
            "partial_every": partial_every}


# Ranges by model: (states, precision, taxa, patterns, share of draws).  The
# product taxa x patterns is kept at or below the largest listed case's.
RANGES = [
    (4, "fp32", (16, 2048), (100, 20000), 0.34),
    (20, "fp32", (16, 512), (100, 10000), 0.24),
    (61, "fp32", (12, 200), (100, 3000), 0.16),
    (122, "fp32", (12, 128), (100, 2000), 0.08),
    (4, "fp64", (8, 512), (100, 4000), 0.10),
    (61, "fp64", (8, 64), (100, 640), 0.08),
]
CEILING = {(4, "fp32"): 2048 * 20000, (20, "fp32"): 256 * 5000, (61, "fp32"): 128 * 2000,
           (122, "fp32"): 128 * 2000, (4, "fp64"): 256 * 3001, (61, "fp64"): 61 * 601}


def draw(rng):
    x, total = rng.random() * sum(r[4] for r in RANGES), 0.0
    for states, precision, taxa, pats, share in RANGES:
        total += share
        if x <= total:
            break
    tips = int(round(math.exp(rng.uniform(*map(math.log, taxa)))))
    top = min(pats[1], CEILING[(states, precision)] // tips)
    patterns = int(round(math.exp(rng.uniform(math.log(pats[0]), math.log(max(top, pats[0] + 1))))))
    cats = rng.choice([4, 4, 4, 4, 1])  # Gamma 4 everywhere in use, else one rate
    mean_t = rng.choice([0.002, 0.02, 0.05, 0.1])
    partial = rng.choice([0, 0, 0, 0, 0, 4]) if precision == "fp32" else 0
    c = case("", rng.choice(["device", "host", "autograd"]), tips, patterns, states, cats,
             precision, mean_t, partial)
    del c["name"]
    return c


# -- inputs ------------------------------------------------------------------

def yule(n, rng):
    """Random rooted binary tree: a uniformly chosen leaf splits until there
    are n.  Tips 0..n-1 in random order, parents numbered after their
    children, root 2n-2.  Returns the parent array."""
    kids, leaves = {0: None}, [0]
    while len(leaves) < n:
        i = int(rng.integers(len(leaves)))
        a = len(kids)
        kids[leaves[i]] = (a, a + 1)
        kids[a] = kids[a + 1] = None
        leaves[i] = a
        leaves.append(a + 1)
    # children have larger temporary numbers than their parents
    label, tips, inner = {}, iter(rng.permutation(n).tolist()), n
    for v in range(2 * n - 2, -1, -1):
        if kids[v] is None:
            label[v] = next(tips)
        else:
            label[v], inner = inner, inner + 1
    parent = np.full(2 * n - 1, -1, dtype=np.int32)
    for v, ch in kids.items():
        if ch is not None:
            parent[label[ch[0]]] = parent[label[ch[1]]] = label[v]
    return parent


def scaled(ex, pi):
    """Generator with rates ex_ij pi_j, mean rate 1."""
    q = ex * pi[None, :]
    np.fill_diagonal(q, 0.0)
    np.fill_diagonal(q, -q.sum(axis=1))
    return q / -float(pi @ np.diag(q))


CODE = "FFLLSSSSYY**CC*WLLLLPPPPHHQQRRRRIIIMTTTTNNKKSSRRVVVVAAAADDEEGGGG"
CODONS = [(i // 16, i // 4 % 4, i % 4) for i in range(64) if CODE[i] != "*"]  # order TCAG
AMINO = [a for a in CODE if a != "*"]


def codon_exchange(kappa, omega):
    """GY94-style exchangeabilities: one position differs; kappa for a
    transition (T-C, A-G), omega for a change of amino acid."""
    ex = np.zeros((61, 61))
    for i in range(61):
        for j in range(i):
            diff = [(x, y) for x, y in zip(CODONS[i], CODONS[j]) if x != y]
            if len(diff) == 1:
                ex[i, j] = (kappa if diff[0][0] // 2 == diff[0][1] // 2 else 1.0) * \
                    (omega if AMINO[i] != AMINO[j] else 1.0)
    return ex + ex.T


def model(c, rng):
    """(Q, pi): JC69 (one category) or HKY85; a 20-state model with Gamma(1)
    exchangeabilities; codons with omega 0.3, kappa 2; or two codon classes
    (omega 0.1 and 1) that switch at rate 0.5."""
    s = c["states"]
    if s == 4:
        pi = rng.dirichlet([10.0] * 4) if c["cats"] > 1 else np.full(4, 0.25)
        ex = np.ones((4, 4))
        if c["cats"] > 1:
            ex[0, 2] = ex[2, 0] = ex[1, 3] = ex[3, 1] = 4.0
        return scaled(ex, pi), pi
    if s == 20:
        ex = np.triu(rng.gamma(1.0, 1.0, (20, 20)), 1)
        pi = np.maximum(rng.dirichlet(np.ones(20)), 1e-3)
        pi /= pi.sum()
        return scaled(ex + ex.T, pi), pi
    pi = np.maximum(rng.dirichlet(np.ones(61)), 1e-4)
    pi /= pi.sum()
    if s == 61:
        return scaled(codon_exchange(2.0, 0.3), pi), pi
    ex, i = np.zeros((122, 122)), np.arange(61)
    for k, omega in enumerate((0.1, 1.0)):
        e = codon_exchange(2.0, omega)
        rate = float(pi @ (e * pi[None, :]).sum(axis=1))
        ex[61 * k:61 * k + 61, 61 * k:61 * k + 61] = 2.0 * e / rate
    ex[i, 61 + i] = ex[61 + i, i] = 0.5 / pi
    pi2 = np.concatenate([pi, pi]) / 2
    return scaled(ex, pi2), pi2


# Means of the four equal bins of a Gamma(0.5) rate with mean 1.
GAMMA4 = np.array([0.03338775, 0.25191592, 0.82026848, 2.89442785])


def inputs(c, seed):
    """The problem as host arrays, from the seed alone: tree, branch lengths
    (log, FP32 values for the FP32 path), model, simulated tip states with
    about 2% gaps, weights 1..5, and partial vectors where asked for."""
    rng = np.random.default_rng([int(seed), c["tips"], c["patterns"], c["states"]])
    n, pats, s, r = c["tips"], c["patterns"], c["states"], c["cats"]
    parent = yule(n, rng)
    log_t = np.log(np.maximum(rng.exponential(c["mean_t"], 2 * n - 2), 1e-8))
    if c["precision"] == "fp32":
        log_t = log_t.astype(np.float32)
    Q, pi = model(c, rng)
    rates = np.ones(1) if r == 1 else GAMMA4
    # States down the tree, every site of a depth at once on the GPU.
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)
    P = transition(Q, rates, np.exp(log_t.astype(np.float64)))
    cum = P.cumsum(-1).float()  # [branch, category, from, to]
    cat = torch.randint(r, (pats,), generator=gen, device=DEV)
    state = torch.zeros(2 * n - 1, pats, dtype=torch.long, device=DEV)
    state[2 * n - 2] = torch.multinomial(torch.tensor(pi, device=DEV), pats, True, generator=gen)
    depth = np.zeros(2 * n - 1, dtype=np.int64)
    for v in range(2 * n - 3, -1, -1):  # parents are numbered above their internal children
        if v >= n:
            depth[v] = depth[parent[v]] + 1
    depth[:n] = depth[parent[:n]] + 1
    for d in range(1, int(depth.max()) + 1):
        for v in np.array_split(np.nonzero(depth == d)[0], max(1, s * pats * (depth == d).sum() // 2 ** 28)):
            vt, pt = torch.tensor(v, device=DEV), torch.tensor(parent[v].astype(np.int64), device=DEV)
            row = cum[vt[:, None], cat[None, :], state[pt]]  # [nodes, patterns, states]
            u = torch.rand(row.shape[:2], generator=gen, device=DEV)
            state[vt] = (u[..., None] > row).sum(-1).clamp_(max=s - 1)
    tips = state[:n]
    tips = torch.where(torch.rand(tips.shape, generator=gen, device=DEV) < 0.02,
                       torch.full_like(tips, s), tips)
    tips = tips.to(torch.uint8).cpu().numpy()
    weights = rng.integers(1, 6, pats).astype(np.float64)
    partials = {}
    if c["partial_every"]:
        for x in range(0, n, c["partial_every"]):
            v = np.zeros((pats, s + 1))
            v[np.arange(pats), tips[x]] = 1.0
            v = v[:, :s] + (tips[x] == s)[:, None]
            # an ambiguous residue is compatible with some other states too
            some = rng.random(pats) < 0.1
            v[some] = np.maximum(v[some], rng.random((int(some.sum()), s)) < 2.0 / s)
            partials[x] = v
    return dict(parent=parent, log_t=log_t, Q=Q, pi=pi, rates=rates,
                cat_weights=np.full(r, 1.0 / r), tips=tips, weights=weights, partials=partials)


def transition(Q, rates, t):
    """exp(rate t Q) for every branch and category, FP64, by torch."""
    q = torch.tensor(Q, device=DEV)
    rt = torch.tensor(np.outer(t, rates), device=DEV)
    out = torch.empty(*rt.shape, *q.shape, dtype=torch.float64, device=DEV)
    for i in range(0, len(t), 512):
        out[i:i + 512] = torch.linalg.matrix_exp(rt[i:i + 512, :, None, None] * q)
    return out


def prepare(c, seed):
    """A context with the problem resident, and the parameters that a pass
    starts from."""
    x = inputs(c, seed)
    n = c["tips"]
    ctx = pg.PhyloContext(n, c["patterns"], c["states"], c["cats"], c["precision"],
                          tip_partials=bool(x["partials"]))
    ctx.set_tree(x["parent"])
    ctx.set_tip_states(x["tips"])
    for tip, v in x["partials"].items():
        ctx.set_tip_partials(tip, v)
    ctx.set_pattern_weights(x["weights"])
    ctx.set_rate_matrix(x["Q"], x["pi"])
    ctx.set_categories(x["rates"], x["cat_weights"])
    log_t = torch.tensor(x["log_t"], device=DEV, requires_grad=c["way"] == "autograd")
    return {"way": c["way"], "fp32": c["precision"] == "fp32", "ctx": ctx, "log_t": log_t,
            "t": np.exp(x["log_t"].astype(np.float64))}


# -- one pass ----------------------------------------------------------------

def run(state):
    """{"logL": ..., "grad": ...}: d log P / d t ("autograd": d / d log t)."""
    ctx, log_t = state["ctx"], state["log_t"]
    if state["way"] == "host":
        ctx.set_branch_lengths(state["t"])
        logL, grad = ctx.evaluate()
        dtype = np.float32 if state["fp32"] else np.float64
        return {"logL": dtype(logL), "grad": grad.astype(dtype, copy=False)}
    if state["way"] == "autograd":
        logL = pg.branch_loglik(log_t.double(), ctx)
        (grad,) = torch.autograd.grad(logL, log_t)
        return {"logL": logL.detach().to(log_t.dtype), "grad": grad}
    ctx.set_branch_lengths(torch.exp(log_t.double()))
    out = ctx.evaluate_device().to(log_t.dtype, copy=True)
    return {"logL": out[0], "grad": out[1:]}


# -- what a pass cannot do without -------------------------------------------

def work(c):
    """Inputs once (tip states or vectors, weights, lengths, model), results
    once, and the products of the pruning recursions: one S x S matrix by
    vector per (internal node, pattern, category) up the tree, two down it;
    a tip's product is a column.  Matrices: S^3 per (branch, category)."""
    n, pats, s, r = c["tips"], c["patterns"], c["states"], c["cats"]
    e = 8 if c["precision"] == "fp64" else 4
    vec = -(-n // c["partial_every"]) if c["partial_every"] else 0
    read = (n - vec) * pats + vec * pats * s * e + pats * e + (2 * n - 2) * 8 + s * s * 8
    flops = 3 * (n - 2) * 2.0 * s * s * r * pats + (2 * n - 2) * r * 2.0 * s ** 3
    return {"bytes": read + (2 * n - 1) * 8, "flops": flops}


# -- the same in 64 bits -----------------------------------------------------

def exact(c, seed):
    """log P and its gradient by plain pruning in FP64 (torch on the GPU):
    partials up the tree, their complements down it, each rescaled per
    (node, pattern) with the logarithms of the scales kept."""
    x = inputs(c, seed)
    n, pats, s, r = c["tips"], c["patterns"], c["states"], c["cats"]
    root, parent = 2 * n - 2, x["parent"]
    Q, pi, rates, w = (torch.tensor(x[k], device=DEV) for k in ("Q", "pi", "rates", "cat_weights"))
    t = torch.exp(torch.tensor(x["log_t"], device=DEV).double())
    P = transition(x["Q"], x["rates"], t.cpu().numpy())
    kids = [[] for _ in range(root + 1)]
    for v in range(root):
        kids[parent[v]].append(v)
    tips = torch.tensor(x["tips"].astype(np.int64), device=DEV)

    def up(v):  # P_v p_v, [category, pattern, state]
        if v >= n:
            return post[v] @ P[v].transpose(1, 2)
        if v in x["partials"]:
            return torch.tensor(x["partials"][v], device=DEV)[None] @ P[v].transpose(1, 2)
        cols = torch.cat([P[v], P[v].new_ones(r, s, 1)], -1)  # the gap: all ones
        return cols[:, :, tips[v]].transpose(1, 2)

    def scale(p):
        m = p.amax(dim=(0, 2))
        return p / m[None, :, None], torch.log(m)

    post, logs, u = {}, torch.zeros(pats, dtype=torch.float64, device=DEV), {}
    for k in range(n, root + 1):  # children are numbered below their parents
        for v in kids[k]:
            u[v] = up(v)
        post[k], ln = scale(u[kids[k][0]] * u[kids[k][1]])
        logs += ln
        for v in kids[k]:
            post.pop(v, None)
    like = torch.einsum("r,s,rcs->c", w, pi, post.pop(root))
    W = torch.tensor(x["weights"], device=DEV)
    logL = (W * (torch.log(like) + logs)).sum()
    grad = torch.zeros(root, dtype=torch.float64, device=DEV)
    pre = {root: pi.expand(r, pats, s)}
    for k in range(root, n - 1, -1):
        q, (i, j) = pre.pop(k), kids[k]
        for v, sib in ((i, j), (j, i)):
            a = q * u[sib]
            den = torch.einsum("r,rcs,rcs->c", w, a, u[v])
            num = torch.einsum("r,rcs->c", w * rates, (a @ Q) * u[v])
            grad[v] = (W * num / den).sum()
            if v >= n:
                pre[v] = scale(a @ P[v])[0]
        del u[i], u[j]
    if c["way"] == "autograd":
        grad = grad * t
    return {"logL": logL, "grad": grad}
