"""Timed cases of the solver: what a user of the library has it do, from one
tiny program to a store larger than the L2 cache.

Each case goes through the binding's public entry points
(paper_1909_01786_gb300.aspgpu).  Programs are drawn here from the seed alone,
with the laws of the repository's synthetic workloads (tiny programs of 20
atoms; random rules with bodies of 1..4 literals, half of them negated;
grounded 3-colouring).  Where a call has to end in a known way they are
planted: an interpretation M is drawn first and the rules are drawn around it,
so that M is an answer set and every part of M is a consistent partial
assignment.  Sizes depend on the case only, contents on the seed only.

Answers are comparable between two runs of the same code: enumerations run to
the end and come back in a fixed order, and a search of a program that cannot
be decided in seconds runs until its first conflict, up to which every
decision and every propagation closure is determined by the program.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1909_01786_gb300 import aspgpu, heuristic


# ------------------------------------------------------------------ programs

def _program(n_atoms, head, atoms, negated, size):
    """Rules given as head [m], atoms [m, K], negated [m, K] and body size [m]
    in the form that the binding takes."""
    used = np.arange(atoms.shape[1])[None, :] < size[:, None]
    pos, neg = used & ~negated, used & negated
    off = lambda x: np.concatenate([[0], np.cumsum(x.sum(1))]).astype(np.int64)  # noqa: E731
    return SimpleNamespace(n_atoms=int(n_atoms), head=head.astype(np.int32),
                           pos_off=off(pos), pos=atoms[pos].astype(np.int32),
                           neg_off=off(neg), neg=atoms[neg].astype(np.int32))


def _bodies(rng, n_atoms, m, law):
    """m bodies of distinct atoms: law "random" has 1..4 literals, each negated
    with probability 1/2; law "tiny" has 0..2 positive and 0..2 negative ones."""
    atoms = rng.integers(0, n_atoms, (m, 4))
    while True:
        s = np.sort(atoms, axis=1)
        bad = np.nonzero((s[:, 1:] == s[:, :-1]).any(1))[0]
        if not bad.size:
            break
        atoms[bad] = rng.integers(0, n_atoms, (bad.size, 4))
    if law == "tiny":
        p, q = rng.integers(0, 3, m), rng.integers(0, 3, m)
        return atoms, np.arange(4)[None, :] >= p[:, None], p + q
    return atoms, rng.random((m, 4)) < 0.5, rng.integers(1, 5, m)


def random_program(rng, n_atoms, n_rules):
    atoms, negated, size = _bodies(rng, n_atoms, n_rules, "random")
    return _program(n_atoms, rng.integers(0, n_atoms, n_rules), atoms, negated, size)


def tiny_program(rng, n_atoms, n_rules, n_constraints):
    atoms, negated, size = _bodies(rng, n_atoms, n_rules + n_constraints, "tiny")
    head = rng.integers(0, n_atoms, n_rules + n_constraints)
    head[n_rules:], size[n_rules:] = -1, 2
    negated[n_rules:] = rng.random((n_constraints, 4)) < 0.5
    return _program(n_atoms, head, atoms, negated, size)


def planted_program(rng, n_atoms, n_rules, n_constraints=0, law="random"):
    """(program, M): M holds about three atoms in ten and is an answer set.
    Each atom of M has one rule that derives it from earlier atoms of M and
    from atoms outside M; any other rule whose body holds in M has its head
    moved into M; constraints do not hold in M."""
    inside = rng.permutation(n_atoms)[:max(1, (3 * n_atoms) // 10)]
    outside = np.setdiff1d(np.arange(n_atoms), inside)
    M = np.zeros(n_atoms, bool)
    M[inside] = True
    m = n_rules + n_constraints
    atoms, negated, size = _bodies(rng, n_atoms, m, law)
    head = rng.integers(0, n_atoms, m)
    head[n_rules:], size[n_rules:] = -1, np.maximum(size[n_rules:], 2)
    k = inside.size                              # rules 0 .. k-1 derive M
    head[:k] = inside
    negated[:k] |= (np.arange(k) == 0)[:, None]
    earlier = inside[(rng.random((k, 4)) * np.arange(k)[:, None]).astype(np.int64)]
    atoms[:k] = np.where(negated[:k], outside[rng.integers(0, outside.size, (k, 4))], earlier)
    used = np.arange(4)[None, :] < size[:, None]
    holds = (~used | (M[atoms] != negated)).all(1)
    move = np.nonzero(holds[:n_rules])[0]
    move = move[move >= k]
    head[move] = inside[rng.integers(0, k, move.size)]
    flip = n_rules + np.nonzero(holds[n_rules:])[0]
    negated[flip, 0] ^= True
    order = rng.permutation(m)
    return _program(n_atoms, head[order], atoms[order], negated[order], size[order]), M


def colouring_program(rng, n, degree):
    """3-colouring of a graph with a planted colouring: col(v, c) = 3v + c and
    ncol(v, c) = 3n + 3v + c in even negative loops, one colour per vertex, no
    edge of one colour.  The first triangle's colours are fixed."""
    colour = np.concatenate([[0, 1, 2], rng.permutation(np.arange(n - 3) % 3)])
    edges = {(0, 1), (0, 2), (1, 2)}
    def link(u, v):
        if u != v and colour[u] != colour[v]:
            edges.add((min(u, v), max(u, v)))
    for v in range(3, n):                        # every vertex has a neighbour
        other = np.nonzero(colour[:v] != colour[v])[0]
        link(int(other[rng.integers(0, other.size)]), v)
    while 2 * len(edges) < degree * n:
        link(*(int(x) for x in rng.integers(0, n, 2)))
    rules = []
    for v in range(n):
        for c in range(3):
            rules += [(3 * v + c, [], [3 * n + 3 * v + c]), (3 * n + 3 * v + c, [], [3 * v + c])]
        rules.append((-1, [], [3 * v, 3 * v + 1, 3 * v + 2]))
        rules += [(-1, [3 * v + a, 3 * v + b], []) for a, b in ((0, 1), (0, 2), (1, 2))]
    rules += [(-1, [3 * u + c, 3 * v + c], []) for u, v in sorted(edges) for c in range(3)]
    rules += [(-1, [], [3 * v + v]) for v in range(3)]
    head = np.array([r[0] for r in rules])
    size = np.array([len(r[1]) + len(r[2]) for r in rules])
    atoms = np.zeros((len(rules), 4), np.int64)
    negated = np.zeros((len(rules), 4), bool)
    for i, (_, p, q) in enumerate(rules):
        atoms[i, :size[i]], negated[i, len(p):size[i]] = p + q, True
    return _program(6 * n, head, atoms, negated, size)


def body_variables(p, M):
    """The solver variables b_r of the rules whose body holds in M."""
    count = lambda bad, off: np.concatenate([[0], np.cumsum(bad)])[off]  # noqa: E731
    wrong = np.diff(count(~M[p.pos], p.pos_off)) + np.diff(count(M[p.neg], p.neg_off))
    rules = np.argsort(p.head, kind="stable")    # the library's order of headed rules
    rules = rules[p.head[rules] >= 0]
    return p.n_atoms + 3 * np.nonzero(wrong[rules] == 0)[0]


def _partial(rng, p, M, depth, n_vars):
    """A partial assignment as deep in the search: `depth` decisions Tb_r."""
    b = rng.permutation(body_variables(p, M))[:depth]
    out = np.zeros(n_vars, np.int8)
    out[b] = 1
    return out


# --------------------------------------------------------------------- cases

def listed():
    return [
        # every answer set of a tiny program: the smallest call, one CTA
        dict(name="solve_tiny", kind="enumerate", atoms=20, rules=40, constraints=3),
        # every 3-colouring of a small graph: many short searches after one another
        dict(name="solve_colouring", kind="colour", vertices=50, degree=6.0),
        # first answer set of random programs (hopeless within seconds, so to
        # the first conflict): a program of one small grid, a medium one under
        # the frontier by units, and the benchmark's program
        dict(name="search_2k", kind="search", atoms=2_000, rules=8_000, frontier=0, learning=0, heuristic=0),
        dict(name="search_20k_units", kind="search", atoms=20_000, rules=50_000, frontier=2, learning=0, heuristic=0),
        dict(name="search_100k", kind="search", atoms=100_000, rules=400_000, frontier=0, learning=0, heuristic=0),
        # the closure of a partial assignment given on the host, of a program
        # whose store is larger than the L2 cache
        dict(name="propagate_400k", kind="propagate", atoms=400_000, rules=1_600_000, depth=1_024),
        # the same on device buffers without allocation, as a loop that must
        # not enter the allocator calls it: small, and the largest served
        dict(name="noalloc_1k", kind="noalloc", atoms=1_000, rules=4_000, depth=4),
        dict(name="noalloc_80k", kind="noalloc", atoms=80_000, rules=320_000, depth=256),
        # many programs in one launch: tiny ones enumerated, and uneven ones
        # (200 to 20000 atoms) solved for a first answer set
        dict(name="batch_tiny", kind="batch_tiny", programs=1_000, config=-1),
        dict(name="batch_uneven", kind="batch", programs=128, smallest=200, largest=20_000, config=-1),
        # the learned heuristic: training on traces, scores of candidates
        dict(name="train_200k", kind="train", samples=200_000, epochs=2),
        dict(name="score_1m", kind="score", samples=1_000_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["enumerate", "colour", "search", "search", "propagate", "propagate", "noalloc", "noalloc",
                       "batch_tiny", "batch", "train", "score"])
    if kind == "enumerate":
        n = rng.randint(12, 28)
        return dict(kind=kind, atoms=n, rules=2 * n + rng.randint(0, 9), constraints=rng.randint(0, 4))
    if kind == "colour":
        return dict(kind=kind, vertices=rng.randint(24, 50), degree=rng.choice([6.0, 6.5, 7.0]))
    if kind == "search":
        n = _log(rng, 1_000, 100_000)
        return dict(kind=kind, atoms=n, rules=int(n * rng.uniform(2.5, 4.0)), frontier=rng.choice([0, 0, 2]),
                    learning=rng.choice([0, 0, 1]), heuristic=rng.choice([0, 0, 4]))
    if kind == "propagate":
        n = _log(rng, 50, 400_000)
        return dict(kind=kind, atoms=n, rules=int(n * rng.uniform(2.0, 4.0)), depth=_log(rng, 1, max(2, n // 100)))
    if kind == "noalloc":
        n = _log(rng, 50, 80_000)
        return dict(kind=kind, atoms=n, rules=int(n * rng.uniform(2.0, 4.0)), depth=_log(rng, 1, max(2, n // 100)))
    if kind == "batch_tiny":
        return dict(kind=kind, programs=_log(rng, 16, 1_000), config=rng.choice([-1, -1, 0, 1]))
    if kind == "batch":
        return dict(kind=kind, programs=rng.randint(8, 128), smallest=rng.randint(100, 400),
                    largest=_log(rng, 1_000, 20_000), config=rng.choice([-1, -1, 0, 1]))
    if kind == "train":
        return dict(kind=kind, samples=_log(rng, 500, 200_000), epochs=rng.randint(1, 2))
    return dict(kind=kind, samples=_log(rng, 100, 1_000_000))


#: rows kept of an enumeration; every listed or drawn enumeration has fewer
ROWS = {"enumerate": 256, "colour": 2048, "batch_tiny": 64}


def _mlp_inputs(case, seed):
    """Standardised features, labels of a noisy teacher (about two in three
    are right, as for decision traces), and initial weights."""
    rng = np.random.default_rng([seed, 3])
    X = rng.standard_normal((case["samples"], aspgpu.MLP_FEATURES), dtype=np.float32)
    X[:, 14:] = 0.0                              # the two features that are always zero
    z = X[:, :8] @ rng.standard_normal(8).astype(np.float32) + X[:, 9] * X[:, 11]
    y = (rng.random(case["samples"]) < 1.0 / (1.0 + np.exp(-0.5 * z))).astype(np.float32)
    return X, y, heuristic.init_weights(seed)


def _uneven(case):
    """Atom counts of an uneven batch, spread evenly over their logarithm."""
    n = np.exp(np.linspace(math.log(case["smallest"]), math.log(case["largest"]), case["programs"]))
    return [int(round(x)) for x in n]


def prepare(case, seed):
    kind, rng = case["kind"], np.random.default_rng([seed, 1])
    s = SimpleNamespace(kind=kind, case=case)
    if kind == "enumerate":
        p, _ = planted_program(rng, case["atoms"], case["rules"], case["constraints"], "tiny")
        s.P = aspgpu.Program(p)
    elif kind == "colour":
        s.P = aspgpu.Program(colouring_program(rng, case["vertices"], case["degree"]))
    elif kind == "search":
        s.P = aspgpu.Program(random_program(rng, case["atoms"], case["rules"]), conflict_budget=1,
                             frontier=case["frontier"], learning=case["learning"], heuristic=case["heuristic"])
    elif kind in ("propagate", "noalloc"):
        p, M = planted_program(rng, case["atoms"], case["rules"])
        s.P = aspgpu.Program(p)
        s.partial = _partial(rng, p, M, case["depth"], s.P.n_vars)
        if kind == "noalloc":
            s.partial = torch.from_numpy(s.partial).cuda()
            s.closure = torch.empty_like(s.partial)
            s.conflict = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind == "batch_tiny":
        opt = dict(deps_levels=64, learned_capacity=1 << 16)
        s.P = [aspgpu.Program(tiny_program(rng, 20, 40, 3), **opt) for _ in range(case["programs"])]
        s.plan = aspgpu.BatchPlan(s.P, max_models_each=0, cap_each=ROWS[kind], config=case["config"])
    elif kind == "batch":
        # half of them planted at 2.5 rules per atom, half random at 1.5, where
        # about half have no answer set; every one is decided after a few conflicts
        opt = dict(deps_levels=1024, learned_capacity=1 << 20, conflict_budget=2000, time_budget_ms=2000)
        ps = [planted_program(rng, n, (5 * n) // 2)[0] if i % 2 else random_program(rng, n, (3 * n) // 2)
              for i, n in enumerate(_uneven(case))]
        s.P = [aspgpu.Program(p, **opt) for p in ps]
        s.plan = aspgpu.BatchPlan(s.P, max_models_each=1, cap_each=1, config=case["config"])
    else:
        s.X, s.y, s.w = _mlp_inputs(case, seed)
    return s


def _rows(out, models):
    """The answer sets in a fixed order, in a buffer of fixed size."""
    out[:len(models)] = np.unique(models, axis=0) if len(models) > 1 else models
    return out


def run(s):
    if s.kind in ("enumerate", "colour"):
        status, models, n = s.P.solve(max_models=0, cap=ROWS[s.kind])
        return status, n, _rows(np.zeros((ROWS[s.kind], s.P.n_atoms), np.uint8), models)
    if s.kind == "search":
        status, models, n = s.P.solve(max_models=1, cap=1)
        st = s.P.stats()
        return (status, n, _rows(np.zeros((1, s.P.n_atoms), np.uint8), models),
                [st[k] for k in ("n_literals", "decisions", "max_level", "conflicts", "completions")])
    if s.kind == "propagate":
        return s.P.propagate(s.partial)
    if s.kind == "noalloc":
        code = s.P.propagate_noalloc(s.partial.data_ptr(), s.closure.data_ptr(), s.conflict.data_ptr())
        return code, s.closure, s.conflict
    if s.kind in ("batch_tiny", "batch"):
        status, n, models = s.plan.run()
        rows = ROWS.get(s.kind, 1)
        return status, n, np.concatenate([_rows(np.zeros((rows, p.n_atoms), np.uint8), m).reshape(-1)
                                          for p, m in zip(s.P, models)])
    if s.kind == "train":
        return aspgpu.train_mlp(s.X, s.y, s.w, epochs=s.case["epochs"])
    return aspgpu.mlp_score(s.w, s.X)


def work(case):
    kind = case["kind"]
    # a rule of b body literals has 11 + 3 b literals in the completion, an
    # atom one; each is 4 bytes, and bodies have 2.5 literals (tiny ones 2)
    store = lambda atoms, rules, body=2.5: 4.0 * (atoms + (11 + 3 * body) * rules)  # noqa: E731
    if kind == "enumerate":
        return dict(bytes=store(case["atoms"], case["rules"], 2) + 8 * case["constraints"], flops=0)
    if kind == "colour":
        n = case["vertices"]
        return dict(bytes=store(6 * n, 6 * n, 1) + 4 * (9 * n + 3 * case["degree"] * n), flops=0)
    if kind == "search":
        return dict(bytes=store(case["atoms"], case["rules"]) + case["atoms"] / 8, flops=0)
    if kind in ("propagate", "noalloc"):
        return dict(bytes=store(case["atoms"], case["rules"]) + 2 * (case["atoms"] + 3 * case["rules"]), flops=0)
    if kind == "batch_tiny":
        return dict(bytes=case["programs"] * store(20, 40, 2), flops=0)
    if kind == "batch":
        return dict(bytes=sum(store(n, (2.5 if i % 2 else 1.5) * n) for i, n in enumerate(_uneven(case))), flops=0)
    n, weights = case["samples"], 16 * 64 + 64
    if kind == "train":
        return dict(bytes=68 * n + 8 * aspgpu.MLP_PARAMS, flops=6 * weights * n * case["epochs"])
    return dict(bytes=68 * n, flops=2 * weights * n)


def _split(w):
    return w[:1024].reshape(64, 16), w[1024:1088], w[1088:1152], w[1152]


def exact(case, seed):
    """The MLP in 64 bits: training as momentum SGD (0.9) on the mean binary
    cross-entropy over minibatches of 4096 rows in order, and scores under
    weights rounded to bf16.  The other cases return whole numbers only."""
    if case["kind"] not in ("train", "score"):
        return None
    X, y, w = _mlp_inputs(case, seed)
    X, y = X.astype(np.float64), y.astype(np.float64)
    if case["kind"] == "score":
        W1, b1, w2, b2 = _split(torch.from_numpy(w).to(torch.bfloat16).double().numpy())
        return np.maximum(X @ W1.T + b1, 0.0) @ w2 + b2
    w, v, lr = w.astype(np.float64), np.zeros(w.size), float(np.float32(0.05))
    momentum = float(np.float32(0.9))
    for _ in range(case["epochs"]):
        for i in range(0, len(X), 4096):
            x, t = X[i:i + 4096], y[i:i + 4096]
            W1, b1, w2, b2 = _split(w)
            a = x @ W1.T + b1
            h = np.maximum(a, 0.0)
            d = (1.0 / (1.0 + np.exp(-(h @ w2 + b2))) - t) / len(x)
            da = (a > 0.0) * d[:, None] * w2
            v = momentum * v + np.concatenate([(da.T @ x).reshape(-1), da.sum(0), h.T @ d, [d.sum()]])
            w = w - lr * v
    return w
