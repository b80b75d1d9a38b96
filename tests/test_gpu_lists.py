"""Propagation through the occurrence lists, packed batch results and the MLP
kernels at the edges of their ranges (needs a GB300): nogoods of up to and of
more than eight literals, one CTA, narrow rounds, list rounds and sweeps, inputs
from none to every variable, batches across the packing scan's blocks, sample
counts around the training cluster's and the scoring tile's shares, rows that
are not 16-byte aligned."""
import numpy as np
import pytest

import oracle
from synth.programs import program_seed, random_program, tiny_program

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1909_01786_gb300 import aspgpu, heuristic
    aspgpu.lib()
    return torch, aspgpu, heuristic


def _perm(prog):
    """oracle variable index for each GPU variable (headed rules by head atom,
    ties in input order, against input order)"""
    headed = np.nonzero(prog.head >= 0)[0]
    o = np.argsort(prog.head[headed], kind="stable")
    aux = prog.n_atoms + 3 * o[:, None] + np.arange(3)
    return np.concatenate([np.arange(prog.n_atoms), aux.reshape(-1)])


def _noalloc(torch, P, partial, shift):
    """asp_propagate_noalloc on buffers `shift` bytes past an aligned address"""
    src = torch.zeros(P.n_vars + 8, dtype=torch.int8, device="cuda")
    dst = torch.full((P.n_vars + 8,), 7, dtype=torch.int8, device="cuda")
    conf = torch.full((1,), 7, dtype=torch.int32, device="cuda")
    src[shift:shift + P.n_vars] = torch.from_numpy(partial).cuda()
    torch.cuda.synchronize()
    assert P.propagate_noalloc(src.data_ptr() + shift, dst.data_ptr() + shift, conf.data_ptr()) == 0
    torch.cuda.synchronize()
    out = dst.cpu().numpy()
    assert (out[:shift] == 7).all() and (out[shift + P.n_vars:] == 7).all()
    return bool(conf.item()), out[shift:shift + P.n_vars]


# one CTA: mean support nogoods of 3, 11 (rows) and 21 literals (long); the grid:
# 4 rules per atom, 10 per atom
@pytest.mark.parametrize("atoms,rules", [(40, 70), (150, 1500), (100, 2000), (5000, 20000), (2000, 20000)])
@pytest.mark.parametrize("frontier", [0, 2])
def test_closures_equal_the_oracle(env, atoms, rules, frontier):
    torch, gpu, _ = env
    prog = random_program(atoms, rules, program_seed(1201, atoms + rules))
    P = gpu.Program(prog, frontier=frontier)
    st = P.stats()                               # nothing counted before the first solve
    assert st["rounds"] == st["propagations"] == st["literal_checks"] == 0
    perm = _perm(prog)
    rng = np.random.default_rng(atoms)
    partial = np.zeros(P.n_vars, np.int8)
    closed = 0
    for k in (0, 1, 3, 3, 3, atoms // 2, atoms):
        if k:
            # a few more atoms on top of the last closure without a conflict
            open_atoms = np.nonzero(partial[:atoms] == 0)[0]
            pick = rng.choice(open_atoms, size=min(k, open_atoms.size), replace=False)
            partial = partial.copy()
            partial[pick] = rng.choice([-1, 1], size=pick.size)
        opart = np.zeros(P.n_vars, np.int8)
        opart[perm] = partial
        want_conflict, want, _, _ = oracle.up_closure(prog, opart)
        conflict, got = P.propagate(partial)
        nconflict, ngot = _noalloc(torch, P, partial, k % 8)
        assert conflict == nconflict == bool(want_conflict)
        if want_conflict:
            partial = np.zeros(P.n_vars, np.int8) if not closed else closure
            continue
        assert (got == want[perm]).all() and (ngot == want[perm]).all()
        closed += 1
        closure = partial = got
    assert closed
    # the closure is its own closure, with every assigned variable in the input
    assert (P.propagate(closure)[1] == closure).all()
    assert (_noalloc(torch, P, closure, 0)[1] == closure).all()


@pytest.mark.parametrize("n", [1, 3, 256, 300])
@pytest.mark.parametrize("config", [-1, 0, 1])
def test_batches_equal_single_solves(env, n, config):
    _, gpu, _ = env
    progs = [random_program(30 + 5 * (i % 50), 60 + 10 * (i % 50), program_seed(1202, i)) if i % 3 == 0 else tiny_program(i)
             for i in range(n)]
    P = [gpu.Program(p, learned_capacity=1 << 16, deps_levels=256) for p in progs]
    plan = gpu.BatchPlan(P, max_models_each=2, cap_each=2, config=config)
    for _ in range(2):
        st, nm, models = plan.run()
        for i, p in enumerate(progs):
            assert nm[i] == len(models[i]) and st[i] == (gpu.SAT if nm[i] else gpu.UNSAT)
            assert len({bytes(m) for m in models[i]}) == nm[i]
            assert all(oracle.is_answer_set(p, m) for m in models[i])
    plan.close()
    for i in range(0, n, 17):
        s, m, k = P[i].solve(2, cap=2)
        assert (s, k) == (st[i], nm[i])


def _train64(X, y, w, epochs, lr):
    w, v = w.astype(np.float64), np.zeros(w.size)
    for _ in range(epochs):
        for i in range(0, len(X), 4096):
            x, t = X[i:i + 4096].astype(np.float64), y[i:i + 4096]
            W1, b1, w2, b2 = w[:1024].reshape(64, 16), w[1024:1088], w[1088:1152], w[1152]
            a = x @ W1.T + b1
            h = np.maximum(a, 0.0)
            d = (1.0 / (1.0 + np.exp(-(h @ w2 + b2))) - t) / len(x)
            da = (a > 0.0) * d[:, None] * w2
            v = 0.9 * v + np.concatenate([(da.T @ x).reshape(-1), da.sum(0), h.T @ d, [d.sum()]])
            w = w - lr * v
    return w


def _misaligned(a):
    """the same values 4 bytes past a 16-byte boundary"""
    buf = np.empty(a.size + 8, np.float32)
    shift = (4 - buf.ctypes.data % 16) % 16 // 4
    out = buf[shift:shift + a.size].reshape(a.shape)
    out[...] = a
    assert out.ctypes.data % 16 == 4
    return out


@pytest.mark.parametrize("n", [1, 15, 255, 257, 4095, 4097, 8200])
def test_training_equals_float64_steps(env, n):
    """Two epochs.  A gradient entry is a mean of terms below 5 summed in fp32 in
    chains of at most 16 + 16 + 16 additions (error below 48 x 2^-24 x 5 =
    1.5e-5); six momentum steps of 0.05 keep the weights within 5e-5, and a
    sample that rounding puts across a ReLU kink adds at most
    0.05 x 5 / 4096 = 6e-5: 2e-4 in all."""
    _, gpu, H = env
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 16)).astype(np.float32)
    y = (rng.random(n) < 0.4).astype(np.float32)
    w = H.init_weights(n)
    got = gpu.train_mlp(X, y, w, epochs=2, learning_rate=0.05)
    assert np.abs(got - _train64(X, y, w, 2, float(np.float32(0.05)))).max() < 2e-4
    assert (gpu.train_mlp(X, y, w, epochs=2, learning_rate=0.05) == got).all()
    assert (gpu.train_mlp(_misaligned(X), _misaligned(y), w, epochs=2, learning_rate=0.05) == got).all()
    assert (gpu.train_mlp(X, y, w, epochs=0) == w).all()


@pytest.mark.parametrize("n", [1, 511, 512, 513, 1025, (1 << 20) + 3])
def test_scores_of_every_row(env, n):
    """bf16 weights, fp32 sums of 16 and 64 terms: 1e-5 of the magnitudes summed"""
    _, gpu, H = env
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 16)).astype(np.float32)
    w = H.init_weights(7)
    u = w.view(np.uint32).astype(np.uint64)
    wb = ((((u + 0x7FFF + ((u >> 16) & 1)) >> 16) << 16).astype(np.uint32)).view(np.float32).astype(np.float64)
    W1, b1, w2, b2 = wb[:1024].reshape(64, 16), wb[1024:1088], wb[1088:1152], wb[1152]
    got = gpu.mlp_score(w, X)
    want = np.maximum(X @ W1.T + b1, 0.0) @ w2 + b2
    bound = 1e-5 * ((np.abs(X) @ np.abs(W1).T + np.abs(b1)) @ np.abs(w2) + abs(b2) + 1.0)
    assert (np.abs(got - want) <= bound).all()
    assert (gpu.mlp_score(w, _misaligned(X)) == got).all()
