"""The caller's device memory (needs a GB300): a program whose occurrence lists
cannot be allocated is propagated by sweeps; memory need be aligned to 8 bytes
only; propagation allocates nothing; a batch without room for every model copies
them program by program."""
import numpy as np
import pytest

import oracle
from synth.programs import coloring_program, from_rules, program_seed, random_program, tiny_program

from test_gpu_fwd_learning import _check_at_conflict, _completion
from test_gpu_lists import _noalloc, _perm

pytestmark = pytest.mark.gpu

ASP_E_OOM = -3


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1909_01786_gb300 import aspgpu
    aspgpu.lib()
    return torch, aspgpu


def _schedule(gpu, programs):
    plan = gpu.BatchPlan(programs, config=0)
    out = plan.info()["frontier"]
    plan.close()
    return out


def _without_lists(gpu, prog, which=0, **options):
    """The program loaded while one of the allocations fails that a load
    survives (the first such, or the `which`-th after it)."""
    L = gpu.lib()
    try:
        for nth in range(1, 64):
            assert L.asp_debug_fail_alloc(nth) == 0
            try:
                P = gpu.Program(prog, **options)
            except gpu.AspError as e:
                assert e.code == ASP_E_OOM
                continue
            break
        if which:
            assert L.asp_debug_fail_alloc(nth + which) == 0
            P = gpu.Program(prog, **options)
    finally:
        L.asp_debug_fail_alloc(0)
    return P


@pytest.mark.parametrize("which", [0, 1, 2])
def test_any_of_the_lists_allocations_may_fail(env, which):
    _, gpu = env
    prog = random_program(60, 120, program_seed(1301, 0))
    assert _schedule(gpu, [gpu.Program(prog)]) == "units"
    P = _without_lists(gpu, prog, which)
    assert _schedule(gpu, [P]) == "full"
    assert _schedule(gpu, [gpu.Program(prog), P]) == "full"


# one CTA (with nogoods of more than 15 literals), a grid
@pytest.mark.parametrize("atoms,rules", [(40, 70), (100, 2000), (5000, 20000)])
@pytest.mark.parametrize("frontier", [0, 2])
def test_closures_without_lists(env, atoms, rules, frontier):
    torch, gpu = env
    prog = random_program(atoms, rules, program_seed(1302, atoms))
    P = _without_lists(gpu, prog, frontier=frontier)
    perm = _perm(prog)
    rng = np.random.default_rng(atoms)
    agreed = 0
    for k in (0, 1, 2, 3, 5, atoms // 4):
        partial = np.zeros(P.n_vars, np.int8)
        pick = rng.choice(atoms, size=k, replace=False)
        partial[pick] = rng.choice([-1, 1], size=k)
        opart = np.zeros(P.n_vars, np.int8)
        opart[perm] = partial
        want_conflict, want, _, _ = oracle.up_closure(prog, opart)
        conflict, got = P.propagate(partial)
        nconflict, ngot = _noalloc(torch, P, partial, k % 8)
        assert conflict == nconflict == bool(want_conflict)
        if not want_conflict:
            agreed += 1
            assert (got == want[perm]).all() and (ngot == want[perm]).all()
    assert agreed


@pytest.mark.parametrize("options", [dict(), dict(frontier=2), dict(learning=1, frontier=2), dict(grid_ctas=5), dict(grid_ctas=5, learning=1)])
def test_answer_sets_without_lists(env, options):
    _, gpu = env
    for prog in [tiny_program(i) for i in (3, 77, 151, 402)] + [coloring_program(20, 4.0, seed_index=1)]:
        _, want, n = gpu.Program(prog).solve(0, cap=1 << 12)
        assert all(oracle.is_answer_set(prog, m) for m in want[:50])
        status, models, k = _without_lists(gpu, prog, **options).solve(0, cap=1 << 12)
        assert k == n and status == (gpu.SAT if n else gpu.UNSAT)
        assert {bytes(m) for m in models} == {bytes(m) for m in want}


@pytest.mark.parametrize("grid", [1, 0])
@pytest.mark.parametrize("k", [1, 9])
def test_learning_without_lists(env, grid, k):
    _, gpu = env
    prog = random_program(2000, 5000, program_seed(705, 2))
    P = _without_lists(gpu, prog, grid_ctas=grid, conflict_budget=k)
    status, _, _ = P.solve(1, cap=1)
    assert status == gpu.UNKNOWN and P.stats()["conflicts"] == k
    compared, reasons = _check_at_conflict(gpu, P, prog, _completion(prog), 0)
    assert compared > 0 and reasons > 0


@pytest.mark.parametrize("config", [-1, 0, 1])
def test_batches_with_some_lists_missing(env, config):
    _, gpu = env
    progs = [tiny_program(i) for i in range(12)] + [random_program(200, 400, program_seed(1303, i)) for i in range(4)]
    P = [gpu.Program(p) if i % 2 else _without_lists(gpu, p) for i, p in enumerate(progs)]
    plan = gpu.BatchPlan(P, max_models_each=0, cap_each=1 << 12, config=config)
    assert plan.info()["frontier"] == "full"
    st, nm, models = plan.run()
    for i, p in enumerate(progs):
        s, want, n = gpu.Program(p).solve(0, cap=1 << 12)
        assert (st[i], nm[i]) == (s, n) and n <= 1 << 12
        assert {bytes(m) for m in models[i]} == {bytes(m) for m in want}


def _allocator(gpu, monkeypatch, allow=lambda n: True, shift=0):
    """Program loads take their memory `shift` bytes past what PyTorch gives,
    where allow(bytes) says so, else none."""
    class Hooks(gpu._TorchAllocator):
        def __init__(self, torch, device, stream):
            def alloc(n, ctx):
                if not allow(n):
                    return None
                return torch.cuda.caching_allocator_alloc(int(n) + shift, device=device, stream=stream) + shift

            def free(p, n, ctx):
                torch.cuda.caching_allocator_delete(p - shift)

            self.c_alloc, self.c_free = gpu._ALLOC(alloc), gpu._FREE(free)

    monkeypatch.setattr(gpu, "_TorchAllocator", Hooks)


@pytest.mark.parametrize("atoms,rules", [(40, 70), (100, 2000), (5000, 20000)])
def test_memory_aligned_to_eight_bytes(env, monkeypatch, atoms, rules):
    torch, gpu = env
    prog = random_program(atoms, rules, program_seed(1304, atoms))
    Q = gpu.Program(prog, conflict_budget=20)
    _allocator(gpu, monkeypatch, shift=8)
    P = gpu.Program(prog, conflict_budget=20)
    partial = np.zeros(P.n_vars, np.int8)
    partial[:2] = -1
    want_conflict, want = Q.propagate(partial)
    conflict, got = P.propagate(partial)
    nconflict, ngot = _noalloc(torch, P, partial, 0)
    assert conflict == nconflict == want_conflict
    if not conflict:
        assert (got == want).all() and (ngot == want).all()
    status, models, _ = P.solve(1, cap=1)
    plan = gpu.BatchPlan([P], config=0)
    st, nm, rows = plan.run()
    for s, ms in ((status, models), (st[0], rows[0])):
        assert s in (gpu.SAT, gpu.UNSAT, gpu.UNKNOWN)
        assert all(oracle.is_answer_set(prog, m) for m in ms)
    assert Q.solve(1, cap=1)[0] in (status, gpu.UNKNOWN) or status == gpu.UNKNOWN


@pytest.mark.parametrize("prog", [from_rules(1, []), from_rules(1, [(0, [], [])]), from_rules(2, [(0, [], [1]), (1, [], [0])]),
                                  random_program(40, 70, program_seed(1305, 0)), random_program(5000, 20000, program_seed(1305, 1))],
                         ids=lambda prog: f"{prog.n_atoms}-{prog.n_rules}")
def test_propagation_allocates_nothing(env, monkeypatch, prog):
    _, gpu = env
    left = [True]
    _allocator(gpu, monkeypatch, allow=lambda n: left[0])
    P = gpu.Program(prog)
    left[0] = False
    partial = np.zeros(P.n_vars, np.int8)
    partial[0] = -1
    opart = np.zeros(P.n_vars, np.int8)
    opart[_perm(prog)] = partial
    want_conflict, want, _, _ = oracle.up_closure(prog, opart)
    for _ in range(2):
        conflict, got = P.propagate(partial)
        assert conflict == bool(want_conflict)
        if not conflict:
            assert (got == want[_perm(prog)]).all()


def _batch_in_little_memory(gpu, monkeypatch, progs, cap):
    """The batch's plan where no block of 100 kB or more can be had."""
    small = [False]
    _allocator(gpu, monkeypatch, allow=lambda n: n < 100_000 or not small[0])
    P = [gpu.Program(p) for p in progs]
    small[0] = True
    return P, gpu.BatchPlan(P, max_models_each=0, cap_each=cap, config=0)


def _choices(k):
    """2^k answer sets"""
    return from_rules(2 * k, [(a, [], [a ^ 1]) for a in range(2 * k)])


def _check_batch(gpu, progs, plan, cap):
    st, nm, models = plan.run()
    for i, p in enumerate(progs):
        s, want, n = gpu.Program(p, torch_memory=False).solve(0, cap=cap)
        assert (st[i], nm[i]) == (s, n) and n <= cap
        assert {bytes(m) for m in models[i]} == {bytes(m) for m in want}


def test_batch_without_room_for_its_models(env, monkeypatch):
    """Room for 12 x 2048 rows would be 197 kB."""
    _, gpu = env
    progs = [tiny_program(i) for i in (3, 77, 151, 402, 555, 918)] + [tiny_program(i) for i in range(5, 11)]
    _, plan = _batch_in_little_memory(gpu, monkeypatch, progs, 2048)
    for _ in range(2):
        _check_batch(gpu, progs, plan, 2048)


def test_batch_rows_after_a_larger_solve(env, monkeypatch):
    """A solve with a larger cap takes another model buffer; the batch's rows
    stay where its launch writes them."""
    _, gpu = env
    progs = [_choices(k) for k in range(12)]
    P, plan = _batch_in_little_memory(gpu, monkeypatch, progs, 2048)
    for p in P:
        p.solve(1, cap=4096)
    _check_batch(gpu, progs, plan, 2048)
