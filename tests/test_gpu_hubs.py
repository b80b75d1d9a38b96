"""Atoms that occur in many rules (needs a GB300): their occurrence lists are
too long for one warp.  One CTA shares them out to its warps, a grid sweeps the
store instead; lists just below and above either line, more of them than the
queue of long lists holds, and rounds whose lists are long only together."""
import numpy as np
import pytest

import oracle
from synth.programs import from_rules

from test_gpu_fwd_learning import _check_at_conflict, _completion
from test_gpu_learning import _check_conflict
from test_gpu_lists import _noalloc, _perm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1909_01786_gb300 import aspgpu
    aspgpu.lib()
    return torch, aspgpu


def _hubs(hubs, each, pool, filler, seed):
    """A choice 0 / 1; hub i :- 0; `each` rules z :- hub, not w for every hub,
    z and w drawn from `pool` atoms, and `filler` rules over those alone."""
    rng = np.random.default_rng(seed)
    rules = [(0, [], [1]), (1, [], [0])] + [(2 + i, [0], []) for i in range(hubs)]
    base = 2 + hubs
    for i in range(hubs):
        rules += [(base + int(z), [2 + i], [base + int(w)]) for z, w in rng.integers(0, pool, (each, 2))]
    rules += [(base + int(z), [base + int(a)], [base + int(w)]) for z, a, w in rng.integers(0, pool, (filler, 3))]
    return from_rules(base + pool, rules)


# hubs, rules of each, atoms, other rules; CTAs (0: one for small programs, else
# the whole GPU).  A hub's list has a nogood more than its rules.
CASES = [(1, 254, 300, 600, 0), (1, 255, 300, 600, 0), (1, 256, 300, 600, 0), (1, 1500, 500, 300, 0), (3, 500, 500, 200, 0),
         (16, 260, 800, 0, 0), (17, 260, 800, 0, 0), (40, 257, 900, 0, 1),
         (1, 125, 4000, 9000, 0), (1, 140, 4000, 9000, 0), (1, 3000, 4000, 9000, 0), (60, 100, 4000, 9000, 0), (300, 60, 6000, 6000, 0), (300, 200, 6000, 1000, 0),
         (20, 300, 3000, 3000, 2), (300, 100, 3000, 3000, 2)]


@pytest.mark.parametrize("hubs,each,pool,filler,grid", CASES)
@pytest.mark.parametrize("frontier", [0, 2])
def test_closures_with_hubs_equal_the_oracle(env, hubs, each, pool, filler, grid, frontier):
    torch, gpu = env
    prog = _hubs(hubs, each, pool, filler, hubs * each)
    P = gpu.Program(prog, frontier=frontier, grid_ctas=grid)
    perm = _perm(prog)
    rng = np.random.default_rng(each)
    agreed = 0
    for first, more in ((1, 0), (-1, 0), (1, 5), (1, 40)):
        partial = np.zeros(P.n_vars, np.int8)
        partial[0] = first
        pick = 2 + hubs + rng.choice(pool, size=more, replace=False)
        partial[pick] = rng.choice([-1, 1], size=more)
        opart = np.zeros(P.n_vars, np.int8)
        opart[perm] = partial
        want_conflict, want, _, _ = oracle.up_closure(prog, opart)
        conflict, got = P.propagate(partial)
        nconflict, ngot = _noalloc(torch, P, partial, 0)
        assert conflict == nconflict == bool(want_conflict)
        if not want_conflict:
            agreed += 1
            assert (got == want[perm]).all() and (ngot == want[perm]).all()
    assert agreed


@pytest.mark.parametrize("hubs,each,pool,filler,grid", [(1, 1500, 500, 300, 0), (17, 260, 800, 0, 0), (1, 3000, 4000, 9000, 0),
                                                        (300, 60, 6000, 6000, 0), (300, 100, 3000, 3000, 2)])
@pytest.mark.parametrize("k", [1, 5])
@pytest.mark.parametrize("learning", [0, 1])
def test_learning_with_hubs(env, hubs, each, pool, filler, grid, k, learning):
    _, gpu = env
    prog = _hubs(hubs, each, pool, filler, k)
    P = gpu.Program(prog, grid_ctas=grid, conflict_budget=k, learning=learning)
    status, _, _ = P.solve(1, cap=1)
    if status != gpu.UNKNOWN or P.stats()["conflicts"] != k:
        pytest.skip("search ended before the k-th conflict")
    if learning:
        _check_conflict(gpu, P)
        return
    compared, reasons = _check_at_conflict(gpu, P, prog, _completion(prog), 0)
    assert compared > 0 and reasons > 0


@pytest.mark.parametrize("learning", [0, 1])
@pytest.mark.parametrize("k", [1, 4, 12])
def test_list_rounds_by_lanes_above_the_root(env, learning, k):
    """Deciding atom 0 claims the 300 hubs' bodies at once, more than one CTA
    follows alone and few enough for lists; two CTAs of one warp each follow them
    a lane per occurrence, and the lanes write the claims' bitmaps."""
    _, gpu = env
    prog = _hubs(300, 40, 1500, 1500, k)
    P = gpu.Program(prog, grid_ctas=2, block_threads=32, conflict_budget=k, learning=learning)
    status, _, _ = P.solve(1, cap=1)
    s = P.stats()
    if status != gpu.UNKNOWN or s["conflicts"] != k:
        pytest.skip("search ended before the k-th conflict")
    if learning:
        _check_conflict(gpu, P)
    else:
        compared, reasons = _check_at_conflict(gpu, P, prog, _completion(prog), 0)
        assert compared > 300 and reasons > 300


def test_a_hub_costs_a_sweep_not_a_walk(env):
    """80k rules of one hub: a warp alone walks its list in several ms, and the
    grid sweeps the store in tens of us."""
    _, gpu = env
    P = gpu.Program(_hubs(1, 80_000, 40_000, 160_000, 1))
    partial = np.zeros(P.n_vars, np.int8)
    partial[0] = 1
    times = []
    for _ in range(3):
        assert not P.propagate(partial)[0]
        times.append(P.stats()["ns_total"])
    assert min(times) < 1.5e6, times


def test_a_hub_costs_a_sweep_without_allocation(env):
    """The same through asp_propagate_noalloc."""
    torch, gpu = env
    P = gpu.Program(_hubs(1, 80_000, 40_000, 160_000, 1))
    d = torch.zeros(P.n_vars, dtype=torch.int8, device="cuda")
    d[0] = 1
    out, conflict = torch.empty_like(d), torch.zeros(1, dtype=torch.int32, device="cuda")
    times = []
    for _ in range(4):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        assert P.propagate_noalloc(d.data_ptr(), out.data_ptr(), conflict.data_ptr()) == 0
        end.record()
        torch.cuda.synchronize()
        assert conflict.item() == 0
        times.append(start.elapsed_time(end))
    assert min(times) < 2.0, times
