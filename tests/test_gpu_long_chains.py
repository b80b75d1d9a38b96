"""Long chains of implications (needs a GB300): a choice starts
a_i :- a_(i-1), one variable after another for three rounds an atom, so one
CTA follows hundreds of thousands of rounds.  The time budget holds meanwhile,
and the other CTAs' barrier limit bounds a phase of it, not the whole chain."""
import numpy as np
import pytest

from synth.programs import from_rules

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1909_01786_gb300 import aspgpu
    aspgpu.lib()
    return aspgpu


def _chain(n):
    """0 :- not 1.  1 :- not 0.  i :- i - 1 (2 :- 0)."""
    return from_rules(n, [(0, [], [1]), (1, [], [0]), (2, [0], [])] + [(i, [i - 1], []) for i in range(3, n)])


@pytest.mark.parametrize("grid", [0, 1])
def test_time_budget_holds_on_a_chain(gpu, grid):
    """The whole chain takes more than 500 ms; the search stops within one
    phase (about 3 ms) of its budget."""
    P = gpu.Program(_chain(100_000), grid_ctas=grid, time_budget_ms=100)
    status, _, n = P.solve(1, cap=1)
    s = P.stats()
    assert status == gpu.UNKNOWN and n == 0
    assert 95e6 < s["ns_total"] < 150e6, s["ns_total"]


def test_time_budget_holds_in_the_stability_step(gpu):
    """One CTA: the assignment is total after about 600 ms, and the least model
    of the chain then takes seconds, a pass per atom; the search stops within
    a phase of passes of its budget."""
    P = gpu.Program(_chain(100_000), grid_ctas=1, time_budget_ms=1_500)
    status, _, n = P.solve(1, cap=1)
    s = P.stats()
    assert status == gpu.UNKNOWN and n == 0 and s["ns_stability"] > 0
    assert 1495e6 < s["ns_total"] < 1600e6, s["ns_total"]


@pytest.mark.parametrize("atom", [0, 1])
def test_barrier_limit_does_not_bound_a_chain(gpu, atom):
    """A limit of 100 ms against a chain of about 500 ms.  Atom 0 true makes
    every atom but 1 true, atom 1 true makes all others false."""
    n = 100_000
    P = gpu.Program(_chain(n))
    assert gpu.lib().asp_debug_barrier(P.handle, -1, 100) == 0
    partial = np.zeros(P.n_vars, np.int8)
    partial[atom] = 1
    conflict, closure = P.propagate(partial)
    want = np.full(n, 1 if atom == 0 else -1, np.int8)
    want[1 - atom], want[atom] = -1, 1
    assert not conflict and (closure[:n] == want).all()
    assert (closure != 0).all()


@pytest.mark.parametrize("grid", [0, 1])
def test_chain_answer_sets(gpu, grid):
    """Both answer sets: everything but atom 1, and atom 1 alone."""
    n = 3_000
    status, models, k = gpu.Program(_chain(n), grid_ctas=grid).solve(0, cap=4)
    want = np.ones((2, n), np.uint8)
    want[0, 1], want[1] = 0, 0
    want[1, 1] = 1
    assert status == gpu.SAT and k == 2
    assert {bytes(m) for m in models} == {bytes(m) for m in want}
