"""Loading programs with far more atoms than rules (needs a GB300): few
literals and very many of them without an occurrence."""
import time

import numpy as np
import pytest

import oracle
from synth.programs import Program, program_seed, random_program

from test_gpu_lists import _perm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1909_01786_gb300 import aspgpu
    aspgpu.lib()
    return aspgpu


def _sparse(atoms, rules):
    """`rules` random rules over 60 atoms, and further atoms without a rule"""
    p = random_program(60, rules, program_seed(1401, rules))
    return Program(atoms, p.head, p.pos_off, p.pos, p.neg_off, p.neg)


# 300 variables more for 100 rules; one block builds the lists of up to 8192
# literals of up to 32768 variables
@pytest.mark.parametrize("atoms,rules", [(60, 100), (32_467, 100), (32_468, 100), (32_469, 100), (100_000, 100), (60, 400), (9000, 400),
                                         (60, 600), (100_000, 600)])
def test_closures_of_sparse_programs(gpu, atoms, rules):
    prog = _sparse(atoms, rules)
    P = gpu.Program(prog)
    perm = _perm(prog)
    rng = np.random.default_rng(atoms)
    agreed = 0
    for k in (0, 1, 4):
        partial = np.zeros(P.n_vars, np.int8)
        pick = rng.choice(60, size=k, replace=False)
        partial[pick] = -1
        opart = np.zeros(P.n_vars, np.int8)
        opart[perm] = partial
        want_conflict, want, _, _ = oracle.up_closure(prog, opart)
        conflict, got = P.propagate(partial)
        assert conflict == bool(want_conflict)
        if not conflict:
            agreed += 1
            assert (got == want[perm]).all()
    assert agreed


def test_many_atoms_and_few_rules_load_as_fast_as_with_more(gpu):
    """4M atoms: nearly all lists are empty, whoever builds them (one block took
    7 ms longer, of 42)."""
    best = {}
    progs = {rules: _sparse(4_000_000, rules) for rules in (200, 1000)}
    for _ in range(8):
        for rules, prog in progs.items():
            t = time.perf_counter()
            P = gpu.Program(prog, learned_capacity=1 << 16, deps_levels=64)
            t = time.perf_counter() - t
            P.close()
            best[rules] = min(t, best.get(rules, t))
    assert best[200] < 1.11 * best[1000], best
