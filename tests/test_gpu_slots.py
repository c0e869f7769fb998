"""Sweeps whose colour classes overlap: the slots of a variable's list that hold no literal of the
previous class are counted before that class is published, the others after. Formulas at the edges
of that split, bit for bit against the oracle."""
import numpy as np
import pytest

import nmc_inputs as W
import oracle as O

pytestmark = pytest.mark.gpu


def _path(n):
    """A chain of 2-clauses: two classes, every occurrence holds a literal of the other one."""
    s = W.splitmix64(5, 2 * n) & np.uint64(1)
    a = np.arange(1, n, dtype=np.int32)
    lits = np.stack([a, a + 1], 1) * np.where(s[: 2 * (n - 1)].reshape(-1, 2), 1, -1)
    return np.ascontiguousarray(lits.astype(np.int32))


def _units(n):
    """Unit clauses only: one class, no other literals."""
    return (np.arange(n, dtype=np.int32)[:, None] + 1) * np.where(np.arange(n)[:, None] % 3, 1, -1).astype(np.int32)


FORMULAS = {
    "path": lambda: (_path(700), 700),
    "units": lambda: (_units(70), 70),
    "3sat_few_classes": lambda: (W.random_ksat(4001, 4.2, 3, 31), 4001),
    "4sat_partial_groups": lambda: (W.random_ksat(1030, 9.6, 4, 32), 1030),
    "6sat": lambda: (W.random_ksat(301, 12.0, 6, 33), 301),
}


@pytest.mark.parametrize("name", sorted(FORMULAS))
@pytest.mark.parametrize("ctas,lanes", [(1, 1), (2, 1), (8, 1), (1, 4), (4, 4), (2, 8)])
def test_overlapped_classes_match_oracle(monkeypatch, name, ctas, lanes):
    import paper_2111_13628_gb300 as nmc
    monkeypatch.setenv("NMC_BATCH_CTAS", str(ctas))
    monkeypatch.setenv("NMC_BATCH_LANES", str(lanes))
    lits, n = FORMULAS[name]()
    T, R = 6, 37
    beta = W.beta_inhomogeneous_linear(n, T, 0.3, 3.0, 0.3, 0.5, 34)
    beta[::7, ::2] = np.inf  # held units: lanes without an attempt
    want = O.ksat_anneal(lits, n, beta, 0, T, seed=35, replicas=R)
    with nmc.Context(0) as ctx:
        inst = ctx.load_ksat(lits, n)
        ctx.set_schedule(inst, beta)
        got = ctx.anneal(inst, R, 0, T, seed=35)
    for key in ("states", "energies", "best_energies", "best_states"):
        assert np.array_equal(got[key], want[key]), key
