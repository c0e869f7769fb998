"""Both forms of the QAP swap change, entries up to 127 (row differences in signed bytes) and
beyond, at the edges of the launch shapes and of the entry range, bit for bit against the oracle."""
import numpy as np
import pytest

import nmc_inputs as W
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 16, 17, 33, 64, 127, 128, 129, 160, 193, 255, 256])
@pytest.mark.parametrize("f_max,d_max", [(127, 127), (128, 127), (99, 128), (255, 255)])
def test_narrow_and_wide_entries(n, f_max, d_max):
    import paper_2111_13628_gb300 as nmc
    F, _ = W.random_qap(n, 71 + n, max_entry=f_max, flow_zero_frac=0.3)
    _, D = W.random_qap(n, 72 + n, max_entry=d_max)
    F[0, 1] = F[1, 0] = f_max  # the largest entries are present
    D[0, 1] = D[1, 0] = d_max
    T, R = 3, 37
    beta = W.beta_scaled_linear(n, T, 0.001, 0.05, 0.5, 1.5, 73)
    want = O.qap_anneal(F, D, beta, 0, T, seed=74, replicas=R)
    with nmc.Context(0) as ctx:
        inst = ctx.load_qap(F, D)
        ctx.set_schedule(inst, beta)
        got = ctx.anneal(inst, R, 0, T, seed=74)
    for a, b in (("states", "perms"), ("energies", "energies"),
                 ("best_energies", "best_energies"), ("best_states", "best_perms")):
        assert np.array_equal(got[a], want[b]), a


@pytest.mark.parametrize("n", [2, 5, 33, 64, 130, 256])
@pytest.mark.parametrize("temps", ["zero", "largest", "mixed"])
def test_largest_uphill_change(n, temps):
    """Acceptance by the largest change a draw allows: inverse temperatures 0 (every change), the
    largest (none uphill), and per facility from 0 over the steps of the table to held."""
    import paper_2111_13628_gb300 as nmc
    F, D = W.random_qap(n, 81 + n)
    T, R = 5, 70
    if temps == "mixed":
        u = W.Stream(82).unit(n * T).reshape(n, T)
        beta = (10.0 ** (-6.0 + 8.0 * u)).astype(np.float32)
        beta[::5] = 0.0
        beta[3::7, ::2] = np.inf
    else:
        beta = W.beta_constant(n, T, 0.0 if temps == "zero" else 65535.0)
    want = O.qap_anneal(F, D, beta, 0, T, seed=83, replicas=R)
    with nmc.Context(0) as ctx:
        inst = ctx.load_qap(F, D)
        ctx.set_schedule(inst, beta)
        got = ctx.anneal(inst, R, 0, T, seed=83)
    for a, b in (("states", "perms"), ("energies", "energies"),
                 ("best_energies", "best_energies"), ("best_states", "best_perms")):
        assert np.array_equal(got[a], want[b]), a
