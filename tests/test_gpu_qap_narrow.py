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
