"""The two forms of the LBP iteration against the oracle: products of e^{-2u} (fields that fit the
range of a double) and sums of u (larger beta or bias). Tolerance 1e-9 as in test_gpu_lbp.py: both
forms differ from the oracle by a few ulp a step, and a convergent iteration contracts that."""
import numpy as np
import pytest

import nmc_inputs as W
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,alpha,n", [(1, 0.5, 40), (2, 1.2, 90), (3, 4.0, 200), (4, 9.0, 150),
                                       (5, 12.0, 60), (8, 6.0, 50)])
@pytest.mark.parametrize("beta,eps", [(0.0, None), (1.0, None), (3.5, 0.5), (6.0, 1.0), (1.0, 900.0)])
def test_both_forms_match_oracle(k, alpha, n, beta, eps):
    import paper_2111_13628_gb300 as nmc
    lits = W.random_ksat(n, alpha, k, 61)
    lits[::5, -1] = 0 if k > 1 else lits[::5, -1]  # padding slots
    S = 3
    x = (W.splitmix64(62, S * n) & np.uint64(1)).astype(np.uint8).reshape(S, n)
    e = None if eps is None else np.full(n, eps)
    lam = [0.5, 0.2]
    with nmc.Context(0) as ctx:
        inst = ctx.load_ksat(lits, n)
        got = ctx.cnf_lbp(inst, x, beta, lam, 1e-8, 40, eps=e)
    for s in range(S):
        want = O.cnf_lbp(lits, n, x[s], beta, lam, 1e-8, 40, eps=e)
        if want["n_done"] == 0:
            continue  # never converged: nothing contracts the rounding differences
        assert got["n_done"][s] == want["n_done"]
        assert np.array_equal(got["iters"][s], want["iters"])
        for key in ("marg", "corr"):
            np.testing.assert_allclose(got[key][s], want[key], rtol=0, atol=1e-9)
        np.testing.assert_allclose([got["p"][s], got["q1"][s]], [want["p"], want["q1"]], rtol=0,
                                   atol=1e-9)
