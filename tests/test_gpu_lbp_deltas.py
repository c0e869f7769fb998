"""The largest change of a message per seed and lambda (`deltas`), which decides convergence, and the
product form near its limit of beta = 4, against the oracle. Tolerance 1e-9 as in test_gpu_lbp.py: a
message's rounding is amplified to about 2^-53 e^{2 beta} = 3e-13 at beta = 4, a few iterations add
a few times that."""
import numpy as np
import pytest

import nmc_inputs as W
import oracle as O

pytestmark = pytest.mark.gpu
TOL = 1e-9


def _run(lits, n, x, beta, lam, tol, max_iter, eps):
    import paper_2111_13628_gb300 as nmc
    with nmc.Context(0) as ctx:
        inst = ctx.load_ksat(lits, n)
        got = ctx.cnf_lbp(inst, x, beta, lam, tol, max_iter, eps=eps)
    want = [O.cnf_lbp(lits, n, x[s], beta, lam, tol, max_iter, eps=eps) for s in range(len(x))]
    for s, w in enumerate(want):
        assert got["n_done"][s] == w["n_done"]
        assert np.array_equal(got["iters"][s], w["iters"])
        for key in ("marg", "corr", "deltas"):
            np.testing.assert_allclose(got[key][s], w[key], rtol=0, atol=TOL, err_msg=key)
    return want


@pytest.mark.parametrize("beta", [2.5, 3.5, 4.0])
@pytest.mark.parametrize("draw", [98, 101, 107, 109])
def test_largest_change_among_nearly_equal_ones(beta, draw):
    """Components (a or b), (not b), (not b or d) whose first message to a grows from near 0 to near beta.
    The amounts differ by parts in 10^7 from one component to the next, while the messages before and
    after, w = e^{-2u}, both differ by parts in 10 (the bias of d sets the field of b that gives
    the amount). Many equal seeds, so that no wave of threads holds all components of one."""
    import paper_2111_13628_gb300 as nmc
    C, S = 400, 1024
    s = W.Stream(draw)
    c = -np.expm1(-2.0 * beta)
    e_b = beta * (0.45 + 0.15 * s.unit(C))
    change = 0.92 * beta * (1.0 + 2e-7 * np.argsort(s.unit(C)))
    w_old = 1.0 - c / (1.0 + np.exp(2.0 * e_b))
    E = c / (1.0 - w_old * np.exp(-2.0 * change)) - 1.0
    u_d = e_b - beta - 0.5 * np.log(E)
    e_d = 0.5 * np.log(c / -np.expm1(-2.0 * u_d) - 1.0)
    assert np.isfinite(e_d).all()
    v = 3 * np.arange(C, dtype=np.int32)
    z = np.zeros(C, np.int32)
    lits = np.concatenate([np.stack([v + 1, v + 2], 1), np.stack([-(v + 2), z], 1), np.stack([-(v + 2), v + 3], 1)])
    lits = np.ascontiguousarray(lits[::-1]).astype(np.int32)
    n = 3 * C
    eps = np.zeros(n)
    eps[1::3], eps[2::3] = e_b, e_d
    with nmc.Context(0) as ctx:
        inst = ctx.load_ksat(lits, n)
        got = ctx.cnf_lbp(inst, np.ones((S, n), np.uint8), beta, [1.0], 1e-8, 1, eps=eps)["deltas"]
    want = O.cnf_lbp(lits, n, np.ones(n, np.uint8), beta, [1.0], 1e-8, 1, eps=eps)["deltas"][0]
    assert abs(want - change.max()) < TOL
    assert np.abs(got - want).max() < TOL


@pytest.mark.parametrize("k,alpha", [(3, 2.5), (3, 4.2), (4, 9.6), (5, 12.0), (8, 20.0)])
@pytest.mark.parametrize("beta", [1.0, 3.5, 4.0, 4.5])
@pytest.mark.parametrize("max_iter", [1, 3])
def test_before_convergence(k, alpha, beta, max_iter):
    n = 150
    lits = W.random_ksat(n, alpha, k, 93)
    x = (W.splitmix64(94, 3 * n) & np.uint64(1)).astype(np.uint8).reshape(3, n)
    want = _run(lits, n, x, beta, [0.4, 0.1], 1e-8, max_iter, np.full(n, 0.5))
    assert all(w["n_done"] == 0 for w in want)


@pytest.mark.parametrize("k,alpha", [(3, 1.5), (4, 2.5), (5, 2.5)])
@pytest.mark.parametrize("beta", [3.5, 4.0])
def test_converged_near_the_limit(k, alpha, beta):
    n = 120
    lits = W.random_ksat(n, alpha, k, 91)
    x = (W.splitmix64(92, 3 * n) & np.uint64(1)).astype(np.uint8).reshape(3, n)
    want = _run(lits, n, x, beta, [0.4, 0.2], 1e-8, 60, np.full(n, 0.5))
    assert all(w["n_done"] == 2 for w in want)


@pytest.mark.parametrize("k,alpha", [(2, 1.2), (3, 3.0), (4, 4.0)])
@pytest.mark.parametrize("beta,bias", [(0.5, 320.0), (1.0, 300.0), (4.0, 150.0), (2.0, 18.0)])
def test_fields_near_the_end_of_the_range(k, alpha, beta, bias):
    """|field| up to just below 340, where e^{+-2 field} and products of 1 - m reach the ends of what the
    product form holds; every third variable without a bias."""
    n = 150
    lits = W.random_ksat(n, alpha, k, 97)
    assert beta * np.bincount(np.abs(lits).reshape(-1) - 1).max() + bias < 340.0
    x = (W.splitmix64(98, 3 * n) & np.uint64(1)).astype(np.uint8).reshape(3, n)
    eps = np.full(n, bias)
    eps[::3] = 0.0
    eps[1::3] *= np.linspace(-1.0, 1.0, len(eps[1::3]))
    _run(lits, n, x, beta, [1.0, 0.5], 1e-8, 4, eps)
