"""The product form of the LBP iteration where fields are small: without a bias and at small beta
every message is far below 1, and its relative precision has to survive.

The reference is plain belief propagation in extended precision (the oracle's correlations, sums over
a clause's configurations, carry an absolute error of 6e-17). Tolerance: a message u <= u0 = -1/2 ln(1 -
c 2^-(k-1)) (about; every literal false with probability 1/2) takes some 3 k roundings, a field sums at
most `deg` messages, each again rounded: |error| <= 64 deg u0 2^-53 for k <= 4. Correlations are
-+c 2^-k to leading order: |error| <= 64 c 2^-53."""
import numpy as np
import pytest

import nmc_inputs as W
import oracle as O

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _reference(lits, n, beta, iters):
    """Marginals and correlations without a bias after `iters` iterations."""
    m, k = lits.shape
    var, sg = np.abs(lits) - 1, np.sign(lits).astype(LD)
    c = -np.expm1(-2 * LD(beta))
    h, u = np.zeros((m, k), LD), None
    for it in range(iters + 1):
        if it:
            field = np.zeros(n, LD)
            np.add.at(field, var.reshape(-1), (sg * u).reshape(-1))
            h = sg * (field[var] - sg * u)
        f = 1 / (1 + np.exp(2 * h))
        u = np.stack([-np.log1p(-c * np.delete(f, i, 1).prod(1)) / 2 for i in range(k)], 1)
    field = np.zeros(n, LD)
    np.add.at(field, var.reshape(-1), (sg * u).reshape(-1))
    viol = f.prod(1)
    return np.tanh(field), ((sg * np.tanh(h)).prod(1) - c * (-sg).prod(1) * viol) / (1 - c * viol)


@pytest.mark.parametrize("k,alpha,n", [(2, 1.5, 90), (3, 4.0, 200), (4, 9.6, 300)])
@pytest.mark.parametrize("beta", [1e-6, 1e-3, 0.1])
def test_small_fields_keep_their_relative_precision(k, alpha, n, beta):
    import paper_2111_13628_gb300 as nmc
    lits = W.random_ksat(n, alpha, k, 63)
    x = (W.splitmix64(64, 2 * n) & np.uint64(1)).astype(np.uint8).reshape(2, n)
    tol = max(1e-13 * beta, 1e-14)  # above the form's limit of 2e-15 at beta = 0.1
    eps = np.zeros(n)
    with nmc.Context(0) as ctx:
        inst = ctx.load_ksat(lits, n)
        got = ctx.cnf_lbp(inst, x, beta, [0.1], tol, 12, eps=eps)
    c = -np.expm1(-2.0 * beta)
    u0 = -0.5 * np.log1p(-c * 2.0 ** (1 - k))
    deg = np.bincount(np.abs(lits).reshape(-1) - 1, minlength=n).max()
    iters = O.cnf_lbp(lits, n, x[0], beta, [0.1], tol, 12, eps=eps)["iters"][0]
    marg, corr = _reference(lits, n, beta, int(iters))
    for s in range(2):
        assert got["iters"][s][0] == iters
        assert np.abs(got["marg"][s] - marg).max() <= 64 * deg * u0 * 2.0 ** -53
        assert np.abs(got["corr"][s] - corr).max() <= 64 * c * 2.0 ** -53
