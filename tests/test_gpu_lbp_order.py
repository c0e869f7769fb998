"""A seed's LBP results do not depend on the other seeds of the call: the same bits alone, among a few
and among many (the launches differ: several lanes per variable where there is little to do)."""
import numpy as np
import pytest

import nmc_inputs as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,alpha,many", [(700, 4, 9.6, 64), (301, 3, 4.2, 200), (90, 5, 12.0, 500)])
def test_same_bits_alone_and_among_others(n, k, alpha, many):
    import paper_2111_13628_gb300 as nmc
    assert n * many >= 152 * 256 > n * 3  # both kinds of launch
    lits = W.random_ksat(n, alpha, k, 65)
    x = (W.splitmix64(66, many * n) & np.uint64(1)).astype(np.uint8).reshape(many, n)
    keys = ("marg", "corr", "iters", "deltas", "n_done", "p", "q1")
    with nmc.Context(0) as ctx:
        inst = ctx.load_ksat(lits, n)
        run = lambda rows: ctx.cnf_lbp(inst, np.ascontiguousarray(x[rows]), 1.0, [0.4, 0.1], 1e-8, 60)
        everyone = run(slice(None))
        for rows in ([0], [many - 1], [3, many // 2, 1]):
            few = run(rows)
            for key in keys:
                assert np.array_equal(few[key], everyone[key][rows]), key
