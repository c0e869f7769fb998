"""The batched kernel's wait between the CTAs of a word, run out on purpose with a short limit (an arrival
that never comes): every work item of the launch is reported, and the context stays usable."""
import numpy as np
import pytest

import nmc_inputs as W

pytestmark = pytest.mark.gpu


def test_expired_step_wait_marks_every_item(monkeypatch):
    import paper_2111_13628_gb300 as nmc
    with nmc.Context(0) as ctx:
        assert ctx.selftest_wait_timeout(40) == nmc.NMC_ETIMEOUT
        # sweeps on clusters of CTAs are still right, and report no wait
        n, T = 500, 6
        inst = ctx.load_ksat(W.random_ksat(n, 9.6, 4, 3), n)
        ctx.set_schedule(inst, W.beta_constant(n, T, 1.0))
        out = []
        for ctas in ("4", "1"):
            monkeypatch.setenv("NMC_BATCH_CTAS", ctas)
            out.append(ctx.anneal(inst, 70, 0, T, seed=4))
    for key in ("states", "energies", "best_energies", "best_states"):
        assert np.array_equal(out[0][key], out[1][key]), key
