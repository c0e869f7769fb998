"""Server ticks whose words get different shapes (CTAs a word, lanes a variable): mixed sizes, clause
lengths and slice lengths, up to more words than the GPU holds at once, bit for bit against the same
requests run one by one."""
import numpy as np
import pytest

import nmc_inputs as W

pytestmark = pytest.mark.gpu
KEYS = ("states", "energies", "best_energies", "best_states")
ALPHA = {3: 4.2, 4: 9.6, 6: 12.0}


@pytest.mark.parametrize("specs", [
    [(40, 3, 33), (9001, 4, 70)],                                                # one tiny, one long
    [(23, 3, 1), (700, 6, 90), (1500, 4, 32), (6001, 4, 250), (12007, 3, 160)],  # every shape
    [(300, 6, 64), (8000, 3, 256), (6999, 4, 128), (7001, 6, 128)],              # both widths large
    [(150, 4, 2048), (900, 6, 1024), (2000, 3, 1024), (3001, 4, 1024)],          # 160 words
], ids=["two", "all", "widths", "many"])
def test_requests_in_mixed_shapes_equal_single_runs(specs):
    import paper_2111_13628_gb300 as nmc
    T, reqs, want = 40, [], []
    with nmc.Context(0) as ctx:
        for i, (n, k, R) in enumerate(specs):
            reqs.append(dict(lits=W.random_ksat(n, ALPHA[k], k, 40 + i), n_vars=n, replicas=R, seed=60 + i,
                             beta=W.beta_inhomogeneous_linear(n, T, 0.3, 3.0, 0.3, 0.5, 50 + i)))
            inst = ctx.load_ksat(reqs[-1]["lits"], n)
            ctx.set_schedule(inst, reqs[-1]["beta"])
            want.append(ctx.anneal(inst, R, 0, T, 60 + i))
    with nmc.Server(0, slice_log2=20) as srv:  # several ticks for each request
        ids = [srv.submit_ksat(**r) for r in reqs]
        for i in ids:
            for _ in range(600):
                if srv.poll(i, wait_ms=200) not in (0, 1):
                    break
        got = [srv.result(i)[0] for i in ids]
    for g, w in zip(got, want):
        for key in KEYS:
            assert np.array_equal(g[key], w[key]), key
