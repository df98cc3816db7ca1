"""Large int8 batches, whose threads take runs of row pairs, against the oracle: rows of whole groups and of partial ones,
runs of two neighbouring lengths, columns shorter than a run, and the groups over the rows' ends."""
import numpy as np
import pytest

import oracle
import paper_0903_3053_gb300 as mc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extents", [[(4096, 514), (16, 8), (8, 2)], [(4094, 514), (10, 4), (14, 6), (4, 4)], [(2000, 1050), (2002, 1050)],
                                     [(8, 50000)] * 3 + [(4104, 514)], [(12, 20002)] * 2 + [(4090, 516)]])
def test_int8_runs_of_row_pairs_against_oracle(extents):
    assert sum((x // 8) * (y // 2) for x, y in extents) >= 1 << 17  # the threshold of the runs
    chains = [mc.ising(e, 0.42 + 0.01 * k, seed=31, chain_id=k) for k, e in enumerate(extents)]
    b = mc.Batch(chains, layout=mc.MC_LAYOUT_INT8, series_capacity=4)
    b.set_mode(mc.MC_MODE_GRID)
    b.sweep(3, 1)
    rec = b.read_series()
    for k, c in enumerate(chains):
        s = oracle.ising_init(c.L, c.seed, c.chain_id, True)
        E, M = oracle.ising_run(s, c.beta, c.seed, c.chain_id, 0, 3)
        np.testing.assert_array_equal(b.get_config(k), s)
        np.testing.assert_array_equal(rec["E"][k], E)
        np.testing.assert_array_equal(rec["M"][k], M)
    b.close()
