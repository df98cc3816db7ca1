"""Calls long enough to run as several chunks on a new context: the random numbers of each go on where the one before
ended."""
import numpy as np
import pytest

import oracle
import paper_0903_3053_gb300 as mc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout,shape", [(mc.MC_LAYOUT_INT8, (64, 64)), (mc.MC_LAYOUT_INT8, (62, 66)),
                                          (mc.MC_LAYOUT_MSC32, (128, 64))])
def test_ising_chunks_of_a_call_against_oracle(layout, shape):
    """600 sweeps in one call: grid launches in chunks of 256, 256 and 88."""
    s = oracle.ising_init(shape, seed=17, chain=2, hot=True)
    E, M = oracle.ising_run(s, 0.4406868, 17, 2, 0, 600)
    b = mc.Batch([mc.ising(shape, 0.4406868, seed=17, chain_id=2)], layout=layout, series_capacity=600)
    b.set_mode(mc.MC_MODE_GRID)
    b.sweep(600, 1)
    rec = b.read_series()
    np.testing.assert_array_equal(b.get_config(0), s)
    np.testing.assert_array_equal(rec["E"][0], E)
    np.testing.assert_array_equal(rec["M"][0], M)
    b.close()


def test_su2_chunks_of_a_call():
    """300 sweeps in one call (chunks of 256 and 44) and as two calls of 150: the same links and records."""
    out = []
    for calls in ((300,), (150, 150)):
        b = mc.Batch([mc.su2((4, 4, 6, 4), 2.3, seed=19, chain_id=1)], series_capacity=300)
        b.set_mode(mc.MC_MODE_GRID)
        for n in calls:
            b.sweep(n, 1)
        out.append((b.get_config(0), b.read_series()))
        b.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
