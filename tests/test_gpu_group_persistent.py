"""The persistent launch of a group (a split cost, or MC_GROUP_FAIR_SHARE): bit-identical to each context's own
sweeps, and so to the oracle, for every cluster size, block size and split of the chains into
shared rounds (one chain on all CTAs of a cluster) and packed ones (one chain per CTA)."""
import numpy as np
import pytest

import oracle
import paper_0903_3053_gb300 as mc
from test_gpu_batch import assert_same, mixed_batches, snapshot

pytestmark = pytest.mark.gpu
FAIR = mc.MC_GROUP_FAIR_SHARE


@pytest.fixture(scope="module")
def reference():
    bs = mixed_batches()
    for b in bs:
        b.set_mode(mc.MC_MODE_GRID, 256)
        b.sweep(4, 2)
        b.sweep(2, 2)
    return snapshot(bs)


# the chains' costs are 24 .. 983040 and their sum 2.2e6: 1e5 shares four of eleven, 1e4 all but four
@pytest.mark.parametrize("C,threads,split", [(1, 256, FAIR), (1, 64, 0.0), (2, 128, FAIR), (4, 256, FAIR), (8, 128, FAIR),
                                             (16, 128, FAIR), (2, 64, 1e5), (4, 96, 1e4), (8, 256, 1e5), (16, 256, 1e4)])
def test_persistent_group_matches_context_sweeps(reference, C, threads, split):
    bs = mixed_batches()
    g = mc.Group(bs)
    g.configure(C, threads, split)
    assert g.schedule() == (0, 0)
    g.sweep(4, 2)
    g.sweep(2, 2)
    assert min(g.schedule()) >= 1
    assert_same(snapshot(bs), reference)
    g.close()


@pytest.mark.parametrize("C,split", [(1, FAIR), (2, FAIR), (4, 0.0), (4, 5000.0)])
def test_persistent_group_chains_against_oracle(C, split):
    """Both layouts, thresholds of zero among them (beta = 3: T4; 6: both)."""
    chains = [mc.ising(32, 0.4406868, seed=5, chain_id=9), mc.ising((64, 32), 0.3, seed=6, chain_id=1),
              mc.ising((62, 10), 0.5, seed=4, chain_id=6)]
    msc = [mc.ising(128, 0.5, seed=7, chain_id=4), mc.ising((128, 64), 3.0, seed=8, chain_id=2),
           mc.ising(64, 6.0, seed=9, chain_id=3)]
    b1 = mc.Batch(chains, layout=mc.MC_LAYOUT_INT8, series_capacity=8)
    b2 = mc.Batch(msc, layout=mc.MC_LAYOUT_MSC32, series_capacity=8)
    g = mc.Group([b1, b2])
    g.configure(C, 128, split)
    g.sweep(10, 5)
    for b, cs in ((b1, chains), (b2, msc)):
        rec = b.read_series()
        for k, c in enumerate(cs):
            s = oracle.ising_init(c.L, c.seed, c.chain_id, True)
            E, M = oracle.ising_run(s, c.beta, c.seed, c.chain_id, 0, 10)
            np.testing.assert_array_equal(b.get_config(k), s)
            np.testing.assert_array_equal(rec["E"][k], E[4::5])
            np.testing.assert_array_equal(rec["M"][k], M[4::5])
    g.close()


@pytest.mark.parametrize("C,split", [(1, FAIR), (4, FAIR), (4, 0.0), (2, 3e5)])
def test_persistent_group_with_overrelaxation(C, split):
    """The contexts' compound sweeps, also after the overrelaxation count changes between calls and after calls of the
    side-by-side form in between."""
    def make():
        return mc.Batch([mc.su2((4, 4, 4, 4), 2.3, seed=41, chain_id=0), mc.su2((6, 4, 4, 8), 2.0, seed=42, chain_id=1)],
                        series_capacity=16)
    steps = ((2, 3), (1, 2), (0, 1), (3, 2))  # overrelaxation count, sweeps
    ref = make()
    ref.set_mode(mc.MC_MODE_GRID, 256)
    for n_or, n in steps:
        ref.set_overrelax(n_or)
        ref.sweep(n, 1)
    b = make()
    g = mc.Group([b])
    for i, (n_or, n) in enumerate(steps):
        if i != 1:  # the second step with the first one's schedule
            g.configure(C, 256, mc.MC_GROUP_SIDE_BY_SIDE if i == 2 else split)
        b.set_overrelax(n_or)
        g.sweep(n, 1)
    assert_same(snapshot([b]), snapshot([ref]))
    g.close()


@pytest.mark.parametrize("layout", [mc.MC_LAYOUT_INT8, mc.MC_LAYOUT_MSC32])
def test_paper_lattice_in_one_persistent_launch(layout):
    """1024 x 512 (Sec. 2.3), hot start, beta_c, 10 measured sweeps, shared by a cluster."""
    s = oracle.ising_init((1024, 512), seed=1, chain=0, hot=True)
    E, M = oracle.ising_run(s, 0.4406868, 1, 0, 0, 10)
    b = mc.Batch([mc.ising((1024, 512), 0.4406868, seed=1, chain_id=0)], layout=layout, series_capacity=16)
    g = mc.Group([b])
    g.configure(4, 256, FAIR)
    g.sweep(10, 1)
    rec = b.read_series()
    np.testing.assert_array_equal(b.get_config(0), s)
    np.testing.assert_array_equal(rec["E"][0], E)
    np.testing.assert_array_equal(rec["M"][0], M)
    g.close()
    b.close()
