"""The colour order's choice between its two kernels by what the chains have been through (ensemble, weight
steps, given weights, snapshots): the same trajectories whichever runs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,W,n,sweeps", [(8, 16, 4096, 3), (6, 32, 2048, 4), (7, 32, 2500, 3)])
def test_results_do_not_depend_on_the_chains_history(L, W, n, sweeps):
    from paper_2011_08560_gb300 import eamc

    def context(kind):
        ctx = eamc.Context(seed=41)
        ctx.set_sweep_order(eamc.EA_ORDER_COLOUR)
        if W != 32:
            ctx.set_tile_width(L, W)
        ctx.init_disorder(3, L, n, rid0=3)
        ctx.set_ensemble(0, n, kind)
        return ctx

    first = context(eamc.EA_POWERLAW)
    for _ in range(4):
        first.run_sweeps(20)
        first.update_weights()
    weights = first.get_weights()
    runs = []
    for kind in (eamc.EA_POWERLAW, eamc.EA_FLAT):   # given weights: a chain's kind does not enter its sweeps
        ctx = context(kind)
        ctx.set_weights(0, weights)
        ctx.run_sweeps(sweeps, count_roundtrips=True)
        if kind == eamc.EA_POWERLAW:                # the rest from a snapshot
            saved = ctx.snapshot()
            ctx = eamc.Context(seed=41)
            ctx.restore(saved)
            ctx.set_sweep_order(eamc.EA_ORDER_COLOUR)
        ctx.run_sweeps(sweeps, count_roundtrips=True)
        ctx.check()
        runs.append([*ctx.state(), ctx.histograms(), ctx.roundtrips_array()])
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
