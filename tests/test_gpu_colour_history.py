"""What the colour order's choice of kernel knows of the chains: weight steps wherever they are made, and
weights that are given.  4096 chains of L = 8 in tiles of 16: the lane kernel is faster on power-law
chains in their first steps (68 against 89 attempts/ns) and on flat ones, the warp kernel on iterated
power-law chains (100 against 89).  Only the choice is tested; no time is."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, L, WARP, LANE = 4096, 8, 1, 2  # EA_COLOUR_WARP, EA_COLOUR_LANE


@pytest.fixture(scope="module")
def eamc():
    import torch
    from paper_2011_08560_gb300 import eamc as m
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the figures are of 152 SMs")
    return m


def _context(eamc, kinds=None, n=N):
    import torch
    ctx = eamc.Context(seed=41, stream=torch.cuda.Stream().cuda_stream)
    ctx.set_sweep_order(eamc.EA_ORDER_COLOUR)
    ctx.set_tile_width(L, 16)
    kinds = [eamc.EA_POWERLAW] if kinds is None else kinds
    for k, kind in enumerate(kinds):
        first = ctx.init_disorder(3, L, n // len(kinds), rid0=3, stream=k)
        ctx.set_ensemble(first, n // len(kinds), kind)
    return ctx


def _iterate(ctx, steps, sweeps=1):
    for _ in range(steps):
        ctx.run_sweeps(sweeps)
        ctx.update_weights()


def test_steps_are_counted_wherever_they_are_made(eamc):
    ctx = _context(eamc)
    assert ctx.colour_kernel() == LANE
    _iterate(ctx, 3)
    assert ctx.colour_kernel() == LANE
    _iterate(ctx, 37)
    assert ctx.colour_kernel() == WARP
    ctx.reset_chains(np.arange(N), np.arange(N) + 3, np.zeros(N, dtype=int))  # unit weights again
    assert ctx.colour_kernel() == LANE

    graph = _context(eamc)
    graph.graph_capture(n_iter=10, sweeps_per_iter=1, update_weights=True)
    graph.graph_launch(1)
    assert graph.colour_kernel() == LANE
    graph.graph_launch(3)
    assert graph.colour_kernel() == WARP
    plain = _context(eamc)
    plain.graph_capture(n_iter=40, sweeps_per_iter=1, update_weights=False)
    plain.graph_launch(1)
    assert plain.colour_kernel() == LANE

    subset = _context(eamc)
    for _ in range(40):
        subset.run_sweeps(1)
        subset.update_weights_subset(np.arange(0, N, 2))
    assert subset.colour_kernel() == LANE                                    # half of the chains
    for _ in range(40):
        subset.update_weights_subset(np.arange(1, N, 2))
    assert subset.colour_kernel() == WARP


def test_flat_chains_count_by_their_share(eamc):
    mixed = _context(eamc, [eamc.EA_POWERLAW, eamc.EA_FLAT])
    _iterate(mixed, 27)
    assert mixed.colour_kernel() == LANE
    flat = _context(eamc, [eamc.EA_FLAT])
    _iterate(flat, 40)
    assert flat.colour_kernel() == LANE


def test_given_weights_count_as_what_they_are(eamc):
    """Weights given every step from the first, as by a recursion on the host, a snapshot early and late,
    thresholds, weights copied within a context."""
    donor = _context(eamc)
    assert donor.colour_kernel() == LANE
    for steps, kernel in ((2, LANE), (38, WARP)):
        _iterate(donor, steps, 60)
        given = _context(eamc)
        given.set_weights(0, donor.get_weights())
        assert given.colour_kernel() == kernel
        given = _context(eamc)
        given.set_thresholds(0, donor.get_thresholds())
        assert given.colour_kernel() == kernel
        saved = eamc.Context(seed=41)
        saved.restore(donor.snapshot())
        saved.set_sweep_order(eamc.EA_ORDER_COLOUR)
        assert saved.colour_kernel() == kernel
    given.set_weights(0, np.zeros_like(donor.get_weights()))
    assert given.colour_kernel() == LANE

    ctx = _context(eamc, n=N // 2)
    _iterate(ctx, 40)
    new = ctx.init_disorder(3, L, N // 2, rid0=3, stream=9)
    assert ctx.colour_kernel() == LANE                                       # half of the chains are new
    ctx.copy_weights(np.arange(N // 2), new + np.arange(N // 2))
    assert ctx.colour_kernel() == WARP
    ctx.build_ensemble(0, N, eamc.EA_FLAT)
    assert ctx.colour_kernel() == LANE
