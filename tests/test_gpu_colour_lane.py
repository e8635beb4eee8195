"""The colour order's lane-per-chain kernel, chosen outright, through the oracle cases of the colour
order (small batches otherwise run a warp per chain), and which kernel large batches take by
themselves, with the trajectories of the other one."""
import types

import numpy as np
import pytest

from tests import test_gpu_colour as cases
from tests.test_gpu_colour import eamc  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.fixture
def lane(eamc):  # noqa: F811
    """The binding with contexts that run the colour order one lane per chain."""
    used = []

    class Context(eamc.Context):
        def __init__(self, *args, **kw):
            super().__init__(*args, **kw)
            self.set_colour_kernel(eamc.EA_COLOUR_LANE)

        def run_sweeps(self, *args, **kw):
            super().run_sweeps(*args, **kw)
            used.append(self.colour_kernel())

        def graph_capture(self, *args, **kw):
            super().graph_capture(*args, **kw)
            used.append(self.colour_kernel())

    module = types.SimpleNamespace(**vars(eamc))
    module.Context = Context
    yield module
    assert used and set(used) == {eamc.EA_COLOUR_LANE}


def _params(test):
    return [m for m in test.pytestmark if m.name == "parametrize"][0].args


SWEEPS, WIDTHS = _params(cases.test_colour_sweeps_bit_exact), _params(cases.test_narrow_colour_tiles_bit_exact)


@pytest.mark.parametrize(SWEEPS[0], SWEEPS[1] + [(2, 3, 40, 300, 0), (2, 7, 33, 150, 0), (2, 9, 5, 80, 0),
                                                 (2, 11, 34, 60, 0), (3, 9, 33, 8, 0), (3, 11, 33, 5, 0)])
def test_sweeps(lane, orc, dim, L, n, sweeps, cpc):
    cases.test_colour_sweeps_bit_exact(lane, orc, dim, L, n, sweeps, cpc)


@pytest.mark.parametrize(WIDTHS[0], WIDTHS[1])
def test_narrow_tiles(lane, orc, L, width, n, sweeps):
    cases.test_narrow_colour_tiles_bit_exact(lane, orc, L, width, n, sweeps)


@pytest.mark.parametrize("shapes", [((4, 16, 17), (6, 16, 18), (8, 16, 10)), ((5, 16, 9), (6, 16, 12), (8, 16, 7)),
                                    ((5, 16, 20), (7, 16, 20)), ((8, 32, 40), (9, 32, 33)), ((3, 32, 9), (7, 16, 33)),
                                    ((4, 8, 11), (6, 16, 18), (8, 8, 10)), ((5, 8, 9), (6, 8, 12), (8, 16, 7)),
                                    ((9, 8, 9), (11, 4, 5)), ((10, 8, 9), (12, 4, 6)), ((4, 8, 9), (7, 8, 9), (12, 4, 3))])
def test_mixed_contexts(lane, orc, shapes):
    """Every form of the kernel: even sizes, odd ones, both, and the small even sizes' narrow tiles."""
    cases.test_small_narrow_tiles_in_mixed_contexts(lane, orc, shapes)


def test_split_launches_and_graphs(lane, orc):
    cases.test_block_sizes_split_launches_and_graph_agree(lane, orc)


def test_berg_and_mixed_sizes(lane, orc):
    cases.test_colour_berg_mixed_sizes_and_narrow_tiles(lane, orc)


def test_snapshot_resume(lane, orc):
    cases.test_colour_snapshot_resume_and_narrow_tiles(lane, orc)


def test_kernel_queries(eamc):  # noqa: F811
    ctx = eamc.Context(seed=1)
    with pytest.raises(eamc.EamcError):
        ctx.colour_kernel()                         # no chains yet
    with pytest.raises(eamc.EamcError):
        ctx.set_colour_kernel(3)
    ctx.init_disorder(3, 8, 9)
    assert ctx.colour_kernel() == eamc.EA_COLOUR_WARP
    ctx.set_colour_kernel(eamc.EA_COLOUR_LANE)
    assert ctx.colour_kernel() == eamc.EA_COLOUR_LANE
    ctx.set_colour_kernel(eamc.EA_COLOUR_AUTO)
    assert ctx.colour_kernel() == eamc.EA_COLOUR_WARP


@pytest.mark.parametrize("dim,L,width,n", [(3, 3, 32, 4096), (3, 4, 32, 4864), (3, 5, 32, 4864), (3, 6, 32, 4096),
                                           (3, 7, 32, 4864), (3, 8, 32, 4864), (3, 9, 32, 4864), (3, 10, 32, 4864),
                                           (3, 11, 32, 4864), (3, 12, 32, 4864), (3, 4, 16, 2432), (3, 6, 16, 2300),
                                           (3, 7, 16, 2432), (3, 8, 16, 2432), (3, 10, 8, 1216), (2, 6, 32, 4864), (2, 7, 32, 4864)])
def test_large_batches_take_it_and_agree(eamc, dim, L, width, n):  # noqa: F811
    """Chains in their first weight steps, full SMs: the library takes the lane kernel, and the same
    batch one warp per chain has the same trajectories."""
    import torch

    def run(kernel):
        ctx = eamc.Context(seed=29)
        ctx.set_sweep_order(eamc.EA_ORDER_COLOUR)
        ctx.set_colour_kernel(kernel)
        if width != 32:
            ctx.set_tile_width(L, width)
        ctx.init_disorder(dim, L, n, rid0=7)
        took = ctx.colour_kernel()
        ctx.run_sweeps(3)
        ctx.update_weights()
        ctx.run_sweeps(3, count_roundtrips=True)
        ctx.check()
        out = [*ctx.state(), ctx.histograms(), ctx.roundtrips_array(), ctx.get_weights()]
        ctx.close()
        return took, out

    took, own = run(eamc.EA_COLOUR_AUTO)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert took == eamc.EA_COLOUR_LANE
    other, want = run(eamc.EA_COLOUR_LANE + eamc.EA_COLOUR_WARP - took)
    assert other != took
    for a, b in zip(own, want):
        assert np.array_equal(a, b)
