"""The two colour-order kernels (one warp per chain, one lane per chain) give the same trajectories:
chains of a batch large enough for the lane kernel against the same chains in a small batch, which
the warp kernel runs (every other test of the colour order holds that one against the oracle)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [((3, 32, 4096),), ((4, 32, 4864),), ((6, 32, 4096),), ((6, 16, 2300),),
                                    ((8, 16, 2048),), ((10, 32, 4864),), ((12, 32, 4864),),
                                    ((3, 32, 2432), (4, 32, 2419))])
def test_large_and_small_batches_agree(shapes):
    from paper_2011_08560_gb300 import eamc

    def run(groups):
        ctx = eamc.Context(seed=29)
        ctx.set_sweep_order(eamc.EA_ORDER_COLOUR)
        for L, width, n, rid0 in groups:
            if width != 32:
                ctx.set_tile_width(L, width)
            first = ctx.init_disorder(3, L, n, rid0=rid0, stream=L)
            ctx.set_ensemble(first, n, eamc.EA_POWERLAW)
        for _ in range(2):
            ctx.run_sweeps(6)
            ctx.update_weights()
        ctx.run_sweeps(5, count_roundtrips=True)
        ctx.check()
        return ctx

    large = run([(L, w, n, 100) for L, w, n in shapes])
    at = 0
    for L, width, n in shapes:
        k = 33
        for chain0, rid0 in ((at, 100), (at + n - k, 100 + n - k)):
            small = run([(L, width, k, rid0)])
            assert np.array_equal(large.roundtrips_array(chain0, k), small.roundtrips_array())
            S, E, t = large.state(chain0, k)
            S2, E2, t2 = small.state()
            assert np.array_equal(S[:, :L ** 3], S2) and np.array_equal(E, E2) and np.array_equal(t, t2)
            assert np.array_equal(large.histograms(chain0, k), small.histograms())
            assert np.array_equal(large.get_weights(chain0, k), small.get_weights())
            small.close()
        at += n
    large.close()
