"""Full tiles swept in parts, a block each (lexicographic order, L >= 7), against the same tiles whole
(whose trajectories the other tests hold against the oracle)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n", [(7, 33), (8, 70), (8, 2432), (9, 40), (10, 65), (11, 35), (12, 37)])
def test_full_tiles_in_parts_agree(L, n):
    """Lexicographic order: full tiles run in parts of 16, 8 or 4 chains while each part has an SM to
    itself; the work-queue launch runs them whole.  Same chains, same results, last tiles ragged."""
    from paper_2011_08560_gb300 import eamc

    def run(persistent):
        ctx = eamc.Context(seed=31)
        ctx.init_disorder(3, L, n, rid0=7)
        ctx.set_ensemble(0, n, eamc.EA_POWERLAW)
        ctx.set_launch(persistent=persistent)
        for _ in range(2):
            ctx.run_sweeps(5)
            ctx.update_weights()
        ctx.run_sweeps(4, count_roundtrips=True)
        ctx.check()
        return ctx

    parts, whole = run(False), run(True)
    for a, b in zip(parts.state(), whole.state()):
        assert np.array_equal(a, b)
    assert np.array_equal(parts.histograms(), whole.histograms())
    assert np.array_equal(parts.roundtrips_array(), whole.roundtrips_array())
    assert np.array_equal(parts.get_weights(), whole.get_weights())


@pytest.mark.parametrize("L,n", [(8, 70), (10, 40), (12, 37)])
def test_parts_in_a_captured_graph_and_in_split_launches(L, n):
    """The captured iteration loop and launches of a few sweeps each, parts throughout: the same as
    direct calls."""
    import torch
    from paper_2011_08560_gb300 import eamc

    def run(graph, per_launch):
        stream = torch.cuda.Stream()
        ctx = eamc.Context(seed=32, stream=stream.cuda_stream)
        ctx.init_disorder(3, L, n)
        ctx.set_ensemble(0, n, eamc.EA_POWERLAW)
        ctx.set_launch(sweeps_per_launch=per_launch)
        if graph:
            ctx.graph_capture(n_iter=2, sweeps_per_iter=5, count_roundtrips=True, update_weights=True)
            ctx.graph_launch(1)
        else:
            for _ in range(2):
                ctx.run_sweeps(5, count_roundtrips=True)
                ctx.update_weights()
        ctx.synchronize()
        ctx.check()
        return [*ctx.state(), ctx.histograms(), ctx.roundtrips_array(), ctx.get_weights()]

    want = run(False, 0)
    for graph, per_launch in ((True, 0), (False, 2), (True, 3)):
        for a, b in zip(run(graph, per_launch), want):
            assert np.array_equal(a, b)
