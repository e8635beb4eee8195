"""Parallel tempering with as many slots in one block as its shared memory holds: a temperature count
that is a prime above the cluster size keeps all slots in one block."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 11


@pytest.mark.parametrize("dim,L,M", [(2, 8, 59), (3, 4, 59), (2, 7, 61)])
def test_pt_many_slots_in_one_block(orc, dim, L, M):
    from paper_2011_08560_gb300 import eamc
    n, betas = 2, list(np.linspace(0.2, 3.0, M))
    ctx = eamc.Context(seed=SEED)
    ctx.pt_init(dim, L, n, betas)
    ctx.pt_set_rt_bounds(np.full(n, -80, np.int32), np.full(n, -30, np.int32))
    reals = [orc.PTRealization(dim, L, SEED, r, betas) for r in range(n)]
    ctx.pt_run(6, count_roundtrips=True)
    S, E, lab, _ = ctx.pt_state()
    for r, p in enumerate(reals):
        p.sweeps(6, count_rt=True, e_g=-80, e_hot=-30)
        assert np.array_equal(E[r], p.E) and np.array_equal(lab[r], p.label)
        assert np.array_equal(S[r].reshape(-1), p.S)
    assert np.array_equal(ctx.pt_swap_counts(), np.sum([p.swap_acc for p in reals], axis=0))
