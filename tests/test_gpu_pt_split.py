"""Parallel tempering with temperature counts that do not divide among the CTAs of a cluster (the last
CTA has empty slots), and batches of few and of many CTAs at each kind of lattice.  Sampled
realizations against the oracle, bit by bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 13


@pytest.mark.parametrize("dim,L,n,M,sweeps", [
    (3, 4, 3, 9, 8), (3, 3, 40, 17, 9), (2, 5, 33, 11, 9), (3, 5, 2, 20, 5), (2, 4, 5, 33, 6),
    (3, 8, 2, 17, 3), (3, 6, 2, 57, 2), (2, 12, 3, 64, 2),
    (3, 7, 608, 8, 3), (3, 8, 992, 12, 3), (3, 6, 640, 8, 3), (3, 9, 610, 8, 2), (3, 10, 450, 8, 2),
    (3, 7, 65, 8, 3), (3, 6, 35, 3, 4), (3, 9, 33, 10, 2), (3, 11, 2, 5, 2), (3, 12, 2, 17, 1),
])
def test_pt_uneven_splits_and_block_forms(orc, dim, L, n, M, sweeps):
    from paper_2011_08560_gb300 import eamc
    betas = list(np.geomspace(0.25, 2.5, M))
    e_g, e_hot = -int(1.2 * L ** dim), -int(0.5 * L ** dim)
    ctx = eamc.Context(seed=SEED)
    ctx.pt_init(dim, L, n, betas)
    ctx.pt_set_rt_bounds(np.full(n, e_g, np.int32), np.full(n, e_hot, np.int32))
    ctx.pt_run(sweeps, count_roundtrips=True)
    ctx.pt_run(1, count_roundtrips=True)
    S, E, lab, _ = ctx.pt_state()
    R = ctx.pt_roundtrips()
    picked = sorted({0, n // 2, n - 1})
    reals = [orc.PTRealization(dim, L, SEED, r, betas) for r in picked]
    for r, p in zip(picked, reals):
        p.sweeps(sweeps + 1, count_rt=True, e_g=e_g, e_hot=e_hot)
        assert np.array_equal(E[r], p.E) and np.array_equal(lab[r], p.label)
        assert np.array_equal(S[r].reshape(-1), p.S)
        for l in range(M):
            want = p.rt[l].as_dict()
            assert all(R[r][l][f] == want[f] for f in ("phase", "n_rt", "t_first", "t_last", "e_min"))
    if n <= 3:
        assert np.array_equal(ctx.pt_swap_counts(), np.sum([p.swap_acc for p in reals], axis=0))
    ctx.close()
