"""Parallel tempering of batches whose groups fill the SMs: a prime temperature count keeps all its slots
in one block as long as that block's shared memory holds them, and is split unevenly where it does not.
Sampled realizations against the oracle, bit by bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 17
SMEM_MAX = 227 << 10  # shared memory of a block


@pytest.mark.parametrize("dim,L,n,M,one_block", [
    (2, 8, 3904, 59, True), (3, 4, 3904, 59, True), (2, 7, 3904, 61, True), (3, 7, 3904, 47, True),
    (3, 8, 4096, 43, False), (3, 10, 4096, 31, False),
])
def test_pt_prime_temperature_counts_of_large_batches(orc, dim, L, n, M, one_block):
    import torch
    from paper_2011_08560_gb300 import eamc
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    ctas, slots, smem = eamc.pt_split(dim, L, n, M, n_sm)
    if n_sm == 152:
        assert (ctas == 1) == one_block
    assert smem <= SMEM_MAX
    betas = list(np.geomspace(0.25, 2.5, M))
    e_g, e_hot, sweeps = -int(1.2 * L ** dim), -int(0.5 * L ** dim), 2
    ctx = eamc.Context(seed=SEED)
    ctx.pt_init(dim, L, n, betas)
    ctx.pt_set_rt_bounds(np.full(n, e_g, np.int32), np.full(n, e_hot, np.int32))
    ctx.pt_run(sweeps, count_roundtrips=True)
    S, E, lab, _ = ctx.pt_state()
    R = ctx.pt_roundtrips()
    for r in (0, n // 2 + 5, n - 1):
        p = orc.PTRealization(dim, L, SEED, r, betas)
        p.sweeps(sweeps, count_rt=True, e_g=e_g, e_hot=e_hot)
        assert np.array_equal(E[r], p.E) and np.array_equal(lab[r], p.label)
        assert np.array_equal(S[r].reshape(-1), p.S)
        for l in range(M):
            want = p.rt[l].as_dict()
            assert all(R[r][l][f] == want[f] for f in ("phase", "n_rt", "t_first", "t_last", "e_min"))
    ctx.close()
