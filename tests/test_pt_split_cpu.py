"""The split of a parallel-tempering batch over CTAs, as the library plans it (host code, no GPU)."""
import pytest

SMEM_MAX = 227 << 10  # shared memory of a block


@pytest.fixture(scope="module")
def split():
    from paper_2011_08560_gb300 import build, eamc
    build.build()
    return eamc.pt_split


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("L", range(3, 13))
def test_every_split_fits_in_shared_memory(split, dim, L):
    """Whatever the number of realizations: the groups of 32 are fewer or more than the SMs."""
    for M in range(2, 65):
        for groups in (1, 2, 8, 16, 18, 19, 20, 32, 38, 64, 76, 128, 152, 153, 304, 1024):
            ctas, slots, smem = split(dim, L, 32 * groups, M, 152)
            assert 1 <= ctas <= 8 and (ctas - 1) * slots < M <= ctas * slots, (M, groups)
            assert smem <= SMEM_MAX, (M, groups, ctas, smem)


def test_refused_batches(split):
    from paper_2011_08560_gb300 import eamc
    for dim, L, n, M in ((4, 8, 1, 8), (3, 2, 1, 8), (3, 13, 1, 8), (3, 8, 0, 8), (3, 8, 1, 1), (3, 8, 1, 65)):
        with pytest.raises(eamc.EamcError):
            split(dim, L, n, M, 152)
