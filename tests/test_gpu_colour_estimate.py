"""The kernel that the library takes for the colour order is the one that measures faster (152 SMs).  Only
the choice is tested; no time is."""
import pytest

pytestmark = pytest.mark.gpu

WARP, LANE = 1, 2  # EA_COLOUR_WARP, EA_COLOUR_LANE


def _choice(dim, L, width, n, power, steps):
    import torch
    from paper_2011_08560_gb300 import eamc
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the figures are of 152 SMs")
    ctx = eamc.Context(seed=3)
    ctx.set_sweep_order(eamc.EA_ORDER_COLOUR)
    if width != 32:
        ctx.set_tile_width(L, width)
    ctx.init_disorder(dim, L, n)
    ctx.set_ensemble(0, n, eamc.EA_POWERLAW if power else eamc.EA_FLAT)
    for _ in range(steps):
        ctx.run_sweeps(1)
        ctx.update_weights()
    kernel = ctx.colour_kernel()
    ctx.close()
    return kernel


# attempts/ns, warp against lane, where they differ by 5 % or more
@pytest.mark.parametrize("dim,L,width,n,power,steps,faster", [
    (2, 3, 32, 256, True, 1, LANE), (2, 3, 32, 1024, True, 1, LANE), (2, 4, 32, 1024, True, 1, LANE),   # 1.3 / 1.7, 4.3 / 7.0, 12 / 19
    (2, 4, 32, 2048, True, 1, LANE), (2, 5, 32, 512, True, 1, WARP), (2, 5, 32, 1024, True, 1, LANE),   # 16 / 37, 6.6 / 6.3, 11 / 13
    (2, 6, 32, 1024, True, 1, WARP), (2, 6, 32, 2048, True, 1, LANE), (2, 7, 32, 1024, True, 1, WARP),  # 24 / 21, 32 / 42, 20 / 17
    (2, 7, 32, 2048, True, 27, LANE), (2, 8, 32, 1024, True, 1, WARP), (2, 8, 32, 2048, True, 27, LANE),  # 29 / 33, 40 / 32, 58 / 65
    (2, 9, 32, 1536, True, 1, WARP), (2, 9, 32, 3072, True, 1, LANE), (2, 10, 32, 1024, True, 1, WARP),  # 38 / 32, 41 / 64, 37 / 27
    (2, 11, 32, 3072, True, 1, LANE), (2, 12, 32, 1024, False, 1, WARP), (2, 12, 32, 3072, True, 1, LANE),  # 40 / 71, 40 / 32, 52 / 96
    (3, 9, 32, 4864, True, 10, WARP), (3, 9, 32, 4864, True, 1, LANE), (3, 7, 32, 4864, True, 10, WARP),  # 76 / 69, 63 / 69, 75 / 64
    (3, 6, 32, 2048, True, 27, WARP), (3, 6, 32, 2048, True, 1, LANE), (3, 8, 16, 4096, True, 27, WARP),  # 70 / 65, 51 / 65, 94 / 89
    (3, 8, 16, 4096, True, 1, LANE), (3, 8, 16, 2432, True, 27, LANE), (3, 4, 16, 2432, False, 1, LANE),  # 68 / 89, 99 / 105, 58 / 65
    (3, 3, 32, 2432, True, 1, LANE), (3, 5, 32, 4864, True, 27, LANE), (3, 12, 32, 2048, True, 1, WARP),  # 20 / 23, 60 / 68, 53 / 39
])
def test_the_faster_kernel_is_taken(dim, L, width, n, power, steps, faster):
    assert _choice(dim, L, width, n, power, steps) == faster


# contexts of several sizes, power law, first weight step: (L, width, chains)
@pytest.mark.parametrize("dim,groups,faster", [
    (3, [(4, 8, 200), (6, 8, 200), (8, 8, 200), (10, 8, 200), (12, 4, 200)], LANE),    # 11 / 17.5
    (3, [(4, 8, 60), (6, 8, 60), (8, 8, 60), (10, 8, 60), (12, 4, 60)], WARP),         # 6.0 / 5.2
    (3, [(4, 32, 200), (6, 32, 200), (8, 32, 200), (10, 32, 200), (12, 32, 200)], WARP),  # 11 / 2.6
    (3, [(7, 8, 333), (8, 8, 333), (9, 8, 333)], LANE), (3, [(8, 8, 500), (9, 8, 500)], WARP),  # 15 / 24, 33 / 26
    (3, [(8, 32, 500), (10, 32, 500)], WARP), (3, [(5, 8, 2048), (7, 8, 2048)], WARP),    # 32 / 13, 51 / 27
    (3, [(L, 8 if L < 11 else 4, 111) for L in range(4, 13)], LANE), (3, [(6, 32, 2048), (8, 32, 2048)], WARP),  # 6.8 / 15, 63 / 18
    (2, [(4, 32, 200), (6, 32, 200), (8, 32, 200), (10, 32, 200), (12, 32, 200)], LANE),  # 6.9 / 15
    (2, [(4, 32, 600), (6, 32, 600), (8, 32, 600), (10, 32, 600), (12, 32, 600)], LANE),  # 17 / 45
    (2, [(8, 32, 500), (12, 32, 500)], WARP),  # 31 / 22
])
def test_the_faster_kernel_is_taken_for_several_sizes(dim, groups, faster):
    import torch
    from paper_2011_08560_gb300 import eamc
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the figures are of 152 SMs")
    ctx = eamc.Context(seed=3)
    ctx.set_sweep_order(eamc.EA_ORDER_COLOUR)
    for L, width, n in groups:
        if width != 32:
            ctx.set_tile_width(L, width)
        ctx.set_ensemble(ctx.init_disorder(dim, L, n), n, eamc.EA_POWERLAW)
    ctx.run_sweeps(1)
    ctx.update_weights()
    kernel = ctx.colour_kernel()
    ctx.close()
    assert kernel == faster
