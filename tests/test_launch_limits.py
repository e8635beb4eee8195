"""The shared-memory limits of the kernels hold for every context of a process: several host threads,
streams and devices.  A kernel's limit belongs to the kernel and the device, so a record of it in one
process-wide variable, or a call that lowers it, breaks another thread's launch."""
import re
import threading
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2011_08560_gb300" / "csrc"


def test_no_launch_state_in_process_wide_variables():
    found = []
    for f in sorted(CSRC.glob("*.cu*")):
        for k, line in enumerate(f.read_text().splitlines(), 1):
            if re.match(r"\s+static\s+(?!const\b|constexpr\b|thread_local\b|__)[\w:<> ]+[ *&]\w+(\[[^\]]*\])?\s*(=|\{|;)", line):
                found.append(f"{f.name}:{k}: {line.strip()}")
    assert not found, found


def test_every_tile_fits_the_limit():
    from paper_2011_08560_gb300 import build, eamc
    build.build()
    sizes = [eamc.tile_width_info(dim, L, w)[0] for dim in (2, 3) for L in range(3, 13)
             for w in [32] + eamc.narrow_widths(dim, L)]
    assert max(sizes) <= 225 * 1024


def _pt(stream, M, runs):
    from paper_2011_08560_gb300 import eamc
    ctx = eamc.Context(seed=5, stream=stream)
    ctx.pt_init(3, 6, 40, list(np.geomspace(0.3, 2.0, M)))
    for _ in range(runs):
        ctx.pt_run(1)
    out = [*ctx.pt_state(spins=False)[1:3]]
    ctx.close()
    return out


def _lex(stream, L, width, n, persistent, runs):
    from paper_2011_08560_gb300 import eamc
    ctx = eamc.Context(seed=6, stream=stream)
    if width != 32:
        ctx.set_tile_width(L, width)
    ctx.init_disorder(3, L, n)
    ctx.set_launch(persistent=persistent)
    for _ in range(runs):
        ctx.run_sweeps(1)
    out = [*ctx.state()]
    ctx.close()
    return out


@pytest.mark.gpu
def test_threads_with_small_and_large_blocks():
    """Blocks of little and of much shared memory of the same kernels from four host threads at once:
    the results of each alone."""
    import torch
    work = [(_pt, (2, 400)), (_pt, (61, 400)), (_lex, (8, 16, 64, False, 100)), (_lex, (7, 32, 64, False, 100)),
            (_lex, (4, 32, 64, True, 100)), (_lex, (10, 32, 40, False, 40))]
    alone = [f(torch.cuda.Stream().cuda_stream, *a) for f, a in work]
    for pair in ((0, 1, 0, 1), (2, 3, 4, 5), (0, 1, 2, 5)):
        got, streams = [None] * len(pair), [torch.cuda.Stream() for _ in pair]

        def call(k, job):
            f, a = work[job]
            try:
                got[k] = f(streams[k].cuda_stream, *a)
            except Exception as e:  # seen by the comparison below
                got[k] = e

        threads = [threading.Thread(target=call, args=(k, job)) for k, job in enumerate(pair)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for k, job in enumerate(pair):
            assert not isinstance(got[k], Exception), (job, got[k])
            for a, b in zip(got[k], alone[job]):
                assert np.array_equal(a, b), job
