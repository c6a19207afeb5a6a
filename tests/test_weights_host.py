"""What a context asks of its caller's memory (host only): the workspace holds the state of a step, whatever the
number of neighbours; the pair weights of multi-step calls have a buffer of their own that nobody has to give."""
import ctypes

import pytest

from paper_2108_09488_gb300 import inputs

FAKE = 1 << 40          # 256-aligned placeholder device addresses; never dereferenced here


def test_workspace_does_not_grow_with_the_neighbours(adelib):
    """Bytes per particle: keys, ranks, two permutations (16), two sorted copies (32), cell tables and partials."""
    for p in (inputs.Plume(3, 128, 2.0), inputs.Plume(3, 64, 2.0), inputs.Plume(2, 1024, 3.0425),
              inputs.Plume(2, 2048, 1.5)):
        assert adelib.workspace_bytes(adelib.params_for(p), p.n) < 100 * p.n
    plumes = inputs.batched_2d(64, seed=20210821)
    n = [p.n for p in plumes]
    assert adelib.batch_workspace_bytes([adelib.params_for(p) for p in plumes], n) < 100 * sum(n)
    p = inputs.Plume(2, 512, 2.1225)
    assert adelib.sweep_workspace_bytes(adelib.params_for(p), p.n, 8) < (100 + 8 * 8) * p.n


def test_weights_need_a_size_asked_for_and_a_buffer_that_fits(adelib):
    p = inputs.lattice_2d_64()
    prm = adelib.params_for(p)
    ctx = adelib.init_particles(prm, p.n, FAKE, FAKE + (1 << 30), FAKE + (2 << 30), adelib.workspace_bytes(prm, p.n))
    lib = adelib.load()
    try:
        assert lib.ade_set_weights(ctx, FAKE + (3 << 30), 1 << 30) == -6      # no size asked for
        assert lib.ade_set_weights(ctx, FAKE + (3 << 30) + 8, 1 << 30) == -1
        assert lib.ade_set_weights(ctx, None, 0) == 0
        assert lib.ade_set_weights(None, None, 0) == -1
        nbytes = ctypes.c_size_t(7)
        assert lib.ade_weights_bytes(ctx, 0, ctypes.byref(nbytes), None) == 0 and nbytes.value > 4 * 20 * p.n   # estimated
        assert lib.ade_set_weights(ctx, FAKE + (3 << 30), 256) == -5
        assert lib.ade_weights_bytes(None, 0, ctypes.byref(nbytes), None) == -1
        assert lib.ade_weights_bytes(ctx, 0, None, None) == -1
    finally:
        adelib.destroy(ctx)


@pytest.mark.parametrize("over", [dict(flags=1), dict(vmax=0.2)])
def test_no_weights_where_they_are_not_kept(adelib, over):
    p = inputs.lattice_2d_64()
    prm = adelib.params_for(p, **over)
    ctx = adelib.init_particles(prm, p.n, FAKE, FAKE + (1 << 30), FAKE + (2 << 30), adelib.workspace_bytes(prm, p.n))
    try:
        nbytes = ctypes.c_size_t(7)
        assert adelib.load().ade_weights_bytes(ctx, 1, ctypes.byref(nbytes), None) == 0
        assert nbytes.value == 0
    finally:
        adelib.destroy(ctx)
