"""The adjoint's workspace (host only): checkpoints and the segment's states take one FP32 value per particle and
state, the working fields and FP64 partials a fixed number of bytes per particle beside them."""
import ctypes

import pytest

from paper_2108_09488_gb300 import inputs

FAKE = 1 << 40          # 256-aligned placeholder device addresses; never dereferenced here


@pytest.mark.parametrize("nsteps,every", [(400, 40), (400, 5), (50, 50), (1, 1)])
def test_one_value_per_particle_and_state(adelib, nsteps, every):
    p = inputs.Plume(2, 512, 1.3)
    prm = adelib.params_for(p)
    ctx = adelib.init_particles(prm, p.n, FAKE, FAKE + (1 << 30), FAKE + (2 << 30), adelib.workspace_bytes(prm, p.n))
    try:
        nbytes = ctypes.c_size_t(0)
        assert adelib.load().ade_adjoint_workspace_bytes(ctx, nsteps, every, ctypes.byref(nbytes)) == 0
        states = -(-nsteps // every) + 1 + min(every, nsteps)
        partials = 48 * (p.n // 128 + 1000) * min(every, nsteps)
        assert nbytes.value <= 4 * p.n * states + partials + 60 * p.n
    finally:
        adelib.destroy(ctx)
