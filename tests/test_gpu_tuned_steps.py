"""Autotuned contexts: the bits of a run do not depend on how its steps are split into calls, whichever walk the
tuner has chosen (a walk whose sums the kept pair weights do not reproduce keeps to itself)."""
import numpy as np
import pytest

from paper_2108_09488_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(adelib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return adelib


PLUMES = {
    "2d-64": lambda: inputs.Plume(2, 64, 1.3),
    "2d-300-jitter": lambda: inputs.Plume(2, 300, 1.9, jitter=0.4, seed=1),
    "2d-160-wide": lambda: inputs.Plume(2, 160, 14.0, jitter=0.4, seed=1),      # 2,700 neighbours: tiles win
    "2d-320-wide": lambda: inputs.Plume(2, 320, 8.0, jitter=0.4, seed=1),       # 800 neighbours, 102,400 particles
    "3d-45-jitter": lambda: inputs.Plume(3, 45, 1.8, jitter=0.3, seed=1),
}


@pytest.mark.parametrize("name", sorted(PLUMES))
def test_split_of_a_tuned_run(lib, name):
    p = PLUMES[name]()
    xq, C = p.initial_state()
    C = C + np.float32(0.05)
    a = lib.Simulation(lib.params_for(p), xq, C)
    a.autotune()
    first = a.checkpoint()
    a.step(4)
    if a.info.variant not in (0, 3, 5, 6):      # tiled or branched: the tuned walk steps, not the table
        assert a._weights is None
    xa, Ca = a.state()
    for split in ((1, 1, 1, 1), (1, 3)):
        a.restore(first)
        for n in split:
            a.run(n)
        xb, Cb = a.state()
        assert np.array_equal(xa, xb) and np.array_equal(Ca.view(np.uint32), Cb.view(np.uint32)), (split, a.info.variant)
