"""Run calls of ever different lengths: replayed, freshly captured and launched steps give the same bits (a context keeps
three captured graphs at most)."""
import numpy as np
import pytest

from paper_2108_09488_gb300 import inputs

pytestmark = pytest.mark.gpu

CALLS = [5, 7, 7, 7, 5, 2, 2, 1, 1, 33, 33, 40, 64, 8, 31, 31, 3, 1]


@pytest.fixture(scope="module")
def lib(adelib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return adelib


def _bits(a, b):
    return np.array_equal(a.view(np.uint32), b.view(np.uint32))


def test_single_batch_and_sweep_runs_of_varied_length(lib):
    p, q = inputs.Plume(2, 70, 1.5, jitter=0.3, seed=1), inputs.Plume(2, 41, 1.4)
    state = [x.initial_state() for x in (p, q)]
    a, b = (lib.Simulation(lib.params_for(p), *state[0]) for _ in range(2))
    ba, bb = (lib.Batch([lib.params_for(p), lib.params_for(q)], [s[0] for s in state], [s[1] for s in state]) for _ in range(2))
    sa, sb = (lib.Sweep(lib.params_for(p), state[0][0], np.stack([state[0][1]] * 3), [(1e-2, 1e-3, 1e-6)] * 3) for _ in range(2))
    for n in CALLS:
        for x in (a, ba, sa):
            x.run(n)
        for x in (b, bb, sb):
            x.step(n)
        assert _bits(a.state()[1], b.state()[1]), n
        assert all(_bits(ba.state(k)[1], bb.state(k)[1]) for k in (0, 1)), n
        assert _bits(sa.state()[1], sb.state()[1]), n
    assert a.stats().step == sum(CALLS)

