"""ade_get_cells after steps: the list of the positions the last step started from, also when the caller's positions
have changed since (the list is the library's, the positions are the caller's)."""
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


@pytest.mark.parametrize("call", ["step", "run"])
@pytest.mark.parametrize("n", [1, 2, 5, 32, 34])
@pytest.mark.parametrize("dim", [2, 3])
def test_cells_are_those_of_the_last_step_whatever_happened_to_the_positions(lib, dim, n, call):
    p = inputs.Plume(2, 61, 1.7, jitter=0.4, seed=1) if dim == 2 else inputs.Plume(3, 17, 1.6, jitter=0.4, seed=1)
    xq, C = p.initial_state()
    sims = [lib.Simulation(lib.params_for(p), xq, C) for _ in range(4)]
    if n > 1:
        sims[0].step(n - 1)
    sims[0].build_cells()                 # the absolute grid's list where the last step starts
    ref = sims[0].cells()
    for s in sims[1:]:
        for _ in range(2 if call == "run" else 1):      # (a graph's replay)
            s.restore(blob) if (blob := getattr(s, "_blob", None)) else setattr(s, "_blob", s.checkpoint())
            getattr(s, call)(n)
    sims[2].xq.zero_()                    # the caller's own write
    sims[3].restore(sims[3]._blob)
    for s in sims[1:]:
        for a, b in zip(s.cells(), ref):
            assert np.array_equal(a, b)
    for a, b in zip(sims[1].cells(), ref):     # asked for again
        assert np.array_equal(a, b)
