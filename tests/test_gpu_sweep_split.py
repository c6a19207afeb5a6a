"""A sweep's bits do not depend on how its steps are split into calls, on launched or replayed steps, or on the
weights buffer: single steps compute the pair weights on the fly, longer calls take them from the table.  Sizes
where the two paths meet: one group (1, 2, 4, 8 sets: one step is too short for the table), several groups,
both kernels, both dimensions, unequal boxes, support edges that fall on lattice sites."""
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


def _bits(a, b):
    return np.array_equal(np.asarray(a).view(np.uint32), np.asarray(b).view(np.uint32))


CASES = {   # dim, side, h / dx, kernel, jitter, box
    "2d-lattice": (2, 64, 2.0, 0, 0.0, None),          # the support is exactly 4 spacings
    "2d-jitter": (2, 97, 1.7, 0, 0.4, None),
    "2d-c4-unequal": (2, 70, 3.3, 1, 0.3, (1.0, 0.6)),
    "3d-c4": (3, 21, 2.9, 1, 0.3, None),
    "3d-lattice": (3, 20, 1.5, 0, 0.0, None),
}


@pytest.mark.parametrize("sets", [1, 2, 4, 8, 11])
@pytest.mark.parametrize("name", sorted(CASES))
def test_bits_do_not_depend_on_the_split(lib, name, sets):
    dim, side, hf, kernel, jitter, box = CASES[name]
    plume = inputs.Plume(dim=dim, side=side, h_over_dx=hf, kernel=kernel, jitter=jitter, seed=2)
    box = np.ones(dim) if box is None else np.asarray(box)
    xq = inputs.to_fixed(plume.positions() * box, box)
    C = (0.05 + inputs.gaussian_plume(inputs.from_fixed(xq, box), box, 0.4 * box, 0.1)).astype(np.float32)
    Cs = np.stack([C * np.float32(1.0 + 0.1 * k) for k in range(sets)])
    theta = [(1e-2 * (k + 1) / sets, 1e-3, 1e-6 * k) for k in range(sets)]
    p = lib.params(dim=dim, h=plume.h * box.min(), alpha_L=1e-2, alpha_T=1e-3, D_m=1e-6, v=plume.velocity,
                   mass=box.prod() / xq.shape[1], box=box, kernel=kernel, dt=1e-4)
    sw = [lib.Sweep(p, xq, Cs, theta) for _ in range(4)]
    sw[0].run(33)                       # graphs of 32 steps and 1
    sw[1].step(33)
    for n in (1, 1, 2, 13, 16):
        sw[2].run(n)
    sw[3]._weights_asked = 2            # no buffer: every step on the fly
    sw[3].run(33)
    x0, C0 = sw[0].state()
    for s in sw[1:]:
        x, c = s.state()
        assert _bits(x, x0) and _bits(c, C0)
