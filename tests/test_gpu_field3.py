"""Velocity-field evaluations in 3D against the FP64 oracle at the edges of the kernel's layout: sets just
below and above the size where four warps stop sharing a chunk, lists that fill many times over (a
dense blob), ragged and empty pencils, a shuffled order, an unequal box, both kernels and every cell grid.

Tolerance: the pair terms and the partial sums of one list (40 entries) are FP32, a rounding of 2^-24 per
operation and about 30 of them a pair, the rest is compensated: 1e-5 of the largest rate, as in 2D."""
import numpy as np
import pytest

from paper_2108_09488_gb300 import inputs

pytestmark = pytest.mark.gpu
RATE_TOL = 1e-5
VMAX = 0.2


@pytest.fixture(scope="module")
def lib(adelib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return adelib


def _set(side, h_dx, jitter, kernel=0, blob=0, box=(1.0, 1.0, 1.0), shuffle=False, seed=3):
    plume = inputs.Plume(dim=3, side=side, h_over_dx=h_dx, kernel=kernel, jitter=jitter, seed=seed)
    rng = np.random.default_rng(seed)
    x = plume.positions()
    if blob:
        x = np.concatenate([x, np.mod(rng.normal(0.02, 0.02, size=(blob, 3)), 1.0)])
    box = np.asarray(box)
    xq = inputs.to_fixed(x * box, box)
    if shuffle:
        xq = np.ascontiguousarray(xq[:, rng.permutation(xq.shape[1])])
    xf = inputs.from_fixed(xq, box)
    C = inputs.gaussian_plume(xf, box, 0.3 * box, 0.1).astype(np.float32)
    v = inputs.velocity_field(xf, box, speed=0.1, amplitude=0.5, seed=9)
    kw = dict(dim=3, h=plume.h * box.min(), alpha_L=1e-2, alpha_T=1e-3, D_m=1e-6, v=plume.velocity,
              mass=box.prod() / xq.shape[1], box=box, kernel=kernel, vmax=VMAX)
    return xq, xf, C, v, kw


CASES = {
    "61-four-warps": lambda: _set(61, 1.7, 0.3),
    "62-one-warp": lambda: _set(62, 1.7, 0.3),
    "20-c4-shuffled": lambda: _set(20, 3.1, 0.4, kernel=1, shuffle=True),
    "19-blob": lambda: _set(19, 1.6, 0.45, blob=3000),
    "18-unequal-box": lambda: _set(18, 1.7, 0.45, box=(1.0, 0.55, 0.8)),
    "16-sparse": lambda: _set(16, 0.55, 0.45),
}


@pytest.mark.parametrize("k", [0, 1, 3])
@pytest.mark.parametrize("name", sorted(CASES))
def test_rate_and_step_against_the_oracle(lib, orc, name, k):
    if name == "20-c4-shuffled" and k == 1:
        pytest.skip("refused: the box holds fewer than three cells of one support radius and the drift")
    xq, x, C, v, kw = CASES[name]()
    sim = lib.Simulation(lib.params(cell_subdiv=k, **kw), xq, C)
    sim.set_velocity_field(v)
    args = (np.ascontiguousarray(v.T, dtype=np.float64), C.astype(np.float64), kw["mass"], 1.0, kw["box"],
            kw["kernel"], sim.info.support, 5.0, kw["alpha_L"], kw["alpha_T"], kw["D_m"])
    sel = np.random.default_rng(1).choice(x.shape[0], min(x.shape[0], 3000), replace=False).astype(np.int32)
    r_orc, _ = orc.rate_at(sel, x, *args)
    r = sim.rate().cpu().numpy()
    assert np.max(np.abs(r[sel] - r_orc)) <= RATE_TOL * np.max(np.abs(r))
    if k:
        return
    sim.step(1)
    xq1, C1 = sim.state()
    xo, Co, _ = orc.step(x, *args, sim.info.dt)
    dC = Co - C
    tol = RATE_TOL * np.max(np.abs(dC)) + np.max(np.abs(Co)) * 2.0 ** -24
    assert np.max(np.abs(C1.astype(np.float64) - C - dC)) <= tol
    d = np.abs(inputs.from_fixed(xq1, kw["box"]) - xo)
    assert np.minimum(d, kw["box"] - d).max() <= 2.0 ** -32
