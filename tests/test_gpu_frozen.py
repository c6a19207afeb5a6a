"""Steps of one call that keep the pair weights (uniform flow: the separations do not change) against
the walks that evaluate every pair anew: the same bits, over the edges of the weight table's layout
(chunks of 32 particles of one pencil, rows over the periodic seam, empty pencils, a table that runs
out of room), both dimensions and kernels, unequal boxes and Cattaneo's form."""
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


def _set(dim, side, h_dx, jitter=0.0, kernel=0, seed=1, order=False, blob=0, box=None):
    plume = inputs.Plume(dim=dim, side=side, h_over_dx=h_dx, kernel=kernel, jitter=jitter, seed=seed)
    x = plume.positions()
    rng = np.random.default_rng(seed)
    if blob:
        x = np.concatenate([x, np.mod(rng.normal(0.4, 0.01, size=(blob, dim)), 1.0)])
    box = np.ones(dim) if box is None else np.asarray(box)
    xq = inputs.to_fixed(x * box, box)
    if order:
        xq = np.ascontiguousarray(xq[:, rng.permutation(xq.shape[1])])
    C = inputs.gaussian_plume(inputs.from_fixed(xq, box), box, np.full(dim, 0.3) * box, 0.1).astype(np.float32)
    kw = dict(dim=dim, h=plume.h * box.min(), alpha_L=1e-2, alpha_T=1e-3, D_m=1e-6, v=plume.velocity,
              mass=box.prod() / xq.shape[1], box=box, kernel=kernel)
    return xq, C, kw


CASES = {
    "2d-lattice-33": lambda: _set(2, 33, 1.3),
    "2d-lattice-64-c4": lambda: _set(2, 64, 4.2, kernel=1),
    "2d-jitter-127": lambda: _set(2, 127, 1.9, jitter=0.45),
    "2d-jitter-shuffled-97": lambda: _set(2, 97, 2.4, jitter=0.3, order=True),
    "2d-blob-no-room": lambda: _set(2, 61, 1.6, jitter=0.2, blob=2500),
    "2d-unequal-box": lambda: _set(2, 80, 2.0, jitter=0.45, box=(1.0, 0.55)),
    "3d-lattice-20": lambda: _set(3, 20, 1.3),
    "3d-jitter-23-c4": lambda: _set(3, 23, 3.1, jitter=0.4, kernel=1, order=True),
    "2d-sparse": lambda: _set(2, 16, 0.55, jitter=0.45),
}


@pytest.mark.parametrize("tau", [0.0, 2e-3])
@pytest.mark.parametrize("k", [1, 2, 4])
@pytest.mark.parametrize("name", sorted(CASES))
def test_kept_weights_give_the_walks_bits(lib, name, k, tau):
    xq, C, kw = CASES[name]()
    if tau:
        kw["dt"] = 1e-3
    a = lib.Simulation(lib.params(cell_subdiv=k, tau=tau, **kw), xq, C)
    b = lib.Simulation(lib.params(cell_subdiv=k, tau=tau, flags=lib.FLAG_DIRECT, **kw), xq, C)
    if tau:
        a.set_flux()
        b.set_flux()
    for n in (3, 5):        # a second call starts from a moved frame
        st = a.run(n)
        ref = b.run(n)      # one step after another: the same per-warp partials of the statistics
        assert _bits(a.state()[0], b.state()[0]) and _bits(a.state()[1], b.state()[1])
        if tau:
            assert _bits(a.flux().cpu().numpy(), b.flux().cpu().numpy())
        assert (st.mass, st.c_min, st.c_max, st.status) == (ref.mass, ref.c_min, ref.c_max, ref.status)


def test_run_split_into_calls_gives_the_same_bits(lib):
    """37 steps as one call (a graph of 32 and one of 5), as launched steps, and split unevenly."""
    xq, C, kw = CASES["2d-jitter-127"]()
    sims = [lib.Simulation(lib.params(**kw), xq, C) for _ in range(3)]
    sims[0].run(37)
    sims[1].step(37)
    for n in (1, 9, 2, 25):
        sims[2].run(n)
    for s in sims[1:]:
        assert _bits(sims[0].state()[0], s.state()[0]) and _bits(sims[0].state()[1], s.state()[1])


def test_cells_after_steps_are_those_of_the_last_steps_start(lib):
    xq, C, kw = CASES["2d-jitter-127"]()
    a, b = (lib.Simulation(lib.params(**kw), xq, C) for _ in range(2))
    a.run(6)
    b.run(5)
    b.build_cells()
    for x, y in zip(a.cells(), b.cells()):
        assert np.array_equal(x, y)
    a.run(2)                # and the next steps go on from the moved frame
    b.run(3)
    assert _bits(a.state()[1], b.state()[1])


def test_nonfinite_concentration_is_reported(lib):
    xq, C, kw = CASES["2d-lattice-33"]()
    C = C.copy()
    C[7] = np.nan
    sim = lib.Simulation(lib.params(**kw), xq, C)
    sim.step(4)
    assert sim.stats().status == -3


@pytest.mark.parametrize("dim", [2, 3])
def test_batch_kept_weights_give_the_walks_bits(lib, dim):
    """Uneven plumes (one with a blob that leaves the table), several steps per call, against
    single-plume contexts stepped by the direct walk."""
    if dim == 2:
        parts = [_set(2, 33, 1.3), _set(2, 20, 1.7, jitter=0.4, blob=1500), _set(2, 90, 2.4, jitter=0.3, order=True),
                 _set(2, 64, 1.2)]
    else:
        parts = [_set(3, 20, 1.3), _set(3, 12, 1.2, jitter=0.4, order=True)]
    plist = [lib.params(**kw) for _, _, kw in parts]
    b = lib.Batch(plist, [x for x, _, _ in parts], [c for _, c, _ in parts])
    for n in (3, 34):
        b.run(n)
        b.step(2)
    for i, (xq, C, kw) in enumerate(parts):
        s = lib.Simulation(lib.params(cell_subdiv=b.plume_info(i).cell_subdiv, flags=lib.FLAG_DIRECT, **kw), xq, C)
        s.step(41)
        xb, Cb = b.state(i)
        assert _bits(xb, s.state()[0]) and _bits(Cb, s.state()[1]), i


@pytest.mark.parametrize("sets", [1, 3, 11])
@pytest.mark.parametrize("name", ["2d-blob-no-room", "2d-unequal-box", "3d-jitter-23-c4", "2d-lattice-33", "2d-sparse"])
def test_sweep_steps_match_single_plumes(lib, name, sets):
    """Steps of a sweep (stored weights g_L, g_T) against single-plume contexts of every set: the two
    forms of a pair's weight differ by a few FP32 roundings, 1e-5 of the increment per step as for
    every rate, and C is rounded once per half step."""
    xq, C, kw = CASES[name]()
    kw = dict(kw, dt=2e-4)
    theta = [(1e-2 * (k + 1) / sets, 1e-3, 1e-6 * k) for k in range(sets)]
    Cs = np.stack([C * np.float32(1.0 + 0.1 * k) for k in range(sets)])
    sw = lib.Sweep(lib.params(**kw), xq, Cs, theta)
    for n in (1, 2):
        sw.run(n)
    xs, out = sw.state()
    for k, th in enumerate(theta):
        p = dict(kw, alpha_L=th[0], alpha_T=th[1], D_m=th[2])
        sim = lib.Simulation(lib.params(flags=lib.FLAG_DIRECT, **p), xq, Cs[k])
        sim.step(3)
        x1, C1 = sim.state()
        assert _bits(xs, x1)
        inc = np.abs(C1.astype(np.float64) - Cs[k]).max()
        tol = 3 * 1e-5 * inc + 6 * np.abs(C1).max() * 2.0 ** -24
        assert np.abs(out[k].astype(np.float64) - C1).max() <= tol, k
