"""Sets that fill a small part of the box, or a few long rows of cells: most rows (pencils) of cells are empty
and a few hold nearly all particles.  The kernels that go by chunks of one pencil (kept pair weights,
sweep, adjoint, 3D velocity field) against the direct walk and the oracle."""
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


def _lattice(dims, dx, jitter, seed):
    rng = np.random.default_rng(seed)
    g = np.meshgrid(*[np.arange(k) + 0.5 for k in dims], indexing="ij")
    x = np.stack([a.ravel() for a in g], axis=1)
    return np.mod((x + rng.uniform(-jitter, jitter, x.shape)) * dx, 1.0)


SETS = {   # positions, spacing, h / spacing
    "slab-2d": lambda: (_lattice((97, 7), 1 / 97, 0.3, 1), 1 / 97, 1.6),
    "rows-2d": lambda: (np.concatenate([_lattice((90, 2), 1 / 90, 0.2, 2), _lattice((90, 2), 1 / 90, 0.2, 3) + [0, 0.5]]),
                        1 / 90, 1.4),
    "column-2d": lambda: (_lattice((5, 101), 1 / 101, 0.3, 4), 1 / 101, 1.5),
    "slab-3d": lambda: (_lattice((31, 6, 5), 1 / 31, 0.3, 5), 1 / 31, 1.4),
    "corner-3d": lambda: (_lattice((9, 9, 9), 1 / 40, 0.3, 6), 1 / 40, 1.5),
    "clumps-3d": lambda: (np.concatenate([_lattice((6, 6, 6), 1 / 48, 0.3, 7), _lattice((6, 6, 6), 1 / 96, 0.3, 8) + 0.6]),
                          1 / 48, 1.4),
}


def _problem(name, **over):
    x, dx, hf = SETS[name]()
    n, dim = x.shape
    # (the mass of the particles' own density and a short step: the explicit step is stable on every set)
    order = np.random.default_rng(9).permutation(n)
    xq = inputs.to_fixed(x[order], np.ones(dim))
    C = (0.1 + np.random.default_rng(10).uniform(size=n)).astype(np.float32)
    kw = dict(dim=dim, h=hf * dx, alpha_L=1e-2, alpha_T=1e-3, D_m=1e-6, v=np.full(dim, 0.1 / np.sqrt(dim)),
              mass=dx ** dim, dt=1e-4)
    kw.update(over)
    return xq, C, kw


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("name", sorted(SETS))
def test_kept_weights_give_the_walks_bits(lib, name, k):
    xq, C, kw = _problem(name)
    a = lib.Simulation(lib.params(cell_subdiv=k, **kw), xq, C)
    b = lib.Simulation(lib.params(cell_subdiv=k, flags=lib.FLAG_DIRECT, **kw), xq, C)
    a.run(4)
    b.run(4)
    assert _bits(a.state()[0], b.state()[0]) and _bits(a.state()[1], b.state()[1])


@pytest.mark.parametrize("side,h_dx", [(60, 11.0), (113, 9.0), (40, 6.0)])
def test_long_chunks_on_few_warps(lib, side, h_dx):
    """Sets of a few hundred chunks with hundreds of neighbours."""
    p = inputs.Plume(2, side, h_dx, jitter=0.4, seed=3)
    xq, C = p.initial_state()
    a = lib.Simulation(lib.params_for(p), xq, C)
    b = lib.Simulation(lib.params_for(p, cell_subdiv=a.info.cell_subdiv, flags=lib.FLAG_DIRECT), xq, C)
    for n in (2, 3):
        a.run(n)
        b.run(n)
        assert _bits(a.state()[0], b.state()[0]) and _bits(a.state()[1], b.state()[1])


@pytest.mark.parametrize("name", sorted(SETS))
def test_adjoint_matches_the_oracle(lib, orc, name):
    """J and dJ/d(alpha_L, alpha_T, D_m) at the bars of the adjoint's tests (1e-5, 1e-4)."""
    xq, C, kw = _problem(name)
    sim = lib.Simulation(lib.params(**kw), xq, C)
    theta = np.array([kw["alpha_L"], kw["alpha_T"], kw["D_m"]])
    target = 0.5 * C.astype(np.float64)
    o = dict(m=kw["mass"], rho=1.0, box=np.ones(kw["dim"]), kind=0, H=2.0 * kw["h"], gamma=kw["dim"] + 2.0,
             dt=sim.info.dt, nsteps=6)
    x = inputs.from_fixed(xq, np.ones(kw["dim"]))
    Jo, go = orc.misfit_gradient_tlm(x, np.asarray(kw["v"]), C.astype(np.float64), theta=theta, target=target, **o)
    J, g, _, _ = sim.adjoint(target.astype(np.float32), 6, 4)
    assert J == pytest.approx(Jo, rel=1e-5)
    for k in range(3):
        assert g[k] == pytest.approx(go[k], rel=1e-4)


@pytest.mark.parametrize("name", [n for n in sorted(SETS) if n.endswith("3d")])
def test_velocity_field_rate_matches_the_oracle(lib, orc, name):
    xq, C, kw = _problem(name, vmax=0.2)
    x = inputs.from_fixed(xq, np.ones(3))
    v = inputs.velocity_field(x, np.ones(3), seed=3)
    v = (v * min(1.0, 0.19 / np.sqrt((v.astype(np.float64) ** 2).sum(axis=0)).max())).astype(np.float32)
    sim = lib.Simulation(lib.params(**kw), xq, C)
    sim.set_velocity_field(v)
    got = sim.rate().cpu().numpy().astype(np.float64)
    ref, _ = orc.rate(x, np.ascontiguousarray(v.T, dtype=np.float64), C.astype(np.float64), kw["mass"], 1.0, np.ones(3), 0,
                      sim.info.support, 5.0, kw["alpha_L"], kw["alpha_T"], kw["D_m"])
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()
    st = sim.run(2)       # the statistics' partials of every warp
    _, C2 = sim.state()
    assert st.c_min == C2.min() and st.c_max == C2.max()
    assert st.mass == pytest.approx(C2.astype(np.float64).sum() * kw["mass"], rel=1e-12)


def test_more_particles_than_65535_blocks_of_one_pencil(lib):
    """A channel of three pencils of 8.7 million particles each."""
    n, Lx, Ly = 26_000_000, 65_000.0, 3.0
    rng = np.random.default_rng(12)
    box = np.array([Lx, Ly])
    xq = rng.integers(0, 1 << 32, size=(2, n), dtype=np.uint32)
    C = (0.5 + rng.uniform(size=n)).astype(np.float32)
    kw = dict(dim=2, h=0.5, alpha_L=1e-2, alpha_T=1e-3, D_m=1e-6, v=(0.1, 0.0), mass=Lx * Ly / n, box=box,
              cell_subdiv=1, dt=1e-2)
    b = lib.Simulation(lib.params(flags=lib.FLAG_DIRECT, **kw), xq, C)
    b.step(1)
    C1 = b.state()[1]
    b.step(1)
    C2 = b.state()[1]
    b.close()
    a = lib.Simulation(lib.params(**kw), xq, C)
    J, _, _, fin = a.adjoint(np.zeros(n, np.float32), 1, 1, want_dC0=False, want_final=True)
    assert J == pytest.approx(0.5 * (C1.astype(np.float64) ** 2).sum(), rel=1e-6)
    assert np.abs(fin.cpu().numpy() - C1).max() <= 1e-6 * np.abs(C1).max()
    a.step(2)
    assert _bits(a.state()[1], C2)
