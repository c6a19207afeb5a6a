"""The weights buffer of multi-step calls: its size follows what the set needs, a part of it (or none) gives the
same results, and it is asked for outside of captures only."""
import ctypes

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


def _ask(lib, obj, kind="", counted=1):
    return obj._weights_bytes(kind, counted)


def _give(lib, obj, nbytes, torch):
    """A buffer of nbytes set, and the context's own question marked as answered."""
    obj._weights = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    obj._weights_asked = 2
    obj._set_weights((obj._weights.data_ptr() + 255) // 256 * 256, nbytes)


def _set(dim, side, h_dx, jitter=0.0, kernel=0, blob=0, box=None):
    plume = inputs.Plume(dim=dim, side=side, h_over_dx=h_dx, kernel=kernel, jitter=jitter, seed=1)
    x = plume.positions()
    if blob:
        x = np.concatenate([x, np.mod(np.random.default_rng(1).normal(0.4, 0.01, size=(blob, dim)), 1.0)])
    box = np.ones(dim) if box is None else np.asarray(box)
    xq = inputs.to_fixed(x * box, box)
    C = (0.1 + inputs.gaussian_plume(inputs.from_fixed(xq, box), box, np.full(dim, 0.3) * box, 0.1)).astype(np.float32)
    return xq, C, dict(dim=dim, h=plume.h * box.min(), alpha_L=1e-2, alpha_T=1e-3, D_m=1e-6, v=plume.velocity,
                       mass=box.prod() / xq.shape[1], box=box, kernel=kernel, dt=1e-4)


CASES = {
    "2d-jitter": lambda: _set(2, 127, 1.9, jitter=0.45),
    "2d-blob": lambda: _set(2, 61, 1.6, jitter=0.2, blob=2500),
    "2d-unequal": lambda: _set(2, 80, 2.0, jitter=0.45, box=(1.0, 0.55)),
    "3d-c4": lambda: _set(3, 23, 3.1, jitter=0.4, kernel=1),
}


@pytest.mark.parametrize("part", [0.0, 0.3, 0.9, 1.0])
@pytest.mark.parametrize("name", sorted(CASES))
def test_a_part_of_the_buffer_gives_the_same_bits(lib, name, part):
    import torch
    xq, C, kw = CASES[name]()
    a = lib.Simulation(lib.params(**kw), xq, C)
    b = lib.Simulation(lib.params(flags=lib.FLAG_DIRECT, cell_subdiv=a.info.cell_subdiv, **kw), xq, C)
    full, n = _ask(lib, a), xq.shape[1]
    fixed = 48 * n           # more than the part that is not weights, whatever the grid
    _give(lib, a, max(fixed, int(full * part) // 128 * 128), torch)
    for k in (3, 2):
        a.run(k)
        b.run(k)
        assert _bits(a.state()[0], b.state()[0]) and _bits(a.state()[1], b.state()[1])


def test_a_buffer_below_the_fixed_part_is_refused(lib):
    import torch
    xq, C, kw = CASES["2d-jitter"]()
    a = lib.Simulation(lib.params(**kw), xq, C)
    _ask(lib, a)
    buf = torch.empty(1 << 16, dtype=torch.uint8, device="cuda")
    assert lib.load().ade_set_weights(a.ctx, buf.data_ptr(), 1 << 16) == -5


def test_size_follows_the_pairs(lib):
    """4 bytes per pair and the rows' idle ends: a lattice's chunks need the same, so little is added; an irregular
    set's rows are as long as their longest lane."""
    for p, low, high in ((inputs.Plume(2, 512, 2.1225), 1.0, 2.2), (inputs.Plume(3, 64, 2.0), 1.0, 2.2),
                         (inputs.Plume(3, 64, 1.7, jitter=0.4, seed=1), 1.0, 5.0)):
        xq, C = p.initial_state()
        s = lib.Simulation(lib.params_for(p), xq, C)
        pairs = s.count_pairs()
        weights = _ask(lib, s) - 60 * p.n        # without the slots and the concentrations
        assert low * 4 * pairs < weights < high * 4 * pairs


def test_single_steps_and_rates_take_no_buffer(lib):
    xq, C, kw = CASES["2d-jitter"]()
    a = lib.Simulation(lib.params(**kw), xq, C)
    a.rate()
    a.step(1)
    a.run(1)
    assert a._weights is None
    a.run(2)
    estimate = a._weights.numel()
    a.run(2)                 # from the second call on, the size the set needs
    assert a._weights.numel() < estimate
    counted = a._weights
    a.run(3)
    assert a._weights is counted


@pytest.mark.parametrize("part", [0.0, 0.4, 1.0])
def test_batch_with_a_part_of_the_buffer(lib, part):
    import torch
    parts = [_set(2, 33, 1.3), _set(2, 20, 1.7, jitter=0.4, blob=1500), _set(2, 90, 2.4, jitter=0.3)]
    plist = [lib.params(**kw) for _, _, kw in parts]
    b = lib.Batch(plist, [x for x, _, _ in parts], [c for _, c, _ in parts])
    n = sum(x.shape[1] for x, _, _ in parts)
    _give(lib, b, max(48 * n, int(_ask(lib, b, "batch_") * part) // 128 * 128), torch)
    b.run(3)
    for i, (xq, C, kw) in enumerate(parts):
        s = lib.Simulation(lib.params(cell_subdiv=b.plume_info(i).cell_subdiv, flags=lib.FLAG_DIRECT, **kw), xq, C)
        s.step(3)
        xb, Cb = b.state(i)
        assert _bits(xb, s.state()[0]) and _bits(Cb, s.state()[1]), i


@pytest.mark.parametrize("part", [None, 0.0, 0.4, 1.0])
@pytest.mark.parametrize("name", sorted(CASES))
def test_sweep_with_a_part_of_the_buffer(lib, name, part):
    """Against single plumes, as tests/test_gpu_frozen.py; part None: no buffer, every step on the fly."""
    import torch
    xq, C, kw = CASES[name]()
    theta = [(1e-2, 1e-3, 1e-6), (3e-3, 2e-3, 0.0), (2e-2, 1e-3, 1e-5)]
    sw = lib.Sweep(lib.params(**kw), xq, np.stack([C] * 3), theta)
    if part is None:
        sw._weights_asked = 2
    else:
        _give(lib, sw, max((100 + 16 * 4) * xq.shape[1], int(_ask(lib, sw, "sweep_") * part) // 128 * 128), torch)
    sw.run(4)
    xs, out = sw.state()
    for k, th in enumerate(theta):
        sim = lib.Simulation(lib.params(flags=lib.FLAG_DIRECT, **dict(kw, alpha_L=th[0], alpha_T=th[1], D_m=th[2])), xq, C)
        sim.step(4)
        x1, C1 = sim.state()
        assert _bits(xs, x1)
        inc = np.abs(C1.astype(np.float64) - C).max()
        assert np.abs(out[k].astype(np.float64) - C1).max() <= 4 * 1e-5 * inc + 8 * np.abs(C1).max() * 2.0 ** -24


@pytest.mark.parametrize("part", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("name", sorted(CASES))
def test_adjoint_with_a_part_of_the_weights(lib, orc, name, part):
    """J and dJ/d(alpha_L, alpha_T, D_m) at the bars of the adjoint's tests (1e-5, 1e-4)."""
    xq, C, kw = CASES[name]()
    sim = lib.Simulation(lib.params(**kw), xq, C)
    sim._adjoint_weights, sim._adjoint_asked = int(_ask(lib, sim, "adjoint_") * part) // 128 * 128, 2
    target = 0.5 * C.astype(np.float64)
    o = dict(m=kw["mass"], rho=1.0, box=kw["box"], kind=kw["kernel"], H=sim.info.support, gamma=kw["dim"] + 2.0, dt=kw["dt"], nsteps=5)
    Jo, go = orc.misfit_gradient_tlm(inputs.from_fixed(xq, kw["box"]), np.asarray(kw["v"]), C.astype(np.float64),
                                     theta=np.array([kw["alpha_L"], kw["alpha_T"], kw["D_m"]]), target=target, **o)
    J, g, _, _ = sim.adjoint(target.astype(np.float32), 5, 3)
    assert J == pytest.approx(Jo, rel=1e-5)
    for k in range(3):
        assert g[k] == pytest.approx(go[k], rel=1e-4)


def test_capture_before_the_first_multi_step_call(lib):
    """The size is not asked for inside a capture (it waits); the captured steps run without the buffer."""
    import torch
    xq, C, kw = CASES["2d-jitter"]()
    a, b = (lib.Simulation(lib.params(**kw), xq, C) for _ in range(2))
    a.step(1)
    b.step(1)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        n = ctypes.c_size_t(0)
        assert lib.load().ade_weights_bytes(a.ctx, 1, ctypes.byref(n), a.stream) == -6
        a.step(3)
    g.replay()
    b.step(3)
    assert _bits(a.state()[1], b.state()[1])
    a.step(3)                # and outside it is asked for
    b.step(3)
    assert a._weights is not None and _bits(a.state()[1], b.state()[1])


def test_a_captured_call_keeps_its_buffer(lib):
    """The buffer that a captured call uses stays allocated when later calls get one of another size (or the grid is
    tuned): the caller's graph can be replayed and writes nowhere else."""
    import torch
    xq, C, kw = CASES["2d-jitter"]()
    a, b = (lib.Simulation(lib.params(**kw), xq, C) for _ in range(2))
    a.step(3)                                   # the estimated buffer
    first = a._weights.data_ptr()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        a.step(2)
    a.step(3)                                   # the counted one
    assert a._weights.data_ptr() != first
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    others = [torch.zeros(8 << 20, dtype=torch.uint8, device="cuda") for _ in range(16)]
    g.replay()
    b.step(3)
    b.step(3)
    b.step(2)
    assert _bits(a.state()[1], b.state()[1])
    assert not any(o.any() for o in others)
    assert any(w.data_ptr() == first for w in a._weights_captured)


@pytest.mark.parametrize("dim,side,h_dx", [(3, 20, 1.5), (3, 13, 1.5), (2, 100, 1.2)])
def test_every_slot_is_written(lib, dim, side, h_dx):
    """Numbers that no chunk has (a count leaves them at the end, gaps lie in between) are marked as such in a
    buffer that arrives with anything in it: {first particle, pencil's first, pencil's end, pencil}, all 0."""
    import torch
    xq, C, kw = _set(dim, side, h_dx, jitter=0.3)
    a = lib.Simulation(lib.params(**kw), xq, C)
    b = lib.Simulation(lib.params(cell_subdiv=a.info.cell_subdiv, flags=lib.FLAG_DIRECT, **kw), xq, C)
    nbytes = _ask(lib, a)
    _give(lib, a, nbytes, torch)
    a._weights.fill_(0xff)
    a.step(2)
    b.step(2)
    assert _bits(a.state()[1], b.state()[1])
    nc, n = a.info.nc, len(C)
    numbers = (n >> 5) + nc[1] * nc[2]
    at = -a._weights.data_ptr() % 256 + 256      # the counter's line, then the slots
    slots = a._weights[at:at + 32 * numbers].cpu().numpy().view(np.int32).reshape(numbers, 8)[:, 4:]
    none = slots[slots[:, 0] >= slots[:, 2]]
    assert len(none) > 0 and not none.any()
    first, _, pe, pencil = slots[slots[:, 0] < slots[:, 2]].T
    length = np.minimum(first + 32, pe) - first
    assert np.array_equal(first, np.cumsum(length) - length) and length.sum() == n
    assert (length > 0).all() and (np.diff(pencil) >= 0).all()
