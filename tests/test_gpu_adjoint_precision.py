"""dJ/d(alpha_L, alpha_T, D_m) on lattices, where the same few separations recur in every pair and step, so that a
rounding of a weight or a constant biases the whole gradient: against the FP64 oracle's rates in the adjoint's own
steps, with the states (C, the half step, the adjoint states and L u) rounded to FP32 where the library keeps
them so.  Those roundings alone move the gradient by up to 1.4e-7 (the plain FP64 gradient is no reference for
less); with weights to 32 bits and the constants (time step, prefactor, dispersion coefficients, box ratios) to
FP64 what is left beside them are the roundings inside the rows' FP32 sums, which differ from particle to particle.

Bar: half a unit in FP32's last place, 2^-24."""
import numpy as np
import pytest

from paper_2108_09488_gb300 import inputs

pytestmark = pytest.mark.gpu
BAR = 2.0 ** -24


@pytest.fixture(scope="module")
def lib(adelib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return adelib


def _gradient(R, C, target, theta, dt, nsteps):
    """dJ/dtheta by the adjoint (tests/test_gpu_adjoint.py's formulas) with R(C, theta) in FP64 and FP32 states."""
    f32 = lambda x: x.astype(np.float32).astype(np.float64)
    states = [C.astype(np.float64)]
    for _ in range(nsteps):
        h = f32(states[-1] + 0.5 * dt * R(states[-1], theta))
        states.append(f32(states[-1] + dt * R(h, theta)))
    p = f32(states[-1] - target.astype(np.float64))
    g = np.zeros(3)
    for u in reversed(states[:-1]):
        a, b = f32(R(u, theta)), R(p, theta)
        for k in range(3):
            e = np.eye(3)[k]
            ru = R(u, e)
            g[k] += dt * np.dot(p, ru) + 0.5 * dt * dt * (np.dot(p, R(a, e)) + np.dot(b, ru))
        p = f32(p + dt * R(f32(p + 0.5 * dt * b), theta))
    return g


@pytest.mark.parametrize("dim,side,h_dx,kernel,box", [(2, 491, 1.505, 0, None), (2, 300, 2.9, 1, (1.0, 0.7)), (2, 512, 1.3, 0, None),
                                                       (3, 48, 1.3, 0, None), (3, 45, 2.7, 1, None)])
def test_gradient_on_lattices(lib, orc, dim, side, h_dx, kernel, box):
    p = inputs.Plume(dim, side, h_dx, kernel=kernel)
    box = np.ones(dim) if box is None else np.asarray(box)
    x = p.positions() + 0.3 * p.dx
    xq = inputs.to_fixed(x * box, box)
    xf = inputs.from_fixed(xq, box)
    C = (0.05 + inputs.gaussian_plume(xf, box, 0.4 * box, 0.1)).astype(np.float32)
    target = (0.05 + 0.8 * inputs.gaussian_plume(xf, box, 0.55 * box, 0.2)).astype(np.float32)
    kw = dict(dim=dim, h=p.h * box.min(), alpha_L=1e-2, alpha_T=1e-3, D_m=1e-6, v=p.velocity, mass=box.prod() / p.n, box=box, kernel=kernel)
    sim = lib.Simulation(lib.params(**kw), xq, C)
    n = 10
    R = lambda c, th: orc._R(xf, p.velocity, c, kw["mass"], 1.0, box, kernel, sim.info.support, dim + 2.0, th)
    go = _gradient(R, C, target, np.array([1e-2, 1e-3, 1e-6]), sim.info.dt, n)
    _, g, _, _ = sim.adjoint(target, n, 4)
    rel = [abs(g[k] - go[k]) / abs(go[k]) for k in range(3)]
    print(dim, side, h_dx, kernel, ["%.2e" % r for r in rel])
    assert max(rel) <= BAR
