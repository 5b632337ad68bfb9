"""The filter of the fluid-driven mesh on the GPU, over the windows that a configuration may ask for.

One step moves a node by dt w, so w is read off the nodes: 400 cells of width 1, dt w up to 0.5, and
the node's rounding (2^-45 at 400) against the oracle's filter. Tolerance: two roundings of a node,
and dt w times the (2 H + 1) 2^-53 that a sum of 2 H + 1 terms may be off."""
import numpy as np
import pytest

import oracle
from paper_2208_06588_gb300 import binding as B

pytestmark = pytest.mark.gpu
N = 400


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_06588_gb300 import build
    build.build()
    B.lib()


def flow(kind, scale, rng):
    """Cell velocities of magnitude up to `scale`."""
    if kind == "uniform":
        return np.full(N, scale)
    if kind == "random":
        return scale * rng.uniform(-1.0, 1.0, N)
    u = scale * np.sin(np.linspace(0.0, 9.0, N))
    u[N // 2:] *= 1e-9  # fast water beside nearly still water
    return u


def solver(u, dt, sigma, half):
    x = np.arange(N + 1.0)
    s = B.Solver(B.make_config(mesh="fluid_gauss", bc="transmissive", gauss_sigma=sigma, gauss_half=half, dt_fixed=dt))
    s.set_problem(x, np.ones(N), u, np.zeros(N), None, q0_is_eta=True)
    return s, x


def reference(u, sigma, half):
    P = oracle.Params(mesh="fluid_gauss", bc="transmissive", gauss_sigma=sigma, gauss_half=half)
    return oracle.fluid_velocity(P, np.ones(N), u, np.zeros(N))


@pytest.mark.parametrize("half", [0, 1, 24, 31, 32, 42, 48, 63, 64])
@pytest.mark.parametrize("sigma", [0.7, 8.0, 64.0, 1e4])
def test_windows(half, sigma):
    rng = np.random.default_rng(half)
    for kind in ("uniform", "random", "mixed"):
        for scale in (0.999, -1.999, rng.uniform(1.0, 2.0) * 2.0 ** -30, -rng.uniform(1.0, 2.0) * 2.0 ** 5):
            u = flow(kind, scale, rng)
            dt = 0.5 / np.abs(u).max()
            s, x = solver(u, dt, sigma, half)
            assert s.advance(1) == 1
            got = s.state()["x"]
            s.close()
            w = reference(u, sigma, half)
            tol = 2.0 * 2.0 ** -44 + 0.5 * (2 * half + 2) * 2.0 ** -53
            assert np.abs(got - (x + dt * w)).max() <= tol, (kind, scale)


def test_two_contexts_keep_their_own_weights():
    """Contexts of different windows stepped in turn move their meshes as each does alone."""
    rng = np.random.default_rng(2)
    u = flow("random", 1.0, rng)
    windows = [(1.5, 4), (40.0, 60)]
    alone = []
    for sigma, half in windows:
        s, _ = solver(u, 0.05, sigma, half)
        s.advance(4)
        alone.append(s.state())
        s.close()
    both = [solver(u, 0.05, *w)[0] for w in windows]
    for _ in range(4):
        for s in both:
            assert s.advance(1) == 1
    for s, ref in zip(both, alone):
        got = s.state()
        s.close()
        for k in ("eta", "hu", "x"):
            assert np.array_equal(got[k], ref[k]), k
