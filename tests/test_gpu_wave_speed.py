"""The scalars of a step are rounded once per operation: sqrt(g h) of uniform water is the correctly rounded root (the
differences of a constant are exact zeros, so the edge depth is h itself)."""
import numpy as np
import pytest

from paper_2208_06588_gb300 import binding as B

pytestmark = pytest.mark.gpu
G = 9.812


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_06588_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("scheme", ["hydrostatic", "nonwb", "special"])
def test_wave_speed_is_the_correctly_rounded_root(scheme):
    import torch
    n, cfg = 5, B.make_config(g=G, scheme=scheme)
    z = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    out = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3)]
    rng = np.random.default_rng(4)
    for h in np.exp(rng.uniform(np.log(1e-3), np.log(1e4), 300)):
        A = B.swale_rhs_noalloc(cfg, torch.cuda.current_stream().cuda_stream, n, z[:n] + h, z[:n], z[:n], z[:n] + 0.25, z,
                                1.0, *out)
        assert A == np.sqrt(G * h), h


@pytest.mark.parametrize("tiles", [None, (128, 64, 0, 0)])
def test_time_step_is_the_rounded_quotient(tiles):
    """dt = cfl J / alpha of uniform still water on a static mesh, by whole steps and by the stage kernels; J a power of
    two."""
    n, rng = 20, np.random.default_rng(5)
    x, z = np.arange(n + 1) / 32.0, np.zeros(n)
    for h, cfl in zip(np.exp(rng.uniform(np.log(1e-2), np.log(1e3), 100)), rng.uniform(0.05, 0.9, 100)):
        s = B.Solver(B.make_config(g=G, cfl=cfl))
        s.set_problem(x, z + h, z, z, None, q0_is_eta=True)
        if tiles:
            B.swale_set_tiles(s.ctx, *tiles)
        dt = s.step()
        s.close()
        assert dt == cfl * (1.0 / 32.0) / np.sqrt(G * h), (h, cfl)
