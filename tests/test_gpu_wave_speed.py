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
