"""The special scheme on a moving mesh: the width reciprocals of a cell's neighbours do not depend on
which blocks of the launch have run already. Launch shapes (one pass, several waves, persistent grids)
and a run whose mesh cache is dropped before every step (swale_save / swale_load) agree bit for bit."""
import numpy as np
import pytest

from paper_2208_06588_gb300 import binding as B

pytestmark = pytest.mark.gpu
KEYS = ("eta", "hu", "b", "x", "t")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_06588_gb300 import build
    build.build()
    B.lib()


def solver(n, mesh, bc):
    x = np.linspace(0.0, 1.0, n + 1)
    xc = 0.5 * (x[1:] + x[:-1])
    b = 0.3 * np.exp(-((xc - 0.6) / 0.15) ** 2)
    h = 1.0 + 0.05 * np.sin(2 * np.pi * xc)
    P = 0.05 * np.sin(2 * np.pi * x)
    P[0] = P[-1] = 0.0
    s = B.Solver(B.make_config(scheme="special", mesh=mesh, bc=bc, mesh_T=0.5))
    s.set_problem(x, h + b, 0.2 * h, b, P, q0_is_eta=True)
    return s


def finish(s):
    out = s.state() | {"status": s.status()}
    s.close()
    assert out["status"][0] == 0
    return out


@pytest.mark.parametrize("n,bc", [(200, "reflective"), (400003, "periodic")])
@pytest.mark.parametrize("mesh", ["profile", "linear", "static"])
def test_launch_shapes_and_a_dropped_cache_agree(n, bc, mesh, tmp_path):
    steps = 5
    s = solver(n, mesh, bc)
    assert s.advance(steps) == steps
    ref = finish(s)
    for tiles in ((64, 64, 0, 0), (256, 256, 0, 0), (128, 64, 152, 152), (64, 128, 3, 7)):
        s = solver(n, mesh, bc)
        B.swale_set_tiles(s.ctx, *tiles)
        assert s.advance(steps) == steps
        got = finish(s)
        assert got["status"] == ref["status"]
        for k in KEYS:
            assert np.array_equal(got[k], ref[k]), (tiles, k)
    s = solver(n, mesh, bc)
    f = str(tmp_path / "state")
    for _ in range(steps):
        B.swale_save(s.ctx, f)
        B.swale_load(s.ctx, f)
        assert s.advance(1) == 1
    got = finish(s)
    for k in KEYS:
        assert np.array_equal(got[k], ref[k]), k
