"""The grid-wide waits of whole-step launches run out (swale_set_wait_test with a poll limit): the state is that of the
last good step, whichever wait of whichever step it was, and the context goes on. Nothing faults: the kernel returns a
status."""
import numpy as np
import pytest

from paper_2208_06588_gb300 import binding as B

pytestmark = pytest.mark.gpu
KEYS = ("h", "hu", "b", "eta", "x", "t")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_06588_gb300 import build
    build.build()
    B.lib()


def solver(n, mesh):
    x = np.linspace(0.0, 1.0, n + 1)
    xc = 0.5 * (x[1:] + x[:-1])
    b = 0.3 * np.exp(-((xc - 0.6) / 0.15) ** 2)
    P = 0.05 * np.sin(2 * np.pi * x)
    P[0] = P[-1] = 0.0
    s = B.Solver(B.make_config(mesh=mesh, bc="reflective", mesh_T=0.5))
    s.set_problem(x, 1.0 + 0.2 * (xc < 0.4), 0.1 * np.sin(2 * np.pi * xc), b, P, q0_is_eta=True)
    return s


def arrays(path, n):
    """The cell and node arrays of a saved state: before the scalars (whose size is the file's fourth word) and the
    projected bottom's two words."""
    data = open(path, "rb").read()
    end = len(data) - 8 - int.from_bytes(data[12:16], "little")
    return data[end - 8 * (4 * n + 2 * (n + 1)):end]


@pytest.mark.parametrize("n,mesh", [(16300, "profile"), (16300, "static"), (90000, "linear")])
def test_state_is_that_of_the_last_good_step(n, mesh, tmp_path):
    # One poll runs out at once; larger limits may let waits pass and run out later in a step or not at all.
    for tries in (1, 2, 3, 4, 6, 8):
        s = solver(n, mesh)
        assert s.advance(5) == 5
        B.swale_set_wait_test(s.ctx, tries, 0)
        timed_out = False
        try:
            s.advance(40)
        except B.SwaleError as err:
            assert err.code == -7
            timed_out = True
        assert timed_out or tries > 1
        B.swale_set_wait_test(s.ctx, 0, 0)
        bits, steps, _ = s.status()
        got = s.state()
        assert bool(bits & B.BIT_TIMEOUT) == timed_out and (5 <= steps < 45 if timed_out else steps == 45)
        r = solver(n, mesh)
        assert r.advance(steps) == steps
        ref = r.state()
        for k in KEYS:
            assert np.array_equal(got[k], ref[k]), (tries, k)
        # the widths too, as a saved state holds them
        f = str(tmp_path / "state")
        B.swale_save(r.ctx, f)
        good = arrays(f, n)
        B.swale_save(s.ctx, f)
        assert arrays(f, n) == good, tries
        s.close()
        r.close()


def test_context_goes_on_with_a_new_problem():
    s = solver(5000, "profile")
    B.swale_set_wait_test(s.ctx, 1, 0)
    with pytest.raises(B.SwaleError):
        s.advance(3)
    B.swale_set_wait_test(s.ctx, 0, 0)
    x = np.linspace(0.0, 1.0, 5001)
    r = solver(5000, "profile")
    g = r.state()
    s.set_problem(x, g["eta"], g["hu"], g["b"], 0.05 * np.sin(2 * np.pi * x) * (x > 0) * (x < 1), q0_is_eta=True)
    assert s.advance(7) == 7 and r.advance(7) == 7
    a, b = s.state(), r.state()
    s.close()
    r.close()
    for k in KEYS:
        assert np.array_equal(a[k], b[k]), k
