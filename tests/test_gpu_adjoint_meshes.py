"""Gradients on static and linear meshes: with and without the tape, for one-step, ragged and single
segments, on a fresh context and on one that has stepped, all the same and the oracle's tangent along a
direction. Device memory is left full of large values first, so that an array read before it is written
shows."""
import numpy as np
import pytest

import oracle
from paper_2208_06588_gb300 import binding as B
from paper_2208_06588_gb300 import workloads as W

pytestmark = pytest.mark.gpu
N, STEPS = 250, 13
GX = np.array([0.13, 0.41, 0.62, 0.88])


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_06588_gb300 import build
    build.build()
    B.lib()


def litter():
    """Fills and frees 2 GB of device memory."""
    import torch
    t = torch.full((1 << 28,), 3.0e3, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    del t
    torch.cuda.empty_cache()


def problem(mesh):
    pr = W.gaussian_basin(N=N, seed=17)
    pr.mesh = mesh
    pr.hu = 0.3 * pr.h * np.sin(np.pi * 0.5 * (pr.x[1:] + pr.x[:-1]))
    pr.profile = 0.4 * np.sin(2 * np.pi * pr.x)  # node velocities of the linear motion
    pr.profile[0] = pr.profile[-1] = 0.0
    return pr


def gradient(pr, obs, ckpt, tape, before):
    """(J, gradients) of the STEPS steps after `before` steps by the stage kernels (whose mesh cache is then full),
    and the state it leaves."""
    litter()
    s = B.Solver(B.make_config(g=pr.g, cfl=pr.cfl, eps_weno=pr.eps_weno, bc=pr.bc, mesh=pr.mesh, dt_fixed=pr.dt_fixed))
    s.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
    if before:
        B.swale_set_tiles(s.ctx, 128, 64, 0, 0)
        assert s.advance(before) == before
    B.swale_set_adjoint_tape(s.ctx, tape)
    J, g = np.zeros(1), [np.zeros(N) for _ in range(3)]
    B.swale_adjoint(s.ctx, STEPS, ckpt, GX.size, GX, obs, J, *g)
    st = s.state()
    s.close()
    return [J, *g], st


def tangent(pr, obs, before, d):
    """J, dJ along d = (dE, dM, dB) by the oracle's tangent-linear steps."""
    P = oracle.Params(g=pr.g, cfl=pr.cfl, eps_weno=pr.eps_weno, bc=pr.bc, mesh=pr.mesh, dt_fixed=pr.dt_fixed)
    st = oracle.State(pr.E, pr.hu, pr.b, pr.J, pr.x)
    if before:
        oracle.run(P, st, pr.profile, nsteps=before)
    rec = oracle.run(P, st.copy(), pr.profile, nsteps=STEPS, record=True)
    J = dJ = 0.0
    for n in range(STEPS):
        dt = rec["dts"][n]
        *d, _ = oracle.tangent(P, st, pr.profile, rec["dts"][n:n + 1], rec["alphas"][3 * n:3 * n + 3], *d)
        c = np.clip(np.searchsorted(st.x, GX, side="right") - 1, 0, N - 1)
        r = (st.E[c] - st.B[c]) - obs[n]
        J += dt * np.sum(r * r)
        dJ += 2.0 * dt * np.sum(r * (d[0][c] - d[2][c]))
    return J, dJ


@pytest.mark.parametrize("mesh", ["static", "linear"])
@pytest.mark.parametrize("before", [0, 4])
def test_gradient_does_not_depend_on_tape_and_segments(mesh, before):
    pr = problem(mesh)
    rng = np.random.default_rng(3)
    obs = 0.6 + 0.05 * rng.normal(size=(STEPS, GX.size))
    ref, end = gradient(pr, obs, STEPS, 0, before)
    d = [rng.normal(size=N) for _ in range(3)]
    Jo, dJ = tangent(pr, obs, before, [v.copy() for v in d])
    scale = sum(np.abs(g) @ np.abs(v) for g, v in zip(ref[1:], d))
    assert abs(ref[0][0] - Jo) <= 1e-11 * Jo
    assert abs(sum(g @ v for g, v in zip(ref[1:], d)) - dJ) <= 1e-12 * scale
    for tape in (0, 1):
        for ckpt in (1, 5, STEPS):
            got, st = gradient(pr, obs, ckpt, tape, before)
            assert abs(got[0][0] - ref[0][0]) <= 1e-14 * ref[0][0], (tape, ckpt)
            for a, b in zip(got[1:], ref[1:]):
                assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max(), (tape, ckpt)
            for k in ("eta", "hu", "b", "x", "t"):
                assert np.array_equal(st[k], end[k]), (tape, ckpt, k)


def test_static_gradient_after_a_moving_one(monkeypatch):
    """Small enough that the call's memory is that of the call before, where a moving mesh left its node
    velocities; a context held open keeps the allocation in place."""
    import sys
    for name, v in (("N", 40), ("STEPS", 3), ("litter", lambda: None)):
        monkeypatch.setattr(sys.modules[__name__], name, v)
    obs = 0.6 + 0.05 * np.random.default_rng(3).normal(size=(STEPS, GX.size))
    pr = problem("static")
    keep = B.Solver(B.make_config())
    keep.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
    for tape in (0, 1):
        ref, _ = gradient(pr, obs, STEPS, tape, 0)
        gradient(problem("linear"), obs, STEPS, tape, 0)
        got, _ = gradient(pr, obs, STEPS, tape, 0)
        assert abs(got[0][0] - ref[0][0]) <= 1e-14 * ref[0][0]
        for a, b in zip(got[1:], ref[1:]):
            assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
    keep.close()
