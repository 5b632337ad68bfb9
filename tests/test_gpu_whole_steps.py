"""Small meshes run whole steps in one launch (k_steps). Its results are those of the stage kernels,
bit for bit: an explicit launch shape (swale_set_tiles) keeps a context on the stage kernels.

The sizes sit at the edges of a block's 122 cells and at the smallest meshes; the largest have as
many blocks as are taken (five per SM). (The error contract on this path: test_gpu_errors.py, whose
meshes are small.)"""
import numpy as np
import pytest

from paper_2208_06588_gb300 import binding as B
from paper_2208_06588_gb300 import workloads as W

pytestmark = pytest.mark.gpu
KEYS = ("eta", "hu", "b", "x", "t")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_06588_gb300 import build
    build.build()
    B.lib()


def problem(n, bc, mesh, seed=0, dry=False):
    rng = np.random.default_rng(100 + n + seed)
    x = np.concatenate([[0.0], np.cumsum(rng.uniform(0.7, 1.3, n))])
    x /= x[-1]
    xc = 0.5 * (x[1:] + x[:-1])
    b = 0.3 * np.exp(-((xc - 0.6) / 0.15) ** 2) + (0.8 * (xc > 0.8) if dry else 0.0)
    h = np.maximum(0.0, 1.0 + 0.2 * np.where(xc < 0.4, 1.0, 0.0) + 0.05 * np.sin(9 * xc) - b) if dry else \
        1.0 + 0.2 * (xc < 0.4) + 0.05 * np.sin(2 * np.pi * xc)
    hu = 0.1 * h * np.sin(2 * np.pi * xc)
    P = 0.02 * np.sin(2 * np.pi * x) * (1.0 if mesh == "profile" else 0.3)
    P[0] = P[-1] = 0.0
    return dict(x=x, E=h + b, hu=hu, b=b, P=P), dict(bc=bc, mesh=mesh, mesh_T=0.7, cfl=0.1 if dry else 0.5)


def run(p, cfg, steps, tiles=None, ones=False):
    s = B.Solver(B.make_config(**cfg))
    s.set_problem(p["x"], p["E"], p["hu"], p["b"], p["P"], q0_is_eta=True)
    if tiles:
        B.swale_set_tiles(s.ctx, *tiles)
    n = sum(s.step() >= 0 for _ in range(steps)) if ones else s.advance(steps)
    out = s.state() | {"flags": s.flags(), "n": n, "dt": s.status()[2]}
    s.close()
    return out


def same(a, b):
    for k in KEYS:
        assert np.array_equal(a[k], b[k]), k
    assert np.array_equal(a["flags"], b["flags"]) and a["n"] == b["n"] and a["dt"] == b["dt"]


@pytest.mark.parametrize("n", [5, 6, 121, 122, 123, 244, 245, 1000])
@pytest.mark.parametrize("bc,mesh,scheme", [("periodic", "profile", "hydrostatic"), ("transmissive", "static", "hydrostatic"),
                                            ("reflective", "linear", "hydrostatic"), ("periodic", "static", "nonwb"),
                                            ("reflective", "profile", "nonwb")])
def test_whole_steps_equal_the_stage_kernels(n, bc, mesh, scheme):
    p, cfg = problem(n, bc, mesh)
    cfg["scheme"] = scheme
    same(run(p, cfg, 13), run(p, cfg, 13, (64, 128, 0, 0)))


@pytest.mark.parametrize("opts", [dict(alpha_bound=1), dict(beta_dx_global=0), dict(dt_fixed=1e-4), dict(limit_hu=1)])
def test_options(opts):
    p, cfg = problem(300, "reflective", "profile", dry=True)
    cfg.update(opts)
    same(run(p, cfg, 10), run(p, cfg, 10, (128, 64, 0, 0)))
    same(run(p, cfg, 10, ones=True) | {"n": 10}, run(p, cfg, 10, (256, 64, 0, 0)))


def test_largest_mesh_and_mixed_paths():
    """As many blocks as are taken; then a few steps on each path in turn."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p, cfg = problem(122 * sms, "transmissive", "profile")
    ref = run(p, cfg, 9, (128, 64, 0, 0))
    same(run(p, cfg, 9), ref)
    s = B.Solver(B.make_config(**cfg))
    s.set_problem(p["x"], p["E"], p["hu"], p["b"], p["P"], q0_is_eta=True)
    s.advance(3)
    B.swale_set_tiles(s.ctx, 256, 64, 0, 0)
    s.advance(2)
    B.swale_set_tiles(s.ctx, 128, 128, 0, 0)
    s.advance(4)
    g = s.state()
    s.close()
    for k in KEYS:
        assert np.array_equal(g[k], ref[k]), k


@pytest.mark.parametrize("per_sm", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("scheme,mesh", [("hydrostatic", "profile"), ("nonwb", "static")])
def test_blocks_per_multiprocessor(per_sm, scheme, mesh):
    """The largest mesh of each number of blocks on an SM, one cell more (the next number, after the last
    the stage kernels)."""
    import torch
    n = 122 * per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    for m in (n, n + 1):
        p, cfg = problem(m, "periodic", mesh)
        cfg["scheme"] = scheme
        same(run(p, cfg, 3), run(p, cfg, 3, (64, 128, 0, 0)))


def test_batch_of_small_instances_and_an_end_time():
    """Instances of uneven size in one launch, each to the end time with its own steps."""
    sizes = [5, 122, 123, 260, 31, 500]
    ps = [problem(n, "reflective", "profile", seed=i, dry=i == 3)[0] for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    cat = lambda k: np.concatenate([p[k] for p in ps])  # noqa: E731
    cfl = np.array([0.1 if i == 3 else 0.5 for i in range(len(sizes))])
    got = []
    for tiles in (None, (64, 64, 0, 0)):
        s = B.Solver(B.make_config(bc="reflective", mesh="profile", mesh_T=0.7, t_end=0.02))
        s.N, s.B = int(off[-1]), len(sizes)
        B.swale_batch_set_problem(s.ctx, len(sizes), off, cat("x"), cat("E"), cat("hu"), cat("b"), cat("P"), cfl, 1)
        if tiles:
            B.swale_set_tiles(s.ctx, *tiles)
        n = s.advance(100000)
        got.append(s.batch_state() | {"n": n})
        s.close()
    for k in ("eta", "hu", "b", "x", "t"):
        assert np.array_equal(got[0][k], got[1][k]), k
    assert got[0]["n"] == got[1]["n"] and np.all(got[0]["t"] == 0.02)


@pytest.mark.parametrize("n", [5, 6, 121, 122, 123, 1000, 4096, 8192, 8193, 20011])
@pytest.mark.parametrize("scheme,bc", [("hydrostatic", "periodic"), ("nonwb", "reflective"), ("special", "transmissive")])
def test_rhs_in_one_launch_equals_the_stage_kernels(n, scheme, bc):
    """swale_rhs_noalloc in one launch against its in-place form, which runs the stage kernels (every
    cell read before the first is written): the same arithmetic, up to the special scheme's point-wise
    source, whose sums the compiler may fuse differently (1e-13 of the largest value)."""
    import torch
    p, cfg = problem(n, bc, "static", dry=n > 200)
    cfg = B.make_config(**dict(cfg, scheme=scheme))
    d = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in p.items()}
    J = d["x"][1:] - d["x"][:-1]
    w = 0.1 * torch.sin(7 * d["x"])
    stream = torch.cuda.current_stream().cuda_stream
    for want_A in (False, True):
        out = [torch.empty_like(d["E"]) for _ in range(3)]
        fl = torch.empty(n, dtype=torch.uint8, device="cuda")
        A = B.swale_rhs_noalloc(cfg, stream, n, d["E"], d["hu"], d["b"], J, w, 6.0, *out, fl, want_A=want_A)
        RM = d["hu"].clone()
        ref = [torch.empty_like(RM), RM, torch.empty_like(RM)]
        fr = torch.empty_like(fl)
        Ar = B.swale_rhs_noalloc(cfg, stream, n, d["E"], RM, d["b"], J, w, 6.0, *ref, fr, want_A=want_A)
        torch.cuda.synchronize()
        assert torch.equal(fl, fr) and A == Ar
        for a, r in zip(out, ref):
            tol = 1e-13 * float(r.abs().max()) if scheme == "special" else 0.0
            assert float((a - r).abs().max()) <= tol
