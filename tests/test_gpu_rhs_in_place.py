"""swale_rhs_noalloc with outputs that overlap an input: the results are those of a call with separate
arrays, bit for bit. And a call with separate arrays has the stage kernels' results (swale_rhs): bit for bit,
up to the special scheme's point-wise source (1e-13 of the largest value; its sums may be fused differently)."""
import numpy as np
import pytest

from paper_2208_06588_gb300 import binding as B

pytestmark = pytest.mark.gpu
SIZES = [5, 122, 123, 1000, 8192, 8193, 65536]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_06588_gb300 import build
    build.build()
    B.lib()


def inputs(n):
    rng = np.random.default_rng(n)
    x = np.concatenate([[0.0], np.cumsum(rng.uniform(0.6, 1.4, n))]) / n
    xc = 0.5 * (x[1:] + x[:-1])
    b = 0.5 + 0.3 * np.sin(5 * xc) + 0.2 * (xc > 0.6)
    h = 1.0 + 0.4 * np.cos(3 * xc) + 0.5 * (xc < 0.3)
    h[n // 2:n // 2 + 3] = 0.0
    return dict(E=h + b, M=0.3 * h * np.sin(7 * xc), B=b, J=np.diff(x), w=0.05 * np.sin(9 * x))


def call(cfg, n, d, out, flags, want_A):
    import torch
    return B.swale_rhs_noalloc(cfg, torch.cuda.current_stream().cuda_stream, n, *(d[k] for k in "EMBJw"), 7.5, *out,
                               flags, want_A=want_A)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("scheme", ["hydrostatic", "nonwb", "special"])
def test_in_place(n, scheme):
    import torch
    cfg = B.make_config(bc="reflective", scheme=scheme)
    host = inputs(n)

    def fresh():
        return {k: torch.from_numpy(v.copy()).cuda() for k, v in host.items()}

    def empty():
        return torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")

    fl, fr = (torch.full((n,), 9, dtype=torch.uint8, device="cuda") for _ in range(2))
    ref = [empty() for _ in range(3)]
    A = call(cfg, n, fresh(), ref, fr, True)
    # the stage kernels
    ctx = B.swale_create(cfg)
    st, fs = [np.zeros(n) for _ in range(3)], np.zeros(n, dtype=np.uint8)
    As, _ = B.swale_rhs(ctx, n, *(host[k] for k in "EMBJw"), 7.5, *st, fs)
    B.swale_destroy(ctx)
    assert A == As and np.array_equal(fr.cpu().numpy(), fs)
    for a, r in zip(ref, st):
        tol = 1e-13 * np.abs(r).max() if scheme == "special" else 0.0
        assert np.abs(a.cpu().numpy() - r).max() <= tol
    # every output on every input, alone; all three on three inputs; an output that begins inside an input
    cases = [{o: k} for o in range(3) for k in "EMBJw"] + [dict(zip(range(3), p)) for p in ("EMB", "JwE", "BEM")]
    for places in cases:
        for want_A in (False, True):
            d = fresh()
            out = [d[places[o]][:n] if o in places else empty() for o in range(3)]
            got = call(cfg, n, d, out, fl, want_A)
            assert torch.equal(fl, fr) and (not want_A or got == A)
            for a, r in zip(out, ref):
                assert torch.equal(a, r), places
    for k in "EMBJw":
        for shift in (1, n - 1):
            d = fresh()
            big = torch.cat([d[k], torch.zeros(n, dtype=torch.float64, device="cuda")])
            d[k] = big[:d[k].numel()]
            out = [empty(), big[shift:shift + n], empty()]
            call(cfg, n, d, out, fl, False)
            for a, r in zip(out, ref):
                assert torch.equal(a, r), (k, shift)


@pytest.mark.parametrize("n", [300, 9000])
@pytest.mark.parametrize("bad", [-1.0, -1e-300, float("nan")])
def test_a_bad_width_spoils_its_neighbours_only(n, bad):
    """One width is not positive, as an integrator's mesh may come out: cells away from it have the stage kernels'
    values (the jump's indicators use the largest width)."""
    import torch
    d = inputs(n)
    at = n // 2 + 20
    d["J"][at] = bad if bad != -1.0 else -d["J"][at]
    cfg = B.make_config(bc="reflective")
    out = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3)]
    fl = torch.empty(n, dtype=torch.uint8, device="cuda")
    call(cfg, n, {k: torch.from_numpy(v).cuda() for k, v in d.items()}, out, fl, False)
    ctx = B.swale_create(cfg)
    ref, fr = [np.zeros(n) for _ in range(3)], np.zeros(n, dtype=np.uint8)
    B.swale_rhs(ctx, n, *(d[k] for k in "EMBJw"), 7.5, *ref, fr)
    B.swale_destroy(ctx)
    far = np.abs(np.arange(n) - at) > 8
    assert fr[far].max() > 0 and np.array_equal(fl.cpu().numpy()[far], fr[far])
    for a, r in zip(out, ref):
        assert np.isfinite(r[far]).all() and np.array_equal(a.cpu().numpy()[far], r[far])
