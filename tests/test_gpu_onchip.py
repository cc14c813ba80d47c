"""The on-chip CG engine (csrc/hh_onchip.cu): lattices whose vectors stay in
shared memory for a whole solve, cut into tiles over (x, tau) for d = 1 and
(z, tau) for d = 3.

Against the oracle's operator (true residual of every solution, 1e-10) and the
grid engine (HH_ENGINE_ONCHIP=0), which runs the same CG: the two take the same
steps, so their counts differ by rounding only and their solutions by the
solver tolerance.  Sizes at the edges of the tiling: tiles of one site or one
plane, N_x = 2 and N_tau = 2, odd extents that leave uneven tiles, several
tiles per SM (3 and 4 right-hand sides), the largest that fit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import workloads  # noqa: E402

H = workloads.T_HOP * workloads.DTAU
A = workloads.A_HS


@pytest.fixture(scope="module")
def hh():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1007_3432_gb300 as pkg
    from paper_1007_3432_gb300 import build
    build.build()
    pkg.load()
    return pkg


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _solve(hh, monkeypatch, onchip, d, nx, ntau, precision, b, sigma, x0=None, **kw):
    monkeypatch.setenv("HH_ENGINE_ONCHIP", str(onchip))
    with hh.Context(d, nx, ntau, precision=precision, **kw) as ctx:
        ctx.set_field(dev(sigma))
        x = torch.full(b.shape, 3.0, dtype=torch.float64, device="cuda") if x0 is None else dev(x0.copy())
        ctx.counters_reset()
        rc, info = ctx.solve(dev(b), x, b.shape[0], guess=x0 is not None, allow=(hh.binding.HH_ENOCONV,))
        cnt = ctx.counters()
        cnt["layout"] = ctx.solver_layout(b.shape[0])
        # which engine ran: no silent fall-back to the other
        assert cnt["layout"]["onchip_launches"] == cnt["layout"]["onchip"] <= (onchip != 0), cnt
        return rc, info, x.cpu().numpy(), cnt


SHAPES = [(1, 2, 2), (1, 2, 7), (1, 3, 2), (1, 17, 5), (1, 33, 40), (1, 300, 11), (1, 731, 24), (3, 2, 2), (3, 2, 9),
          (3, 3, 5), (3, 5, 16), (3, 8, 20), (3, 13, 10), (3, 16, 17)]


# HH_ENGINE_ONCHIP: 1 the form the layout rule takes, 2 the tile form (vectors in
# shared memory), 3 the column form (vectors in registers) where a layout has one.
@pytest.mark.parametrize("form", [1, 2, 3])
@pytest.mark.parametrize("precision,cheb", [("fp64", 0), ("mixed", 0), ("fp64", 4)])
@pytest.mark.parametrize("d,nx,ntau", SHAPES)
@pytest.mark.parametrize("n_rhs", [1, 4])
def test_onchip_solve_matches_oracle_and_grid_engine(hh, monkeypatch, d, nx, ntau, precision, cheb, n_rhs, form):
    n = nx ** d * ntau
    sigma = workloads.sigma_field(n, seed=1500 + nx + ntau)
    b = np.stack([workloads.source(n, seed=1501, rhs=a) for a in range(n_rhs)])
    kw = dict(cheb_degree=cheb, cheb_eps=1e-3)
    rc, info, x, cnt = _solve(hh, monkeypatch, form, d, nx, ntau, precision, b, sigma, **kw)
    rc0, info0, x0, cnt0 = _solve(hh, monkeypatch, 0, d, nx, ntau, precision, b, sigma, **kw)
    lay = cnt["layout"]
    if form == 3 and (d, nx, ntau, n_rhs) == (3, 16, 17, 4):
        assert lay["onchip"] == 0
        pytest.skip("no column layout: 16 planes of 256 sites in 17 slices, four times, need two rows per block")
    assert lay["onchip"] == 1 and (form == 1 or (lay["slices"] > 0) == (form == 3)), lay
    # a mixed on-chip solve is one launch more (the grid engine, for a hand-over)
    assert cnt["kernel_launches"] == cnt0["kernel_launches"] + (1 if precision == "mixed" else 0)
    assert rc == 0 and rc0 == 0 and info["converged"] == 1 and info["true_relres"] <= 1e-10
    lat = oracle.lattice(d, nx, ntau)
    L = oracle.links(lat, A, sigma)
    for a in range(n_rhs):
        for sol in (x, x0):
            res = b[a] - oracle.apply_MTM(lat, H, L, sol[a])
            assert np.linalg.norm(res) <= 1.0001e-10 * np.linalg.norm(b[a])
    assert abs(info["iterations"] - info0["iterations"]) <= 2 + 0.03 * info0["iterations"], (info, info0)
    assert np.linalg.norm(x - x0) <= 1e-4 * np.linalg.norm(x0)
    assert cnt["solves"] == n_rhs and cnt["cg_steps"] > 0


# (lattice, right-hand sides, blocks per SM, x in global memory, column form)
LARGE = [(3, 16, 64, "fp64", 2, 1, 1, False), (1, 1024, 160, "fp64", 2, 1, 0, False),
         (3, 17, 33, "fp64", 1, 2, 0, False), (3, 22, 27, "fp64", 1, 2, 1, False),
         (3, 14, 84, "fp64", 2, 2, 1, False), (1, 136, 151, "fp64", 4, 2, 0, True),
         (3, 20, 96, "mixed", 1, 1, 0, False), (1, 2048, 96, "mixed", 3, 1, 0, False),
         (3, 21, 108, "mixed", 1, 1, 1, False), (3, 22, 39, "mixed", 2, 2, 1, False),
         (1, 557, 103, "mixed", 3, 2, 0, True), (3, 8, 157, "mixed", 2, 2, 0, True)]


@pytest.mark.parametrize("d,nx,ntau,precision,n_rhs,per_sm,x_global,column", LARGE)
def test_onchip_large_lattices(hh, monkeypatch, d, nx, ntau, precision, n_rhs, per_sm, x_global, column):
    """Tiles of hundreds to thousands of sites, one and two blocks per SM, x
    in shared and in global memory, in both forms: capped at 60 steps, where
    both engines hold the same iterate up to rounding (FP64: 1e-10; FP32 steps
    between reliable updates: 1e-4 of the iterate)."""
    n = nx ** d * ntau
    sigma = workloads.sigma_field(n, seed=1600 + nx)
    b = np.stack([workloads.source(n, seed=1601, rhs=a) for a in range(n_rhs)])
    rc, info, x, cnt = _solve(hh, monkeypatch, 1, d, nx, ntau, precision, b, sigma, cg_maxit=60)
    lay = cnt["layout"]
    assert (lay["onchip"], lay["blocks_per_sm"], lay["x_global"], lay["slices"] > 0) == (1, per_sm, x_global, column), lay
    rc0, info0, x0, _ = _solve(hh, monkeypatch, 0, d, nx, ntau, precision, b, sigma, cg_maxit=60)
    assert rc == rc0 == hh.binding.HH_ENOCONV and info["iterations"] == info0["iterations"] == 60
    tol = 1e-10 if precision == "fp64" else 1e-4
    assert np.linalg.norm(x - x0) <= tol * np.linalg.norm(x0)
    assert abs(info["true_relres"] - info0["true_relres"]) <= 1e-3 * info0["true_relres"]


@pytest.mark.parametrize("form", [2, 3])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_onchip_guess_and_zero_source(hh, monkeypatch, precision, form):
    d, nx, ntau = 3, 5, 12
    n = nx ** d * ntau
    sigma = workloads.sigma_field(n, seed=1700)
    b = np.stack([workloads.source(n, seed=1701, rhs=a) for a in range(2)])
    b[1] = 0.0
    rc, info, x, cnt = _solve(hh, monkeypatch, form, d, nx, ntau, precision, b, sigma)
    assert cnt["layout"]["onchip"] == 1
    assert rc == 0 and not np.any(x[1]) and info["true_relres"] <= 1e-10
    x0 = x * (1.0 + 1e-6)
    x0[1] = 5.0                      # dropped: b = 0 has the solution 0
    rc2, info2, x2, _ = _solve(hh, monkeypatch, form, d, nx, ntau, precision, b, sigma, x0=x0)
    assert rc2 == 0 and not np.any(x2[1]) and info2["true_relres"] <= 1e-10
    assert info2["iterations"] < info["iterations"]
    assert np.linalg.norm(x2[0] - x[0]) <= 1e-4 * np.linalg.norm(x[0])


@pytest.mark.parametrize("form,order", [(2, 0), (3, 0), (1, 1)])
@pytest.mark.parametrize("d,nx,ntau", [(1, 48, 64), (3, 6, 16)])
def test_onchip_mixed_hands_over_to_fp64_steps(hh, monkeypatch, d, nx, ntau, form, order):
    """With reliable_delta = 0.9 each reliable update follows a drop of 10%,
    which counts as a stall: after two the systems go on with FP64 steps, in
    the grid engine, from the on-chip state (of both forms, and of the
    exact-block form of M)."""
    n = nx ** d * ntau
    sigma = workloads.sigma_field(n, seed=1800)
    b = np.stack([workloads.source(n, seed=1801, rhs=a) for a in range(2)])
    b[1] = 0.0                       # done on the chip; the other goes on
    rc, info, x, cnt = _solve(hh, monkeypatch, form, d, nx, ntau, "mixed", b, sigma, reliable_delta=0.9,
                               link_order=order)
    rc0, info0, x0, cnt0 = _solve(hh, monkeypatch, 0, d, nx, ntau, "mixed", b, sigma, reliable_delta=0.9,
                               link_order=order)
    assert cnt["layout"]["onchip"] == 1 and cnt0["layout"]["onchip"] == 0
    assert cnt["fp64_steps"] > 0 and cnt0["fp64_steps"] > 0, (cnt, cnt0)
    assert abs(cnt["cg_steps"] - cnt0["cg_steps"]) <= 2 + 0.03 * cnt0["cg_steps"]
    assert rc == 0 and info["converged"] == 1 and info["true_relres"] <= 1e-10 and not np.any(x[1])
    lat = oracle.lattice(d, nx, ntau)
    L = oracle.links(lat, A, sigma)
    q = oracle.apply_MTM_ex(lat, H, L, 1, x[0]) if order else oracle.apply_MTM(lat, H, L, x[0])
    res = b[0] - q
    assert np.linalg.norm(res) <= 1.0001e-10 * np.linalg.norm(b[0])


def test_onchip_layouts_alternate_in_one_context(hh, monkeypatch):
    """Solves with 1, 3 and 2 right-hand sides in turn (other tiles each) and
    a repeat give, bit for bit, what a fresh context gives."""
    monkeypatch.setenv("HH_ENGINE_ONCHIP", "1")
    d, nx, ntau = 1, 61, 40
    n = nx * ntau
    sigma = dev(workloads.sigma_field(n, seed=1900))
    b = dev(np.stack([workloads.source(n, seed=1901, rhs=a) for a in range(3)]))

    def one(ctx, k):
        x = torch.zeros(k, n, dtype=torch.float64, device="cuda")
        ctx.counters_reset()
        ctx.solve(b[:k].clone(), x, k)
        assert ctx.solver_layout(k)["onchip_launches"] == 1
        return x.cpu()

    fresh = {}
    for k in (1, 2, 3):
        with hh.Context(d, nx, ntau) as ctx:
            ctx.set_field(sigma)
            fresh[k] = one(ctx, k)
    with hh.Context(d, nx, ntau) as ctx:
        ctx.set_field(sigma)
        for k in (1, 3, 2, 1, 1, 3):
            assert torch.equal(one(ctx, k), fresh[k])


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("d,nx,ntau", [(1, 2, 2), (1, 2, 5), (1, 33, 9), (1, 500, 7), (3, 2, 3), (3, 3, 5), (3, 5, 16),
                                       (3, 10, 12), (3, 16, 6)])
@pytest.mark.parametrize("n_rhs", [1, 3])
def test_onchip_exact_block_first_order(hh, monkeypatch, d, nx, ntau, precision, n_rhs):
    """The exact-block form to first order: its halos are those of the slice
    before and after (corners of the tiles included)."""
    n = nx ** d * ntau
    sigma = workloads.sigma_field(n, seed=2000 + nx + ntau)
    b = np.stack([workloads.source(n, seed=2001, rhs=a) for a in range(n_rhs)])
    rc, info, x, cnt = _solve(hh, monkeypatch, 1, d, nx, ntau, precision, b, sigma, link_order=1)
    rc0, info0, x0, _ = _solve(hh, monkeypatch, 0, d, nx, ntau, precision, b, sigma, link_order=1)
    assert cnt["layout"]["onchip"] == 1
    assert rc == 0 and rc0 == 0 and info["converged"] == 1 and info["true_relres"] <= 1e-10
    lat = oracle.lattice(d, nx, ntau)
    L = oracle.links(lat, A, sigma)
    for a in range(n_rhs):
        res = b[a] - oracle.apply_MTM_ex(lat, H, L, 1, x[a])
        assert np.linalg.norm(res) <= 1.0001e-10 * np.linalg.norm(b[a])
    assert abs(info["iterations"] - info0["iterations"]) <= 2 + 0.03 * info0["iterations"], (info, info0)
    assert np.linalg.norm(x - x0) <= 1e-4 * np.linalg.norm(x0)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_onchip_solve_replays_from_a_graph(hh, monkeypatch, precision):
    """A captured solve goes on from the phase numbers on the device: replays,
    with a plain solve between them, give the plain solve's bits."""
    monkeypatch.setenv("HH_ENGINE_ONCHIP", "1")
    d, nx, ntau = 1, 48, 24
    n = nx * ntau
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        b = dev(workloads.source(n, seed=2100))
        x = torch.zeros_like(b)
        with hh.Context(d, nx, ntau, precision=precision) as ctx:
            ctx.set_field(dev(workloads.sigma_field(n, seed=2101)))
            ctx.solve(b, x, 1)
            assert ctx.solver_layout(1)["onchip_launches"] == 1
            ref = x.clone()
            stream.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                ctx.solve(b, x, 1, info=False)
            for _ in range(2):
                x.zero_()
                g.replay()
                stream.synchronize()
                assert torch.equal(x, ref)
                x.zero_()
                ctx.solve(b, x, 1)
                assert torch.equal(x, ref)


@pytest.mark.parametrize("onchip", [0, 1])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_captured_solve_replays_after_other_solves(hh, monkeypatch, onchip, precision):
    """A captured solve brings its own system and tile tables and, also as the
    context's first solve, runs in the same engine as others: replays after
    solves of other right-hand sides (more of them, from a guess) give its own
    bits; so do those solves after the replay."""
    monkeypatch.setenv("HH_ENGINE_ONCHIP", str(onchip))
    d, nx, ntau = 1, 48, 24
    n = nx * ntau
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sigma = dev(workloads.sigma_field(n, seed=2201))
        b = dev(np.stack([workloads.source(n, seed=2200, rhs=a) for a in range(6)]))
        two, five = torch.zeros_like(b[:2]), torch.zeros_like(b[1:])
        for ref, rhs in ((two, b[:2]), (five, b[1:])):
            with hh.Context(d, nx, ntau, precision=precision, n_pf=5) as ctx:
                ctx.set_field(sigma)
                ctx.solve(rhs, ref, ref.shape[0])
        with hh.Context(d, nx, ntau, precision=precision, n_pf=5) as ctx:
            ctx.set_field(sigma)
            xa, xb = torch.zeros_like(two), torch.zeros_like(five)
            stream.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                ctx.solve(b[:2], xa, 2, info=False)
            assert ctx.solver_layout(2)["onchip_launches"] == onchip
            for guess in (False, True):
                xa.zero_()
                g.replay()
                stream.synchronize()
                assert torch.equal(xa, two)
                xb.zero_()
                ctx.solve(b[1:], xb, 5)
                assert torch.equal(xb, five)
                xa.zero_()
                g.replay()
                stream.synchronize()
                assert torch.equal(xa, two)
                ctx.solve(b[1:], xb, 5, guess=guess)    # the same plan as before the replay
                assert torch.equal(xb, five)


def test_first_solves_allocate_nothing(hh, monkeypatch):
    """Solves take no device memory, the first one and larger ones included:
    another stream's capture may be going on (an allocation would end it)."""
    monkeypatch.setenv("HH_ENGINE_ONCHIP", "1")
    d, nx, ntau = 1, 64, 16
    n = nx * ntau
    b = dev(np.stack([workloads.source(n, seed=2300, rhs=a) for a in range(4)]))
    x = torch.zeros_like(b)
    y = torch.zeros(8, device="cuda")
    own, side = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with hh.Context(d, nx, ntau, stream=own) as ctx:
        ctx.set_field(dev(workloads.sigma_field(n, seed=2301)))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):        # global capture mode
            y += 1.0
            for k in (1, 3, 4):
                ctx.solve(b, x, k, info=False)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.all(y == 1.0)
        rc, info = ctx.solve(b, x, 4)
        assert rc == 0 and info["converged"] == 1
