"""Edges of the kernels' tiles: path counts around a tile and a warp, step counts that leave
a partial chunk, draw counts around the staging and counter widths, every width of the
normal equations. References are computed here in FP64 or are the same paths of a larger run."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2211_17005_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2211_17005_gb300 import api as A, build
    build.build()
    return A


def _clocks(api, seed, M, N, C):
    """The draws' uniforms [M, N, C] (exact in FP32 and FP64)."""
    out = np.empty((M, N, 4 * ((C + 3) // 4)))
    k, l = np.meshgrid(np.arange(M), np.arange(N), indexing="ij")   # noqa: E741
    for b in range((C + 3) // 4):
        ctr = np.stack([k, l, np.zeros_like(k), np.full_like(k, (2 << 24) | b)], axis=-1).astype(np.uint32)
        x = api.philox4x32_10(torch.from_numpy(ctr.reshape(-1, 4).view(np.int32)).cuda(), seed)
        x = x.cpu().numpy().view(np.uint32).reshape(M, N, 4)
        out[:, :, 4 * b:4 * b + 4] = ((x >> 9) + 0.5) * 2.0 ** -23
    return out[:, :, :C]


@pytest.mark.parametrize("name,M,N,n", [("small", 5, 70000, 50), ("small", 33, 1, 5), ("mixed", 37, 33, 250),
                                        ("paper", 129, 3, 20), ("paper", 70, 2, 100),
                                        ("batched", 40, 65, 30)])
def test_default_steps_and_targets_follow_from_thresholds_and_exposures(api, name, M, N, n):
    wl = W.make(name, M=M, N=N, n_steps=n)
    sim = api.Simulation(wl.model, wl.portfolios, wl.grid, M, N, keep_defaults=True)
    sim.run(wl.seed)
    C = wl.model.C
    w = _clocks(api, wl.seed, M, N, C)
    thr = sim.thresholds().cpu().numpy().astype(np.float64)
    idx = sim.defaults().cpu().numpy()
    expo = sim.exposures().cpu().numpy().astype(np.float64)
    I0 = sim.discount_integral().cpu().numpy().astype(np.float64)
    for k in range(M):
        for c in range(C):
            ref = 1 + np.searchsorted(thr[1:, c, k], w[k, :, c], side="left")
            np.testing.assert_array_equal(idx[k, :, c], ref)
    cnt = np.zeros((n + 2, C, M))
    for c in range(C):
        for k in range(M):
            cnt[:, c, k] = np.bincount(idx[k, :, c], minlength=n + 2)[:n + 2]
    got = sim.targets().cpu().numpy().astype(np.float64)
    # nonnegative FP32 terms: every rounding of the n C additions and products is relative
    rtol = (n * C + 16) * 2.0 ** -24
    for pf in range(sim.n_pf):
        loss = (expo[pf, 1:] * cnt[1:n + 1]).sum(1)
        ref = np.exp(I0[:n]) * np.cumsum(loss[::-1], axis=0)[::-1] / N
        np.testing.assert_allclose(got[pf], ref, rtol=rtol, atol=0)
    bits = sim.targets().clone()
    for inner in (2, 4, 8):   # other tiles, and 128 threads' paths per pricing block
        sim.set_tiles(64, 128, inner, 2432, 1)
        sim.run(wl.seed)
        assert torch.equal(sim.targets(), bits)
    sim.close()


@pytest.mark.parametrize("M", [1, 31, 33, 257])
@pytest.mark.parametrize("name,n,S", [("paper", 10, 3), ("small", 25, 1), ("mixed", 10, 1)])
def test_paths_do_not_depend_on_the_tiles(api, name, n, S, M):
    """A short run's paths equal the same paths of a longer one, with four and eight warps a block."""
    big = W.make(name, M=700, N=2, n_steps=n, substeps=S)
    a = api.Simulation(big.model, big.portfolios, big.grid, 700, 2)
    a.run(big.seed)
    b = api.Simulation(big.model, big.portfolios, big.grid, M, 2)
    for tiles in (None, (64, 128, 0, 2432, 1), (128, 256, 0, 2432, 1)):
        if tiles:
            b.set_tiles(*tiles)
        b.run(big.seed)
        for what in ("features", "discount_integral", "thresholds", "exposures", "targets"):
            assert torch.equal(getattr(b, what)(), getattr(a, what)()[..., :M]), (what, tiles)
    a.close()
    b.close()


def _fit64(cols, y):
    """Fitted values of the targets y [nt, M] on the columns [m, M] and a constant, FP64."""
    A = np.concatenate([np.ones((1, cols.shape[1])), cols]).T
    A = A / np.linalg.norm(A, axis=0)
    return (A @ np.linalg.lstsq(A, y.T, rcond=None)[0]).T


@pytest.mark.parametrize("F,M", [(1, 97), (6, 1024), (7, 1025), (14, 4099), (15, 4100), (22, 513), (23, 20000),
                                 (27, 100003), (30, 2049)])
@pytest.mark.parametrize("basis", ["linear", "poly2"])
def test_fit_at_every_width_of_the_normal_equations(api, F, M, basis):
    rng = np.random.default_rng(100 * F + M)
    Y = (0.02 + 0.01 * rng.normal(size=(F, M))).astype(np.float32)
    xi = (0.01 + (Y - 0.02).sum(0) + 0.005 * rng.normal(size=M)).astype(np.float32)
    pred, coef = api.regress(torch.from_numpy(xi).cuda(), torch.from_numpy(Y).cuda(), basis=basis)
    Y64 = Y.astype(np.float64)
    d = Y64[0] - Y64[0].mean()
    ref = _fit64(np.stack([d, d ** 2]) if basis == "poly2" else Y64, xi.astype(np.float64)[None])[0]
    # FP32 runs of at most 256 products and five more additions: 261 roundings of 2^-24 in the
    # normal equations, whose scaled condition number is below 7 here
    assert np.sqrt(np.mean((pred.cpu().numpy() - ref) ** 2)) <= 261 * 2.0 ** -24 * 7 * np.sqrt(np.mean(xi.astype(np.float64) ** 2))
    assert np.all(np.isfinite(coef))


@pytest.mark.parametrize("basis", ["linear", "poly2"])
def test_six_targets_share_the_normal_equations(api, basis):
    wl = W.make("batched", M=1003, N=16, n_steps=20)
    sim = api.Simulation(wl.model, wl.portfolios, wl.grid, wl.M, wl.N)
    sim.run(wl.seed)
    pred, _ = sim.regress_portfolios(basis)
    j = 7
    Y = sim.features()[j].cpu().numpy().astype(np.float64)
    xi = sim.targets()[:, j].cpu().numpy().astype(np.float64)
    d = Y[0] - Y[0].mean()
    ref = _fit64(np.stack([d, d ** 2]) if basis == "poly2" else Y, xi)
    gap = np.sqrt(np.mean((pred[:, j].cpu().numpy() - ref) ** 2, axis=1))
    assert np.all(gap <= 261 * 2.0 ** -24 * 30 * np.sqrt(np.mean(xi ** 2, axis=1))), gap   # correlated factors
    sim.close()


@pytest.mark.parametrize("name,M,N,n", [("mixed", 203, 70, 20), ("small", 67, 5, 25), ("paper", 150, 64, 10)])
def test_alive_statistics_around_the_staged_draws(api, name, M, N, n):
    """The fit at X = 0 equals the least squares over the written-out M N rows."""
    wl = W.make(name, M=M, N=N, n_steps=n)
    sim = api.Simulation(wl.model, wl.portfolios, wl.grid, M, N, keep_defaults=True)
    sim.run(wl.seed)
    pred, _, dropped = sim.regress_alive(0)
    j, C = n // 2, wl.model.C
    idx = sim.defaults().cpu().numpy().astype(np.int64)
    V = np.concatenate([sim.exposures()[0].cpu().numpy(), np.zeros((1, C, M), np.float32)]).astype(np.float64)
    I0 = sim.discount_integral()[j].cpu().numpy().astype(np.float64)
    loss = sum(np.where(idx[:, :, c] > j, V[idx[:, :, c], c, np.arange(M)[:, None]], 0.0) for c in range(C))
    y = (loss * np.exp(I0)[:, None]).reshape(-1)
    X = (idx <= j).astype(np.float64).reshape(-1, C)
    f = sim.features()[j].cpu().numpy().astype(np.float64)
    Y = np.repeat(((f - f.mean(1, keepdims=True)) / f.std(1, keepdims=True)).T, N, axis=0)
    use = X.any(0)
    assert dropped[j] == C - use.sum()
    A = np.concatenate([np.ones((M * N, 1)), Y, X[:, use]], axis=1)
    w = np.linalg.lstsq(A, y, rcond=None)[0]
    ref = A[::N, :1 + f.shape[0]] @ w[:1 + f.shape[0]]
    # as above; the indicators' columns are near multiples of one another at small samples
    assert np.sqrt(np.mean((pred[j].cpu().numpy() - ref) ** 2)) <= 261 * 2.0 ** -24 * 60 * np.sqrt(np.mean(y ** 2))
    sim.close()


def test_adjoint_of_path_ranges_adds_up(api):
    """Path counts that run in several ranges: the gradient is the mean of its parts'."""
    wl = W.make("adjoint", M=70001, n_steps=100)
    pf = api.frozen(wl.model, wl.portfolios[0])
    c, g = api.grad_cva0(wl.model, pf, wl.grid, 70001, wl.seed)
    parts = [(0, 30000), (30000, 39999), (69999, 2)]
    cs, gs = zip(*(api.grad_cva0(wl.model, pf, wl.grid, m, wl.seed, k0=k) for k, m in parts))
    wgt = np.array([m for _, m in parts]) / 70001
    assert c == pytest.approx(float(np.dot(wgt, cs)), rel=1e-9)
    ref = np.tensordot(wgt, np.stack(gs), axes=1)
    # the parts split a period's dates over other blocks: FP32 sums of up to ten terms each
    np.testing.assert_allclose(g, ref, rtol=1e-5, atol=1e-6 * np.abs(ref).max())


@pytest.mark.parametrize("date", [0, 1, 13, 19])
def test_nested_copies_start_at_the_branch_date(api, date):
    wl = W.make("paper", M=130, N=16, n_steps=20, substeps=2)
    sim = api.Simulation(wl.model, wl.portfolios, wl.grid, wl.M, wl.N)
    got = sim.nested_reference(wl.seed, date, 3)
    left = {w: getattr(sim, w)().clone() for w in ("features", "discount_integral", "thresholds", "exposures", "targets")}
    acc = None
    for b in (1, 2, 3):
        sim.run_twin(wl.seed, date, b)
        t = sim.targets()[0, date].clone()
        acc = t if acc is None else acc + t
    for w, v in left.items():   # the last copy stays, whole
        assert torch.equal(getattr(sim, w)(), v), w
    assert torch.allclose(got, acc / 3, rtol=3 * 2.0 ** -24, atol=0)
    sim.close()


@pytest.mark.parametrize("C,M,N", [(1, 70, 15), (1, 33, 64), (2, 37, 130), (3, 65, 127), (3, 40, 64), (4, 5, 2050),
                                   (8, 33, 257), (8, 1, 1), (16, 19, 67)])
def test_kept_default_steps_at_the_edges_of_the_staged_draws(api, C, M, N):
    """Rows of N C bytes of every alignment, draw counts around the staged ones, every tile."""
    model = W.single_swap_model(tuple(0.02 + 0.05 * c for c in range(C)))
    pf = W._swaps(np.random.default_rng(C), 12, 1, C, 1.0, 5.0)
    sim = api.Simulation(model, [pf], W.Grid(5.0, 20), M, N, keep_defaults=True)
    for inner in (0, 2, 4, 8):
        sim.set_tiles(128, 256, inner, 2432, 1)
        sim.defaults().zero_()
        sim.run(3)
        w = _clocks(api, 3, M, N, C)
        thr = sim.thresholds().cpu().numpy().astype(np.float64)
        idx = sim.defaults().cpu().numpy()
        for c in range(C):
            ref = np.stack([1 + np.searchsorted(thr[1:, c, k], w[k, :, c], side="left") for k in range(M)])
            np.testing.assert_array_equal(idx[:, :, c], ref)
    sim.close()


@pytest.mark.parametrize("E,C,CS,M", [(1, 2, 0, 29184), (1, 2, 0, 29185), (1, 1, 1, 30001), (2, 2, 1, 29217),
                                      (3, 5, 3, 9745), (3, 5, 3, 30001)])
@pytest.mark.parametrize("S", [1, 3])
def test_paths_do_not_depend_on_the_number_of_paths(api, E, C, CS, M, S):
    """The forms taken at large path counts (a thread per path, one and four warps per 32 paths) give
    the paths that 64 paths at a time give, branches and restarts included."""
    model = W.small_model() if (E, C, CS) == (1, 2, 0) else W.paper_model(np.random.default_rng(E), E=E, C=C)
    if CS < C and E > 1:   # the last ones of constant intensity
        nu = np.array(model.cir_nu)
        nu[CS:] = 0.0
        model = dataclasses.replace(model, cir_nu=nu, corr=model.corr[:2 * E - 1 + CS, :2 * E - 1 + CS])
    pf = W._swaps(np.random.default_rng(1), 12, E, C, 1.0, 5.0)
    grid = W.Grid(5.0, 10, S)
    big = api.Simulation(model, [pf], grid, M, 2)
    few = api.Simulation(model, [pf], grid, 64, 2)
    what = ("features", "discount_integral", "thresholds")
    for k0 in (0, M - 64):
        runs = [lambda s, k: s.run(5, k0=k), lambda s, k: s.run_twin(5, 4, 2, k0=k),
                lambda s, k: s.nested_reference(5, 4, 2, k0=k)]
        for run in runs:
            run(big, 0)
            run(few, k0)
            for w in what:
                assert torch.equal(getattr(few, w)(), getattr(big, w)()[..., k0:k0 + 64]), w
    big.close()
    few.close()


def test_the_default_tiles_can_be_set(api):
    """Setting the values a simulation starts with leaves it in the forms it starts in (results never
    change, so by the time of the path simulation, where a wrong form takes over twice as long)."""
    wl = W.make("small", M=1 << 19, N=1)
    sim = api.Simulation(wl.model, wl.portfolios, wl.grid, wl.M, 1, profile=True)

    def ms():
        t = []
        for _ in range(7):
            sim.run(1)
            torch.cuda.synchronize()
            t.append(sim.kernel_ms()[0])
        return float(np.median(t))

    ms()
    fresh = ms()
    sim.set_tiles(128, 256, 0, 2432, 0)
    assert ms() < 1.5 * fresh
    sim.close()


@pytest.mark.parametrize("name,M,n,S", [("adjoint", 1, 10, 1), ("adjoint", 9800, 20, 3), ("small", 33, 25, 1),
                                        ("small", 30001, 25, 4), ("adjoint", 70001, 100, 1)])
def test_forward_alone_gives_the_gradients_value(api, name, M, n, S):
    """The forward keeps fewer arrays than the gradient and may take other path ranges: the same
    FP64 terms in another order."""
    wl = W.make(name, M=M, n_steps=n, substeps=S)
    pf = api.frozen(wl.model, wl.portfolios[0])
    c, g = api.grad_cva0(wl.model, pf, wl.grid, M, wl.seed)
    f, none = api.grad_cva0(wl.model, pf, wl.grid, M, wl.seed, forward_only=True)
    assert none is None and np.all(np.isfinite(g))
    assert f == pytest.approx(c, rel=1e-13)


@pytest.mark.parametrize("name,n", [("adjoint", 10), ("small", 25)])
def test_adjoints_of_paths_are_added_in_fp64(api, name, n):
    """A path's adjoints do not depend on the other paths of its thread and block, so the sums of two
    calls are those of one to FP64 rounding (paths 0 and 128 share a thread)."""
    wl = W.make(name, M=129, n_steps=n)
    pf = api.frozen(wl.model, wl.portfolios[0])
    c, g = api.grad_cva0(wl.model, pf, wl.grid, 129, wl.seed)
    c1, g1 = api.grad_cva0(wl.model, pf, wl.grid, 128, wl.seed)
    c2, g2 = api.grad_cva0(wl.model, pf, wl.grid, 1, wl.seed, k0=128)
    assert c * 129 == pytest.approx(c1 * 128 + c2, rel=1e-12)
    ref = g1 * 128 + g2
    np.testing.assert_allclose(g * 129, ref, rtol=1e-12, atol=1e-12 * np.abs(ref).max())


@pytest.mark.parametrize("C", [2, 8])
def test_alive_losses_are_added_in_fp64_beyond_eight_paths(api, C):
    """Losses whose sums over eight paths are exact in FP32 and whose sum over a tile is not: the
    buffers of a simulation are overwritten with them, one counterparty defaulting at step 1 in
    every other draw and the next one, with the loss, at step 3."""
    M, N, n, j = 32, 2, 5, 2
    model = W.single_swap_model(tuple(0.02 + 0.01 * c for c in range(C)))
    pf = W._swaps(np.random.default_rng(2), 10, 1, C, 1.0, 5.0)
    sim = api.Simulation(model, [pf], W.Grid(5.0, n), M, N, keep_defaults=True)
    sim.run(1)
    loss = np.repeat([2.0 ** 30, 1.0, -2.0 ** 30, 1.0], 8)
    y = np.arange(M) % 4 + np.arange(M) // 16
    sim.defaults().fill_(n + 1)
    sim.defaults()[:, 0, 0] = 1
    sim.defaults()[:, 0, 1] = 3
    sim.exposures().zero_()
    sim.exposures()[0, 3, 1] = torch.from_numpy(loss.astype(np.float32)).cuda()
    sim.discount_integral().zero_()
    sim.targets().zero_()
    sim.features()[:, 0] = torch.from_numpy(y.astype(np.float32)).cuda()
    _, coef, dropped = sim.regress_alive(0)
    # unknowns: constant, state, the first counterparty; M N rows, of which M with its default
    A = np.array([[N * M, N * y.sum(), M], [N * y.sum(), N * (y * y).sum(), y.sum()], [M, y.sum(), M]], dtype=np.float64)
    w = np.linalg.solve(A, [0.0, 0.0, loss.sum()])
    assert dropped[j] == C - 1
    rows = np.stack([np.ones(2 * M), np.tile(y, 2), np.repeat([0.0, 1.0], M)], axis=1)   # no loss before, one after
    np.testing.assert_allclose(rows @ coef[j][:3], rows @ w, rtol=1e-9)
    sim.close()


@pytest.mark.parametrize("name,M,n,S,tiles", [
    ("paper", 130, 20, 2, (64, 256, 0, 2432, 0)), ("paper", 700, 100, 1, (64, 128, 0, 2432, 4)),
    ("batched", 130, 20, 1, (64, 256, 0, 2432, 0)), ("batched", 300, 20, 1, (128, 256, 0, 2432, 1)),
    ("batched", 300, 120, 1, (128, 256, 0, 2432, 4)), ("small", 257, 50, 1, (64, 256, 0, 2432, 4)),
    ("small", 30001, 50, 1, (128, 256, 0, 2432, 0)), ("mixed", 70, 40, 1, (128, 256, 0, 2432, 0))])
def test_nested_restart_in_every_form(api, name, M, n, S, tiles):
    """Copies that start at the branch date leave what whole copies leave: every simulation form,
    pricing form and portfolio count, branches at a reset date and inside a period."""
    wl = W.make(name, M=M, N=4, n_steps=n, substeps=S)
    sim = api.Simulation(wl.model, wl.portfolios, wl.grid, M, 4)
    sim.set_tiles(*tiles)
    what = ("features", "discount_integral", "thresholds", "exposures", "targets")
    for date in (n // 5, n // 2 + 1, n - 1):
        sim.nested_reference(wl.seed, date, 2)
        left = {w: getattr(sim, w)().clone() for w in what}
        for w in what:
            getattr(sim, w)().fill_(float("nan"))
        sim.run_twin(wl.seed, date, 2)
        for w in what:
            assert torch.equal(getattr(sim, w)(), left[w]), (w, date)
    sim.close()


@pytest.mark.parametrize("name,basis,M", [("paper", "linear", 70000), ("paper", "linear", 70001), ("small", "linear", 140003),
                                          ("batched", "poly2", 9001)])
def test_fit_of_long_chunks(api, name, basis, M):
    """Chunks of more rows than a lane's FP32 run (256), and several chunks of six targets."""
    wl = W.make(name, M=M, N=2, n_steps=20)
    sim = api.Simulation(wl.model, wl.portfolios, wl.grid, M, 2)
    sim.set_tiles(128, 256, 0, 152 if basis == "linear" else 2432, 0)
    sim.run(wl.seed)
    pred, _ = sim.regress_portfolios(basis)
    j = 7
    Y = sim.features()[j].cpu().numpy().astype(np.float64)
    xi = sim.targets()[:, j].cpu().numpy().astype(np.float64)
    d = Y[0] - Y[0].mean()
    ref = _fit64(np.stack([d, d ** 2]) if basis == "poly2" else Y, xi)
    gap = np.sqrt(np.mean((pred[:, j].cpu().numpy() - ref) ** 2, axis=1))
    assert np.all(gap <= 261 * 2.0 ** -24 * 30 * np.sqrt(np.mean(xi ** 2, axis=1))), gap   # correlated factors
    sim.close()


@pytest.mark.parametrize("K", [1, 3, 16])
def test_checkpoints_of_the_run_time_shapes(api, K):
    """Only these recompute from checkpoints: the interval changes no operation of a path."""
    wl = W.make("mixed", M=300, n_steps=20)
    pf = api.frozen(wl.model, wl.portfolios[1])
    c, g = api.grad_cva0(wl.model, pf, wl.grid, 300, wl.seed, ckpt_every=10)
    ck, gk = api.grad_cva0(wl.model, pf, wl.grid, 300, wl.seed, ckpt_every=K)
    assert ck == pytest.approx(c, rel=1e-12)
    np.testing.assert_allclose(gk, g, rtol=1e-12, atol=1e-12 * np.abs(g).max())
