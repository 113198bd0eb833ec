"""The latent state between its forms over sequences of calls: which arithmetic and form a solve runs
after changes of weights, states and data.  References are the same calls with every entry kept
(FUSE_OPT_LATENT_IMPL = 0), bit for bit, and the FP64 oracle."""
import math

import numpy as np
import pytest

from paper_2210_04184_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle import nlpr  # noqa: E402
from paper_2210_04184_gb300 import build as _build  # noqa: E402
from paper_2210_04184_gb300 import fuse  # noqa: E402
from paper_2210_04184_gb300.fuse import (Fusion, FusionBatch, FUSE_OPT_GRAPH, FUSE_OPT_LATENT_FORM,  # noqa: E402
                                         FUSE_OPT_LATENT_IMPL, FUSE_OPT_RESIDUALS)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()


def small(**kw):
    base = dict(H=40, W=40, L_l=6, L_h=2, L_s=3, d=4, blur_size=5, blur_sigma=1.0, K=1, S=2,
                lam1=1.0, lam2=1e-2, rho=5e-2, h=0.3, seed=17)
    base.update(kw)
    return synth.make_problem(**base)


def dev(a, dtype=torch.float32):
    return torch.tensor(a, dtype=dtype, device="cuda")


@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("foreign", ["weights", "state"])
def test_monitored_solve_of_a_foreign_state(K, foreign):
    # entries left by other weights, or set from another run, are not those of a run on the current
    # thresholds: a monitored iteration on them does not make them so
    p, q = small(K=K, seed=5), small(K=K, seed=6)
    runs = []
    for monitor in (1, 0):
        f = Fusion.from_problem(p, dtype="f32", wdtype="f32")
        f.set_option(FUSE_OPT_RESIDUALS, 1) if monitor else f.set_option(FUSE_OPT_LATENT_IMPL, 0)
        yl, yh = dev(p.Yl), dev(p.Yh)
        f.weights(yh)
        f.solve(yl, yh, 6)
        if foreign == "weights":
            f.weights(dev(q.Yh))
        else:
            st = f.get_state()
            f.weights(dev(q.Yh))
            f.solve(yl, yh, 2)
            f.set_state(st)
        xs = [f.solve(yl, yh, 1, warm=True)[0].clone(), f.solve(yl, yh, 8, warm=True)[0].clone()]
        xs.append(f.get_state())
        runs.append(xs)
        f.close()
    for a, b in zip(*runs):
        assert torch.equal(a, b)


@pytest.mark.parametrize("K", [1, 2])
def test_thresholds_are_rounded_to_nearest(K):
    # thresholds far below the moves of X saturate nearly every entry: |s| is the threshold on the
    # grid, half a step at most from lambda2/rho times the weight
    p = small(K=K, lam2=1e-7)
    f = Fusion.from_problem(p, dtype="f32", wdtype="f32")
    yl, yh = dev(p.Yl), dev(p.Yh)
    f.weights(yh)
    f.solve(yl, yh, 6)
    n, nk, nP, Ls = p.H * p.W, f.nW // 2, (2 * K + 1) ** 2, p.L_s
    mu = (torch.tensor(p.lam2 / p.rho, dtype=torch.float32, device="cuda") * f.get_weights().reshape(f.nW, n)).double()
    s = f.get_state().view(torch.float32)[5 * Ls * n:][:nk * nP * Ls * n].reshape(nk, nP, Ls, n)
    # the centre of the patch (k = 0) has the threshold of its own pixel; the kept offsets are the
    # second half of the window
    s, mu = s[:, nP // 2].abs().double(), mu[nk:, None]
    g = 2.0 ** (math.frexp(p.lam2 / p.rho)[1] - 24)
    off = (s - mu).abs()
    at = off <= g
    assert at.double().mean() > 0.9
    assert (off[at] <= g / 2 * (1 + 1e-9)).all()
    f.close()


def oracle_runs(p, steps):
    """X of the FP64 oracle after each (weights, iterations) of `steps`, continued from one to the next."""
    st, out = None, []
    for om, iters in steps:
        X, st, _ = nlpr.admm(nlpr.to_hwl(p.Yl), nlpr.to_hwl(p.Yh), p.blur, p.d, p.R, p.E, p.K, p.S, p.lam1, p.lam2,
                             p.rho, om, iters, state=st, fast=True)
        out.append(nlpr.to_lhw(X))
    return out


def rel(a, b):
    a = a.double().cpu().numpy()
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# FP32 iterates against the FP64 oracle: the bound of the parity tests
FP32_BOUND = 1e-5


@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("scale", [1.0, 1 / 8, 1 / 64, 1 / 4096, 8.0, 64.0])
@pytest.mark.parametrize("impl", [1, 0])
def test_weights_scaled_under_a_state(K, scale, impl):
    # the entering entries reach far beyond the new thresholds, or not near them
    p = small(K=K)
    om = nlpr.weights(nlpr.to_hwl(p.Yh), p.K, p.S, p.h).astype(np.float32).astype(np.float64)
    f = Fusion.from_problem(p, dtype="f32", wdtype="f32")
    f.set_option(FUSE_OPT_LATENT_IMPL, impl)
    yl, yh = dev(p.Yl), dev(p.Yh)
    steps = [(om, 8), (om * scale, 1), (om * scale, 5), (om, 4)]
    ref = oracle_runs(p, steps)
    for i, (w, iters) in enumerate(steps):
        f.set_weights(dev(w))
        X, _ = f.solve(yl, yh, iters, warm=i > 0)
        assert rel(X, ref[i]) <= FP32_BOUND
    f.close()


@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("factor", [1 / 64, 64.0])
def test_state_of_another_lambda2(K, factor):
    # parameter continuation: the state of a run with lambda2 starts one with lambda2 times the factor
    p = small(K=K)
    q = small(K=K, lam2=p.lam2 * factor)
    om = nlpr.weights(nlpr.to_hwl(p.Yh), p.K, p.S, p.h)
    _, st, _ = nlpr.admm(nlpr.to_hwl(p.Yl), nlpr.to_hwl(p.Yh), p.blur, p.d, p.R, p.E, p.K, p.S, p.lam1, p.lam2, p.rho, om,
                         8, fast=True)
    X1, _, _ = nlpr.admm(nlpr.to_hwl(p.Yl), nlpr.to_hwl(p.Yh), p.blur, p.d, p.R, p.E, p.K, p.S, p.lam1, q.lam2, p.rho, om,
                         6, state=st, fast=True)
    a, b = (Fusion.from_problem(x, dtype="f32", wdtype="f32") for x in (p, q))
    yl, yh = dev(p.Yl), dev(p.Yh)
    a.weights(yh)
    b.weights(yh)
    a.solve(yl, yh, 8)
    b.set_state(a.get_state())
    X, _ = b.solve(yl, yh, 6, warm=True)
    assert rel(X, nlpr.to_lhw(X1)) <= FP32_BOUND
    a.close()
    b.close()


@pytest.mark.parametrize("K", [1, 2])
def test_state_set_before_the_weights(K):
    # a saved state continues bit for bit also where the weights are set after it, or set again
    p = small(K=K)
    a, b = (Fusion.from_problem(p, dtype="f32", wdtype="f32") for _ in range(2))
    yl, yh = dev(p.Yl), dev(p.Yh)
    a.weights(yh)
    a.solve(yl, yh, 5)
    st = a.get_state()
    a.weights(yh)
    Xa, _ = a.solve(yl, yh, 7, warm=True)
    b.set_state(st)
    b.weights(yh)
    Xb, _ = b.solve(yl, yh, 7, warm=True)
    X, _ = b.solve(yl, yh, 12)
    assert torch.equal(Xa, X) and torch.equal(Xb, X)
    a.close()
    b.close()


def test_captured_solves():
    # a solve captured by the caller (direct launches) and replayed after other calls: the thresholds, the
    # state and its form are those of the replay's time
    p, q = small(K=2, seed=5), small(K=2, seed=6)
    yl, yh, g2 = dev(p.Yl), dev(p.Yh), dev(q.Yh)

    def context():
        f = Fusion.from_problem(p, dtype="f32", wdtype="f32")
        f.set_option(FUSE_OPT_GRAPH, 0)
        return f

    ref = context()
    f, guide = context(), yh.clone()
    for warm in (False, True):                            # every buffer and loop of the calls to come
        f.weights(guide)
        f.solve(yl, yh, 5, warm=warm)
    f.sync()
    cold, warm, both = (torch.cuda.CUDAGraph() for _ in range(3))
    with torch.cuda.graph(cold):
        Xc, _ = f.solve(yl, yh, 5)
    with torch.cuda.graph(warm):
        Xw, _ = f.solve(yl, yh, 5, warm=True)
    with torch.cuda.graph(both):
        f.weights(guide)
        Xb, _ = f.solve(yl, yh, 5)
    torch.cuda.synchronize()

    def equal(x, y):
        torch.cuda.synchronize()
        assert torch.equal(x, y)

    for g in (yh, g2):
        f.weights(g)                                      # direct, then replays of solves captured before it
        ref.weights(g)
        cold.replay()
        equal(Xc, ref.solve(yl, yh, 5)[0])
        warm.replay()
        warm.replay()
        equal(Xw, ref.solve(yl, yh, 10, warm=True)[0])
        assert torch.equal(f.get_state(), ref.get_state())  # direct, after the replays
        warm.replay()
        equal(Xw, ref.solve(yl, yh, 5, warm=True)[0])
        equal(f.solve(yl, yh, 3, warm=True)[0], ref.solve(yl, yh, 3, warm=True)[0])
        guide.copy_(g2 if g is yh else yh)                # weights within the replay
        both.replay()
        ref.weights(guide)
        equal(Xb, ref.solve(yl, yh, 5)[0])
        equal(f.solve(yl, yh, 4, warm=True)[0], ref.solve(yl, yh, 4, warm=True)[0])
    f.close()
    ref.close()


def _given(nW, H, W, value):
    """Symmetric weights in (0, 1], one pair of them `value`."""
    g = torch.Generator().manual_seed(3)
    w = torch.rand(nW, H, W, generator=g) * 0.9 + 0.1
    S = (math.isqrt(nW + 1) - 1) // 2
    offs = [(a, b) for a in range(-S, S + 1) for b in range(-S, S + 1) if (a, b) != (0, 0)]
    for i, t in enumerate(offs[:nW // 2]):                # omega_{i,-tau} = omega_{i+tau,tau}
        w[i] = torch.roll(w[nW - 1 - i], (t[0], t[1]), (0, 1))
    w[nW - 1, 7, 9] = value
    a, b = offs[0]
    w[0, (7 + a) % H, (9 + b) % W] = value
    return w


# (problem, scale of the data, one weight, whether the grid carries them): FP32_BOUND is what the former
# arithmetic is held to at every one of them
RANGES = [
    (dict(), 1.0, 0.5, True),
    (dict(lam2=1.0, rho=5e-2), 1.0, 0.5, False),          # lambda2/rho = 20
    (dict(lam2=2.0, rho=5e-2), 1.0, 0.5, False),          # 40
    (dict(lam2=2.0, rho=5e-2), 1e3, 0.5, True),
    (dict(), 1e-2, 0.5, False),
    (dict(), 1e-4, 0.5, False),
    (dict(), 1e4, 0.5, True),
    (dict(), 1.0, 1e2, False),
    (dict(), 1.0, 1e4, False),
    (dict(), 1.0, 1e8, False),
    (dict(lam2=0.0), 1e-4, 0.5, True),                    # thresholds of zero
]


@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("dtype,bound", [("f32", FP32_BOUND), ("f64", 1e-11)])
@pytest.mark.parametrize("kw,scale,weight,grid", RANGES)
def test_grid_only_where_it_carries_the_inputs(K, dtype, bound, kw, scale, weight, grid):
    p = small(K=K, **kw)
    p.Yl, p.Yh = p.Yl * scale, p.Yh * scale
    td = torch.float64 if dtype == "f64" else torch.float32
    w = _given((2 * p.S + 1) ** 2 - 1, p.H, p.W, weight).to(td)
    Xo = oracle_runs(p, [(w.double().numpy(), 30)])[0]
    got = {}
    for impl in (1, 0, 2):
        f = Fusion.from_problem(p, dtype=dtype, wdtype=dtype)
        f.set_option(FUSE_OPT_LATENT_IMPL, impl)
        f.set_weights(w.cuda())
        X, _ = f.solve(dev(p.Yl, td), dev(p.Yh, td), 30)
        assert f.get_option(FUSE_OPT_LATENT_FORM) == ({1: 2, 0: 1, 2: 0}[impl] if grid else 0)
        assert rel(X, Xo) <= bound
        got[impl] = (X.clone(), f.get_state())
        f.close()
    assert torch.equal(got[1][0], got[0][0]) and torch.equal(got[1][1], got[0][1])
    if not grid:                                          # the former arithmetic, bit for bit
        assert torch.equal(got[1][0], got[2][0]) and torch.equal(got[1][1], got[2][1])


@pytest.mark.parametrize("bad", ["inf", "nan", "negative", "guide"])
def test_weights_that_are_no_thresholds(bad):
    # infinite or not a number: no threshold, as entries have it; FP32 and FP64 alike
    p = small(K=2)
    for dtype in ("f32", "f64"):
        td = torch.float64 if dtype == "f64" else torch.float32
        out = []
        for impl in (1, 2):
            f = Fusion.from_problem(p, dtype=dtype, wdtype=dtype)
            f.set_option(FUSE_OPT_LATENT_IMPL, impl)
            if bad == "guide":
                g = dev(p.Yh, td)
                g[0, 3, 4] = float("nan")
                f.weights(g)
            else:
                v = {"inf": float("inf"), "nan": float("nan"), "negative": -0.5}[bad]
                f.set_weights(_given(f.nW, p.H, p.W, v).to(td).cuda())
            out.append(f.solve(dev(p.Yl, td), dev(p.Yh, td), 12)[0].clone())
            assert f.get_option(FUSE_OPT_LATENT_FORM) == 0 and torch.isfinite(out[-1]).all()
            f.weights(dev(p.Yh, td))                      # ordinary ones again
            f.solve(dev(p.Yl, td), dev(p.Yh, td), 2)
            assert f.get_option(FUSE_OPT_LATENT_FORM) == (2 if impl == 1 else 0)
            f.close()
        assert torch.equal(*out)


def test_size_of_the_data():
    # X is what counts: E scaled up makes it smaller than Y_l; samples off a mask do not count
    p = small(K=2)
    for kw, s, form in ((dict(), 1e3, 0), (dict(lam2=2.0), 1e-3, 2), (dict(lam2=2.0), 1.0, 0)):
        q = small(K=2, **kw)
        q.E = q.E * s
        f = Fusion.from_problem(q, dtype="f32", wdtype="f32")
        f.weights(dev(q.Yh))
        f.solve(dev(q.Yl), dev(q.Yh), 3)
        assert f.get_option(FUSE_OPT_LATENT_FORM) == form
        f.close()
    q = small(K=2, d=1, blur_size=1)
    mask = torch.zeros(q.H, q.W, dtype=torch.bool, device="cuda")
    mask[::2, ::3] = True
    xs = []
    for fill in (0.0, float("nan"), 1e9):
        f = Fusion.from_problem(q, dtype="f32", wdtype="f32")
        f.set_mask(mask)
        yl = torch.where(mask, dev(q.Yl), fill)
        f.weights(dev(q.Yh))
        xs.append(f.solve(yl, dev(q.Yh), 5)[0].clone())
        assert f.get_option(FUSE_OPT_LATENT_FORM) == 2
        f.close()
    assert torch.equal(xs[0], xs[1]) and torch.equal(xs[0], xs[2])


def test_continued_with_other_data():
    # frames of a scene that goes dark: the state leaves the grid, and stays off it until a new start
    p = small(K=2)
    om = nlpr.weights(nlpr.to_hwl(p.Yh), p.K, p.S, p.h).astype(np.float32)
    f = Fusion.from_problem(p, dtype="f32", wdtype="f32")
    f.set_weights(dev(om))
    st = None
    for i, (scale, form) in enumerate([(1.0, 2), (0.8, 2), (1e-3, 0), (1.0, 0)]):
        Yl, Yh = p.Yl * scale, p.Yh * scale
        X, _ = f.solve(dev(Yl), dev(Yh), 5, warm=i > 0)
        assert f.get_option(FUSE_OPT_LATENT_FORM) == form
        Xo, st, _ = nlpr.admm(nlpr.to_hwl(Yl), nlpr.to_hwl(Yh), p.blur, p.d, p.R, p.E, p.K, p.S, p.lam1, p.lam2, p.rho,
                              om.astype(np.float64), 5, state=st, fast=True)
        assert rel(X, nlpr.to_lhw(Xo)) <= FP32_BOUND
    f.solve(dev(p.Yl), dev(p.Yh), 5)
    assert f.get_option(FUSE_OPT_LATENT_FORM) == 2
    f.close()


def test_batch_of_both_kinds():
    # problems on the grid and off it in one batch: each as alone
    ps = [small(K=1, S=3, H=h, W=w, L_s=5, seed=30 + i) for i, (h, w) in enumerate([(24, 40), (40, 160), (64, 24)])]
    ps[1].Yl, ps[1].Yh = ps[1].Yl * 1e-3, ps[1].Yh * 1e-3
    ctx = [Fusion.from_problem(p, dtype="f32", wdtype="bf16") for p in ps]
    yl, yh = [dev(p.Yl) for p in ps], [dev(p.Yh) for p in ps]
    ref = []
    for f, a, b in zip(ctx, yl, yh):
        f.weights(b)
        ref.append(f.solve(a, b, 9)[0].clone())
    forms = [f.get_option(FUSE_OPT_LATENT_FORM) for f in ctx]
    assert forms == [2, 0, 2]
    batch = FusionBatch(ctx)
    for _ in range(2):
        Xs, _ = batch.solve(yl, yh, 9)
        batch.sync()
        assert [f.get_option(FUSE_OPT_LATENT_FORM) for f in ctx] == forms
        for x, y in zip(Xs, ref):
            assert torch.equal(x, y)
    batch.close()
    for f, a, b, r in zip(ctx, yl, yh, ref):              # and continue alone
        x = f.solve(a, b, 3, warm=True)[0].clone()
        assert torch.equal(x, f.solve(a, b, 12)[0])
        f.close()


@pytest.mark.parametrize("entries", [(0,), (1, 2), (0, 1, 2, 3)])
def test_batch_of_levels_and_entries(entries):
    # problems that are not on levels (by choice here, or for want of memory) beside others that are: the
    # bits of each are those it has alone
    ps = [small(K=2, S=2, L_s=5, H=h, W=w, seed=40 + h) for h, w in ((32, 64), (40, 40), (48, 160), (24, 24))]
    ctx = [Fusion.from_problem(p, dtype="f32", wdtype="bf16") for p in ps]
    yl, yh = [dev(p.Yl) for p in ps], [dev(p.Yh) for p in ps]
    ref = []
    for i, (f, a, b) in enumerate(zip(ctx, yl, yh)):
        if i in entries:
            f.set_option(FUSE_OPT_LATENT_IMPL, 2)
        f.weights(b)
        ref.append(f.solve(a, b, 6)[0].clone())
    forms = [f.get_option(FUSE_OPT_LATENT_FORM) for f in ctx]
    assert forms == [0 if i in entries else 2 for i in range(4)]
    batch = FusionBatch(ctx)
    for step in range(3):
        if step == 2:
            batch.autotune(yl, yh, 1)
        batch.set_option(FUSE_OPT_GRAPH, int(step != 1))
        Xs, _ = batch.solve(yl, yh, 6)
        batch.sync()
        assert [f.get_option(FUSE_OPT_LATENT_FORM) for f in ctx] == forms
        for x, y in zip(Xs, ref):
            assert torch.equal(x, y)
    batch.close()


@pytest.mark.parametrize("K,dtype", [(1, "f32"), (2, "f32"), (2, "f64")])
def test_saved_states(K, dtype):
    # a state saved to device memory, or through host memory, or at an odd offset, is the same, and what
    # it was saved from goes on as if it had not been
    p = small(K=K)
    td = torch.float64 if dtype == "f64" else torch.float32
    f = Fusion.from_problem(p, dtype=dtype, wdtype=dtype)
    yl, yh = dev(p.Yl, td), dev(p.Yh, td)
    f.weights(yh)
    whole = f.solve(yl, yh, 13)[0].clone()
    f.solve(yl, yh, 6)
    a = f.get_state()
    assert f.get_option(FUSE_OPT_LATENT_FORM) == 2        # still levels
    f.solve(yl, yh, 3, warm=True)
    odd = torch.empty(a.numel() + 1, dtype=torch.uint8, device="cuda")[1:]
    host = torch.empty(a.numel(), dtype=torch.uint8)
    b = f.get_state()
    f.weights(dev(small(K=K, seed=3).Yh, td))             # saved under other weights: the entries of the run
    assert torch.equal(f.get_state(), b)
    f.weights(yh)
    fuse.fuse_get_state(f.ctx, odd.data_ptr())
    fuse.fuse_get_state(f.ctx, host.data_ptr())
    assert torch.equal(odd, b) and torch.equal(host.cuda(), b)
    assert torch.equal(f.solve(yl, yh, 4, warm=True)[0], whole)
    f.set_state(a)
    assert torch.equal(f.get_state(), a)                  # of a state not looked at yet
    assert torch.equal(f.solve(yl, yh, 7, warm=True)[0], whole)
    f.close()


@pytest.mark.parametrize("K", [1, 2])
def test_monitored_calls_of_every_length(K):
    # calls of few iterations stay entries between their monitored ones, long ones form levels: the
    # same bits as without the monitor, and the monitor's own results
    p = small(K=K)
    f, g = (Fusion.from_problem(p, dtype="f32", wdtype="f32") for _ in range(2))
    e = Fusion.from_problem(p, dtype="f32", wdtype="f32")
    f.set_option(FUSE_OPT_RESIDUALS, 1)
    e.set_option(FUSE_OPT_RESIDUALS, 1)
    yl, yh = dev(p.Yl), dev(p.Yh)
    for c in (f, g, e):
        c.weights(yh)
    done = 0
    for i, it in enumerate((1, 1, 2, 3, 20, 1, 9, 25, 4)):
        X = f.solve(yl, yh, it, warm=i > 0)[0].clone()
        assert torch.equal(X, g.solve(yl, yh, it, warm=i > 0)[0])
        done += it
        e.solve(yl, yh, done)
        assert f.residuals() == e.residuals()
    assert torch.equal(f.get_state(), g.get_state())
    for c in (f, g, e):
        c.close()


def test_first_solve_while_another_thread_captures():
    # the first solve of a context allocates the levels' buffers: a capture that another thread has under
    # way, in the mode that forbids allocations everywhere, goes on, and the solve is on levels
    import threading
    p = small(K=2)
    yl, yh = dev(p.Yl), dev(p.Yh)
    ref, f = (Fusion.from_problem(p, dtype="f32", wdtype="f32") for _ in range(2))
    ref.weights(yh)
    want = ref.solve(yl, yh, 5)[0].clone()
    X, mine, a, errors = torch.empty_like(want), torch.cuda.Stream(), torch.ones(64, device="cuda"), []
    f.weights(yh)
    fuse.fuse_set_option(f.ctx, FUSE_OPT_GRAPH, 0)
    torch.cuda.synchronize()

    def run():
        try:
            fuse.fuse_set_stream(f.ctx, mine.cuda_stream)
            fuse.fuse_solve(f.ctx, yl.data_ptr(), yh.data_ptr(), 5, 0, X.data_ptr(), None)
        except Exception as e:                            # noqa: BLE001
            errors.append(e)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="global"):
        b = a * 2.0
        t = threading.Thread(target=run)
        t.start()
        t.join()
        b = b + 1.0
    g.replay()
    torch.cuda.synchronize()
    assert not errors and torch.equal(X, want) and (b == 3.0).all()
    assert f.get_option(FUSE_OPT_LATENT_FORM) == 2
    f.close()
    ref.close()


def test_captured_batch():
    # a batch solve captured by the caller: thresholds and forms are those of the replay's time
    ps = [small(K=2, H=32, W=64, seed=5), small(K=2, H=40, W=40, seed=6)]
    ctx = [Fusion.from_problem(p, dtype="f32", wdtype="bf16") for p in ps]
    yl, yh = [dev(p.Yl) for p in ps], [dev(p.Yh) for p in ps]
    guides = [[dev(small(H=p.H, W=p.W, seed=s).Yh) for p in ps] for s in (7, 8)]
    stream = torch.cuda.Stream()                          # a batch keeps the stream it is created with
    for f, b in zip(ctx, yh):
        f.weights(b)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        batch = FusionBatch(ctx)
        batch.set_option(FUSE_OPT_GRAPH, 0)
        batch.solve(yl, yh, 5)
        batch.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        Xs, _ = batch.solve(yl, yh, 5)
    for scale, form in ((1.0, 2), (1e-3, 0), (1.0, 2)):   # the data too
        for gs in guides:
            for f, w in zip(ctx, gs):
                f.weights(w)
            for a, p in zip(yl, ps):
                a.copy_(dev(p.Yl) * scale)
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            got = [x.clone() for x in Xs]
            for f, a, b, x in zip(ctx, yl, yh, got):
                assert f.get_option(FUSE_OPT_LATENT_FORM) == form
                assert torch.equal(x, f.solve(a, b, 5)[0])
    batch.close()


@pytest.mark.parametrize("K,dtype", [(1, "f32"), (2, "f32"), (1, "f64"), (2, "f64")])
@pytest.mark.parametrize("how", ["levels", "entries", "monitored", "host"])
def test_stored_entries_stay_within_their_thresholds(K, dtype, how):
    # a threshold that the grid rounds up: an entry at it is stored as the threshold itself
    p = small(K=K, lam2=1e-3)
    td = torch.float64 if dtype == "f64" else torch.float32
    f = Fusion.from_problem(p, dtype=dtype, wdtype=dtype)
    if how == "entries":
        f.set_option(FUSE_OPT_LATENT_IMPL, 0)
    if how == "monitored":
        f.set_option(FUSE_OPT_RESIDUALS, 1)
    yl, yh = dev(p.Yl, td), dev(p.Yh, td)
    f.weights(yh)
    f.solve(yl, yh, 6)
    n, nk, nP, Ls = p.H * p.W, f.nW // 2, (2 * K + 1) ** 2, p.L_s
    om = torch.tensor(p.lam2 / p.rho, dtype=td, device="cuda") * f.get_weights()
    if how == "host":                                     # in place, and then to host memory
        buf = torch.empty(fuse.fuse_state_bytes(f.ctx), dtype=torch.uint8)
        fuse.fuse_get_state(f.ctx, buf.data_ptr())
        st = buf.cuda()
    else:
        st = f.get_state()
    s = st.view(td)[5 * Ls * n:][:nk * nP * Ls * n].reshape(nk, nP, Ls, p.H, p.W).abs()
    hit = 0.0
    for k, (a, b) in enumerate((a, b) for a in range(-K, K + 1) for b in range(-K, K + 1)):
        mu = torch.roll(om[nk:], (-a, -b), (1, 2))[:, None]          # omega_tau(m + k)
        assert (s[:, k] <= mu).all()
        hit += (s[:, k] == mu).double().mean().item() / nP
    assert hit > 0.1                                      # the test's point: some are at theirs
    X = f.solve(yl, yh, 5, warm=True)[0].clone()
    assert torch.equal(X, f.solve(yl, yh, 11)[0])
    f.close()


def test_without_memory_for_the_levels(monkeypatch):
    # a context that gets no buffers for levels (an allocation failure armed and never reached has that
    # effect) runs entries, alone and beside others in a batch, and takes up a state that was levels
    p = small(K=2)
    yl, yh = dev(p.Yl), dev(p.Yh)
    a = Fusion.from_problem(p, dtype="f32", wdtype="bf16")
    monkeypatch.setenv("FUSE_FAULT_ALLOC", "1000000")
    f, g = (Fusion.from_problem(p, dtype="f32", wdtype="bf16") for _ in range(2))
    monkeypatch.delenv("FUSE_FAULT_ALLOC")
    g.set_option(FUSE_OPT_LATENT_IMPL, 2)
    for c in (a, f, g):
        c.weights(yh)
    X = f.solve(yl, yh, 9)[0].clone()
    assert f.get_option(FUSE_OPT_LATENT_FORM) == 0
    assert torch.equal(X, g.solve(yl, yh, 9)[0])
    Xa = a.solve(yl, yh, 9)[0].clone()
    batch = FusionBatch([a, f])
    Xs, _ = batch.solve([yl, yl], [yh, yh], 9)
    batch.sync()
    assert torch.equal(Xs[0], Xa) and torch.equal(Xs[1], X)
    assert [c.get_option(FUSE_OPT_LATENT_FORM) for c in (a, f)] == [2, 0]
    f.set_state(a.get_state())
    om = a.get_weights().double().cpu().numpy()
    ref = oracle_runs(p, [(om, 15)])[0]
    assert rel(f.solve(yl, yh, 6, warm=True)[0], ref) <= FP32_BOUND
    a.set_state(f.get_state())                            # and back: not entries of the grid
    assert torch.equal(a.solve(yl, yh, 4, warm=True)[0], f.solve(yl, yh, 4, warm=True)[0])
    assert a.get_option(FUSE_OPT_LATENT_FORM) == 0
    batch.close()
    for c in (a, f, g):
        c.close()
