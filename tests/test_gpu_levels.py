"""Solves that keep the latent state as levels against solves that keep every entry
(FUSE_OPT_LATENT_IMPL = 0): the state lives on the same grid, where the update and its sums are exact, so
X and the saved state are equal bit for bit.  Sizes at the edges of the level kernels: widths that are
no multiple of a warp, several pixel chunks per row, band groups with a remainder, the smallest and
largest windows, big moves (data far above the thresholds), thresholds of zero, weights above one, not
finite or negative."""
import numpy as np
import pytest

from paper_2210_04184_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2210_04184_gb300 import build as _build  # noqa: E402
from paper_2210_04184_gb300.fuse import (Fusion, FusionBatch, FUSE_OPT_GRAPH, FUSE_OPT_HALF_WINDOW,  # noqa: E402
                                         FUSE_OPT_LATENT_IMPL, FUSE_OPT_X_UPDATE)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()


def small(**kw):
    base = dict(H=40, W=40, L_l=6, L_h=2, L_s=3, d=4, blur_size=5, blur_sigma=1.0, K=1, S=2,
                lam1=1.0, lam2=1e-2, rho=5e-2, h=0.3, seed=17)
    base.update(kw)
    return synth.make_problem(**base)


def context(p, entries, dtype="f32", wdtype="f32", opts=(), weights=None, scale=1.0):
    f = Fusion.from_problem(p, dtype=dtype, wdtype=wdtype)
    for o, v in opts:
        f.set_option(o, v)
    if entries:
        f.set_option(FUSE_OPT_LATENT_IMPL, 0)
    td = torch.float64 if dtype == "f64" else torch.float32
    yl = torch.tensor(p.Yl * scale, dtype=td, device="cuda")
    yh = torch.tensor(p.Yh * scale, dtype=td, device="cuda")
    if weights is None:
        f.weights(torch.tensor(p.Yh, dtype=td, device="cuda"))
    else:
        f.set_weights(weights(f.nW, p.H, p.W).to(f.wtdtype).cuda())
    return f, yl, yh


def both(p, iters, **kw):
    out = []
    for entries in (0, 1):
        f, yl, yh = context(p, entries, **kw)
        X, _ = f.solve(yl, yh, iters)
        f.sync()
        out.append((X.clone(), f.get_state()))
        f.close()
    return out


@pytest.mark.parametrize("half", [1, 0])
@pytest.mark.parametrize("dtype,wdtype", [("f32", "f32"), ("f32", "bf16"), ("f64", "f64")])
@pytest.mark.parametrize("size", [dict(H=16, W=20, S=1), dict(H=20, W=36, K=2, S=3, L_s=5),
                                  dict(H=24, W=160, K=2, S=1), dict(H=12, W=400, S=2, L_l=40, L_s=33),
                                  dict(H=32, W=32, K=1, S=13, L_s=2)])
def test_levels_equal_entries(size, dtype, wdtype, half):
    p = small(**size)
    a, b = both(p, 12, dtype=dtype, wdtype=wdtype, opts=[(FUSE_OPT_HALF_WINDOW, half)])
    assert torch.equal(a[0], b[0])
    assert torch.equal(a[1], b[1])


@pytest.mark.parametrize("kw", [dict(lam2=0.0), dict(lam2=2.0), dict(lam2=1e-7)])
@pytest.mark.parametrize("scale", [1.0, 3e4, 1e-3])
def test_thresholds_far_from_the_data(kw, scale):
    # thresholds of zero, far above and far below the moves of X (codes of X beyond 2^32 included)
    p = small(K=2, S=2, **kw)
    a, b = both(p, 10, scale=scale)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def _mixed(nW, H, W):
    g = torch.Generator().manual_seed(3)
    w = torch.rand(nW, H, W, generator=g) * 40.0
    w[0, 0, :5] = torch.tensor([float("nan"), float("inf"), 0.0, -0.5, 1e-30])
    return w


@pytest.mark.parametrize("dtype,wdtype", [("f32", "bf16"), ("f32", "f32"), ("f64", "f64")])
def test_given_weights(dtype, wdtype):
    p = small(K=2, S=2, H=24, W=36)
    a, b = both(p, 8, dtype=dtype, wdtype=wdtype, weights=_mixed)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert torch.isfinite(a[0]).all()


@pytest.mark.parametrize("graph", [1, 0])
def test_warm_continuations(graph):
    # warm solves after a saved and restored state, after new weights and after a state of other
    # weights: levels where the state allows it, entries otherwise, the same bits throughout
    p, q = small(K=2, S=2, seed=5), small(K=2, S=2, seed=6)
    runs = []
    for entries in (0, 1):
        f, yl, yh = context(p, entries, opts=[(FUSE_OPT_GRAPH, graph)])
        g = torch.tensor(q.Yh, dtype=torch.float32, device="cuda")
        xs = [f.solve(yl, yh, 5)[0].clone(), f.solve(yl, yh, 3, warm=True)[0].clone()]
        st = f.get_state()
        xs.append(f.solve(yl, yh, 4, warm=True)[0].clone())
        f.set_state(st)
        xs.append(f.solve(yl, yh, 4, warm=True)[0].clone())
        assert torch.equal(xs[2], xs[3])
        f.weights(g)                                      # the state stays, its thresholds change
        xs.append(f.solve(yl, yh, 4, warm=True)[0].clone())
        f.set_state(st)                                   # a state of other weights
        xs.append(f.solve(yl, yh, 4, warm=True)[0].clone())
        xs.append(f.solve(yl, yh, 5)[0].clone())          # cold again
        f.weights(g)
        s1 = f.get_state()                                # saved after the weights were set again
        xs.append(s1)
        runs.append(xs)
        f.close()
    for a, b in zip(*runs):
        assert torch.equal(a, b)


def test_variant_x_update_and_batches():
    # the variant's first iteration has a nonzero X; a batch with a remainder of bands
    p = small(K=2, S=2, L_s=5)
    a, b = both(p, 9, opts=[(FUSE_OPT_X_UPDATE, 1)])
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    ps = [small(K=2, S=3, L_s=5, H=h, W=w, seed=30 + i) for i, (h, w) in enumerate([(24, 40), (40, 160), (64, 24)])]
    ref = [both(x, 7)[1][0] for x in ps]
    ctx = [context(x, 0) for x in ps]
    batch = FusionBatch([c[0] for c in ctx])
    for _ in range(2):
        Xs, _ = batch.solve([c[1] for c in ctx], [c[2] for c in ctx], 7)
        batch.sync()
        for x, y in zip(Xs, ref):
            assert torch.equal(x, y)
    batch.close()


def test_non_finite_data_stays_non_finite():
    p = small()
    f, yl, yh = context(p, 0)
    yl[0, 0, 0] = float("nan")
    X, _ = f.solve(yl, yh, 4)
    f.sync()
    assert not torch.isfinite(X).all()
    yl[0, 0, 0] = 0.5
    X, _ = f.solve(yl, yh, 4)
    f.sync()
    assert torch.isfinite(X).all()
    f.close()


def test_reference_is_close():
    # the grid is as fine as FP32: against FP64 contexts on the same problem
    p = small(K=2, S=3, H=48, W=64, L_l=8, L_h=3, L_s=4)
    X32 = both(p, 30)[0][0].double().cpu().numpy()
    X64 = both(p, 30, dtype="f64", wdtype="f64")[0][0].cpu().numpy()
    assert np.linalg.norm(X32 - X64) <= 2e-6 * np.linalg.norm(X64)
