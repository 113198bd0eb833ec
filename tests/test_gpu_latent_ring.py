"""Entries through the bulk-copy ring (FUSE_OPT_LATENT_IMPL = 2), which every state that is not kept as
levels runs: its launch shapes, its precision against the oracle, batches, and the choice between the
forms."""
import numpy as np
import pytest

from paper_2210_04184_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle import nlpr  # noqa: E402
from paper_2210_04184_gb300 import build as _build  # noqa: E402
from paper_2210_04184_gb300 import fuse  # noqa: E402
from paper_2210_04184_gb300.fuse import (Fusion, FusionBatch, FuseError, FUSE_OPT_HALF_WINDOW,  # noqa: E402
                                         FUSE_OPT_LATENT_BANDS, FUSE_OPT_LATENT_FORM, FUSE_OPT_LATENT_IMPL,
                                         FUSE_OPT_LATENT_STAGES, FUSE_OPT_LATENT_THREADS, FUSE_OPT_WAIT_LIMIT)

ENTRIES, LEVELS = 0, 2          # FUSE_OPT_LATENT_FORM


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()


def small(**kw):
    base = dict(H=48, W=64, L_l=8, L_h=3, L_s=4, d=4, blur_size=9, blur_sigma=1.7, K=2, S=3,
                lam1=1.0, lam2=1e-2, rho=5e-2, h=0.3, seed=11)
    base.update(kw)
    return synth.make_problem(**base)


def context(p, dtype="f32", wdtype="f32", opts=()):
    td = torch.float64 if dtype == "f64" else torch.float32
    f = Fusion.from_problem(p, dtype=dtype, wdtype=wdtype)
    for o, v in opts:
        f.set_option(o, v)
    yl, yh = (torch.tensor(a, dtype=td, device="cuda") for a in (p.Yl, p.Yh))
    f.weights(yh)
    return f, yl, yh


def solve(p, iters, form=ENTRIES, **kw):
    f, yl, yh = context(p, **kw)
    X, _ = f.solve(yl, yh, iters)
    f.sync()
    assert f.get_option(FUSE_OPT_LATENT_FORM) == form
    out = X.double().cpu().numpy()
    f.close()
    return out


def oracle(p, iters):
    om = nlpr.weights(nlpr.to_hwl(p.Yh), p.K, p.S, p.h)
    X, _, _ = nlpr.admm(nlpr.to_hwl(p.Yl), nlpr.to_hwl(p.Yh), p.blur, p.d, p.R, p.E, p.K, p.S, p.lam1, p.lam2, p.rho, om,
                        iters, fast=True)
    return nlpr.to_lhw(X)


@pytest.mark.parametrize("threads,stages,bands", [(32, 2, 1), (64, 3, 3), (256, 4, 2), (128, 16, 1), (256, 8, 4),
                                                   (256, 6, 64)])
def test_ring_shapes_bitwise_equal(threads, stages, bands):
    p = small()
    ref = solve(p, 6, opts=[(FUSE_OPT_LATENT_IMPL, 2)])
    got = solve(p, 6, opts=[(FUSE_OPT_LATENT_IMPL, 2), (FUSE_OPT_LATENT_THREADS, threads),
                            (FUSE_OPT_LATENT_STAGES, stages), (FUSE_OPT_LATENT_BANDS, bands)])
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("half", [1, 0])
@pytest.mark.parametrize("K,S,W", [(1, 2, 40), (2, 1, 64), (2, 3, 160)])
@pytest.mark.parametrize("dtype,bound", [("f32", 1e-5), ("f64", 1e-11)])
def test_ring_and_levels_parity(K, S, W, half, dtype, bound):
    p = small(H=32, W=W, K=K, S=S)
    ref = oracle(p, 25)
    for impl, form in ((2, ENTRIES), (1, LEVELS)):
        X = solve(p, 25, form, dtype=dtype, wdtype=dtype, opts=[(FUSE_OPT_HALF_WINDOW, half), (FUSE_OPT_LATENT_IMPL, impl)])
        assert np.linalg.norm(X - ref) <= bound * np.linalg.norm(ref)


@pytest.mark.parametrize("dtype,wdtype", [("f32", "bf16"), ("f64", "f64")])
def test_batch_of_entries(dtype, wdtype):
    opts = [(FUSE_OPT_LATENT_IMPL, 2)]
    ps = [small(K=1, S=2, L_s=5, H=h, W=w, seed=100 + i) for i, (h, w) in enumerate([(40, 40), (48, 64), (96, 96), (32, 24)])]
    ref = [solve(p, 12, dtype=dtype, wdtype=wdtype, opts=opts) for p in ps]
    ctx = [context(p, dtype, wdtype, opts) for p in ps]
    batch = FusionBatch([c[0] for c in ctx])
    for shape in ((256, 6, 2), (64, 3, 1), (128, 4, 5)):
        for o, v in zip((FUSE_OPT_LATENT_THREADS, FUSE_OPT_LATENT_STAGES, FUSE_OPT_LATENT_BANDS), shape):
            batch.set_option(o, v)
        Xs, _ = batch.solve([c[1] for c in ctx], [c[2] for c in ctx], 12)
        batch.sync()
        for c, x, y in zip(ctx, Xs, ref):
            assert c[0].get_option(FUSE_OPT_LATENT_FORM) == ENTRIES
            assert np.array_equal(x.double().cpu().numpy(), y)
    batch.close()


def test_short_wait_limit_of_the_ring():
    # one poll per wait: every copy lands in time and the result is the same, or the solve reports
    # the timeout; the context works again afterwards
    p = small()
    ref = solve(p, 3, opts=[(FUSE_OPT_LATENT_IMPL, 2)])
    f, yl, yh = context(p, opts=[(FUSE_OPT_LATENT_IMPL, 2), (FUSE_OPT_WAIT_LIMIT, 1)])
    X, _ = f.solve(yl, yh, 3)
    try:
        f.sync()
        assert np.array_equal(X.double().cpu().numpy(), ref)
    except FuseError as e:
        assert e.status == fuse.FUSE_ETIMEOUT
        fuse.fuse_reset_error(f.ctx)
    f.set_option(FUSE_OPT_WAIT_LIMIT, 1 << 22)
    X, _ = f.solve(yl, yh, 3)
    f.sync()
    assert np.array_equal(X.double().cpu().numpy(), ref)
    f.close()


def test_choice_of_the_form():
    # W = 36: the ring does not fit FP32 rows, levels need none
    p = small(W=36)
    f, yl, yh = context(p)
    X = f.solve(yl, yh, 5)[0].clone()
    assert f.get_option(FUSE_OPT_LATENT_FORM) == LEVELS
    f.set_option(FUSE_OPT_LATENT_IMPL, 0)
    assert torch.equal(f.solve(yl, yh, 5)[0], X) and f.get_option(FUSE_OPT_LATENT_FORM) == 1
    f.set_option(FUSE_OPT_LATENT_IMPL, 1)
    assert torch.equal(f.solve(yl, yh, 5)[0], X) and f.get_option(FUSE_OPT_LATENT_FORM) == LEVELS
    with pytest.raises(FuseError):
        f.set_option(FUSE_OPT_LATENT_IMPL, 2)
    fuse.fuse_reset_error(f.ctx)
    assert torch.equal(f.solve(yl, yh, 5)[0], X) and f.get_option(FUSE_OPT_LATENT_FORM) == LEVELS
    f.close()
    # FP32 with 3 x 3 patches and a 3 x 3 search stays entries
    solve(small(K=1, S=1), 4)
