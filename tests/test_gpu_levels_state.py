"""The latent state between its forms over sequences of calls: which arithmetic and form a solve runs
after changes of weights, states and data.  References are the same calls with every entry kept
(FUSE_OPT_LATENT_IMPL = 0), bit for bit, and the FP64 oracle."""
import math

import pytest

from paper_2210_04184_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2210_04184_gb300 import build as _build  # noqa: E402
from paper_2210_04184_gb300.fuse import Fusion, FUSE_OPT_LATENT_IMPL, FUSE_OPT_RESIDUALS  # noqa: E402


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
