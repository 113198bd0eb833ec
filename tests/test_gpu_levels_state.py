"""The latent state between its forms over sequences of calls: which arithmetic and form a solve runs
after changes of weights, states and data.  References are the same calls with every entry kept
(FUSE_OPT_LATENT_IMPL = 0), bit for bit, and the FP64 oracle."""
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
