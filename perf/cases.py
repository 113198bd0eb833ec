"""Performance cases of the fusion solver: what a user's program asks of it, as plain dicts.

A case names the call a program makes (`kind`), the sizes and the options; `prepare` builds what
such a program has in hand on the GPU before the call (images of the imaging model Y_l = S B Z,
Y_h = Z R in [0, 1]-scaled units, the subspace basis, the solver context), `run` is one pass
through the public entry points, and `exact` the same result from plain torch in float64.

Kinds:
  solve     Fusion.weights + Fusion.solve from a zero start: guide weights, `iters` iterations, X and Z
  batch     Fusion.weights of every problem + FusionBatch.solve over problems of uneven sizes
  host      FusionBatch.run_host: pinned host images in, weights, solve, every Z back in host memory
  unrolled  Fusion.unrolled and its backward: X and the gradients of an MSE loss against Z
"""
import math

import numpy as np
import torch

from paper_2210_04184_gb300.fuse import Fusion, FusionBatch

# image sides with factors 2, 3 and 5 that a ratio of 4 divides
SIDES = [32, 36, 40, 48, 60, 64, 72, 80, 96, 100, 108, 120, 128, 144, 160, 180, 192, 200, 216, 240, 256, 288, 300,
         320, 360, 384, 400, 432, 480, 512]
# (lambda2, rho, h) of the workloads and of the parity tests
PARAMS = {"workload": (1e-3, 1e-2, 0.15), "strong": (1e-2, 5e-2, 0.3)}


def _solve(name, H, W, L_l, L_h, L_s, K, S, iters, dtype="f32", wdtype="bf16", ratio=4, blur=9, sigma=1.7, snr=35.0,
           mask=0.0, identity=False, params="workload"):
    return dict(name=name, kind="solve", H=H, W=W, L_l=L_l, L_h=L_h, L_s=L_s, K=K, S=S, iters=iters, dtype=dtype,
                wdtype=wdtype, ratio=ratio, blur=blur, sigma=sigma, snr=snr, mask=mask, identity=identity,
                params=params)


def listed():
    return [
        # a small tile of a preview or a parameter search: launches and latency count
        _solve("tile_48", 48, 64, 8, 3, 4, 1, 2, 10, blur=5, sigma=1.0),
        # pansharpening of a 128 x 128 MS + PAN scene in FP64 (E = I), the whole 50-iteration run
        _solve("pansharpen_128_f64", 128, 128, 4, 1, 4, 1, 2, 50, dtype="f64", wdtype="f64", snr=40.0, identity=True),
        # HS + MS fusion, 256 x 256, 93 bands, the whole 100-iteration run
        _solve("hsms_256", 256, 256, 93, 4, 20, 2, 3, 100),
        # the same scene in FP64, as a reference run against which FP32 results are checked
        _solve("hsms_128_f64", 128, 128, 93, 4, 20, 2, 3, 20, dtype="f64", wdtype="f64"),
        # an HS + MS crop whose sides are neither powers of two nor multiples of 8, FP32 weights
        _solve("crop_200x180", 200, 180, 31, 3, 11, 2, 2, 40, wdtype="f32", params="strong"),
        # hyperspectral sharpening with a PAN guide at the largest size and search window, as many
        # iterations as one refinement of a warm-up takes
        _solve("hspan_512", 512, 512, 128, 1, 20, 2, 5, 24, blur=11, sigma=2.0, snr=30.0),
        # guided inpainting: every fifth pixel observed, no blur
        _solve("inpaint_256", 256, 256, 31, 3, 8, 1, 3, 60, ratio=1, blur=1, sigma=1.0, mask=0.2),
        # a set of scene tiles of uneven sizes solved together
        dict(name="batch_24", kind="batch", sizes="256,96,384,192,128,320,384,96,256,128,192,320,"
                                                  "256,384,96,128,320,192,384,256,128,96,192,320",
             L_l=31, L_h=3, L_s=8, K=1, S=3, iters=40, dtype="f32", wdtype="bf16", ratio=4, blur=9, sigma=1.7,
             snr=35.0, mask=0.0, identity=False, params="workload"),
        # a service's request: a few tiles from host memory, every result back in host memory
        dict(name="host_6", kind="host", sizes="128,192,96,256,128,96", L_l=31, L_h=3, L_s=8, K=1, S=3, iters=50,
             dtype="f32", wdtype="bf16", ratio=4, blur=9, sigma=1.7, snr=35.0, mask=0.0, identity=False,
             params="workload"),
        # one training step's solver part: 20 unrolled iterations and their reverse pass
        dict(name="unrolled_256", kind="unrolled", H=256, W=256, L_l=31, L_h=3, L_s=8, K=1, S=1, iters=20,
             dtype="f32", wdtype="f32", ratio=4, blur=9, sigma=1.5, snr=35.0, mask=0.0, identity=False,
             params="workload", guide=False),
    ]


def _latent_work(c):
    """Latent entries of a pass (kept offsets x patch x bands x pixels x iterations)."""
    nk = ((2 * c["S"] + 1) ** 2 - 1) // 2
    return nk * (2 * c["K"] + 1) ** 2 * c["L_s"] * sum(h * w for h, w in _sizes(c)) * c["iters"]


def _sizes(c):
    if "sizes" in c:
        return [(int(s), int(s)) for s in c["sizes"].split(",")]
    return [(c["H"], c["W"])]


def draw(rng):
    """One more case of the same ranges: sides 32 to 512, 3 to 20 subspace bands, patches 3 x 3 and
    5 x 5, search windows 3 x 3 to 11 x 11, both precisions."""
    limit = _latent_work([c for c in listed() if c["name"] == "hspan_512"][0])
    while True:
        kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "batch", "host", "unrolled"])
        c = dict(kind=kind, L_l=rng.randint(8, 128), L_h=rng.choice([1, 3, 4]), K=rng.choice([1, 1, 2, 2]),
                 S=rng.choice([1, 2, 3, 3, 5]), iters=rng.randint(8, 60), dtype="f32",
                 wdtype=rng.choice(["bf16", "bf16", "f32"]), ratio=4, blur=rng.choice([5, 7, 9, 11]),
                 sigma=round(rng.uniform(1.0, 2.0), 2), snr=rng.choice([30.0, 35.0, 40.0]), mask=0.0, identity=False,
                 params=rng.choice(sorted(PARAMS)))
        c["L_s"] = rng.randint(3, min(20, c["L_l"]))
        if kind in ("batch", "host"):
            sides = [s for s in SIDES if s % 8 == 0 and s <= 384]
            c["sizes"] = ",".join(str(_log_pick(rng, sides)) for _ in range(rng.randint(3, 16)))
        else:
            c["H"], c["W"] = _log_pick(rng, SIDES), _log_pick(rng, SIDES)
        if kind == "solve":
            form = rng.choice(["f32", "f32", "f64", "mask"])
            if form == "f64":
                c["dtype"] = c["wdtype"] = "f64"
            if form == "mask":
                c.update(ratio=1, blur=1, sigma=1.0, mask=round(rng.uniform(0.1, 0.5), 2))
        if kind == "unrolled":
            c.update(wdtype="f32", S=rng.choice([1, 2]), iters=rng.randint(4, 20), guide=rng.random() < 0.3)
            c["L_s"] = min(c["L_s"], 12)
        cost = _latent_work(c) * (2 if c["dtype"] == "f64" else 1) * (4 if kind == "unrolled" else 1)
        # a pass no dearer than the largest listed one, and a reverse-pass tape of a few GB
        if cost <= limit and (kind != "unrolled" or _latent_work(c) * 4 <= 6e9) and min(map(min, _sizes(c))) >= 32:
            return c


def _log_pick(rng, sides):
    x = math.exp(rng.uniform(math.log(sides[0]), math.log(sides[-1] * 1.02)))
    return min(sides, key=lambda s: abs(math.log(s / x)))


# ---- inputs ---------------------------------------------------------------------------------


def _gauss(size, sigma):
    u = np.arange(-(size // 2), size // 2 + 1, dtype=np.float64)
    g = np.exp(-(u[:, None] ** 2 + u[None, :] ** 2) / (2.0 * sigma * sigma))
    return g / g.sum()


def _blur_hat(blur, H, W, device):
    b = torch.zeros(H, W, dtype=torch.float64, device=device)
    r = blur.shape[0] // 2
    for i in range(blur.shape[0]):
        for j in range(blur.shape[1]):
            b[(i - r) % H, (j - r) % W] += float(blur[i, j])
    return torch.fft.fft2(b)


def _field(gen, H, W, device):
    """A smooth periodic random field with tiled texture over random rectangles, in [0, 1]."""
    corr = max(H, W) / 16.0
    fy = torch.fft.fftfreq(H, dtype=torch.float64, device=device)[:, None]
    fx = torch.fft.fftfreq(W, dtype=torch.float64, device=device)[None, :]
    noise = torch.randn(H, W, dtype=torch.float64, device=device, generator=gen)
    f = torch.fft.ifft2(torch.fft.fft2(noise) * torch.exp(-2.0 * (math.pi * corr) ** 2 * (fy ** 2 + fx ** 2))).real
    f = (f - f.min()) / (f.max() - f.min())
    tile = torch.rand(16, 16, dtype=torch.float64, device=device, generator=gen)
    tex = tile.repeat(-(-H // 16), -(-W // 16))[:H, :W]
    u = torch.rand(6, 4, dtype=torch.float64, device=device, generator=gen)
    y = torch.arange(H, device=device, dtype=torch.float64)[:, None]
    x = torch.arange(W, device=device, dtype=torch.float64)[None, :]
    m = torch.zeros(H, W, dtype=torch.bool, device=device)
    for r in range(6):
        hh, ww = H / 8 + u[r, 2] * (H / 3 - H / 8), W / 8 + u[r, 3] * (W / 3 - W / 8)
        m |= (torch.remainder(y - u[r, 0] * H, H) < hh) & (torch.remainder(x - u[r, 1] * W, W) < ww)
    f = torch.where(m, 0.35 * f + 0.65 * tex, f)
    return (f - f.min()) / (f.max() - f.min())


def _noise(gen, Y, snr):
    sig = (Y.pow(2).mean(dim=(1, 2)) / 10.0 ** (snr / 10.0)).sqrt()
    return Y + sig[:, None, None] * torch.randn(Y.shape, dtype=Y.dtype, device=Y.device, generator=gen)


def _problem(c, H, W, seed):
    """Scene Z, images Y_l and Y_h, blur, R, E and the sampling mask (float64 on the GPU)."""
    device = "cuda"
    gen = torch.Generator(device=device).manual_seed(seed)
    L = c["L_l"]
    if c["identity"]:
        Z = torch.stack([_field(gen, H, W, device) for _ in range(L)])
        R = torch.rand(L, c["L_h"], dtype=torch.float64, device=device, generator=gen)
        R = R / R.sum(0, keepdim=True)
    else:
        # mixtures of 6 smooth spectra (sums of 3 Gaussians over the bands) with textured abundances
        b = torch.arange(L, dtype=torch.float64, device=device)
        u = torch.rand(6, 3, 3, dtype=torch.float64, device=device, generator=gen)
        ctr, wid, amp = u[..., 0] * L, L / 12 + u[..., 1] * (L / 3 - L / 12), 0.2 + 0.8 * u[..., 2]
        spec = (amp[..., None] * torch.exp(-0.5 * ((b - ctr[..., None]) / wid[..., None]) ** 2)).sum(1)
        ab = torch.softmax(torch.stack([4.0 * _field(gen, H, W, device) for _ in range(6)]), dim=0)
        Z = torch.einsum("ehw,el->lhw", ab, spec)
        Z = (Z - Z.min()) / (Z.max() - Z.min())
        if c["L_h"] == 1:
            R = (1.0 + b / L)[:, None]
        else:
            cen = (torch.arange(c["L_h"], dtype=torch.float64, device=device) + 0.5) * L / c["L_h"]
            R = torch.exp(-0.5 * ((b[:, None] - cen[None, :]) / (L / 8.0)) ** 2)
        R = R / R.sum(0, keepdim=True)
    blur = _gauss(c["blur"], c["sigma"])
    Yh = _noise(gen, torch.einsum("lhw,lk->khw", Z, R), c["snr"])
    d = c["ratio"]
    BZ = torch.fft.ifft2(torch.fft.fft2(Z) * _blur_hat(blur, H, W, device)).real
    Yl = _noise(gen, BZ[:, ::d, ::d].contiguous(), c["snr"])
    mask = torch.rand(H, W, dtype=torch.float64, device=device, generator=gen) < c["mask"] if c["mask"] else None
    if c["identity"]:
        E = np.eye(L)
    else:
        M = Yl.reshape(L, -1)
        _, v = np.linalg.eigh((M @ M.T).cpu().numpy())
        E = v[:, ::-1][:, :c["L_s"]].T.copy()
        for r in range(E.shape[0]):
            if E[r, np.argmax(np.abs(E[r]))] < 0:
                E[r] = -E[r]
    return dict(H=H, W=W, Z=Z, Yl=Yl, Yh=Yh, R=R.cpu().numpy(), E=E, blur=blur, mask=mask)


def _problems(c, seed):
    return [_problem(c, h, w, 1009 * seed + 31 * i + 7) for i, (h, w) in enumerate(_sizes(c))]


def _context(c, p):
    lam2, rho, h = PARAMS[c["params"]]
    f = Fusion(H=p["H"], W=p["W"], L_l=c["L_l"], L_h=c["L_h"], L_s=c["L_s"], blur=p["blur"], ratio=c["ratio"],
               R=p["R"], E=p["E"], K=c["K"], S=c["S"], lam1=1.0, lam2=lam2, rho=rho, h=h, dtype=c["dtype"],
               wdtype=c["wdtype"])
    if p["mask"] is not None:
        f.set_mask(p["mask"])
    return f


def prepare(case, seed):
    """The program's images (in its precision), its solver contexts and, for a batch, the batch."""
    td = torch.float64 if case["dtype"] == "f64" else torch.float32
    ps = _problems(case, seed)
    st = dict(case=case, fs=[_context(case, p) for p in ps])
    yl, yh = [p["Yl"].to(td).contiguous() for p in ps], [p["Yh"].to(td).contiguous() for p in ps]
    if case["kind"] == "host":
        yl, yh = [a.cpu().pin_memory() for a in yl], [a.cpu().pin_memory() for a in yh]
    if case["kind"] in ("batch", "host"):
        st["batch"] = FusionBatch(st["fs"])
    if case["kind"] == "unrolled":
        st["Z"] = ps[0]["Z"].to(td)
        st["E"] = torch.tensor(ps[0]["E"], dtype=td, device="cuda")
        st["params"] = st["fs"][0].params()
        if not case["guide"]:
            st["fs"][0].weights(yh[0])
    st.update(yl=yl, yh=yh)
    return st


def run(state):
    case, fs, yl, yh = state["case"], state["fs"], state["yl"], state["yh"]
    if case["kind"] == "solve":
        fs[0].weights(yh[0])
        X, Z = fs[0].solve(yl[0], yh[0], case["iters"], want_Z=True)
        return {"X": X, "Z": Z}
    if case["kind"] == "batch":
        for f, g in zip(fs, yh):
            f.weights(g)
        X, Z = state["batch"].solve(yl, yh, case["iters"], want_Z=True)
        return {"X": X, "Z": Z}
    if case["kind"] == "host":
        _, Z = state["batch"].run_host(yl, yh, case["iters"])
        return {"Z": Z}
    a, b = yl[0].detach().requires_grad_(True), yh[0].detach().requires_grad_(True)
    q = state["params"].detach().requires_grad_(True)
    X = fs[0].unrolled(a, b, case["iters"], q, guide=b if case["guide"] else None)
    loss = _loss(X, state["E"], state["Z"])
    loss.backward()
    return {"X": X.detach(), "Yl_grad": a.grad, "Yh_grad": b.grad, "params_grad": q.grad}


def _loss(X, E, Z):
    """MSE of Z = X E against the scene."""
    return (torch.einsum("chw,cl->lhw", X, E) - Z).pow(2).mean()


# ---- work and exact values --------------------------------------------------------------------


def work(case):
    """Images read and written once, and per iteration what separates two global transforms: the
    right-hand side and X written and read, the two scaled duals read and written, and one number
    per kept offset, band and pixel read and written (the least a latent state can hold).  Flops:
    the transforms, the L_s x L_s closed forms and ten per kept offset, band and pixel.  The reverse
    pass counts as two more forward passes."""
    b = 8 if case["dtype"] == "f64" else 4
    nk = ((2 * case["S"] + 1) ** 2 - 1) // 2
    Ls, it = case["L_s"], case["iters"]
    byts = flops = 0.0
    for h, w in _sizes(case):
        n = h * w
        lat = nk * Ls * n
        io = b * (case["L_l"] * n / case["ratio"] ** 2 + case["L_h"] * n + case["L_l"] * n
                  + (Ls * n if case["kind"] != "host" else 0))
        per_b = b * (8 * Ls * n + 2 * lat)
        per_f = 5.0 * Ls * n * math.log2(n) + 4.0 * Ls * Ls * n + 10.0 * lat
        rep = 3 if case["kind"] == "unrolled" else 1
        byts += io + rep * it * per_b
        flops += rep * it * per_f
    return {"bytes": byts, "flops": flops}


def _sh(x, t):
    return torch.roll(x, shifts=t, dims=(-2, -1))


def _admm64(c, p, yl, yh, omega_guide, lam):
    """X after the iterations in float64, as a function of the images and (lambda1, lambda2, rho)."""
    dev = yl.device
    H, W, K, S, Ls, d = p["H"], p["W"], c["K"], c["S"], c["L_s"], c["ratio"]
    h2 = PARAMS[c["params"]][2] ** 2
    lam1, lam2, rho = lam[0], lam[1], lam[2]
    E = torch.tensor(p["E"], dtype=torch.float64, device=dev)
    R = torch.tensor(p["R"], dtype=torch.float64, device=dev)
    patch = [(a, b) for a in range(-K, K + 1) for b in range(-K, K + 1)]
    # one offset of each +-tau pair: the other's term in D^T D and D^T (Q + Sigma) is equal
    kept = [(a, b) for a in range(0, S + 1) for b in range(-S, S + 1) if a > 0 or b > 0]
    om = []
    for t in kept:
        e = (omega_guide - _sh(omega_guide, t)).pow(2).sum(0)
        om.append(torch.exp(-sum(_sh(e, k) for k in patch) / h2))
    bh = _blur_hat(p["blur"], H, W, dev)
    fy = torch.arange(H, dtype=torch.float64, device=dev)[:, None] / H
    fx = torch.arange(W, dtype=torch.float64, device=dev)[None, :] / W
    den = 1.0 + bh.abs() ** 2 + len(patch) * sum(4.0 - 4.0 * torch.cos(2 * math.pi * (fy * a + fx * b)) for a, b in kept)
    eye = torch.eye(Ls, dtype=torch.float64, device=dev)
    ER = E @ R
    M1 = torch.linalg.inv(E @ E.T + rho * eye)
    F = torch.linalg.inv(eye + lam1 / rho * ER @ ER.T)
    samp = torch.zeros(H, W, dtype=torch.bool, device=dev)
    samp[::d, ::d] = True
    if p["mask"] is not None:
        samp = p["mask"]
    D9a = torch.einsum("lhw,cl->chw", _upsample(yl, d, H, W), E)
    D9b = lam1 / rho * torch.einsum("khw,ck->chw", yh, ER)
    mu = [lam2 / rho * torch.stack([_sh(w, (-a, -b)) for a, b in patch])[:, None] for w in om]
    z = torch.zeros(Ls, H, W, dtype=torch.float64, device=dev)
    L1, U1, L2, U2, Rr = z, z, z, z, z
    sig = [torch.zeros(len(patch), 1, 1, 1, dtype=torch.float64, device=dev) for _ in kept]
    X = z
    fft, ifft = torch.fft.fft2, torch.fft.ifft2
    for _ in range(c["iters"]):
        X = ifft(fft(ifft(fft(U1) * bh.conj()).real + U2 + Rr) / den).real
        BX = ifft(fft(X) * bh).real
        w2 = X - L2
        P2 = torch.einsum("jhw,jc->chw", w2 + D9b, F)
        L2, U2 = P2 - w2, 2 * P2 - w2
        w1 = BX - L1
        P1 = torch.where(samp, torch.einsum("jhw,jc->chw", rho * w1 + D9a, M1), w1)
        L1, U1 = P1 - w1, 2 * P1 - w1
        Rr = z
        for i, t in enumerate(kept):
            u = sig[i] - (X - _sh(X, t))
            s = torch.where(u.abs() < mu[i], u, torch.sign(u) * mu[i])
            g = (2 * s - u).sum(0)
            Rr = Rr + 2 * (g - _sh(g, (-t[0], -t[1])))
            sig[i] = s
    return X


def _upsample(yl, d, H, W):
    up = torch.zeros(yl.shape[0], H // d, d, W // d, d, dtype=yl.dtype, device=yl.device)
    one = torch.zeros(d, 1, d, dtype=yl.dtype, device=yl.device)
    one[0, 0, 0] = 1.0
    return (up + yl[:, :, None, :, None] * one).reshape(yl.shape[0], H, W)


def exact(case, seed):
    nk, nP = ((2 * case["S"] + 1) ** 2 - 1) // 2, (2 * case["K"] + 1) ** 2
    state = max(nk * nP * case["L_s"] * h * w * 8 for h, w in _sizes(case))
    # the latent state and, for gradients, one copy of it per saved intermediate and iteration
    if state * (8 * case["iters"] if case["kind"] == "unrolled" else 1) > 3e10:
        return None
    td = torch.float64 if case["dtype"] == "f64" else torch.float32
    lam2, rho, _ = PARAMS[case["params"]]
    lam = torch.tensor([1.0, lam2, rho], dtype=torch.float64, device="cuda")
    X, Z = [], []
    for p in _problems(case, seed):
        # the inputs the program has, in its precision
        yl, yh = p["Yl"].to(td).double(), p["Yh"].to(td).double()
        E = torch.tensor(p["E"], dtype=torch.float64, device="cuda")
        if case["kind"] == "unrolled":
            yl.requires_grad_(True)
            yh.requires_grad_(True)
            lam.requires_grad_(True)
            x = _admm64(case, p, yl, yh, yh if case["guide"] else yh.detach(), lam)
            _loss(x, E, p["Z"].to(td).double()).backward()
            return {"X": x.detach(), "Yl_grad": yl.grad, "Yh_grad": yh.grad, "params_grad": lam.grad.cpu()}
        x = _admm64(case, p, yl, yh, yh, lam)
        X.append(x)
        Z.append(torch.einsum("chw,cl->lhw", x, E))
    if case["kind"] == "solve":
        return {"X": X[0], "Z": Z[0]}
    if case["kind"] == "host":
        return {"Z": [z.cpu() for z in Z]}
    return {"X": X, "Z": Z}
