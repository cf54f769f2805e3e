"""Performance cases of the framework, through its public entry points.

Each case draws a synthetic survey from a seed (exposures, catalog, Poisson counts), binds it as a
user's program does, and `run` makes one call or one chain of calls on it.  The shapes are those of the
repository's workloads: one 41 x 41 x 5 source; a 2048 x 1489 field in five bands with 1000 sources; a
mosaic of overlapping fields with 1-3 bands each; the warm-start network on 32 x 32 x 5 patches.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1611_03404_gb300 as celeste
from paper_1611_03404_gb300 import cnn
from paper_1611_03404_gb300.blockcoord import block_coordinate

# Galaxy profile tables (unit flux, half-light radius 1): exponential (6) and de Vaucouleurs (8).
EXP_NU = [0.0006596951502967703, 0.008499948273535158, 0.056750668148803744, 0.22909140806738018,
          0.4610677000650011, 0.24393058029498293]
EXP_TAU = [0.0026964523198173673, 0.019832622513022816, 0.0868133713693027, 0.2965756227564619,
           0.872162744212001, 2.3672623510096025]
DEV_NU = [0.00016023890226608196, 0.001477650972700837, 0.00773972860823985, 0.028967916143913062,
          0.0835980906908277, 0.1889718131555343, 0.32221770578089337, 0.36686685574562483]
DEV_TAU = [1.8377602381471976e-06, 3.154405920442516e-05, 0.00029861402151766113, 0.002189029452081167,
           0.01433137495816934, 0.09284202670479808, 0.6780991051805976, 8.133158735894337]
TAU = np.array(EXP_TAU + DEV_TAU)
PRIORS = np.array([0.5, 2.0, 1.0, 0.0, 0.25])   # P(galaxy); log flux mean, variance; colour mean, variance
COLOUR_MIX = np.array([[-1, -1, 0, 0], [0, -1, 0, 0], [0, 0, 0, 0], [0, 0, 1, 0], [0, 0, 1, 1]], float)

FIELD_W, FIELD_H = 2048, 1489
# operations per pixel of the value + gradient + Hessian evaluation and of the value alone
FLOPS_FULL, FLOPS_VALUE = 7349, 403
CNN_MACS = 1024 * 32 * 45 + 256 * 64 * 288 + 64 * 64 * 576 + 16 * 64 * 576 + 1024 * 256 + 256 * 27
CNN_PARAMS = 32 * 46 + 64 * 289 + 2 * 64 * 577 + 256 * 1025 + 27 * 257


# ------------------------------------------------------------------------------------------ the cases
def _survey(name, kind, sources, **more):
    case = {"name": name, "kind": kind, "sources": sources, "fields_x": 1, "fields_y": 1, "width": FIELD_W,
            "height": FIELD_H, "bands_min": 5, "bands_max": 5, "rmin": 8, "rmax": 32, "wide": False, "tile": 128,
            "hessian": 0}
    case.update(more)
    return case


def listed():
    return [
        # a program that looks at one light source at a time: launch and latency bound
        _survey("one_source_elbo", "elbo", 1, width=41, height=41, rmin=20, rmax=20),
        _survey("one_source_newton", "newton", 1, width=41, height=41, rmin=20, rmax=20),
        # an optimiser or sampler of the user's own over a field: value, gradient and Hessian per call
        _survey("field_elbo", "elbo", 1000),
        # the same over wide patches of a few overlapping fields, the Hessian's products on tensor cores
        _survey("mosaic_elbo_tf32x3", "elbo", 2000, fields_x=2, bands_min=1, bands_max=3, rmax=64, wide=True,
                hessian=celeste.HESS_TF32X3),
        # line searches and model comparison: values only, in the larger tiles
        _survey("field_value", "value", 1000, tile=256),
        # what the library is for: every source of a field to convergence from the catalog
        _survey("field_newton", "newton", 1000),
        # error bars of a converged field catalog
        _survey("field_covariance", "covariance", 1000),
        # a crowded field's neighbours, rendered again before every pass of block-coordinate ascent
        _survey("crowded_background", "background", 4000),
        # all sources at once, couplings included, from two block-coordinate passes
        _survey("field_joint", "joint", 200, width=768, height=560),
        # the production step on a mosaic: new counts, neighbours, network start, Newton
        _survey("mosaic_pass", "pass", 9000, fields_x=3, fields_y=3, bands_min=1, bands_max=3, rmax=64, wide=True),
        # the network's inference over a catalog, in the library's batches, the last one ragged
        {"name": "network_predict", "kind": "predict", "patches": 20000},
        # one training step of the network at the batch it is trained with
        {"name": "network_train", "kind": "train", "patches": 512},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["elbo", "elbo", "value", "newton", "newton", "covariance", "background", "joint", "pass",
                       "predict", "train"])
    if kind == "predict":
        return {"kind": kind, "patches": _log_int(rng, 1, 20000)}
    if kind == "train":
        return {"kind": kind, "patches": _log_int(rng, 8, 1024)}
    most = {"joint": 200, "pass": 5000, "background": 4000}.get(kind, 2000)
    sources = _log_int(rng, 100 if kind == "pass" else 1, most)
    case = _survey("", kind, sources)
    del case["name"]
    if kind == "pass" or (kind != "joint" and sources >= 200 and rng.random() < 0.3):
        # overlapping fields, 1-3 bands each
        case.update(fields_x=rng.randint(1, 3), fields_y=rng.randint(1, 2), bands_min=1, bands_max=3, rmax=64, wide=True)
        density = sources / (case["fields_x"] * case["fields_y"])
        case["width"] = min(FIELD_W, 64 + int(math.sqrt(density) * rng.uniform(50, 75)))
        case["height"] = min(FIELD_H, 64 + int(math.sqrt(density) * rng.uniform(40, 55)))
    else:
        side = 41 + math.sqrt(sources) * rng.uniform(28, 60)
        case.update(width=min(FIELD_W, int(side * rng.uniform(1.0, 1.3))), height=min(FIELD_H, int(side)),
                    bands_min=rng.choice([1, 3, 5, 5]), rmin=rng.randint(5, 12), rmax=rng.randint(16, 32))
    if kind in ("elbo", "covariance"):
        case["hessian"] = rng.choice([celeste.HESS_FP32, celeste.HESS_FP32, celeste.HESS_BF16X6, celeste.HESS_TF32X3])
    if case["hessian"] == celeste.HESS_FP32:
        case["tile"] = rng.choice([128, 128, 256, 512])
    return case


# ------------------------------------------------------------------------------------- synthetic survey
def _psf(rng):
    """Three Gaussian components as quadratic polynomials over the exposure, widths 1-3 px."""
    psf = np.zeros((3, 6, 6))
    psf[:, 0, 0] = np.log(rng.dirichlet([3.0, 3.0, 3.0]))
    psf[:, 1:3, 0] = rng.normal(0.0, 0.1, (3, 2))
    psf[:, 3:5, 0] = np.log(rng.uniform(1.4, 2.1, (3, 2)))
    psf[:, 5, 0] = np.arctanh(rng.uniform(-0.3, 0.3, 3))
    psf[:, 0, 1:] = rng.uniform(-0.1, 0.1, (3, 5))
    psf[:, 1:6, 1:] = rng.uniform(-0.05, 0.05, (3, 5, 5))
    return psf


def _psf_at(im, pos):
    """PSF of an exposure at pixel positions [P, 2]: weights [P, 3], means [P, 3, 2], covariances [P, 3, 3]."""
    x, y = 2.0 * pos[:, 0] / (im.W - 1) - 1.0, 2.0 * pos[:, 1] / (im.H - 1) - 1.0
    par = np.einsum("kqc,pc->pkq", im.psf, np.stack([np.ones_like(x), x, y, x * x, x * y, y * y], -1))
    w = np.exp(par[..., 0] - par[..., 0].max(-1, keepdims=True))
    sx, sy = np.exp(par[..., 3]), np.exp(par[..., 4])
    return w / w.sum(-1, keepdims=True), par[..., 1:3], np.stack([sx * sx, np.tanh(par[..., 5]) * sx * sy, sy * sy], -1)


def _render(im, pos, gal, shape, flux, device):
    """Expected counts of an exposure: sky plus every true source over 4 sigma of its profile, at most 64 px.
    The sources' light is added in whole 2^-20ths of a count, so the sum does not depend on its order."""
    acc = torch.zeros(im.H * im.W, dtype=torch.int64, device=device)
    w, mean, cov = _psf_at(im, pos)
    A = im.wcs[:4].reshape(2, 2)
    c, s, q2 = np.cos(shape[:, 2]), np.sin(shape[:, 2]), shape[:, 1] ** 2
    g = np.stack([c * c + q2 * s * s, (1 - q2) * c * s, s * s + q2 * c * c], -1) * (shape[:, 3:4] ** 2) * gal[:, None]
    G = A @ np.stack([np.stack([g[:, 0], g[:, 1]], -1), np.stack([g[:, 1], g[:, 2]], -1)], -2) @ A.T
    g = np.stack([G[:, 0, 0], G[:, 0, 1], G[:, 1, 1]], -1)
    nu = np.concatenate([(1 - shape[:, 0:1]) * EXP_NU, shape[:, 0:1] * DEV_NU], 1)
    S = cov[:, :, None, :] + TAU[None, None, :, None] * g[:, None, None, :]                        # [P, 3, 14, 3]
    det = S[..., 0] * S[..., 2] - S[..., 1] ** 2
    amp = im.iota * flux[:, None, None] * w[:, :, None] * nu[:, None, :] / (2 * np.pi * np.sqrt(det))
    P = np.stack([S[..., 2], -S[..., 1], S[..., 0]], -1) / det[..., None]
    half = np.ceil(4 * np.sqrt((cov[..., [0, 2]].max((1, 2)) + np.where(gal, TAU.max() * shape[:, 3] ** 2, 0.0))))
    steps = np.array([8, 12, 16, 24, 32, 48, 64])
    half = steps[np.searchsorted(steps, np.minimum(half, 64))]
    t = lambda a, dt=torch.float32: torch.as_tensor(np.ascontiguousarray(a), device=device, dtype=dt)
    for h in np.unique(half):
        off = torch.arange(-int(h), int(h) + 1, device=device)
        batch = max(1, (1 << 22) // len(off) ** 2)
        sel = np.nonzero(half == h)[0]
        for i in range(0, len(sel), batch):
            k = sel[i:i + batch]
            c0 = np.floor(pos[k] + 0.5)
            f = t(pos[k] - c0)
            X, Y = off.float()[None, None, :] - f[:, 0, None, None], off.float()[None, :, None] - f[:, 1, None, None]
            val = torch.zeros(len(k), len(off), len(off), device=device)
            Pk, ak, mk = t(P[k]), t(amp[k]), t(mean[k])
            for a in range(3):
                dx, dy = X - mk[:, a, 0, None, None], Y - mk[:, a, 1, None, None]
                for j in range(14):
                    p = Pk[:, a, j, :, None, None]
                    val += ak[:, a, j, None, None] * torch.exp(
                        -0.5 * (p[:, 0] * dx * dx + 2 * p[:, 1] * dx * dy + p[:, 2] * dy * dy))
            xs = t(c0[:, 0], torch.int64)[:, None, None] + off[None, None, :]
            ys = t(c0[:, 1], torch.int64)[:, None, None] + off[None, :, None]
            ok = (xs >= 0) & (xs < im.W) & (ys >= 0) & (ys < im.H)
            acc.index_add_(0, (ys * im.W + xs)[ok], (val[ok] * 1048576.0).round().to(torch.int64))
    return im.sky + acc.view(im.H, im.W).double() / 1048576.0


def _make_survey(case, seed, device):
    """Exposures with Poisson counts on the device, and the catalog they are solved from (the truth
    perturbed, as a previous survey's would be)."""
    rng = np.random.default_rng(seed)
    S, W, H, fx, fy = case["sources"], case["width"], case["height"], case["fields_x"], case["fields_y"]
    images = []
    extent = np.array([0.8 * W * (fx - 1) + W, 0.8 * H * (fy - 1) + H])
    for j in range(fy):
        for i in range(fx):
            nb = int(rng.integers(case["bands_min"], case["bands_max"] + 1))
            for b in sorted(rng.choice(5, nb, replace=False)):
                ang, sc = (rng.uniform(-0.02, 0.02), rng.uniform(0.98, 1.02)) if fx * fy > 1 else (0.0, 1.0)
                A = sc * np.array([[math.cos(ang), -math.sin(ang)], [math.sin(ang), math.cos(ang)]])
                centre = np.array([0.8 * W * i + W / 2, 0.8 * H * j + H / 2])
                o = np.array([W, H]) / 2 - A @ centre + rng.uniform(-0.5, 0.5, 2)
                images.append(SimpleNamespace(H=H, W=W, band=int(b), sky=float(np.float32(rng.uniform(50, 200))),
                                              iota=float(np.float32(rng.uniform(100, 300))),
                                              wcs=np.concatenate([A.reshape(-1), o]), psf=_psf(rng)))
    edge = min(20.0, 0.25 * min(W, H)) if S > 1 else 0.48 * min(W, H)
    u = rng.uniform(edge, extent - 1 - edge, (S, 2))
    gal = rng.random(S) < 0.6
    log_r, colour = rng.normal(PRIORS[1], math.sqrt(PRIORS[2]), S), rng.normal(0.0, math.sqrt(PRIORS[4]), (S, 4))
    shape = np.stack([rng.uniform(0, 1, S), rng.uniform(0.3, 1, S), rng.uniform(0, np.pi, S), rng.uniform(0.5, 4, S)], -1)
    if case["wide"]:
        ext = rng.random(S) < 0.02
        shape[ext, 3] = rng.uniform(4, 8, int(ext.sum()))
    flux = np.exp(log_r[:, None] + colour @ COLOUR_MIX.T)

    logit = lambda p: np.log(p) - np.log1p(-p)
    th = np.zeros((S, 27))
    th[:, 0:2] = u + rng.uniform(-0.5, 0.5, (S, 2))
    th[:, 2] = np.where(gal, logit(np.clip(shape[:, 0] + rng.normal(0, 0.1, S), 0.05, 0.95)), 0.0)
    th[:, 3] = np.where(gal, logit(np.clip(shape[:, 1] + rng.normal(0, 0.05, S), 0.1, 0.95)), logit(0.7))
    th[:, 4] = np.where(gal, shape[:, 2] + rng.normal(0, 0.1, S), rng.uniform(0, np.pi, S))
    th[:, 5] = np.where(gal, np.log(shape[:, 3]) + rng.normal(0, 0.1, S), 0.0)
    th[:, 7] = th[:, 9] = log_r + rng.normal(0, 0.2, S)
    th[:, 11:15] = th[:, 19:23] = colour + rng.normal(0, 0.1, (S, 4))
    th[:, [8, 10]] = th[:, 15:19] = th[:, 23:27] = 0.0
    th[:, [8, 10] + list(range(15, 19)) + list(range(23, 27))] = math.log(0.01)

    # patch radius: where the profile in the brightest exposure falls under half the sky noise; on wide
    # patches at least 4 sigma of the widest component
    radius, pixels = np.full(S, float(case["rmin"])), []
    gen = torch.Generator(device=device).manual_seed(int(rng.integers(1 << 62)))
    for im in images:
        pos = u @ im.wcs[:4].reshape(2, 2).T + im.wcs[4:]
        near = ((pos > -64) & (pos < [im.W + 63, im.H + 63])).all(1)
        rate = _render(im, pos[near], gal[near], shape[near], flux[near, im.band], device)
        pixels.append(torch.poisson(rate, generator=gen).float())
        seen = ((pos >= 0) & (pos <= [im.W - 1, im.H - 1])).all(1)
        w, _, cov = _psf_at(im, pos)
        s2 = (w * 0.5 * (cov[..., 0] + cov[..., 2])).sum(-1) + np.where(gal, shape[:, 3] ** 2, 0.0)
        arg = im.iota * flux[:, im.band] / (np.pi * s2 * math.sqrt(im.sky))
        r = np.sqrt(2 * s2 * np.log(np.maximum(arg, 1.0)))
        if case["wide"]:
            r = np.maximum(r, 4 * np.sqrt(cov[..., [0, 2]].max((1, 2)) + np.where(gal, TAU.max() * shape[:, 3] ** 2, 0.0)))
        radius = np.where(seen, np.maximum(radius, r), radius)
    return SimpleNamespace(images=images, u0=th[:, 0:2].copy(), theta0=th, priors=PRIORS, exp_nu=EXP_NU, exp_tau=EXP_TAU,
                           dev_nu=DEV_NU, dev_tau=DEV_TAU, pixels=pixels,
                           radius=np.clip(np.ceil(radius), case["rmin"], case["rmax"]).astype(np.int32))


def _patches(n, seed, device):
    """Network inputs with the values that patch extraction gives (noise of unit scale, a bright centre)."""
    gen = torch.Generator(device=device).manual_seed(seed)
    ax = torch.arange(32, device=device, dtype=torch.float32) - 16
    r2 = ax[:, None] ** 2 + ax[None, :] ** 2
    x = torch.randn(n, 32, 32, 5, device=device, generator=gen, dtype=torch.float32)
    peak = torch.exp(3 * torch.randn(n, 1, 1, 5, device=device, generator=gen, dtype=torch.float32).clamp(-2, 2))
    wid = 1.0 + 3.0 * torch.rand(n, 1, 1, 1, device=device, generator=gen, dtype=torch.float32)
    x = torch.asinh(x + peak * torch.exp(-0.5 * r2[None, :, :, None] / wid ** 2))
    return x.to(torch.bfloat16).view(torch.int16).contiguous()


def _network(seed, device):
    """A network as in the middle of training: weights, biases and moments away from zero."""
    net = cnn.WarmStartCNN(device, seed=seed % (1 << 31))
    gen = torch.Generator(device=device).manual_seed(seed + 1)
    rand = lambda: torch.randn(net.n, device=device, generator=gen, dtype=torch.float32)
    net.params += 0.02 * rand()
    net.params_bf16.copy_(net.params.to(torch.bfloat16).view(torch.int16))
    net.m.copy_(1e-3 * rand())
    net.v.copy_(1e-4 * (1.0 + rand().abs()))
    net.step = 100
    return net


# --------------------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    device = torch.device("cuda")
    kind = case["kind"]
    if kind in ("predict", "train"):
        st = SimpleNamespace(kind=kind, net=_network(seed, device), x=_patches(case["patches"], seed + 2, device))
        if kind == "predict":
            gen = torch.Generator(device=device).manual_seed(seed + 3)
            st.net.set_standardisation(torch.randn(512, 27, device=device, generator=gen, dtype=torch.float32) - 1.0)
        else:
            gen = torch.Generator(device=device).manual_seed(seed + 3)
            st.target = torch.randn(case["patches"], 27, device=device, generator=gen, dtype=torch.float32)
        return st
    scene = _make_survey(case, seed, device)
    prob = celeste.Problem(scene, device=device, tile_pixels=case["tile"], hessian_mode=case["hessian"],
                           device_pixels=scene.pixels)
    theta0 = torch.as_tensor(scene.theta0, device=device).contiguous()
    st = SimpleNamespace(kind=kind, prob=prob, theta0=theta0, theta=theta0.clone(),
                         delta=torch.zeros(len(theta0), dtype=torch.float64, device=device))
    if kind != "joint":
        prob.render_background(theta0)
    if kind == "covariance":     # the converged catalog
        prob.newton_batch(st.theta)
    if kind == "joint":
        st.theta0, _ = block_coordinate(prob, theta0, passes=2, mode=celeste.NBR_WINDOW)
        st.theta0 = st.theta0.contiguous()
        prob.joint_value(st.theta0)   # binds the joint workspace
    if kind == "pass":
        # a network that predicts near the usual log variances and an undecided type
        st.net = _network(seed + 5, device)
        targets = torch.zeros(2, 27, device=device, dtype=torch.float32)
        targets[:, [8, 10] + list(range(15, 19)) + list(range(23, 27))] = -4.0
        st.net.set_standardisation(targets + torch.tensor([[-0.3], [0.3]], device=device))
    return st


def run(st):
    if st.kind == "predict":
        return st.net.predict(st.x)
    if st.kind == "train":
        net = st.net
        y = net.forward(st.x)
        loss, dy = net.mse(y, st.target)
        net.grad.zero_()
        net.backward(st.x, dy)
        net.adamw(1e-3)
        return {"y": y, "loss": loss, "dy": dy, "grad": net.grad, "params": net.params,
                "params_bf16": net.params_bf16.view(torch.bfloat16), "m": net.m, "v": net.v}
    prob = st.prob
    if st.kind == "elbo":
        elbo, grad, hess = prob.elbo_batch(st.theta0)
        return {"elbo": elbo, "grad": grad, "hess": hess}
    if st.kind == "value":
        return {"elbo": prob.elbo_batch(st.theta0, want=celeste.WANT_ELBO)[0]}
    if st.kind == "background":
        # the background is kept inside the problem; the values under it are how a program sees it
        prob.render_background(st.theta0)
        return {"elbo": prob.elbo_batch(st.theta0, want=celeste.WANT_ELBO)[0]}
    if st.kind == "covariance":
        cov, ok = prob.covariance(st.theta)
        return {"cov": cov, "ok": ok}
    st.theta.copy_(st.theta0)
    if st.kind == "joint":
        out = prob.joint_newton(st.theta, max_iter=30)
        return {"theta": st.theta, **out}
    if st.kind == "pass":
        prob.refresh_pixels()
        prob.render_background(st.theta0)
        st.theta.copy_(cnn.warm_start(st.theta0, st.net.predict(prob.extract_patches())))
    else:
        prob.render_background(st.theta0)
    st.delta.zero_()
    delta, iters, status, elbo = prob.newton_batch(st.theta, st.delta)
    return {"theta": st.theta, "delta": delta, "iters": iters, "status": status, "elbo": elbo}


# ------------------------------------------------------------------------------------------ cost of a pass
def work(case):
    kind = case["kind"]
    if kind == "predict":
        n = case["patches"]
        return {"bytes": n * (32 * 32 * 5 * 2 + 27 * 4) + 4 * CNN_PARAMS, "flops": 2 * CNN_MACS * n}
    if kind == "train":
        n = case["patches"]
        # forward, input gradients (none for the first layer), weight gradients; the activations stay on chip at best
        return {"bytes": n * (32 * 32 * 5 * 2 + 4 * 27 * 4) + 30 * CNN_PARAMS,
                "flops": 2 * n * (3 * CNN_MACS - 1024 * 32 * 45)}
    S = case["sources"]
    side = 2 * min(case["rmax"], max(case["rmin"], 23 if case["wide"] else 9)) + 1
    bands = 0.5 * (case["bands_min"] + case["bands_max"])
    px = S * bands * (1.5 if case["fields_x"] * case["fields_y"] > 1 else 1.0) * side * side
    dense = S * side * side / (case["width"] * case["height"] * case["fields_x"] * case["fields_y"])
    moments = 16 * px                       # each pixel's count and fixed terms
    if kind == "elbo":
        return {"bytes": moments + S * 8 * (27 + 1 + 27 + 729), "flops": px * FLOPS_FULL}
    if kind == "value":
        return {"bytes": moments + S * 8 * 28, "flops": px * FLOPS_VALUE}
    if kind == "background":
        return {"bytes": 2 * moments + S * 8 * 28, "flops": px * FLOPS_VALUE * (1 + 4 * dense)}
    if kind == "covariance":
        return {"bytes": moments + S * 8 * (27 + 729), "flops": px * FLOPS_FULL + S * 3 * 27 ** 3}
    # iterative solves: one read of the inputs and one write of the catalog; the iterations' arithmetic
    iters = {"joint": 12, "pass": 14}.get(kind, 17)
    return {"bytes": 2 * moments + S * 8 * 60, "flops": px * (iters * (FLOPS_FULL + FLOPS_VALUE) + FLOPS_VALUE * 4 * dense)}


# --------------------------------------------------------------------------------- the same in 64 bits
def _exact_network(case, seed, device):
    net, x = _network(seed, device), _patches(case["patches"], seed + 2, device)
    x = x.view(torch.bfloat16).double().permute(0, 3, 1, 2)
    shapes = [(32, 3, 3, 5), (64, 3, 3, 32), (64, 3, 3, 64), (64, 3, 3, 64), (256, 1024), (27, 256)]
    weights = net.params_bf16.view(torch.bfloat16).double()
    # weights enter as their BF16 copies, biases in FP32
    p = net.params.double()
    at, views = 0, []
    for s in shapes:
        n = int(np.prod(s))
        p[at:at + n] = weights[at:at + n]
        views.append((at, n, s))
        at += n + s[0]
    p.requires_grad_(case["kind"] == "train")

    def forward(x):
        for k, (a, n, s) in enumerate(views):
            w, b = p[a:a + n].view(s), p[a + n:a + n + s[0]]
            if len(s) == 4:
                x = torch.nn.functional.conv2d(x, w.permute(0, 3, 1, 2), b, stride=1 if k == 0 else 2, padding=1)
            else:
                if k == 4:
                    x = x.permute(0, 2, 3, 1).reshape(len(x), 1024)
                x = x @ w.T + b
            if k < 5:
                x = torch.relu(x)
        return x

    return net, p, forward, x


def _exact_predict(case, seed, device):
    net, _, forward, x = _exact_network(case, seed, device)
    gen = torch.Generator(device=device).manual_seed(seed + 3)
    targets = torch.randn(512, 27, device=device, generator=gen, dtype=torch.float32) - 1.0
    mu, sd = targets.mean(0).double(), targets.std(0).clamp_min(1e-3).double()
    with torch.no_grad():
        return torch.cat([forward(x[i:i + 1024]) for i in range(0, len(x), 1024)]) * sd + mu


def _exact_train(case, seed, device):
    net, p, forward, x = _exact_network(case, seed, device)
    gen = torch.Generator(device=device).manual_seed(seed + 3)
    target = torch.randn(case["patches"], 27, device=device, generator=gen, dtype=torch.float32).double()
    y = forward(x)
    loss = ((y - target) ** 2).mean()
    dy, g = torch.autograd.grad(loss, (y, p))
    m, v = 0.9 * net.m.double() + 0.1 * g, 0.999 * net.v.double() + 0.001 * g * g
    step = 101
    new = net.params.double() * (1 - 1e-3 * 1e-4) - 1e-3 * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return {"y": y.detach(), "loss": loss.detach().view(1), "dy": dy, "grad": g, "params": new, "params_bf16": new, "m": m,
            "v": v}


class _Exposure:
    """The patches of one exposure in 64 bits: which sources it holds, their windows, PSFs and neighbours."""

    def __init__(self, scene, im, device):
        A, o = im.wcs[:4].reshape(2, 2), im.wcs[4:]
        pos = scene.u0 @ A.T + o
        c = np.floor(pos + 0.5)
        self.src = np.nonzero(((c >= 0) & (c <= [im.W - 1, im.H - 1])).all(1))[0]
        R, c = scene.radius[self.src][:, None], c[self.src]
        self.lo = np.maximum(c - R, 0).astype(np.int64)
        self.hi = np.minimum(c + R, [im.W - 1, im.H - 1]).astype(np.int64) + 1
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=device, dtype=torch.float64)
        self.w, self.mean, self.cov = (t(a) for a in _psf_at(im, pos[self.src]))
        self.A, self.o, self.im = t(A), t(o), im
        self.src_t = torch.as_tensor(self.src, device=device)
        self.tau, self.mix, self.device = t(TAU), t(COLOUR_MIX[im.band]), device
        self.nu_e, self.nu_d = t(EXP_NU), t(DEV_NU)

    def neighbours(self, p):
        hit = ((self.lo < self.hi[p]) & (self.hi > self.lo[p])).all(1)
        hit[p] = False
        return np.nonzero(hit)[0]

    def moments(self, theta, patch, X, Y):
        """E[G] and Var[G] of the patches' sources at pixels (X, Y) of the exposure, one patch per pixel."""
        used, at = torch.unique(patch, return_inverse=True)
        th = theta[self.src_t[used]]
        pos = th[:, 0:2] @ self.A.T + self.o
        e, q2, sc = torch.sigmoid(th[:, 2]), torch.sigmoid(th[:, 3]) ** 2, torch.exp(2 * th[:, 5])
        c, s = torch.cos(th[:, 4]), torch.sin(th[:, 4])
        g00, g01, g11 = sc * (c * c + q2 * s * s), sc * (1 - q2) * c * s, sc * (s * s + q2 * c * c)
        a, b, cc, d = self.A[0, 0], self.A[0, 1], self.A[1, 0], self.A[1, 1]
        h00 = a * (a * g00 + b * g01) + b * (a * g01 + b * g11)
        h01 = cc * (a * g00 + b * g01) + d * (a * g01 + b * g11)
        h11 = cc * (cc * g00 + d * g01) + d * (cc * g01 + d * g11)
        cov = self.cov[used]
        dx = X[:, None] - pos[at, 0, None] - self.mean[used][at][:, :, 0]
        dy = Y[:, None] - pos[at, 1, None] - self.mean[used][at][:, :, 1]

        def density(s00, s01, s11, weight, dx, dy):
            det = s00 * s11 - s01 * s01
            n, r = weight / (2 * math.pi * torch.sqrt(det)), -0.5 / det
            p00, p01, p11 = (s11 * r)[at], (-2 * s01 * r)[at], (s00 * r)[at]
            return n[at] * torch.exp((p00 * dx + p01 * dy) * dx + p11 * dy * dy)

        f0 = density(cov[..., 0], cov[..., 1], cov[..., 2], self.w[used], dx, dy).sum(1)
        nu = torch.cat([(1 - e)[:, None] * self.nu_e, e[:, None] * self.nu_d], 1)
        grow = lambda k, h: cov[:, :, None, k] + self.tau * h[:, None, None]
        f1 = density(grow(0, h00), grow(1, h01), grow(2, h11), self.w[used][:, :, None] * nu[:, None, :], dx[:, :, None],
                     dy[:, :, None]).sum((1, 2))
        L1, L2 = [], []
        for r, rho, col, gam in ((7, 8, 11, 15), (9, 10, 19, 23)):
            m = th[:, r] + th[:, col:col + 4] @ self.mix
            v = torch.exp(th[:, rho]) + torch.exp(th[:, gam:gam + 4]) @ (self.mix * self.mix)
            L1.append(torch.exp(m + 0.5 * v)[at])
            L2.append(torch.exp(2 * m + 2 * v)[at])
        a1 = torch.sigmoid(th[:, 6])[at]
        a0 = torch.sigmoid(-th[:, 6])[at]
        EG = a0 * L1[0] * f0 + a1 * L1[1] * f1
        return EG, a0 * L2[0] * f0 * f0 + a1 * L2[1] * f1 * f1 - EG * EG

    def pixels_of(self, patches, within=None):
        """Pixels of the patches (or of `within`'s windows, one per patch): index into the list, X, Y."""
        own = patches if within is None else within
        parts = [np.meshgrid(np.arange(self.lo[w, 0], self.hi[w, 0]), np.arange(self.lo[w, 1], self.hi[w, 1])) for w in own]
        n = [p[0].size for p in parts]
        t = lambda a: torch.as_tensor(a, device=self.device)
        return (t(np.repeat(np.arange(len(own)), n)), t(np.concatenate([p[0].reshape(-1) for p in parts])),
                t(np.concatenate([p[1].reshape(-1) for p in parts])))


def _kl(theta):
    phi, mu_r, var_r, mu_c, var_c = PRIORS
    normal = lambda m, lv, mu, s2: 0.5 * (math.log(s2) - lv + (torch.exp(lv) + (m - mu) ** 2) / s2 - 1.0)
    la1, la0 = torch.nn.functional.logsigmoid(theta[:, 6]), torch.nn.functional.logsigmoid(-theta[:, 6])
    kl = torch.exp(la1) * (la1 - math.log(phi)) + torch.exp(la0) * (la0 - math.log1p(-phi))
    for la, r, rho, col, gam in ((la0, 7, 8, 11, 15), (la1, 9, 10, 19, 23)):
        k = normal(theta[:, r], theta[:, rho], mu_r, var_r) + normal(theta[:, col:col + 4], theta[:, gam:gam + 4], mu_c, var_c).sum(1)
        kl = kl + torch.exp(la) * k
    return kl


def _derivatives(f, theta, order):
    """Per-source value, gradient and Hessian of f(theta) = sum_s f_s(theta_s): [S] values first."""
    th = theta.clone().requires_grad_(order > 0)
    v = f(th)
    if order == 0:
        return v.detach(), None, None
    (g,) = torch.autograd.grad(v.sum(), th, create_graph=order > 1)
    if order == 1:
        return v.detach(), g, None
    rows = [torch.autograd.grad(g[:, j].sum(), th, retain_graph=True, allow_unused=True)[0] for j in range(27)]
    return v.detach(), g.detach(), torch.stack([torch.zeros_like(th) if r is None else r for r in rows], 1)


def _exact_elbo(case, seed, device, order):
    scene = _make_survey(case, seed, device)
    theta = torch.as_tensor(scene.theta0, device=device)
    S = len(theta)
    L, g, H = _derivatives(lambda th: -_kl(th), theta, order)
    for im, pix in zip(scene.images, scene.pixels):
        ex = _Exposure(scene, im, device)
        if not len(ex.src):
            continue
        area = np.prod(ex.hi - ex.lo, axis=1)
        group = np.cumsum(area) // 65536
        for k in np.unique(group):
            patches = np.nonzero(group == k)[0]
            at, X, Y = ex.pixels_of(patches)
            bE, bV = torch.full_like(X, 0, dtype=torch.float64), torch.full_like(X, 0, dtype=torch.float64)
            start = np.concatenate([[0], np.cumsum(area[patches])])
            pairs = [(i, q) for i, p in enumerate(patches) for q in ex.neighbours(p)]
            for c in range(0, len(pairs), 128):
                part = pairs[c:c + 128]
                who, nX, nY = ex.pixels_of(None, [patches[i] for i, _ in part])
                nbr = torch.as_tensor([int(q) for _, q in part], device=device)[who]
                with torch.no_grad():
                    EG, VG = ex.moments(theta, nbr, nX.double(), nY.double())
                dest = torch.as_tensor(np.concatenate([np.arange(start[i], start[i + 1]) for i, _ in part]), device=device)
                bE.index_add_(0, dest, EG)
                bV.index_add_(0, dest, VG)
            x = pix[Y, X].double()
            own = torch.as_tensor(patches, device=device)[at]
            src = ex.src_t[own]

            def f(th):
                EG, VG = ex.moments(th, own, X.double(), Y.double())
                E, V = im.sky + im.iota * (bE + EG), im.iota ** 2 * (bV + VG)
                ell = x * (torch.log(E) - V / (2 * E * E)) - E - torch.lgamma(x + 1)
                return torch.zeros(S, dtype=torch.float64, device=device).index_add(0, src, ell)

            l1, g1, H1 = _derivatives(f, theta, order)
            L = L + l1
            g = g if g is None else g + g1
            H = H if H is None else H + H1
    return L, g, H


def exact(case, seed):
    device, kind = torch.device("cuda"), case["kind"]
    if kind == "predict":
        return _exact_predict(case, seed, device)
    if kind == "train":
        return _exact_train(case, seed, device)
    if kind not in ("elbo", "value", "background"):
        return None     # the end of an iteration, or functions of one: no value that plain arithmetic gives
    px = work(dict(case, kind="value"))["flops"] / FLOPS_VALUE
    order = 0 if kind != "elbo" else (2 if px <= 4e5 else 1)   # the Hessian within 20 s
    elbo, grad, hess = _exact_elbo(case, seed, device, order)
    return {"elbo": elbo, "grad": grad, "hess": hess} if kind == "elbo" else {"elbo": elbo}
