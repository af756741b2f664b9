"""What a program that catalogs a region of sky asks of this library, one pass at a time.

A case is a region (its layout, sources and images), the call made on it and the pixel
precision.  The inputs are the package's synthetic SDSS-shaped draws; the problem handle
is made once and kept, as a fitting program keeps it while it moves the parameters.

A single-precision call (FP32 pixels) accumulates into 64-bit buffers, but its values
carry single precision; the program that asks for it goes on in single precision, so
its results are returned as float32.  Positions stay 64-bit (thousands of pixels to 1e-3).
"""
import math

import numpy as np
import torch

from paper_1801_10277_gb300 import autograd
from paper_1801_10277_gb300 import celeste as cel
from paper_1801_10277_gb300 import synth

# ---------------------------------------------------------------------------------
# the cases


def listed():
    return [
        # the smallest call: one blended pair (a star on a galaxy), 48 x 48 pixels in five
        # bands, as an interactive deblend or the innermost call of another optimiser
        dict(name="pair_grad", layout="pair", call="grad", fp32=True, side=48, n_src=2),
        # a crowded 256 x 256 region, every source overlapping 2 to 12 others: one value and
        # gradient through the differentiable function (forward, then backward)
        dict(name="crowded_autograd", layout="crowded", call="autograd", fp32=True, side=256, n_src=64),
        # the same region's value and gradient in one call: a region task's optimiser step
        dict(name="crowded_grad", layout="crowded", call="grad", fp32=True, side=256, n_src=64),
        # one survey field (five bands of 2048 x 1489, 500 sources): the benchmark's step
        dict(name="field_grad", layout="field", call="grad", fp32=True, width=2048, height=1489, n_src=500,
             bright=0.0),
        # the same through the host arrays of the C interface, as a program without torch calls it
        dict(name="field_grad_host", layout="field", call="host_grad", fp32=True, width=2048, height=1489,
             n_src=500, bright=0.0),
        # a dense field with bright sources (patches up to 101 pixels): the largest evaluation
        dict(name="dense_grad", layout="field", call="grad", fp32=True, width=2048, height=1489, n_src=3125,
             bright=0.1),
        # a repeatedly imaged piece of sky: many small patches per source, a map per patch
        dict(name="stack_grad", layout="stack", call="grad", fp32=True, side=400, n_src=100, epochs=16),
        # the field in double precision: the reference evaluation a fit's polish ends on
        dict(name="field_grad_fp64", layout="field", call="grad", fp32=False, width=2048, height=1489, n_src=500,
             bright=0.0),
        # every source's 44 x 44 Hessian with the gradient: the input of a Newton step and of
        # the curvature-based uncertainties, in single and in double precision
        dict(name="field_hess", layout="field", call="hess", fp32=True, width=2048, height=1489, n_src=500,
             bright=0.0),
        dict(name="crowded_hess_fp64", layout="crowded", call="hess", fp32=False, side=256, n_src=64),
        # block-coordinate Newton, two double-precision iterations per source from a rough
        # start: the refresh of a crowded region's catalog, and what a fit's polish is made of
        dict(name="crowded_fit", layout="crowded", call="fit", fp32=False, side=256, n_src=64, iters=2),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    layout = rng.choice(["pair", "crowded", "field", "field", "field", "stack"])
    call = rng.choice(["grad", "grad", "elbo", "autograd", "host_grad", "hess", "fit"])
    fp32 = call != "fit" and rng.random() < 0.7
    c = dict(layout=layout, call=call, fp32=fp32)
    if call == "fit":
        c["iters"] = rng.randint(1, 2)
    if layout == "pair":
        c.update(side=rng.randint(33, 120), n_src=2)
    elif layout == "crowded":
        c.update(side=rng.randint(200, 300), n_src=log_int(24, 64))
    elif layout == "field":
        heavy = not fp32 or call == "fit"
        c.update(width=log_int(120, 2048), height=log_int(120, 1489), bright=rng.choice([0.0, 0.1]))
        room = c["width"] * c["height"] / 1000.0    # a dense field holds a source per 1000 pixels
        c["n_src"] = log_int(3, max(4, min(300 if heavy else 2500, room)))
    else:
        c.update(side=rng.randint(150, 400), epochs=log_int(2, 16))
        c["n_src"] = log_int(4, 24 if not fp32 else 100)
    if layout != "stack":
        c["n_psf"] = rng.choice([3, 3, 2, 1])
        c["sky_map"] = rng.random() < 0.25
    return c


# ---------------------------------------------------------------------------------
# inputs


def _sources_in_field(rng, c):
    truth, is_gal = synth.draw_truth(rng, c["n_src"], bright_frac=c["bright"])
    truth[:, 0] = rng.uniform(0, c["width"] - 1, size=c["n_src"])
    truth[:, 1] = rng.uniform(0, c["height"] - 1, size=c["n_src"])
    return truth, is_gal


def _sources_in_pair(rng, c):
    truth, _ = synth.draw_truth(rng, 2)
    s = c["side"]
    truth[:, 0:2] = np.array([[0.45, 0.5], [0.58, 0.52]]) * s + rng.uniform(-1, 1, size=(2, 2))
    truth[:, synth.I_R1:synth.I_R1 + 2] = rng.uniform(math.log(10.0), math.log(40.0), size=(2, 1))
    truth[:, synth.I_A] = [1.0, 0.0]
    truth[:, synth.I_A + 1] = [0.0, 1.0]
    return truth, np.array([False, True])


def _sources_in_crowd(rng, c):
    """Clusters of overlapping sources."""
    s, n = c["side"], c["n_src"]
    truth, is_gal = synth.draw_truth(rng, n)
    centres = rng.uniform(0.12 * s, 0.88 * s, size=(12, 2))
    at = centres[rng.integers(12, size=n)] + rng.normal(0, 0.09 * s, size=(n, 2))
    truth[:, 0:2] = np.clip(at, 2, s - 3)
    return truth, is_gal


def _stack_images(rng, c):
    """Epochs of the same sky, each with its own pointing, rotation, scale, PSF, sky,
    calibration and smooth distortion."""
    images, mid, s = [], c["side"] / 2.0 - 8, c["side"]
    for _ in range(c["epochs"]):
        A = (1.0 + rng.normal(0, 3e-3)) * synth._rot(rng.normal(0, 1e-2))
        t = np.array([s / 2.0, s / 2.0]) + rng.uniform(-8, 8, size=2) - A @ np.array([mid, mid])
        wcs = np.array([A[0, 0], A[0, 1], A[1, 0], A[1, 1], t[0], t[1]])
        warp = (mid, mid, mid, *rng.normal(0, 0.3, size=4))
        for b in range(synth.NBANDS):
            images.append(synth.Image(band=b, pixels=np.zeros((s, s), np.float32), sky=rng.uniform(100, 200),
                                      calib=rng.uniform(0.004, 0.006), wcs=wcs.copy(), psf=synth.draw_psf(rng),
                                      warp=warp))
    return images


def _observe(rng, images, truth, is_gal, with_sky_map):
    """Poisson counts around the sky and one round blob per source, drawn on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 62)))
    for im in images:
        H, W = im.height, im.width
        rate = np.full((H, W), im.sky, np.float32)
        if with_sky_map:
            gx, gy = rng.uniform(0, 15, size=2)
            rate += (gx * np.linspace(0, 1, W)[None, :] + gy * np.linspace(0, 1, H)[:, None]).astype(np.float32)
            im.sky_map = rate.copy()
        for s in range(truth.shape[0]):
            lf = synth.band_log_flux(truth[s, synth.I_R1], truth[s, synth.I_C1:synth.I_C1 + 4])[im.band]
            v = synth._blob_var(im.psf, bool(is_gal[s]), truth[s, synth.I_SCALE])
            px, py = synth.pixel_position_full(im, truth[s, 0:2])
            rad = int(math.ceil(5 * math.sqrt(v)))
            x0, x1 = max(0, int(px) - rad), min(W, int(px) + rad + 1)
            y0, y1 = max(0, int(py) - rad), min(H, int(py) + rad + 1)
            if x0 < x1 and y0 < y1:
                peak = math.exp(lf) / im.calib / (2 * math.pi * v)
                rate[y0:y1, x0:x1] += peak * np.outer(np.exp(-(np.arange(y0, y1) - py) ** 2 / (2 * v)),
                                                      np.exp(-(np.arange(x0, x1) - px) ** 2 / (2 * v)))
        im.pixels = torch.poisson(torch.from_numpy(rate).cuda(), generator=gen).cpu().numpy()


def _region(case, seed, observed=True):
    """The synthetic region of a case: images, priors, start, patches, neighbours."""
    c, rng = case, np.random.default_rng(seed)
    if c["layout"] == "stack":
        images = _stack_images(rng, c)
        truth, is_gal = synth.draw_truth(rng, c["n_src"])
        truth[:, 0:2] = rng.uniform(12, c["side"] - 28, size=(c["n_src"], 2))
    else:
        H, W = c.get("height", c.get("side")), c.get("width", c.get("side"))
        images = synth._single_field_images(rng, H, W)
        for im in images:
            im.psf = synth.draw_psf(rng, k=c.get("n_psf", 3))
        place = dict(pair=_sources_in_pair, crowded=_sources_in_crowd, field=_sources_in_field)[c["layout"]]
        truth, is_gal = place(rng, c)
    theta = synth.perturb_start(rng, truth, is_gal)
    if observed:
        _observe(rng, images, truth, is_gal, bool(c.get("sky_map")))
    exp_mix, dev_mix = synth.load_profiles()
    prior_star, prior_r, prior_c = synth.draw_priors(rng)
    po, pa = synth.make_patches(images, theta, is_gal)
    no, nb = synth.make_neighbours(truth.shape[0], po, pa) if observed else (None, None)
    pw = None
    if images[0].warp is not None:
        owner = np.repeat(np.arange(truth.shape[0]), np.diff(po))
        pw = np.stack([synth.linearised_wcs(images[int(pa[p, 0])], theta[owner[p], 0:2]) for p in range(len(pa))])
    return synth.Problem(images=images, exp_mix=exp_mix, dev_mix=dev_mix, prior_star=prior_star, prior_r=prior_r,
                         prior_c=prior_c, theta=theta, truth=truth, patch_offsets=po, patches=pa, nbr_offsets=no,
                         nbrs=nb, patch_wcs=pw)


def prepare(case, seed):
    region = _region(case, seed)
    n, f64 = region.n_src, dict(dtype=torch.float64, device="cuda")
    s = dict(case=case, problem=cel.Problem(region), theta=region.theta,
             precision=cel.FP32 if case["fp32"] else cel.FP64)
    if case["call"] in ("grad", "elbo", "hess", "autograd"):
        s["d_theta"] = torch.from_numpy(region.theta).cuda()
    if case["call"] in ("grad", "elbo"):
        # total, every source's own objective and the gradient, in one buffer
        s["out"] = torch.zeros(1 + n + n * cel.NPARAM, **f64)
        s["total"], s["local"] = s["out"][:1], s["out"][1:1 + n]
        s["grad"] = s["out"][1 + n:].view(n, cel.NPARAM)
    if case["call"] == "hess":
        s["out"] = torch.zeros(n * (1 + cel.NPARAM + cel.NPARAM ** 2), **f64)
        s["local"] = s["out"][:n]
        s["grad"] = s["out"][n:n + n * cel.NPARAM].view(n, cel.NPARAM)
        s["hess"] = s["out"][n + n * cel.NPARAM:].view(n, cel.NPARAM, cel.NPARAM)
    if case["call"] == "autograd":
        s["d_theta"].requires_grad_(True)
    return s


# ---------------------------------------------------------------------------------
# one pass


def _views(flat, n, keys):
    """The named parts of a flat result (see prepare)."""
    size = dict(total=(1,), local=(n,), grad=(n, cel.NPARAM), hess=(n, cel.NPARAM, cel.NPARAM))
    out, at = {}, 0
    for k in keys:
        m = math.prod(size[k])
        out[k] = flat[at:at + m].view(size[k])
        at += m
    return out


def run(state):
    s, p, prec = state, state["problem"], state["precision"]
    call, n = s["case"]["call"], state["problem"].n_src
    single = prec == cel.FP32
    if call == "grad":
        p.elbo_grad_device(s["d_theta"], s["total"], s["local"], s["grad"], precision=prec)
        return _views(s["out"].float() if single else s["out"], n, ("total", "local", "grad"))
    if call == "elbo":
        p.elbo_device(s["d_theta"], s["total"], s["local"], precision=prec)
        out = s["out"][:1 + n]
        return _views(out.float() if single else out, n, ("total", "local"))
    if call == "hess":
        p.hess_device(s["d_theta"], s["local"], s["grad"], s["hess"], precision=prec)
        return _views(s["out"].float() if single else s["out"], n, ("local", "grad", "hess"))
    if call == "autograd":
        s["d_theta"].grad = None
        total = autograd.elbo(s["d_theta"], p, prec)
        total.backward()
        total, grad = total.detach(), s["d_theta"].grad
        return dict(total=total.float() if single else total, grad=grad.float() if single else grad)
    if call == "host_grad":
        total, local, grad = p.elbo_grad(s["theta"], precision=prec)
        kind = np.float32 if single else np.float64
        return dict(total=kind(total), local=local.astype(kind, copy=False), grad=grad.astype(kind, copy=False))
    theta, iters, status, total = p.fit(s["theta"], precision=prec, max_iter=s["case"]["iters"], max_sweeps=1)
    return dict(theta=theta, iters=iters, status=status, total=total)


def work(case):
    """Operations counted from the formulas: per source-pixel (a pixel of a source's patch),
    3 PSF components x 14 profile components give 1,113 for the value and gradient (305 for
    the value alone) and 4,870 with the Hessian.  Bytes: each source-pixel's count once,
    the parameters in, the results out."""
    region = _region(case, 0, observed=False)
    px = float(np.sum(region.patches[:, 3].astype(np.int64) * region.patches[:, 4]))
    n, call = case["n_src"], case["call"]
    size = 4 if case["fp32"] else 8
    flops = dict(elbo=305, hess=4870, fit=4870 * case.get("iters", 1)).get(call, 1113) * px
    results = dict(elbo=1, hess=45 + 44 * 44, fit=44).get(call, 45) * n * size
    return dict(flops=flops, bytes=4 * px + 8 * 44 * n + results)


# ---------------------------------------------------------------------------------
# the same in plain torch, 64 bits


_BETA = ((-1, -1, 0, 0), (0, -1, 0, 0), (0, 0, 0, 0), (0, 0, 1, 0), (0, 0, 1, 1))


class _Plain:
    """ELBO = sum over covered pixels of x (log E - V / (2 E^2)) - E  -  sum_s KL_s, with
    E = sky + sum_s E_s, V = sum_s (E[F_s^2] - E_s^2); written out with autograd tensors."""

    def __init__(self, r):
        f64 = dict(dtype=torch.float64, device="cuda")
        self.r, self.theta = r, torch.from_numpy(r.theta).cuda()
        pa = r.patches.astype(np.int64)
        self.size = pa[:, 3] * pa[:, 4]
        self.owner = torch.from_numpy(np.repeat(np.arange(r.n_src), np.diff(r.patch_offsets))).cuda()
        self.pa = torch.from_numpy(pa).cuda()
        start = np.concatenate([[0], np.cumsum([im.height * im.width for im in r.images])])
        self.start, self.wide = torch.from_numpy(start).cuda(), torch.tensor([im.width for im in r.images]).cuda()
        self.x = torch.cat([torch.from_numpy(im.pixels).reshape(-1) for im in r.images]).cuda()
        self.sky = torch.cat([torch.full((im.height * im.width,), im.sky, dtype=torch.float64) if im.sky_map is None
                              else torch.from_numpy(im.sky_map).double().reshape(-1) for im in r.images]).cuda()
        self.band = torch.tensor([im.band for im in r.images]).cuda()
        self.iota = torch.tensor([1.0 / im.calib for im in r.images], **f64)
        k = max(im.psf.shape[0] for im in r.images)
        psf = np.zeros((len(r.images), k, 6))
        psf[:, :, 3] = psf[:, :, 5] = 1.0            # a component of weight 0 where there are fewer
        for i, im in enumerate(r.images):
            psf[i, :im.psf.shape[0]] = im.psf
        self.psf = torch.tensor(psf, **f64)
        wcs = r.patch_wcs if r.patch_wcs is not None else np.stack([r.images[i].wcs for i in pa[:, 0]])
        self.wcs = torch.tensor(wcs, **f64)
        self.mix = torch.tensor(np.concatenate([r.exp_mix, r.dev_mix]), **f64)
        self.n_exp = r.exp_mix.shape[0]
        self.beta = torch.tensor(_BETA, **f64)
        self.blocks, p = [], 0                        # runs of patches of about 2^17 pixels
        while p < len(pa):
            q = int(np.searchsorted(np.cumsum(self.size[p:]), 1 << 17)) + p + 1
            self.blocks.append((p, min(q, len(pa))))
            p = self.blocks[-1][1]

    def pixels(self, p, q):
        """Patch, position in the image and index among all pixels, of every patch pixel."""
        size = torch.from_numpy(self.size[p:q]).cuda()
        at = torch.repeat_interleave(torch.arange(p, q, device="cuda"), size)
        i = torch.arange(int(size.sum()), device="cuda") - torch.repeat_interleave(torch.cumsum(size, 0) - size, size)
        px, py = self.pa[at, 1] + i % self.pa[at, 3], self.pa[at, 2] + i // self.pa[at, 3]
        img = self.pa[at, 0]
        return at, px.double(), py.double(), self.start[img] + py * self.wide[img] + px

    def light(self, theta, p, q, at, px, py):
        """E_s and E[F_s^2] - E_s^2 of the patches' sources at their pixels."""
        th, img, w = theta[self.owner[p:q]], self.pa[p:q, 0], self.wcs[p:q]
        a = at - p
        mx = w[:, 0] * th[:, 0] + w[:, 1] * th[:, 1] + w[:, 4]
        my = w[:, 2] * th[:, 0] + w[:, 3] * th[:, 1] + w[:, 5]
        cs, sn, s2, r2 = torch.cos(th[:, 4]), torch.sin(th[:, 4]), th[:, 5] ** 2, th[:, 3] ** 2
        W = torch.stack([s2 * (cs * cs + r2 * sn * sn), s2 * (1 - r2) * cs * sn, s2 * (1 - r2) * cs * sn,
                         s2 * (sn * sn + r2 * cs * cs)], 1).view(-1, 2, 2)
        A = w[:, :4].view(-1, 2, 2)
        G = A @ W @ A.transpose(1, 2)
        psf, nu = self.psf[img], torch.cat([self.mix.new_zeros(1), self.mix[:, 1]])   # nu = 0: the star
        c = [psf[:, :, None, 3 + i] + nu * G[:, None, None, i // 2, (i + 1) // 2] for i in range(3)]
        det = c[0] * c[2] - c[1] ** 2
        edev = th[:, 2:3]
        wt = torch.cat([(1 - edev) * self.mix[:self.n_exp, 0], edev * self.mix[self.n_exp:, 0]], 1)
        amp = psf[:, :, None, 0] / (2 * math.pi * torch.sqrt(det)) * torch.cat([torch.ones_like(edev), wt], 1)[:, None]
        inv = [c[2] / det, c[1] / det, c[0] / det]
        dx = (px[:, None] - mx[a, None] - psf[a, :, 1])[:, :, None]
        dy = (py[:, None] - my[a, None] - psf[a, :, 2])[:, :, None]
        f = amp[a] * torch.exp(-0.5 * (inv[0][a] * dx * dx - 2 * inv[1][a] * dx * dy + inv[2][a] * dy * dy))
        g = [f[:, :, 0].sum(1), f[:, :, 1:].sum((1, 2))]
        e = v = 0.0
        for i in range(2):
            beta, iota = self.beta[self.band[img]], self.iota[img]
            m = th[:, 6 + i] + (beta * th[:, 10 + 4 * i:14 + 4 * i]).sum(1)
            s = th[:, 8 + i] + (beta ** 2 * th[:, 18 + 4 * i:22 + 4 * i]).sum(1)
            e = e + (th[:, 26 + i] * iota * torch.exp(m + s / 2))[a] * g[i]
            v = v + (th[:, 26 + i] * iota ** 2 * torch.exp(2 * m + 2 * s))[a] * g[i] ** 2
        return e, v - e * e

    def kl(self, th):
        r, out = self.r, 0.0
        for i, phi in enumerate((r.prior_star, 1 - r.prior_star)):
            mean, var = r.prior_r[i]
            pc = torch.from_numpy(r.prior_c[i]).to(th)
            cov = pc[:, 5:].view(-1, 4, 4)
            prec, c2, k = torch.linalg.inv(cov), th[:, 18 + 4 * i:22 + 4 * i], th[:, 28 + 8 * i:36 + 8 * i]
            d = th[:, None, 10 + 4 * i:14 + 4 * i] - pc[:, 1:5]
            kc = 0.5 * (torch.logdet(cov) - torch.log(c2).sum(1, keepdim=True) - 4
                        + torch.einsum("djj,sj->sd", prec, c2) + torch.einsum("sdj,djl,sdl->sd", d, prec, d))
            r1, r2 = th[:, 6 + i], th[:, 8 + i]
            kr = 0.5 * (math.log(var) - torch.log(r2) + (r2 + (r1 - mean) ** 2) / var - 1)
            out = out + th[:, 26 + i] * (torch.log(th[:, 26 + i] / phi) + kr
                                         + (k * (torch.log(k / pc[:, 0]) + kc)).sum(1))
        return out

    def evaluate(self, order):
        """total, local and, by `order`, the gradient (1) and the Hessians (2) of each source's
        own objective, the other sources held."""
        n, th = self.r.n_src, self.theta
        E, V, seen = self.sky.clone(), torch.zeros_like(self.sky), torch.zeros_like(self.sky, dtype=torch.bool)
        with torch.no_grad():
            for p, q in self.blocks:
                at, px, py, m = self.pixels(p, q)
                e, v = self.light(th, p, q, at, px, py)
                E.index_add_(0, m, e)
                V.index_add_(0, m, v)
                seen[m] = True
            ll = self.x[seen] * (torch.log(E[seen]) - V[seen] / (2 * E[seen] ** 2)) - E[seen]
        t = th.clone().requires_grad_(order > 0)
        kl = self.kl(t)
        total, local = ll.sum() - kl.detach().sum(), -kl.detach()
        grad, hess = torch.zeros_like(th), torch.zeros(n, 44, 44, dtype=th.dtype, device="cuda")

        def add(value, columns):
            """The derivatives of a sum over sources of functions of their own parameters."""
            g, = torch.autograd.grad(value, t, create_graph=order > 1)
            grad.add_(g.detach())
            for k in range(columns if order > 1 else 0):
                h, = torch.autograd.grad(g[:, k].sum(), t, retain_graph=True)
                hess[:, k].add_(h)

        if order:
            add(-kl.sum(), 44)
        for p, q in self.blocks:
            at, px, py, m = self.pixels(p, q)
            e, v = self.light(t, p, q, at, px, py)
            e, v = E[m] - e.detach() + e, V[m] - v.detach() + v
            ll = self.x[m] * (torch.log(e) - v / (2 * e * e)) - e
            local.index_add_(0, self.owner[at], ll.detach())
            if order:
                add(ll.sum(), 28)                     # pixels do not depend on the last 16
        return dict(total=total, local=local, grad=grad, hess=hess)


def exact(case, seed):
    call = case["call"]
    if call == "fit":
        return None
    got = _Plain(_region(case, seed)).evaluate(dict(elbo=0, hess=2).get(call, 1))
    if call == "hess":
        return {k: got[k] for k in ("local", "grad", "hess")}
    if call == "elbo":
        return dict(total=got["total"].view(1), local=got["local"])
    if call == "autograd":
        return dict(total=got["total"], grad=got["grad"])
    return dict(total=got["total"].view(1 if call == "grad" else ()), local=got["local"], grad=got["grad"])
