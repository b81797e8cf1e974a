"""The work that users of libmemsynth have it do, as cases that can be timed.

Every case goes through `memsynth.Context` (or the autograd operator on top of
it), the calls that a program makes: an objective with its gradient, the
operator pair, the dirty and residual maps, the gridded forward, a whole solve.
Inputs are a seeded interferometer observation: antennas in a disk, Earth
rotation tracks, a sky of Gaussians and points under a Gaussian primary beam,
thermal noise, and a positive image near that sky.

The forms in 32 bits and in split 16 bits return their objective, chi^2 and
entropy with 32-bit accuracy; `run` hands them on as float32, and the FP64
form's as they are.
"""
import math

import numpy as np
import torch

from paper_1703_02920_gb300 import memsynth, synth

ARCSEC = math.pi / 648000.0
LAMBDA_PAPER = 0.1  # entropy weight in units of 1/G, as in the configurations

# The array geometry goes with the image size: pixel (arcsec), antennas, disk
# diameter (m) and prior G (Jy/pixel) of the 64, 256, 512 and 1024 pixel
# configurations; other sizes take the scaling between them.
GEOMETRY = {64: (0.2, 20, 300.0), 128: (0.1, 50, 500.0), 256: (0.05, 50, 1000.0), 512: (0.025, 50, 2000.0),
            1024: (0.0125, 64, 3000.0)}


def listed():
    return [
        # the 64 x 64 configuration: 190 baselines x 27 dumps and conjugates;
        # the smallest ordinary evaluation, where launches count
        case("evaluate", 64, "fp16x3", 10260, name="evaluate_64"),
        # the same observation in the FP64 form, the reference of the others
        case("evaluate", 64, "fp64_direct", 10260, name="evaluate_64_fp64"),
        # a mid-size image in the split BF16 form, ragged visibility count,
        # projected gradient as the solver asks for it
        case("evaluate", 128, "bf16x3", 100003, projected=True, name="evaluate_128_bf16"),
        # the 256 x 256 configuration: 1,225 baselines x 816 dumps
        case("evaluate", 256, "fp16x3", 999600, name="evaluate_256"),
        # the 1024 x 1024 configuration at 248 of its dumps (2,016 baselines)
        case("evaluate", 1024, "fp16x3", 499968, name="evaluate_1024"),
        # a spectral cube: independent 256 x 256 images, uneven channels
        case("evaluate", 256, "fp16x3", 400000, channels=6, name="cube_256"),
        # multi-frequency synthesis or a mosaic: one image for all channels
        case("evaluate", 128, "fp16x3", 60001, channels=5, shared=True, name="shared_128"),
        # the differentiable operator: forward, and the adjoint as its backward
        case("operator", 512, "fp16x3", 122501, name="operator_512"),
        # the operator pair on a short observation
        case("operator", 256, "bf16x3", 3001, name="operator_256_small"),
        # residual map, dirty map and PSF of one observation
        case("maps", 256, "fp16x3", 99999, name="maps_256"),
        # the gridded approximation of the forward, padded to twice the image
        case("gridded", 256, "fp16x3", 999600, pad=2, name="gridded_256"),
        # a short solve of the 64 x 64 configuration: CG iterations with their
        # line searches, the loop that every user's run ends in
        case("solve", 64, "fp16x3", 10260, iterations=5, name="solve_64"),
    ]


def case(kind, n, form, z, **more):
    c = {"kind": kind, "n": n, "form": form, "z": z, "channels": 1, "shared": False, "projected": False}
    c.update(more)
    return c


LARGEST = 1024 * 1024 * 499968  # (visibility, pixel) pairs of one pass


def draw(rng):
    kind = rng.choice(["evaluate"] * 6 + ["operator"] * 3 + ["maps", "maps", "gridded", "gridded", "solve"])

    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "solve":
        return case("solve", 64, "fp16x3", spread(2000, 30000), iterations=rng.randint(1, 6))
    if kind == "gridded":
        n, pad = rng.choice([(64, 3), (128, 2), (128, 5), (256, 3), (256, 4), (512, 2), (512, 3), (1024, 2)])
        return case("gridded", n, "fp16x3", spread(3000, 2000000), pad=pad)
    if kind == "evaluate" and rng.random() < 0.2:
        # the direct forms take any multiple of 16
        form = rng.choice(["fp32_direct", "fp64_direct"])
        n = 16 * rng.randint(3, 10)
        top = 4e8 if form == "fp32_direct" else 4e7
        return case("evaluate", n, form, spread(300, int(top / (n * n))), projected=rng.random() < 0.5)
    n = rng.choice([64, 128, 256, 512, 768, 1024])
    form = rng.choice(["fp16x3", "fp16x3", "bf16x3"])
    # the maps take a forward and three adjoints, twice an evaluation's passes
    z = spread(500, min(1500000, LARGEST // (n * n) // (2 if kind == "maps" else 1)))
    if n <= 256 and rng.random() < 0.3:
        return case(kind, n, form, max(z, 2000), channels=rng.randint(2, 9), shared=rng.random() < 0.4)
    return case(kind, n, form, z, projected=kind == "evaluate" and rng.random() < 0.5)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def observation(c, seed):
    """The data set of a case (numpy, host memory, as mem_create takes it) and
    the image that the calls are made at."""
    rng = np.random.Generator(np.random.PCG64([int(seed), c["n"], c["z"]]))
    n = c["n"]
    cell, antennas, disk = GEOMETRY.get(n, (12.8 / n, 50, 1000.0 * n / 256))
    dx, G = cell * ARCSEC, 0.4096 / (n * n)
    enu = synth.antennas_in_disk(rng, antennas, disk)
    baselines = antennas * (antennas - 1) // 2
    # uneven channels: shares spread over a factor of ten
    share = np.exp(rng.uniform(0.0, math.log(10.0), c["channels"]))
    z = np.maximum(1, (c["z"] * share / share.sum()).astype(np.int64)) if c["channels"] > 1 else np.array([c["z"]])
    fwhm = synth.BEAM_FWHM_345
    us, vs, vos, beams, truths = [], [], [], [], []
    comps = synth.continuum_sky(rng)
    for k in range(c["channels"]):
        wavelength = synth.WAVELENGTH * (1.0 + 0.002 * k)
        u, v = synth.earth_rotation_uv(enu, -(-int(z[k]) // baselines) + 1, wavelength)
        u, v = u[: z[k]], v[: z[k]]
        if c["channels"] > 1 and not c["shared"]:
            comps = synth.continuum_sky(rng)
        wide = fwhm * wavelength / synth.WAVELENGTH
        vis = sky_visibilities(comps, u, v, wide)
        vos.append(vis + synth.SIGMA_NOISE * (rng.standard_normal(u.size) + 1j * rng.standard_normal(u.size)))
        us.append(u)
        vs.append(v)
        beams.append(synth.gaussian_beam(n, dx, dx, wide))
        if not (c["shared"] and k):
            truths.append(synth.sky_image(comps, n, dx, dx))
    truth = np.stack(truths)
    # an image on the way to the sky: scaled pixel by pixel, never below G
    image = np.maximum(truth * rng.uniform(0.7, 1.3, truth.shape), G).astype(np.float32)
    zt = int(z.sum())
    ds = synth.Dataset(name="observation", N=n, dx=dx, dy=dx, u=np.concatenate(us), v=np.concatenate(vs),
                       vo=np.concatenate(vos), sigma=synth.SIGMA_NOISE * rng.uniform(0.8, 1.25, zt),
                       pb=np.stack(beams), offsets=np.concatenate([[0], np.cumsum(z)]).astype(np.int64),
                       truth=truth.astype(np.float32), G=G, lam=LAMBDA_PAPER / G, n_iter=1,
                       shared_image=c["shared"])
    y = (rng.standard_normal((zt, 2)) * 0.3).astype(np.float32)
    return ds, np.maximum(image, np.float32(G)), y


def sky_visibilities(comps, u, v, fwhm):
    """synth's closed-form visibilities, on the GPU where there is one."""
    if u.size < 20000 or not torch.cuda.is_available():
        return synth.sky_visibilities(comps, u, v, fwhm)
    sb2 = (fwhm * synth.FWHM_TO_SIGMA) ** 2
    tu, tv = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    out = torch.zeros(u.size, dtype=torch.complex128, device="cuda")
    for g in comps:
        if isinstance(g, synth.Point):
            amp, quad, x, y = g.flux * math.exp(-0.5 * (g.x0 ** 2 + g.y0 ** 2) / sb2), None, g.x0, g.y0
        else:
            S = g.cov()
            Si = np.linalg.inv(S)
            Pi = np.linalg.inv(Si + np.eye(2) / sb2)
            mu = np.array([g.x0, g.y0])
            h = Si @ mu
            x, y = Pi @ h
            amp = g.flux * math.sqrt(np.linalg.det(Pi) / np.linalg.det(S)) * math.exp(0.5 * h @ Pi @ h - 0.5 * mu @ Si @ mu)
            quad = Pi[0, 0] * tu * tu + 2 * Pi[0, 1] * tu * tv + Pi[1, 1] * tv * tv
        phase = -2 * math.pi * (tu * x + tv * y)
        size = torch.full_like(tu, amp) if quad is None else amp * torch.exp(-2 * math.pi ** 2 * quad)
        out += torch.polar(size, phase)
    return out.cpu().numpy()


def prepare(c, seed):
    ds, image, y = observation(c, seed)
    state = {"case": c, "ctx": memsynth.Context(ds, precision=c["form"]), "image": torch.from_numpy(image).cuda(),
             "op": memsynth.MemOperator()}
    if c["kind"] == "operator":
        state["y"] = torch.from_numpy(y).cuda()
        state["image"].requires_grad_(True)
    if c["kind"] == "solve":
        state["image"] = torch.full_like(state["image"], ds.G)
    return state


def run(state):
    c, ctx, image = state["case"], state["ctx"], state["image"]
    if c["kind"] == "evaluate":
        phi, chi2, entropy, grad = ctx.objective_grad(image, projected=c["projected"])
        return {"objective": scalars(c, phi, chi2, entropy), "gradient": grad}
    if c["kind"] == "operator":
        vis = state["op"].apply(image, ctx)
        (grad,) = torch.autograd.grad(vis, image, state["y"])
        return {"visibilities": vis.detach(), "gradient": grad}
    if c["kind"] == "maps":
        return {"residual": ctx.residual_image(image), "dirty": ctx.dirty_image(), "psf": ctx.dirty_image(psf=True)}
    if c["kind"] == "gridded":
        return {"visibilities": ctx.forward_gridded(image, c["pad"])}
    solved, report, _ = ctx.solve(image, c["iterations"])
    return {"image": solved, "objective": scalars(c, report.phi, report.chi2, report.entropy)}


def scalars(c, *values):
    return np.array(values, dtype=np.float64 if c["form"] == "fp64_direct" else np.float32)


def work(c):
    """One multiply-add per (visibility, pixel) pair and operator pass: pixels
    that mirror each other about the image's centre row share their products."""
    n, z, channels = c["n"], c["z"], c["channels"]
    images = 1 if c["shared"] else channels
    pixels = n * n * channels
    pair = 2.0 * z * n * n
    if c["kind"] == "evaluate":  # phases, data and weight; image, beam, gradient
        return {"bytes": 36.0 * z + 4.0 * pixels + 8.0 * images * n * n, "flops": 2 * pair}
    if c["kind"] == "operator":  # phases, y, V; image, beam, gradient
        return {"bytes": 32.0 * z + 4.0 * pixels + 8.0 * images * n * n, "flops": 2 * pair}
    if c["kind"] == "maps":  # a forward and three adjoints
        return {"bytes": 3 * 36.0 * z + 20.0 * pixels, "flops": 4 * pair}
    if c["kind"] == "gridded":  # u, v, V; image, beam; a real 2-D transform
        m = c["pad"] * n
        return {"bytes": 24.0 * z + 8.0 * pixels, "flops": channels * 5.0 * m * m * math.log2(m) + 16.0 * z}
    # about a gradient, a curvature pass and ten line-search passes an iteration
    return {"bytes": c["iterations"] * 13 * 36.0 * z, "flops": (14 * c["iterations"] + 2) * pair}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def turns(t):
    return t - torch.round(t)


def row_factors(freq, d, n):
    """cos and sin of 2 pi freq (k - n/2) d, (visibilities, n)."""
    k = torch.arange(n, dtype=torch.float64, device=freq.device) - n // 2
    a = 2 * math.pi * turns(turns(freq * d)[:, None] * k[None, :])
    return torch.cos(a), torch.sin(a)


def exact_forward(u, v, dx, dy, B):
    out = []
    for i in range(0, u.numel(), 16384):
        cx, sx = row_factors(u[i : i + 16384], dx, B.shape[1])
        cy, sy = row_factors(v[i : i + 16384], dy, B.shape[0])
        tr, ti = cy @ B, sy @ B
        out.append(torch.stack([(cx * tr - sx * ti).sum(1), -(sx * tr + cx * ti).sum(1)], 1))
    return torch.cat(out) if out else torch.zeros((0, 2), dtype=torch.float64, device=B.device)


def exact_adjoint(u, v, dx, dy, y, n):
    out = torch.zeros((n, n), dtype=torch.float64, device=u.device)
    for i in range(0, u.numel(), 16384):
        cx, sx = row_factors(u[i : i + 16384], dx, n)
        cy, sy = row_factors(v[i : i + 16384], dy, n)
        yr, yi = y[i : i + 16384, :1], y[i : i + 16384, 1:]
        out += cy.T @ (yr * cx - yi * sx) - sy.T @ (yr * sx + yi * cx)
    return out


def exact_gridded(u, v, dx, dy, B, pad):
    n = B.shape[0]
    m = pad * n
    o = (m - n) // 2
    padded = torch.zeros((m, m), dtype=torch.float64, device=B.device)
    padded[o : o + n, o : o + n] = B
    F = torch.fft.fft2(torch.fft.ifftshift(padded))
    gu, gv = u * (m * dx), v * (m * dy)
    k, l = torch.floor(gu), torch.floor(gv)
    fx, fy = gu - k, gv - l
    k, l = k.long(), l.long()

    def at(kk, ll):
        return F[ll % m, kk % m]

    V = ((1 - fx) * (1 - fy) * at(k, l) + fx * (1 - fy) * at(k + 1, l) + (1 - fx) * fy * at(k, l + 1)
         + fx * fy * at(k + 1, l + 1))
    return torch.view_as_real(V)


def exact(c, seed):
    if c["kind"] == "solve" or not torch.cuda.is_available():
        return None  # a trajectory: it has no value of its own to be near to
    ds, image, y = observation(c, seed)
    on = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda().double()  # noqa: E731
    n, dx, dy, G, lam = ds.N, ds.dx, ds.dy, ds.G, ds.lam
    u, v, w, beam, img = on(ds.u), on(ds.v), 1.0 / on(ds.sigma) ** 2, on(ds.pb), on(image)
    vo = torch.stack([on(ds.vo.real), on(ds.vo.imag)], 1)
    images = img.shape[0]
    grad, chi2, vis, maps = torch.zeros_like(img), 0.0, [], {"residual": [], "dirty": [], "psf": []}
    for k in range(c["channels"]):
        s = slice(int(ds.offsets[k]), int(ds.offsets[k + 1]))
        i = 0 if c["shared"] else k
        B = beam[k] * img[i]
        if c["kind"] == "gridded":
            vis.append(exact_gridded(u[s], v[s], dx, dy, B, c["pad"]))
            continue
        V = exact_forward(u[s], v[s], dx, dy, B)
        if c["kind"] == "evaluate":
            r = V - vo[s]
            chi2 += 0.5 * float((w[s, None] * r * r).sum())
            grad[i] += beam[k] * exact_adjoint(u[s], v[s], dx, dy, w[s, None] * r, n)
        elif c["kind"] == "operator":
            vis.append(V)
            grad[i] += beam[k] * exact_adjoint(u[s], v[s], dx, dy, on(y)[s], n)
        else:
            weight = (w[s] / w[s].sum())[:, None]
            one = torch.tensor([[1.0, 0.0]], dtype=torch.float64, device=u.device)
            for name, what in (("residual", vo[s] - V), ("dirty", vo[s]), ("psf", one)):
                maps[name].append(exact_adjoint(u[s], v[s], dx, dy, weight * what, n))
    if c["kind"] == "maps":
        return {name: torch.stack(m) for name, m in maps.items()}
    if c["kind"] == "gridded":
        return {"visibilities": torch.cat(vis)}
    if c["kind"] == "operator":
        return {"visibilities": torch.cat(vis), "gradient": grad}
    log = torch.log(img / G)
    entropy = -float((img * log).sum())
    grad += lam * (1.0 + log)
    if c["projected"]:
        grad[(img <= G) & (grad > 0)] = 0.0
    assert grad.shape[0] == images
    return {"objective": np.array([chi2 - lam * entropy, chi2, entropy]), "gradient": grad}
