"""The performance cases of the library: what is timed, on which inputs, and the
FP64 values the results are held against.

Sizes come from the benchmark's workloads (32^3 warp, 64^3 motion capture, 128^3
8-coil operator, 192^3 16-coil CG and warp-only FISTA, 256^3 sweep) and from the
parity tests (ragged, non-cubic grids, rational oversampling); sample counts of the
larger ones are cut so that a plan is made in about a second or two.  Inputs are
synthetic, of the benchmark's kind (ellipsoid phantom, Gaussian-bump motion, coil
maps on a ring, cone trajectories), made on the GPU from the seed.
"""

import json
import math
import os
import tempfile

import numpy as np
import torch

from paper_2501_16713_gb300 import Cnn, Plan, nrsense

DEV = "cuda"
GOLDEN_ANGLE = math.pi * (3.0 - math.sqrt(5.0))
READOUT = 1042  # samples per cone interleave

# Launch choices that autotuning keeps on the 128^3, 8-coil, 4-phase plan, as a
# program with a tuning file on disk loads them (the other plans either run
# autotune themselves or keep the defaults).
TUNED_128 = {"spread_variant": 4, "interp_coils": 4, "interp_tma": 1, "spread_image_warp": 2,
             "fft_pruned": 1, "spread_mma_wpc": 1, "spread_mma_cube": 1, "spread_max_item": 0,
             "interp_image_home": 0, "image_fft_pruned": 1}


def _case(name, kind, shape, coils, phases, samples, **kw):
    c = {"kind": kind, "n0": shape[0], "n1": shape[1], "n2": shape[2], "coils": coils,
         "phases": phases, "samples": samples, "uneven": False, "warp": True, "osf": 2.0,
         "width": 4, "precision": "fp32", "tuning": "default", "steps": 1}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: motion fields applied and undone on a small image, no coils
        _case("warp32", "normal", (32, 32, 32), 0, 1, 0),
        # motion-corrected CG reconstruction of a low-resolution volume, stopped early as a
        # regularisation: launch-bound iterations
        _case("cg64", "cg", (64, 64, 64), 8, 2, 125040, tuning="autotune", steps=6),
        # the benchmark's operator, at its full size: one CG or FISTA step of a reconstruction
        _case("sense128", "normal", (128, 128, 128), 8, 4, 1500480, tuning="file"),
        # the same operator on an acquisition without a round size: ragged axes, few coils and
        # uneven phases, the plan as created
        _case("ragged", "normal", (84, 60, 132), 5, 3, 70001, uneven=True),
        # simulated acquisition: the forward operator of the batched CG workload's geometry
        _case("forward192", "forward", (192, 192, 192), 16, 1, 1200384, warp=False,
              tuning="autotune"),
        # gridding of a large many-coil acquisition, as created: the right-hand side of a solve
        _case("adjoint256", "adjoint", (256, 256, 256), 16, 1, 3000960, warp=False),
        # the wide kernel at reduced oversampling, for memory-limited problems
        _case("wide96", "normal", (96, 80, 64), 8, 2, 150048, osf=1.5, width=6),
        # half-width storage of the coil grids
        _case("bf16_128", "normal", (128, 128, 128), 8, 1, 400128, warp=False, precision="bf16"),
        # motion capture: density compensation, then one weighted reconstruction per heartbeat
        _case("inav64", "recon", (64, 64, 64), 8, 1, 16384, warp=False, tuning="autotune",
              steps=8),
        # a new motion estimate or trajectory: the plan is made anew, then data are gridded
        _case("replan64", "replan", (64, 64, 64), 8, 2, 62520),
        # inversion of a known warp by wavelet-FISTA
        _case("fista_warp192", "fista", (192, 192, 192), 0, 1, 0, steps=6),
        # preconditioner training on residual/error pairs of CG: gradients of a batch, and the
        # network applied to a new residual
        _case("train128", "train", (128, 128, 128), 0, 1, 0, warp=False, steps=2),
    ]


def _even(v):
    return max(12, 2 * int(round(v / 2.0)))


def draw(rng):
    """A case between the listed ones: any kind, sizes over their logarithm, odd coil, phase
    and sample counts among them; at most about 2.2 M gridded points and 0.4 G grid values."""
    kind = rng.choice(["normal", "normal", "normal", "forward", "adjoint", "cg", "recon",
                       "replan", "fista", "train"])
    big = 112 if kind in ("cg", "recon", "replan") else 128 if kind == "train" else 144
    n = math.exp(rng.uniform(math.log(24), math.log(big)))
    if kind == "fista":  # every axis a multiple of 2^levels
        shape = [8 * max(2, round(n * rng.uniform(0.8, 1.25) / 8)) for _ in range(3)]
    elif rng.random() < 0.4:  # cubes of a customary size
        m = min((32, 48, 64, 80, 96, 112, 128, 144), key=lambda v: abs(v - n))
        shape = [m] * 3
    else:
        shape = [_even(n * rng.uniform(0.75, 1.3)) for _ in range(3)]
    nvox = shape[0] * shape[1] * shape[2]
    if kind == "train":
        return _case("", kind, shape, 0, 1, 0, warp=False, steps=rng.randint(1, 4))
    if kind == "fista" or (kind == "normal" and rng.random() < 0.25):
        return _case("", kind, shape, 0, max(1, min(rng.randint(1, 4), 2200000 // nvox)), 0,
                     steps=rng.randint(4, 12) if kind == "fista" else 1)
    width, osf, precision = 4, 2.0, "fp32"
    p = rng.random()
    if p < 0.2:
        width = 6
        if all(v % 4 == 0 for v in shape):
            osf = rng.choice([1.25, 1.5, 2.0])
    elif p < 0.3 and len(set(shape)) == 1 and shape[0] in (32, 64, 128):
        precision = "bf16"
    gvol = nvox * osf ** 3
    coils = max(1, min(rng.choice([1, 2, 3, 4, 5, 6, 8, 8, 12, 16]), int(4.0e8 / gvol)))
    phases = rng.randint(1, 4)
    warp = kind != "recon" and rng.random() < 0.7
    if kind == "recon":
        phases = 1
    if warp:
        phases = max(1, min(phases, 1600000 // nvox))
    samples = max(200, min(int(nvox * math.exp(rng.uniform(math.log(0.05), math.log(0.8)))),
                           1200000 // phases))
    tuning = ("autotune" if kind != "replan" and precision == "fp32" and rng.random() < 0.5
              else "default")
    return _case("", kind, shape, coils, phases, samples, uneven=rng.random() < 0.4, warp=warp,
                 osf=osf, width=width, precision=precision, tuning=tuning,
                 steps=rng.randint(3, 6) if kind == "cg" else rng.randint(4, 12) if kind == "recon"
                 else 1)


# -- inputs ------------------------------------------------------------------


def _shape(case):
    return (case["n0"], case["n1"], case["n2"])


def _counts(case):
    m, P = case["samples"], case["phases"]
    if not case["uneven"]:
        return [m] * P
    # heartbeats fall unevenly into the phases: from half to one and a half of the mean
    return [max(1, int(m * (0.5 + (j + 0.5) / P))) for j in range(P)]


def _axes(shape, dtype=torch.float32):
    return [torch.arange(s, device=DEV, dtype=dtype).reshape([-1 if k == a else 1 for k in range(3)])
            for a, s in enumerate(shape)]


def _u(rng, lo, hi, n=None):
    return rng.uniform(lo, hi, n)


def _phantom(shape, rng, gen):
    """Ellipsoids within the field of view, a smooth phase, and 5 % white noise."""
    ax = _axes(shape)
    img = torch.zeros(shape, device=DEV)
    for _ in range(8):
        d = 0
        for a in range(3):
            c = (0.5 + _u(rng, -0.2, 0.2)) * shape[a]
            d = d + ((ax[a] - c) / (_u(rng, 0.06, 0.2) * shape[a])) ** 2
        img += _u(rng, 0.2, 1.0) * (d <= 1.0)
    ph = _u(rng, -math.pi, math.pi)
    for a in range(3):
        ph = ph + _u(rng, -1.0, 1.0) * (ax[a] / shape[a] - 0.5)
    x = torch.polar(img, ph.expand(shape).contiguous())
    return x + 0.05 * torch.randn(shape, dtype=torch.complex64, device=DEV, generator=gen)


def _displacement(shape, phases, rng, largest):
    """Sums of Gaussian bumps of at most `largest` voxels, plus a rigid shift of at most half."""
    ax = _axes(shape)
    out = torch.empty((phases, 3) + tuple(shape), device=DEV)
    for j in range(phases):
        d = torch.zeros((3,) + tuple(shape), device=DEV)
        for _ in range(6):
            w = _u(rng, 0.05, 0.1) * max(shape)
            g = 1.0
            for a in range(3):
                c = _u(rng, 0.2, 0.8) * shape[a]
                g = g * torch.exp(-((ax[a] - c) ** 2) / (2 * w * w))
            for a in range(3):
                d[a] += _u(rng, -1, 1) * g
        d *= largest / d.square().sum(0).sqrt().max().clamp_min(1e-6)
        for a in range(3):
            d[a] += _u(rng, -0.25, 0.25) * largest
        out[j] = d
    return out


def _coil_maps(shape, coils, rng):
    """Gaussian profiles on a ring, sum of squares one."""
    ax = _axes(shape)
    s = 0.4 * max(shape)
    maps = torch.empty((coils,) + tuple(shape), dtype=torch.complex64, device=DEV)
    for c in range(coils):
        ang = 2 * math.pi * c / coils + _u(rng, -0.1, 0.1)
        ctr = [0.5, 0.5 + 0.6 * math.cos(ang), 0.5 + 0.6 * math.sin(ang)]
        d, ph = 0, _u(rng, -math.pi, math.pi)
        for a in range(3):
            d = d + (ax[a] - ctr[a] * shape[a]) ** 2
            ph = ph + _u(rng, -1.5, 1.5) * (ax[a] / shape[a] - 0.5)
        maps[c] = torch.polar(torch.exp(-d / (2 * s * s)), ph.expand(shape).contiguous())
    return maps / maps.abs().square().sum(0).sqrt()


def _trajectory(counts, rng):
    """Cone interleaves on golden-angle azimuths, dealt to the phases in turn."""
    P = len(counts)
    out = []
    nil = [-(-m // READOUT) for m in counts]
    total = P * max(nil)
    phi = _u(rng, 0, 2 * math.pi)
    for j, m in enumerate(counts):
        # interleaves of phase j spread over the whole set of cone angles
        ids = torch.arange(nil[j], device=DEV, dtype=torch.float64) * (total / nil[j]) + j
        cos_t = 1.0 - 2.0 * ((ids + 0.5) / total).clamp(0, 1)
        sin_t = (1.0 - cos_t ** 2).clamp_min(0).sqrt()
        t = (torch.arange(READOUT, device=DEV, dtype=torch.float64) + 0.5) / READOUT
        ang = (ids * GOLDEN_ANGLE + phi)[:, None] + 8 * math.pi * t[None]
        rad = 0.999 * math.pi * t[None]
        k = torch.stack([(rad * cos_t[:, None]).expand_as(ang), rad * sin_t[:, None] * ang.cos(),
                         rad * sin_t[:, None] * ang.sin()], -1)
        out.append(k.reshape(-1, 3)[:m].float().contiguous())
    return out


def _kdata(coords, coils, gen):
    """Noisy samples whose size falls with the radius in k space."""
    k = torch.cat(coords)
    size = 1.0 / (1.0 + 40.0 * k.square().sum(-1, keepdim=True))
    y = torch.randn((k.shape[0], coils), dtype=torch.complex64, device=DEV, generator=gen)
    return (size + 0.02) * y


def _inputs(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    shape, P, C = _shape(case), case["phases"], case["coils"]
    inp = {"x": _phantom(shape, rng, gen), "disp": None, "coords": None, "smaps": None}
    if case["warp"]:
        inp["disp"] = _displacement(shape, P, rng, min(8.0, 0.06 * max(shape)))
    if C:
        inp["smaps"] = _coil_maps(shape, C, rng)
        inp["coords"] = _trajectory(_counts(case), rng)
    if case["kind"] in ("adjoint", "replan"):
        inp["y"] = _kdata(inp["coords"], C, gen)
    elif case["kind"] == "cg":  # a solve has data that belong to an image, with 3 % noise
        y = _Geo(case).A(inp["x"].to(torch.complex128), inp).to(torch.complex64)
        noise = torch.randn(y.shape, dtype=torch.complex64, device=DEV, generator=gen)
        inp["y"] = (y + 0.03 * y.abs().mean() * noise) / y.abs().max()
    elif case["kind"] == "recon":
        inp["y"] = [_kdata(inp["coords"], C, gen) for _ in range(case["steps"])]
    elif case["kind"] == "fista":
        inp["y"] = torch.stack([inp["x"]] * P)
    elif case["kind"] == "train":
        # a residual is rough, the error that belongs to it smooth
        inp["e"] = [_phantom(shape, rng, gen) for _ in range(case["steps"])]
        inp["r"] = [2.0 * e + torch.randn(shape, dtype=torch.complex64, device=DEV, generator=gen)
                    for e in inp["e"]]
        ch = nrsense.CNN_CHANNELS
        inp["params"] = [((rng.standard_normal((co, ci, 3, 3, 3)) * math.sqrt(2 / (27 * ci))
                           * (0.1 if co == 2 else 1.0)).astype(np.float32), np.zeros(co, np.float32))
                         for ci, co in zip(ch[:-1], ch[1:])]
    return inp


FISTA_LAMBDA = 1e-2
DCF_ITERS = 10


def _lam(case):
    """Tikhonov weight: the order of 1e-2 of the largest eigenvalue of sum A_j^H A_j, which on
    cone trajectories is some thousands of times the mean one (the number of samples); without
    coils 5 % of the phases' sum."""
    return 100.0 * sum(_counts(case)) if case["coils"] else 0.05 * case["phases"]


def _lip(case):
    """Step bound of the warp-only problem: twice the largest eigenvalue of sum T_j^H T_j, which
    is about one per phase and grows where a warp compresses."""
    return 8.0 * case["phases"]


def _make_plan(case, inp):
    osf = case["osf"]
    return Plan(_shape(case), disp=inp["disp"], coords=inp["coords"], smaps=inp["smaps"],
                n_phases=case["phases"], osf=int(osf) if osf == int(osf) else osf,
                width=case["width"], identity_warp=not case["warp"],
                precision=nrsense.BF16_STORE if case["precision"] == "bf16" else nrsense.FP32)


def prepare(case, seed):
    inp = _inputs(case, seed)
    st = {"case": case, "inp": inp}
    if case["kind"] == "train":
        st["net"] = Cnn(_shape(case))
        st["net"].set_params(inp["params"])
    elif case["kind"] != "replan":
        st["plan"] = plan = _make_plan(case, inp)
        if case["tuning"] == "autotune":
            plan.autotune(reps=2)
        elif case["tuning"] == "file":
            with tempfile.TemporaryDirectory() as d:
                path = os.path.join(d, "tuning.json")
                with open(path, "w") as f:
                    json.dump({plan.tuning_key(): TUNED_128}, f)
                plan.autotune(cache=path)
    return st


def run(state):
    case, inp = state["case"], state["inp"]
    kind, plan = case["kind"], state.get("plan")
    if kind == "normal":
        return plan.normal(inp["x"], _lam(case))
    if kind == "forward":
        return plan.forward(inp["x"])
    if kind == "adjoint":
        return plan.adjoint(inp["y"])
    if kind == "cg":
        x, _, _, _, _ = plan.solve_cg(inp["y"], _lam(case), tol=0.0, maxit=case["steps"], graph=True)
        return x
    if kind == "recon":
        w = plan.dcf(0, iters=DCF_ITERS)
        return {"w": w, "img": [plan.adjoint_weighted(y, w) for y in inp["y"]]}
    if kind == "replan":
        plan = _make_plan(case, inp)
        out = plan.adjoint(inp["y"])
        plan.close()
        return out
    if kind == "fista":
        x, _, _ = plan.solve_fista(inp["y"], FISTA_LAMBDA, levels=3, L=_lip(case),
                                   maxit=case["steps"])
        return x
    net = state["net"]
    loss = [net.gradients(r, e, accumulate=k > 0, want_loss=k == 0)
            for k, (r, e) in enumerate(zip(inp["r"], inp["e"]))]
    return {"loss": loss[0], "grads": net.get_grads(), "z": net.apply(inp["r"][0])}


# -- what a pass cannot do without -------------------------------------------


def work(case):
    shape, P, C = _shape(case), case["phases"], case["coils"]
    nv = float(np.prod(shape))
    g = [case["osf"] * s for s in shape]
    gv = float(np.prod(g))
    M = float(sum(_counts(case)))
    W3 = case["width"] ** 3
    lg = math.log2(gv)
    if case["kind"] == "train":
        # per pair forward, backward and weight gradients of the symmetric form's ten
        # convolutions; activations count once in and out of each pass
        mac = 27 * 2 * (2 * 16 + 3 * 256 + 256) * nv
        n = case["steps"]
        return {"bytes": nv * 8 * (2 * n + 2), "flops": 2 * mac * (3 * n + 1)}
    # one direction of T, of G S (flops of the transforms and of the taps)
    t_dir = (5 * gv * lg + 5 * nv * math.log2(nv) + P * nv * W3 * 4) if case["warp"] else 0.0
    k_dir = P * C * 5 * gv * lg * 0.6 + M * C * W3 * 4 + P * C * nv * 8
    geo = (12 * P * nv if case["warp"] else 0) + 8 * C * nv + 12 * M
    img, dat = 8 * nv, 8 * C * M
    kind, n = case["kind"], case["steps"]
    if kind == "normal":
        return {"bytes": 2 * img + geo, "flops": 2 * (t_dir + k_dir)}
    if kind in ("forward", "adjoint", "replan"):
        return {"bytes": img + dat + geo, "flops": t_dir + k_dir}
    if kind == "cg":
        return {"bytes": img + dat + geo, "flops": (2 * n + 1) * (t_dir + k_dir)}
    if kind == "fista":
        return {"bytes": img * (1 + P) + geo, "flops": (2 * n + 1) * t_dir}
    return {"bytes": n * (img + dat) + geo,
            "flops": n * k_dir + DCF_ITERS * 2 * M * W3 * 2}


# -- the same in 64 bits, without the library --------------------------------


class _Geo:
    def __init__(self, case):
        self.n, self.W = _shape(case), case["width"]
        self.g = [int(round(case["osf"] * s)) for s in self.n]
        sigma = self.g[0] / self.n[0]
        self.sigma = sigma
        self.beta = math.pi * math.sqrt((self.W / sigma) ** 2 * (sigma - 0.5) ** 2 - 0.8)
        # 1 / C(m / G) for m in [-N/2, N/2), per axis
        self.dea = []
        for n, g in zip(self.n, self.g):
            a = math.pi * self.W * (np.arange(n) - n // 2) / g
            z2 = self.beta ** 2 - a * a
            zp, zn = np.sqrt(np.maximum(z2, 1e-300)), np.sqrt(np.maximum(-z2, 1e-300))
            first = np.where(z2 > 0, np.sinh(np.where(z2 > 0, zp, 1)) / np.where(z2 > 0, zp, 1),
                             np.sinc(np.where(z2 > 0, 0, zn) / math.pi))
            self.dea.append(torch.from_numpy(1.0 / (self.W * (first - np.sinc(a / math.pi))))
                            .to(DEV))

    def deapod(self, v):
        """Divides by the kernel's transform, indices centred."""
        return (v * self.dea[0][:, None, None] * self.dea[1][None, :, None]
                * self.dea[2][None, None, :])

    def pos(self, a):
        return torch.remainder(torch.arange(self.n[a], device=DEV) - self.n[a] // 2, self.g[a])

    def pad(self, v):
        """Centred block onto the periodic oversampled grid."""
        out = torch.zeros(self.g, dtype=torch.complex128, device=DEV)
        out[self.pos(0)[:, None, None], self.pos(1)[None, :, None], self.pos(2)[None, None, :]] = v
        return out

    def crop(self, u):
        return u[self.pos(0)][:, self.pos(1)][:, :, self.pos(2)]

    def taps(self, q):
        """(linear index, weight) of every tap of the points q (3, M)."""
        W, ax = self.W, []
        for a in range(3):
            base = q[a].floor() - (W // 2 - 1)
            tap = []
            for t in range(W):
                u = 2.0 * (q[a] - base - t) / W
                arg = (1.0 - u * u).clamp_min(0.0)
                wt = torch.special.i0(self.beta * arg.sqrt()) - 1.0
                tap.append((torch.remainder(base + t, self.g[a]).long(), wt))
            ax.append(tap)
        for i0, w0 in ax[0]:
            for i1, w1 in ax[1]:
                lin, w = i0 * self.g[1] + i1, w0 * w1
                for i2, w2 in ax[2]:
                    yield lin * self.g[2] + i2, w * w2

    def interp(self, grids, q):
        """Values of several grids at q, one vector each."""
        flat = [u.reshape(-1) for u in grids]
        out = [torch.zeros(q.shape[1], dtype=grids[0].dtype, device=DEV) for _ in flat]
        for lin, w in self.taps(q):
            for o, u in zip(out, flat):
                o += w * u[lin]
        return out

    def spread(self, vals, q):
        """Several value vectors spread onto grids of their own."""
        out = [torch.zeros(self.g[0] * self.g[1] * self.g[2], dtype=v.dtype, device=DEV)
               for v in vals]
        for lin, w in self.taps(q):
            for o, v in zip(out, vals):
                if v.is_complex():
                    torch.view_as_real(o).index_add_(0, lin, torch.view_as_real(w * v))
                else:
                    o.index_add_(0, lin, w * v)
        return [o.reshape(self.g) for o in out]

    def warp_points(self, d):
        n = torch.stack(torch.meshgrid(*[torch.arange(s, device=DEV, dtype=torch.float64)
                                         for s in self.n], indexing="ij"))
        return (self.sigma * (n + d.double())).reshape(3, -1)

    def T(self, x, disps):
        """The warped image of every phase."""
        s = math.prod(self.g) / math.prod(self.n)
        X = self.deapod(torch.fft.fftshift(torch.fft.fftn(x)))
        u = torch.fft.ifftn(self.pad(X)) * s
        return [self.interp([u], self.warp_points(d))[0].reshape(self.n) for d in disps]

    def TH(self, ms, disps):
        u = 0
        for m, d in zip(ms, disps):
            u = u + self.spread([m.reshape(-1)], self.warp_points(d))[0]
        U = self.deapod(self.crop(torch.fft.fftn(u)))
        return torch.fft.ifftn(torch.fft.ifftshift(U))  # the 1/N of both directions cancel

    def kpoints(self, om):
        g = torch.tensor(self.g, dtype=torch.float64, device=DEV)
        return (om.double() * g / (2 * math.pi)).T.contiguous()

    def GS(self, m, om, smaps):
        out, q = [], self.kpoints(om)
        for c0 in range(0, smaps.shape[0], 4):
            grids = [torch.fft.fftn(self.pad(self.deapod(s.to(torch.complex128) * m)))
                     for s in smaps[c0:c0 + 4]]
            out += self.interp(grids, q)
        return torch.stack(out, 1)

    def GSH(self, y, om, smaps):
        w, q = 0, self.kpoints(om)
        for c0 in range(0, smaps.shape[0], 4):
            grids = self.spread([y[:, c] for c in range(c0, min(c0 + 4, y.shape[1]))], q)
            for s, u in zip(smaps[c0:c0 + 4], grids):
                v = self.deapod(self.crop(torch.fft.ifftn(u, norm="forward")))
                w = w + s.to(torch.complex128).conj() * v
        return w

    def A(self, x, inp):
        P = len(inp["coords"])
        ms = self.T(x, inp["disp"]) if inp["disp"] is not None else [x] * P
        return torch.cat([self.GS(m, om, inp["smaps"]) for m, om in zip(ms, inp["coords"])])

    def AH(self, y, inp):
        ys = torch.split(y, [om.shape[0] for om in inp["coords"]])
        ws = [self.GSH(v, om, inp["smaps"]) for v, om in zip(ys, inp["coords"])]
        return self.TH(ws, inp["disp"]) if inp["disp"] is not None else sum(ws)

    def E(self, x, inp, lam):
        if inp["coords"] is None:
            return self.TH(self.T(x, inp["disp"]), inp["disp"]) + lam * x
        return self.AH(self.A(x, inp), inp) + lam * x


def _haar(x):
    """One level of the orthonormal 3D Haar transform: the eight sub-bands along three new
    leading axes, index 0 of each the low-pass half."""
    for a in range(3):
        lo, hi = x.unfold(a + (x.dim() - 3), 2, 2).unbind(-1)
        x = torch.stack([(lo + hi), (lo - hi)], 0) * math.sqrt(0.5)
    return x


def _haar_inv(x):
    for a in reversed(range(3)):
        lo, hi = x.unbind(0)
        x = torch.stack([lo + hi, lo - hi], -1) * math.sqrt(0.5)
        # x: (..., n_a first of the trailing three axes, ..., 2): interleave along axis a
        d = x.dim() - 1 - 3 + a
        x = x.movedim(-1, d + 1).flatten(d, d + 1)
    return x


def _prox(v, tau, levels):
    def soft(c):
        mag = c.abs()
        return c * (1.0 - tau / mag.clamp_min(1e-300)).clamp_min(0.0)

    if levels == 0:
        return soft(v)
    b = _haar(v)
    low = _prox(b[0, 0, 0].clone(), tau, levels - 1)
    b = soft(b)
    b[0, 0, 0] = low
    return _haar_inv(b)


def _network(u, params):
    """z = u0 + N4^T (I + W5^T W5) N4 u0 of one residual (u: (2, n0, n1, n2)), with the masks of
    the four ReLU layers, as the symmetric form defines it (biases unused)."""
    conv, tr = torch.nn.functional.conv3d, torch.nn.functional.conv_transpose3d
    h, masks = u[None], []
    for w in params[:4]:
        h = conv(h, w, padding=1)
        masks.append((h > 0).to(h.dtype))
        h = h * masks[-1]
    g = h + tr(conv(h, params[4], padding=1), params[4], padding=1)
    for w, m in zip(reversed(params[:4]), reversed(masks)):
        g = tr(g * m, w, padding=1)
    return u + g[0]


def _train_exact(case, inp):
    """Losses, gradients and output in 64 bits (of the BF16-rounded weights, which the kernels
    read); activations unrounded."""
    nv = float(np.prod(_shape(case)))
    ws = [torch.from_numpy(w).to(DEV).bfloat16().double().requires_grad_() for w, _ in inp["params"]]
    real = lambda v: torch.stack([v.real, v.imag]).double()  # noqa: E731
    loss0, z0 = None, None
    for k, (r, e) in enumerate(zip(inp["r"], inp["e"])):
        s = (r.to(torch.complex128).abs().square().sum() / nv).sqrt()
        o = _network(real(r) / s, ws)
        t = real(e)
        loss = 1.0 - (o * t).sum() / (o.norm() * t.norm())
        loss.backward()
        if k == 0:
            loss0, z0 = float(loss), o.detach()
    grads = [(w.grad.cpu().numpy(), None) for w in ws]
    return {"loss": loss0, "grads": grads, "z": torch.complex(z0[0], z0[1])}


def exact(case, seed):
    inp = _inputs(case, seed)
    kind = case["kind"]
    if kind == "train":
        return _train_exact(case, inp)
    passes = {"normal": 2, "cg": 2 * case["steps"] + 1, "fista": 2 * case["steps"] + 1,
              "recon": case["steps"] + 3}.get(kind, 1)
    points = sum(_counts(case)) * case["coils"]
    if case["warp"]:
        points += case["phases"] * float(np.prod(_shape(case)))
    if points * case["width"] ** 3 * passes > 1e11:
        return None  # minutes
    geo = _Geo(case)
    c128 = lambda v: v.to(torch.complex128)  # noqa: E731
    if kind == "normal":
        return geo.E(c128(inp["x"]), inp, _lam(case))
    if kind == "forward":
        return geo.A(c128(inp["x"]), inp)
    if kind in ("adjoint", "replan"):
        return geo.AH(c128(inp["y"]), inp)
    if kind == "recon":
        q = geo.kpoints(inp["coords"][0])
        w = torch.ones(q.shape[1], dtype=torch.float64, device=DEV)
        for _ in range(DCF_ITERS):
            w = w / geo.interp(geo.spread([w], q), q)[0]
        return {"w": w, "img": [geo.AH(c128(y) * w[:, None], inp) for y in inp["y"]]}
    if kind == "cg":
        lam = _lam(case)
        b = geo.AH(c128(inp["y"]), inp)
        x, r = torch.zeros_like(b), b.clone()
        p, rr = r.clone(), r.abs().square().sum()
        for _ in range(case["steps"]):
            Ep = geo.E(p, inp, lam)
            al = rr / (p.conj() * Ep).sum().real
            x, r = x + al * p, r - al * Ep
            new = r.abs().square().sum()
            p, rr = r + (new / rr) * p, new
        return x
    # FISTA: gradient step with L, Haar prox, momentum
    b = geo.TH([c128(v) for v in inp["y"]], inp["disp"])
    x = torch.zeros_like(b)
    z, t, L = x.clone(), 1.0, _lip(case)
    for _ in range(case["steps"]):
        grad = 2.0 * (geo.E(z, inp, 0.0) - b)
        new = _prox(z - grad / L, FISTA_LAMBDA / L, 3)
        t1 = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        z, x, t = new + ((t - 1.0) / t1) * (new - x), new, t1
    return x
