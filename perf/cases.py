"""The work whose time and accuracy count: one entry per way the library is used.

A case names a kind of call (below), the geometry of its problem and the
options that are on.  Objects, displacements, probes and scans follow the
repository's own input recipe (paper_2312_14907_gb300.synth); the measured
counts are Poisson draws of a plain torch forward model, so they do not come
from the library's kernels, and the state a call is made at is a generic one
near the truth, as in the middle of a reconstruction.

Kinds:
  grad      loss and gradient over every frame (options: background, one
            probe per peak, positions off the pixel grid, reproducible sums)
  autograd  the loss as a torch autograd function whose backward recomputes
  steps     optimizer iterations replayed from a captured graph, from a
            restart at the given state
  adam      minibatch Adam iterations resumed from a checkpoint
  batch     loss and gradient of several problems of different sizes
  forward   model intensities of every frame
  host      loss and gradient on page-locked host buffers, counts included
  project   the projection of a displacement field onto unwrapped phases

The loss and df/dalpha of a call are sums of FP32 terms; they are taken as
float32, the type of the variables they serve (as the autograd function
does for its gradients), with the other outputs as the call returns them.
"""
import math

import numpy as np
import torch

from paper_2312_14907_gb300 import mpbp, synth

PHOTONS = 1e4          # expected counts of a frame inside the support
STEP_WEIGHTS = {"w_rho": 1.0, "w_u": 1e-3, "w_alpha": 1e-3}
ADAM = {"lr_u": 0.01, "lr_chi": 0.1, "lr_alpha": 0.1, "beta1": 0.9, "beta2": 0.999, "eps": 1e-8}
ADAM_T = 200           # minibatch steps behind the checkpoint of an adam case
CHUNK = 1 << 24        # frame pixels per chunk of the torch model


def _geometry(n1, n2, m, d, rows, cols, step, **options):
    return dict({"n1": n1, "n2": n2, "m": m, "d": d, "rows": rows, "cols": cols, "step": step}, **options)


def listed():
    return [
        # the smallest problem in use, 147 frames: launches and latency
        dict(name="grad-64-m32", kind="grad", **_geometry(64, 64, 32, 3, 7, 7, 4)),
        # the ordinary interactive size: one evaluation of a line search or
        # of an outside optimizer
        dict(name="grad-256-m64", kind="grad", **_geometry(256, 256, 64, 3, 31, 31, 6)),
        # the largest data set of one GPU: 87,846 frames, the scan
        # overhanging the object
        dict(name="grad-1024-m128", kind="grad", **_geometry(1024, 1024, 128, 6, 121, 121, 8)),
        # the production loop: captured gradient-descent iterations
        dict(name="steps-512-m128", kind="steps", count=3, **_geometry(512, 512, 128, 4, 61, 61, 6)),
        # the paper's own iteration: minibatches of 50 shuffled frames
        dict(name="adam-256-m64-b50", kind="adam", batch=50, count=8, **_geometry(256, 256, 64, 3, 31, 31, 6)),
        # many independent reconstructions of uneven sizes at once
        dict(name="batch-16", kind="batch", count=16, lo=128, hi=512),
        # simulation: the intensities of 14,884 frames (experiment planning, synthetic data)
        dict(name="forward-512-m128", kind="forward", **_geometry(512, 512, 128, 4, 61, 61, 6)),
        # detector counts arriving in host memory, 16 bits each
        dict(name="host16-256-m64", kind="host", counts16=True, **_geometry(256, 256, 64, 3, 31, 31, 6)),
        # a beamline crop: odd ragged grid, irregular scan, one probe per
        # peak, background; the loss inside a torch program
        dict(name="autograd-301x333-m64", kind="autograd", probes=True, bg=True, jitter=True,
             **_geometry(301, 333, 64, 4, 33, 37, 7)),
        # measured scan positions: every frame its own shifted probe
        dict(name="subpixel-512-m128", kind="grad", subpixel=True, **_geometry(512, 512, 128, 3, 41, 41, 9)),
        # the displacement projector that follows an Adam step
        dict(name="project-256", kind="project", **_geometry(256, 256, 64, 3, 31, 31, 6)),
        # a run that has to repeat bit for bit
        dict(name="repeatable-256-m64", kind="grad", repeatable=True, **_geometry(256, 256, 64, 3, 31, 31, 6)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grad"] * 5 + ["steps", "steps", "adam", "adam", "batch", "forward", "host", "autograd",
                                      "autograd", "project"])
    if kind == "batch":
        lo = rng.randrange(128, 257)
        return {"kind": kind, "count": rng.randrange(3, 15), "lo": lo, "hi": rng.randrange(lo, 481)}
    m = rng.choice([32, 64, 64, 128, 128])
    n1 = _log(rng, max(64, 2 * m), 1024)
    n2 = n1 if rng.random() < 0.6 else max(2 * m, min(1024, int(n1 * rng.uniform(0.75, 1.3))))
    c = {"kind": kind, "n1": n1, "n2": n2, "m": m, "d": rng.randrange(2, 7), "step": rng.randrange(4, 11)}
    most = 8e8         # frame pixels
    if kind == "project":
        c["d"] = rng.randrange(2, 4)
    if kind == "host":
        most = 2.4e7
        c["counts16"] = rng.random() < 0.5
    if kind == "forward":
        most = 3e8
    if kind == "autograd":
        most = 4e8
    if kind == "steps":
        c["count"] = rng.randrange(2, 5)
        most /= c["count"]
    if kind == "adam":
        c["batch"], c["count"] = rng.randrange(20, 129), rng.randrange(3, 13)
    if kind in ("grad", "autograd", "forward", "steps", "adam"):
        c["jitter"] = rng.random() < 0.25
        c["probes"] = rng.random() < 0.2
    if kind in ("grad", "autograd", "steps"):
        c["bg"] = rng.random() < 0.2
        if c["bg"]:
            most /= 2
    if kind == "grad":
        option = rng.random()
        if option < 0.2:
            c["subpixel"] = True
            most /= 4
        elif option < 0.4 and m >= 64 and n2 % 2 == 0:
            c["repeatable"] = True
            most /= 3
    over = rng.choice([0, 0, m // 2])      # how far the scan overhangs each edge
    while True:
        c["rows"] = max(2, (n1 + 2 * over - m) // c["step"] + 1)
        c["cols"] = max(2, (n2 + 2 * over - m) // c["step"] + 1)
        if c["d"] * c["rows"] * c["cols"] * m * m <= most or (c["step"] >= m and c["d"] == 2):
            return c
        if c["step"] < m:
            c["step"] += 1
        else:
            c["d"] -= 1


# ---------------------------------------------------------------- inputs

def _directions(d):
    if d <= 3:
        return synth.AXIS_PEAKS[:d].copy()
    if d == 4:
        return synth.PAPER_PEAKS.copy()
    g = np.random.default_rng(synth.SEED_BASE + 5).standard_normal((d, 3))
    return g / np.linalg.norm(g, axis=1, keepdims=True)


def _spec(c, seed):
    m = c["m"]
    return synth.ProblemSpec("case", c["n1"], c["n2"], 3, c["d"], m, c["rows"], c["step"], _directions(c["d"]),
                             synth.SEED_BASE + seed, bumps=8, straight=2, curved=2, sigma=6.0 * m / 32,
                             quad=0.01 * (32.0 / m) ** 2,
                             alpha_true=synth.PAPER_SCALINGS.copy() if c["d"] == 4 else None,
                             probe_per_peak=bool(c.get("probes")))


def _scan(c, seed):
    """A raster over the object, centred; jitter: each position up to 2 pixels off it."""
    r0 = (c["n1"] - ((c["rows"] - 1) * c["step"] + c["m"])) // 2
    c0 = (c["n2"] - ((c["cols"] - 1) * c["step"] + c["m"])) // 2
    r, k = np.meshgrid(r0 + c["step"] * np.arange(c["rows"]), c0 + c["step"] * np.arange(c["cols"]), indexing="ij")
    s = np.stack([r.ravel(), k.ravel()], axis=1)
    if c.get("jitter"):
        s = s + np.random.default_rng(seed + 11).integers(-2, 3, s.shape)
    return s.astype(np.int32)


def _cuda(a, dtype=np.float32):
    return torch.from_numpy(np.ascontiguousarray(a, dtype)).cuda()


class _Inputs:
    """One problem's inputs on the GPU, made from the seed with numpy and torch alone."""

    def __init__(self, c, seed, counts=True):
        self.c, self.seed = c, seed
        self.spec, self.scan = _spec(c, seed), _scan(c, seed)
        m, d = c["m"], c["d"]
        self.gen = torch.Generator(device="cuda").manual_seed(1000 + seed)
        rho, u = (_cuda(a) for a in synth.truth(self.spec))
        alpha = _cuda(synth.alpha_truth(self.spec))
        probe = synth.probe(self.spec)
        probe = probe * math.sqrt(PHOTONS / (m * m * float((np.abs(probe.reshape(-1, m, m)[0]) ** 2).sum())))
        self.probe = _cuda(probe, np.complex64)
        self.offsets = None
        if c.get("subpixel"):
            self.offsets = np.random.default_rng(seed + 12).uniform(-0.5, 0.5, (self.scan.shape[0], 2))
        self.bg = self.y = None
        if counts:
            shape = (d, self.scan.shape[0], m, m)
            if c.get("bg"):
                self.bg = 0.1 * self._rand(shape)
            self.y = torch.empty(shape, device="cuda")
            flat = self.y.view(-1, m, m)
            model = _Model(self, torch.float32)
            for lo, hi in model.chunks():
                mean = model.intensity(model.objects(rho, u, alpha), torch.arange(lo, hi, device="cuda"))
                if self.bg is not None:
                    mean += self.bg.view(-1, m, m)[lo:hi]
                flat[lo:hi] = torch.poisson(mean, generator=self.gen)
        # the state of the call
        self.rho = rho + 0.2 + 0.05 * self._randn(rho.shape)
        self.u = u + 0.05 * self._randn(u.shape)
        self.alpha = alpha * (1.0 + 0.05 * self._randn(alpha.shape))
        self.alpha[0] = 1.0

    def _rand(self, shape):
        return torch.rand(shape, generator=self.gen, device="cuda")

    def _randn(self, shape):
        return torch.randn(shape, generator=self.gen, device="cuda")

    def problem(self):
        p = mpbp.Problem.from_spec(self.spec, self.scan)
        p.set_probe(self.probe)
        if self.offsets is not None:
            p.set_scan_offsets(self.offsets)
        if self.c.get("repeatable"):
            p.set_deterministic(True)
        if self.y is not None:
            p.set_data(self.y, self.bg)
        return p

    def first_step(self):
        """Inverse of the curvature bound of one density pixel: M^2 max|P|^2 x covering frames."""
        c = self.c
        cover = (c["m"] / c["step"]) ** 2 * c["d"]
        return 1.0 / (c["m"] ** 2 * float(self.probe.abs().max()) ** 2 * cover)

    def minibatches(self):
        order = synth.epoch_order(self.c["d"] * self.scan.shape[0], self.seed + 13)
        b = self.c["batch"]
        lists = [order[k:k + b] for k in range(0, len(order), b)][-self.c["count"]:]   # the epoch's end: the last one is ragged
        return [_cuda(x, np.int32) for x in lists]


# ---------------------------------------------------------------- the model in torch

class _Model:
    """Objects, far fields, loss and gradient in plain torch ops at a chosen precision."""

    def __init__(self, x, dtype):
        c, self.x, self.dtype = x.c, x, dtype
        self.cdtype = torch.complex128 if dtype == torch.float64 else torch.complex64
        self.m, self.d, self.J = c["m"], c["d"], x.scan.shape[0]
        self.n1, self.n2, self.pad = c["n1"], c["n2"], c["m"] + 4
        self.G = torch.from_numpy(x.spec.G).cuda().to(dtype)
        self.scan = torch.from_numpy(x.scan.astype(np.int64)).cuda()
        self.k = torch.arange(self.m, device="cuda")
        self.P = x.probe.to(self.cdtype)

    def chunks(self):
        n = self.d * self.J
        b = max(1, CHUNK // (self.m * self.m))
        return [(lo, min(n, lo + b)) for lo in range(0, n, b)]

    def turns(self, u):
        return 2.0 * math.pi * torch.einsum("mc,cij->mij", self.G, u)

    def objects(self, rho, u, alpha):
        phase = self.turns(u)
        O = torch.polar((alpha[:, None, None] * rho).abs(), phase) * torch.sign(alpha[:, None, None] * rho)
        return torch.nn.functional.pad(O, (self.pad,) * 4)

    def index(self, f):
        """Flat index into the padded objects of every pixel of frames f."""
        s = self.scan[f % self.J] + self.pad
        w1, w2 = self.n1 + 2 * self.pad, self.n2 + 2 * self.pad
        rows = (f // self.J)[:, None] * w1 + s[:, :1] + self.k
        return rows[:, :, None] * w2 + (s[:, 1:] + self.k)[:, None, :]

    def probes(self, f):
        P = self.P[f // self.J] if self.P.dim() == 3 else self.P
        if self.x.offsets is None:
            return P
        d = torch.from_numpy(self.x.offsets).cuda()[f % self.J].to(self.dtype)
        q = (torch.fft.fftfreq(self.m, device="cuda", dtype=self.dtype) * 2.0 * math.pi)
        ramp = lambda t: torch.polar(torch.ones_like(t), t)  # noqa: E731
        shift = ramp(-q * d[:, :1])[:, :, None] * ramp(-q * d[:, 1:])[:, None, :]
        return torch.fft.ifft2(torch.fft.fft2(P) * shift)

    def intensity(self, O, f):
        psi = self.probes(f) * O.reshape(-1)[self.index(f)]
        return torch.fft.fft2(psi).abs().square()

    def loss_grad(self, rho, u, alpha, frames=None):
        O = self.objects(rho, u, alpha)
        acc = torch.zeros(O.numel(), 2, dtype=self.dtype, device="cuda")
        loss = torch.zeros((), dtype=torch.float64, device="cuda")
        y, bg = self.x.y.view(-1, self.m, self.m), self.x.bg
        lists = [torch.arange(lo, hi, device="cuda") for lo, hi in self.chunks()] if frames is None else [frames.long()]
        for f in lists:
            P, at = self.probes(f), self.index(f)
            far = torch.fft.fft2(P * O.reshape(-1)[at])
            I = far.real.square() + far.imag.square()
            if bg is not None:
                I = I + bg.view(-1, self.m, self.m)[f].to(self.dtype)
            amp = I.sqrt()
            r = amp - y[f].to(self.dtype).sqrt()
            loss += 0.5 * r.square().sum()
            chi = torch.where(amp > 0, r / amp, torch.zeros_like(r)) * far
            g = torch.view_as_real(P.conj() * torch.fft.ifft2(chi) * (self.m * self.m)).reshape(-1, 2)
            at = at.reshape(-1)
            acc[:, 0].scatter_add_(0, at, g[:, 0])
            acc[:, 1].scatter_add_(0, at, g[:, 1])
        w1, w2, p = self.n1 + 2 * self.pad, self.n2 + 2 * self.pad, self.pad
        A = torch.view_as_complex(acc).view(self.d, w1, w2)[:, p:p + self.n1, p:p + self.n2]
        phase = self.turns(u)
        T = torch.polar(torch.ones_like(phase), -phase) * A
        g_rho = (alpha[:, None, None] * T.real).sum(0)
        g_phi = alpha[:, None, None] * rho * T.imag
        g_u = 2.0 * math.pi * torch.einsum("mc,mij->cij", self.G, g_phi)
        return loss, g_rho, g_u, (rho * T.real).sum((1, 2))


# ---------------------------------------------------------------- batches

def _members(c):
    """The problems of a batch: sides from lo to hi, frames 32, 64 and 128, 3 and 4 peaks, growing scans."""
    out, last = [], max(1, c["count"] - 1)
    for i in range(c["count"]):
        n = 16 * round((c["lo"] + (c["hi"] - c["lo"]) * i / last) / 16)
        m = (32, 64, 128)[i % 3]
        while m > n // 2:
            m //= 2
        side = 15 + (46 * i) // last
        out.append(_geometry(n, n, m, 3 + i % 2, side, side, max(1, (n - m) // (side - 1)), kind="grad"))
    return out


# ---------------------------------------------------------------- prepare and run

class _Sums:
    """The loss and df/dalpha of a call side by side, so that one cast gives both."""

    def __init__(self, d):
        self.both = torch.empty(1 + d, dtype=torch.float64, device="cuda")

    def out(self, g_rho, g_u):
        return self.both[:1], g_rho, g_u, self.both[1:]


def prepare(case, seed):
    c, kind = dict(case), case["kind"]
    if kind == "batch":
        xs = [_Inputs(k, seed * 64 + i) for i, k in enumerate(_members(c))]
        return {"kind": kind, "problems": [x.problem() for x in xs], "states": [(x.rho, x.u, x.alpha) for x in xs]}
    if kind == "project":
        x = _Inputs(c, seed, counts=False)
        return {"kind": kind, "problem": x.problem(), "u": _wrapped_u(x), "mask": _cuda(synth.support_mask(x.spec))}
    x = _Inputs(c, seed, counts=kind != "forward")
    s = {"kind": kind, "rho": x.rho, "u": x.u, "alpha": x.alpha, "sums": _Sums(c["d"])}
    if kind == "host":
        s["problem"] = mpbp.Problem.from_spec(x.spec, x.scan)
        s["problem"].set_probe(x.probe)
        y = x.y.to(torch.uint16) if c["counts16"] else x.y
        s["y"] = y.cpu().pin_memory()
        for k in ("rho", "u", "alpha"):
            s[k] = s[k].cpu().pin_memory()
        s["out"] = tuple(torch.empty(n, dtype=t).pin_memory() for n, t in (
            ((1,), torch.float64), (x.rho.shape, torch.float32), (x.u.shape, torch.float32), ((c["d"],), torch.float64)))
        return s
    p = s["problem"] = x.problem()
    if kind == "autograd":
        for k in ("rho", "u", "alpha"):
            s[k].requires_grad_()
    if kind == "steps":
        s["count"] = c["count"]
        s["start"] = tuple(t.clone() for t in (x.rho, x.u, x.alpha))
        s["state"] = p.step_init(x.first_step(), **STEP_WEIGHTS)
        s["state0"] = s["state"].clone()
        p.step_capture(s["rho"], s["u"], s["alpha"], s["state"])
    if kind == "adam":
        s["mask"] = _cuda(synth.support_mask(x.spec))
        s["lists"] = x.minibatches()
        s["saved"], s["moments"] = _checkpoint(x)
        s["vars"] = tuple(t.clone() for t in s["saved"])
        s["state"] = p.adam_init(**ADAM)
        st = p.read_adam_state(s["state"])
        st.t = ADAM_T
        s["state0"] = torch.frombuffer(bytearray(st), dtype=torch.uint8).cuda()
    return s


def _checkpoint(x):
    """Variables and moments of an Adam run in progress: moments at the scale of a minibatch's gradients."""
    scale = x.c["m"] ** 2 * float(x.probe.abs().max()) ** 2
    g = lambda t: scale * x._randn(t.shape)  # noqa: E731
    at = torch.log(x.alpha.clamp(min=1e-3))
    vars_ = (torch.log(x.rho.clamp(min=0.2)), x.u, at)
    moments = []
    for t in vars_:
        m = 0.1 * g(t)
        v = 0.1 * g(t).square() + 0.05 * scale * scale
        moments += [m, v]
    return vars_, moments[:4] + [1e3 * moments[4].double(), 1e6 * moments[5].double()]


def _wrapped_u(x):
    """A smooth displacement with noise and two lines across which it jumps by a lattice vector, as Adam
    steps on wrapped phases leave it; there is one way to unwrap its phases."""
    spec = x.spec
    rng = np.random.default_rng(x.seed + 14)
    i, j = np.meshgrid(np.arange(spec.n1), np.arange(spec.n2), indexing="ij")
    u = 0.005 * rng.standard_normal((3, spec.n1, spec.n2)).clip(-3, 3)
    n = min(spec.n1, spec.n2)
    for _ in range(8):
        a, b, w = rng.uniform(0, spec.n1), rng.uniform(0, spec.n2), rng.uniform(n / 6, n / 3)
        v = rng.standard_normal(3)
        u += 0.4 * (v / np.linalg.norm(v))[:, None, None] * np.exp(-((i - a) ** 2 + (j - b) ** 2) / (2 * w * w))
    for c in range(2):
        th, a, b = rng.uniform(0, math.pi), rng.uniform(0.2, 0.8) * spec.n1, rng.uniform(0.2, 0.8) * spec.n2
        u[c] += rng.choice([-1.0, 1.0]) * ((i - a) * math.cos(th) > (j - b) * math.sin(th))
    return _cuda(u)


def run(s):
    kind = s["kind"]
    if kind == "batch":
        outs = mpbp.loss_grad_batched(s["problems"], s["states"])
        return [(f.float(), g_rho, g_u, g_alpha.float()) for f, g_rho, g_u, g_alpha in outs]
    p = s["problem"]
    if kind == "project":
        return p.project_displacement(s["u"].clone(), s["mask"])
    if kind == "forward":
        return p.forward(s["rho"], s["u"], s["alpha"])
    if kind == "grad":
        g_rho, g_u = torch.empty_like(s["rho"]), torch.empty_like(s["u"])
        p.loss_grad(s["rho"], s["u"], s["alpha"], out=s["sums"].out(g_rho, g_u))
        return s["sums"].both.float(), g_rho, g_u
    if kind == "host":
        f, g_rho, g_u, g_alpha = p.loss_grad_host(s["rho"], s["u"], s["alpha"], y=s["y"], out=s["out"])
        return torch.cat((f, g_alpha)).float(), g_rho, g_u
    if kind == "autograd":
        x = s["rho"], s["u"], s["alpha"]
        for t in x:
            t.grad = None
        loss = mpbp.mpbp_loss(*x, p, recompute=True)
        loss.backward()
        return loss.detach().float(), x[0].grad, x[1].grad, x[2].grad
    if kind == "steps":
        x = s["rho"], s["u"], s["alpha"]
        for t, t0 in zip(x, s["start"]):
            t.copy_(t0)
        s["state"].copy_(s["state0"])
        for _ in range(s["count"]):
            p.step_replay()
        return x + (s["state"].view(torch.float64)[:4].float(),)    # f_prev, |g|^2, t, f_last
    # adam: resume, then the minibatches
    for t, t0 in zip(s["vars"], s["saved"]):
        t.copy_(t0)
    s["state"].copy_(s["state0"])
    p.adam_set_state(s["moments"])
    for frames in s["lists"]:
        p.adam_step(frames, *s["vars"], s["state"], mask=s["mask"])
    moments = p.adam_get_state()
    return s["vars"] + moments[:4] + tuple(t.float() for t in moments[4:]) + (s["state"].view(torch.float64)[6:7].float(),)


# ---------------------------------------------------------------- work and exact values

def _pixels(c):
    return c["n1"] * c["n2"]


def _io(c):
    """rho, u, alpha read and their gradients written, and the probe."""
    return 8 * (4 * _pixels(c) + c["d"]) + 8 * c["m"] ** 2 * (c["d"] if c.get("probes") else 1)


def _eval(c, frames):
    """One loss and gradient over `frames` frames: counts (and background) read once; two 2-D transforms a frame
    (5 n log2 n each) and 24 flops a pixel; 30 flops a peak and object pixel."""
    mm = c["m"] ** 2
    probes = 8 * mm * c["rows"] * c["cols"] if c.get("subpixel") else 0
    return {"bytes": 4.0 * mm * frames * (2 if c.get("bg") else 1) + probes + _io(c),
            "flops": frames * mm * (10.0 * math.log2(mm) + 24.0) + 30.0 * c["d"] * _pixels(c)}


def _frames(c):
    return c["d"] * c["rows"] * c["cols"]


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        each = [_eval(k, _frames(k)) for k in _members(c)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    if kind == "project":
        return {"bytes": 4.0 * _pixels(c) * (2 * 3 + 1), "flops": _pixels(c) * c["d"] * 60.0}
    if kind == "forward":
        mm = c["m"] ** 2
        return {"bytes": 4.0 * mm * _frames(c) + _io(c) / 2,
                "flops": _frames(c) * mm * (5.0 * math.log2(mm) + 9.0) + 30.0 * c["d"] * _pixels(c)}
    if kind == "host":
        w = _eval(c, _frames(c))
        return dict(w, bytes=(2.0 if c["counts16"] else 4.0) * c["m"] ** 2 * _frames(c) + _io(c))
    if kind == "steps":
        return {k: c["count"] * v for k, v in _eval(c, _frames(c)).items()}
    if kind == "adam":
        n, b = _frames(c), c["batch"]
        sizes = [min(b, n - k) for k in range(0, n, b)][-c["count"]:]
        each = [_eval(c, k) for k in sizes]
        moments = 2.0 * 2 * 4 * 4 * _pixels(c)     # both moments of chi and u read and written
        return {"bytes": sum(e["bytes"] + moments for e in each), "flops": sum(e["flops"] for e in each)}
    return _eval(c, _frames(c))


def _exact_grad(x):
    model = _Model(x, torch.float64)
    return model.loss_grad(x.rho.double(), x.u.double(), x.alpha.double())


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind == "batch":
        out = []
        for i, k in enumerate(_members(c)):
            f, g_rho, g_u, g_alpha = _exact_grad(_Inputs(k, seed * 64 + i))
            out.append((f.view(1), g_rho, g_u, g_alpha))
        return out
    if kind == "project":
        return _exact_projection(_Inputs(c, seed, counts=False))
    x = _Inputs(c, seed, counts=kind != "forward")
    if kind == "forward":
        model = _Model(x, torch.float64)
        O = model.objects(x.rho.double(), x.u.double(), x.alpha.double())
        out = torch.empty(c["d"] * model.J, c["m"], c["m"], dtype=torch.float64, device="cuda")
        for lo, hi in model.chunks():
            out[lo:hi] = model.intensity(O, torch.arange(lo, hi, device="cuda"))
        return out.view(c["d"], model.J, c["m"], c["m"])
    if kind == "steps":
        return _exact_steps(x)
    if kind == "adam":
        return _exact_adam(x)
    f, g_rho, g_u, g_alpha = _exact_grad(x)
    if kind == "autograd":
        return f, g_rho, g_u, g_alpha
    both = torch.cat((f.view(1), g_alpha))
    return (both.cpu(), g_rho.cpu(), g_u.cpu()) if kind == "host" else (both, g_rho, g_u)


def _exact_steps(x):
    """Gradient descent with the lagged Armijo test, alpha_0 held."""
    model, w = _Model(x, torch.float64), (STEP_WEIGHTS["w_rho"], STEP_WEIGHTS["w_u"], STEP_WEIGHTS["w_alpha"])
    now, t, base, f_prev, gn2 = (x.rho.double(), x.u.double(), x.alpha.double()), x.first_step(), None, 0.0, 0.0
    for k in range(x.c["count"]):
        f, *g = model.loss_grad(*now)
        g[2][0] = 0.0
        f = float(f)
        if k == 0 or f <= f_prev - 1e-4 * t * gn2:
            base, f_prev = (now, g), f
            gn2 = sum(wi * float(gi.square().sum()) for wi, gi in zip(w, g))
            t = t * 1.25 if k else t
        else:
            t = t * 0.5
        now = tuple(b - t * wi * gi for b, gi, wi in zip(base[0], base[1], w))
    return now + (torch.tensor([f_prev, gn2, t, f], dtype=torch.float64, device="cuda"),)


def _exact_adam(x):
    model = _Model(x, torch.float64)
    mask = _cuda(synth.support_mask(x.spec)).double()
    lists = x.minibatches()
    v, mom = _checkpoint(x)
    chi, u, at = (t.double() for t in v)
    mom = [t.double() for t in mom]
    b1, b2 = ADAM["beta1"], ADAM["beta2"]
    for k, frames in enumerate(lists):
        rho, alpha = mask * chi.exp(), at.exp()
        alpha[0] = 1.0
        f, g_rho, g_u, g_alpha = model.loss_grad(rho, u, alpha, frames)
        t = ADAM_T + 1 + k
        new = []
        for i, (var, g, lr) in enumerate(((chi, rho * g_rho, ADAM["lr_chi"]), (u, g_u, ADAM["lr_u"]),
                                          (at, alpha * g_alpha, ADAM["lr_alpha"]))):
            m = b1 * mom[2 * i] + (1 - b1) * g
            s = b2 * mom[2 * i + 1] + (1 - b2) * g * g
            step = lr * (m / (1 - b1 ** t)) / ((s / (1 - b2 ** t)).sqrt() + ADAM["eps"])
            if i == 2:     # alpha_0 is no variable
                m[0], s[0], step[0] = mom[4][0], mom[5][0], 0.0
            mom[2 * i], mom[2 * i + 1] = m, s
            new.append(var - step)
        chi, u, at = new
    return (chi, u, at) + tuple(mom) + (f.view(1),)


def _exact_projection(x):
    """u moved onto phases unwrapped inside the support, whose first pixel keeps its wrapped phase."""
    u = _wrapped_u(x).cpu().numpy().astype(np.float64)
    mask = synth.support_mask(x.spec) > 0
    rows, cols = np.flatnonzero(mask.any(1)), np.flatnonzero(mask.any(0))
    box = slice(rows[0], rows[-1] + 1), slice(cols[0], cols[-1] + 1)
    G = x.spec.G
    phase = 2.0 * math.pi * np.einsum("mc,cij->mij", G, u)
    wrapped = np.mod(phase + math.pi, 2.0 * math.pi) - math.pi
    delta = np.zeros_like(phase)
    for k in range(G.shape[0]):
        first = wrapped[k][box]
        flat = first.copy()
        flat[:, 0] = np.unwrap(flat[:, 0])
        flat = np.unwrap(flat, axis=1)
        delta[k][box] = flat - phase[k][box]
    return u + np.einsum("cm,mij->cij", np.linalg.pinv(G), delta) / (2.0 * math.pi)
