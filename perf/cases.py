"""Performance cases of the LM-MEW OSEM library: what a user has it do, through
the Python binding over the C ABI.

Objects are elliptical water bodies with a bone disc and hot lesions, events
are drawn by a small photon simulation (forced detection, first-order
scatter), so the events fall where the detector and the lines put them.  The
scanners are those of this repository's workloads:

* ``lmmew_32``    32 x 32 pixels of 0.8 cm, 32 angles, 32 bins, 16 x 16 scatter cells
* ``lmmew_64``    64 x 64 of 0.6 cm, 60 angles, 64 bins, 64 x 64 scatter cells
* ``lmmew_128``   128 x 128 of 0.3 cm, 120 angles, 128 bins, 64 x 64 scatter cells
* ``paper_study`` 64 x 64 of 0.46 cm, 120 angles, 64 bins, 32 x 32 scatter cells,
  the three photopeak windows

and, for drawn cases, scanners in between with odd angle and bin counts.
"""
import math

import numpy as np
import torch

import paper_2305_17111_gb300 as lm

LINES = (82.0, 154.0, 270.0)            # keV, Ra-223's three main peaks
YIELDS = (0.6, 0.2, 0.2)
KNOTS = (82.0, 154.0, 270.0)
MU_WATER = (0.184, 0.148, 0.121)        # 1/cm at the knots
FWHM_FRAC, E_REF = 0.10, 140.0          # energy resolution: 10 % at 140 keV, ~ E^-1/2
COLL_FWHM0, COLL_SLOPE = 0.3, 0.02      # collimator FWHM at the face and per cm of depth
ME_C2 = 510.99895
TO_SIGMA = 1.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))
WINDOWS = {"wide": ((50.0, 300.0),),
           "peaks": ((68.0, 102.0), (123.0, 184.0), (243.0, 297.0))}

G32 = dict(n=32, pixel_cm=0.8, n_angles=32, n_bins=32, scatter_n=16, windows="wide")
G64 = dict(n=64, pixel_cm=0.6, n_angles=60, n_bins=64, scatter_n=64, windows="wide")
G128 = dict(n=128, pixel_cm=0.3, n_angles=120, n_bins=128, scatter_n=64, windows="wide")
STUDY = dict(n=64, pixel_cm=0.46, n_angles=120, n_bins=64, scatter_n=32, windows="peaks")


def listed():
    return [
        # one projection of a short acquisition or of one bed position: the
        # smallest call, where launches and latency count
        dict(name="forward_32", op="forward", events=2_000, **G32),
        # a whole small reconstruction with its log-likelihood watched
        dict(name="osem_32_loglik", op="osem", events=2_000, subsets=4, iters=1, loglik=True, **G32),
        # forward projection of a full list (likelihood, residuals, simulation checks)
        dict(name="forward_64", op="forward", events=300_000, **G64),
        # back projection of an odd-sized list with the caller's weights
        dict(name="backproject_64", op="backproject", events=123_457, **G64),
        # the 64 x 64 reconstruction as it is run: 8 subsets x 10 iterations
        dict(name="osem_64", op="osem", events=300_000, subsets=8, iters=10, loglik=False, **G64),
        # one noise realisation of the paper's study: ~10^4 events, 4 x 16
        dict(name="osem_study", op="osem", events=10_007, subsets=4, iters=16, loglik=False, **STUDY),
        # noise realisations of the study reconstructed together
        dict(name="batch_study", op="batch", events=10_000, realisations=24, subsets=4, iters=16,
             **STUDY),
        # one iteration over a million events at 128 x 128
        dict(name="osem_128", op="osem", events=1_000_000, subsets=8, iters=1, loglik=False, **G128),
        # a new patient: the model built from an attenuation map, its sensitivities read
        dict(name="model_64", op="model", events=0, subsets=8, **G64),
        # reconstruction with the learned scatter term on the node grid
        dict(name="osem_learned_64", op="osem_learned", events=50_000, subsets=8, iters=1, stride=2,
             **G64),
        # the scatter network evaluated on a block of inputs
        dict(name="net_forward", op="net_forward", rows=500_003),
        # its gradient on one training minibatch
        dict(name="net_gradient", op="net_gradient", rows=16_384),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["forward", "backproject", "osem", "osem", "batch", "model", "osem_learned",
                     "net_forward", "net_gradient"])
    if op == "net_forward":
        return dict(op=op, rows=log_int(1_000, 1_000_000))
    if op == "net_gradient":
        return dict(op=op, rows=log_int(500, 65_536))
    n = rng.choice([24, 32, 48, 64])
    geo = dict(n=n, pixel_cm=rng.choice([25.6, 29.44, 38.4]) / n, n_angles=rng.randint(24, 90),
               n_bins=rng.randint(max(20, n // 2), n + 8), scatter_n=n // rng.choice([1, 2]),
               windows=rng.choice(["wide", "wide", "peaks"]))
    if op in ("forward", "backproject"):
        return dict(op=op, events=log_int(500, 600_000), **geo)
    if op == "model":
        return dict(op=op, events=0, subsets=rng.randint(1, 12), **geo)
    if op == "osem":
        return dict(op=op, events=log_int(1_000, 300_000), subsets=rng.randint(1, 12),
                    iters=rng.randint(1, 10), loglik=False, **geo)
    if op == "batch":
        return dict(op=op, events=log_int(1_000, 20_000), realisations=rng.randint(2, 16),
                    subsets=rng.randint(1, 8), iters=rng.randint(1, 10), **geo)
    return dict(op=op, events=log_int(1_000, 50_000), subsets=rng.randint(1, 8), iters=1,
                stride=rng.randint(2, 4), **geo)


# ------------------------------------------------------------------ inputs
def make_object(case, seed):
    """(rho, activity) as [n, n] float32 arrays: an 11 x 9 cm water ellipse with
    a bone disc and lesions whose places follow the seed."""
    n, h = case["n"], case["pixel_cm"]
    rng = np.random.default_rng(seed)
    scale = min(1.0, n * h / 25.6)
    c = (np.arange(n) + 0.5 - n / 2.0) * h
    y, x = np.meshgrid(c, c, indexing="ij")
    body = (x / (11.0 * scale)) ** 2 + (y / (9.0 * scale)) ** 2 <= 1.0
    rho, act = np.where(body, 1.0, 0.0), np.where(body, 1.0, 0.0)

    def disc(r):
        t, d = rng.uniform(0.0, 2.0 * math.pi), rng.uniform(2.0, 5.5) * scale
        return body & ((x - d * math.cos(t)) ** 2 + (y - d * math.sin(t)) ** 2 <= r * r)

    rho[disc(2.0 * scale)] = 1.6
    for r in (1.4, 1.0):
        act[disc(r * scale)] = 8.0
    return rho.astype(np.float32), act.astype(np.float32)


def _mu(e):
    k, m = KNOTS, MU_WATER
    s0, s1 = (m[1] - m[0]) / (k[1] - k[0]), (m[2] - m[1]) / (k[2] - k[1])
    return torch.where(e < k[1], m[0] + (e - k[0]) * s0, m[1] + (e - k[1]) * s1)


def make_events(case, act, count, seed):
    """(angle, bin, energy) CUDA tensors of `count` detected events."""
    n, h, A, B = case["n"], case["pixel_cm"], case["n_angles"], case["n_bins"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    half, scale = 0.5 * n * h, min(1.0, n * h / 25.6)
    ax, ay = 11.0 * scale, 9.0 * scale
    cdf = torch.from_numpy(np.cumsum(act.reshape(-1), dtype=np.float64)).cuda()
    ycdf = torch.tensor(np.cumsum(YIELDS), device="cuda")
    win = WINDOWS[case["windows"]]
    out, have = [], 0

    def u(k):
        return torch.rand(k, generator=g, device="cuda")

    def chord(x, y, c, s):   # way out of the ellipse along (c, s)
        a = (c / ax) ** 2 + (s / ay) ** 2
        b = x * c / ax ** 2 + y * s / ay ** 2
        d = (x / ax) ** 2 + (y / ay) ** 2 - 1.0
        return (-b + torch.sqrt(torch.clamp(b * b - a * d, min=0.0))) / a

    while have < count:
        k = min(6 * count + 4096, 1 << 22)
        pix = torch.searchsorted(cdf, u(k).double() * cdf[-1]).clamp(max=n * n - 1)
        x = ((pix % n) + u(k) - 0.5 * n) * h
        y = (torch.div(pix, n, rounding_mode="floor") + u(k) - 0.5 * n) * h
        e0 = torch.tensor(LINES, device="cuda")[
            torch.searchsorted(ycdf, u(k).double()).clamp(max=len(LINES) - 1)]
        a = (u(k) * A).long().clamp(max=A - 1)
        th = a * (2.0 * math.pi / A)
        c, s = torch.cos(th), torch.sin(th)
        # unscattered: survive the way out; scattered: one Compton interaction
        # at an exponential distance along a random direction, then out
        phi = u(k) * (2.0 * math.pi)
        dist = -torch.log(u(k).clamp(min=1e-7)) / _mu(e0)
        px, py = x + dist * torch.cos(phi), y + dist * torch.sin(phi)
        scat = (u(k) < 0.6) & ((px / ax) ** 2 + (py / ay) ** 2 < 1.0)
        r = 1.0 / (1.0 + (e0 / ME_C2) * (1.0 - torch.cos(phi - th)))
        kn = r * r * (r + 1.0 / r - torch.sin(phi - th) ** 2) / 2.0
        e1 = torch.where(scat, e0 * r, e0)
        ox, oy = torch.where(scat, px, x), torch.where(scat, py, y)
        keep = u(k) < torch.exp(-_mu(e1) * chord(ox, oy, c, s)) * torch.where(scat, kn, torch.ones_like(kn))
        depth = half - (ox * c + oy * s)
        pos = -ox * s + oy * c + (COLL_FWHM0 + COLL_SLOPE * depth) * TO_SIGMA * torch.randn(
            k, generator=g, device="cuda")
        b = torch.floor((pos + half) / (2.0 * half) * B).long()
        eh = e1 + FWHM_FRAC * torch.sqrt(e1 * E_REF) * TO_SIGMA * torch.randn(
            k, generator=g, device="cuda")
        inside = torch.zeros_like(keep)
        for lo, hi in win:
            inside |= (eh >= lo) & (eh < hi)
        i = torch.nonzero(keep & inside & (b >= 0) & (b < B)).reshape(-1)[: count - have]
        out.append((a[i], b[i], eh[i]))
        have += i.numel()
    return tuple(torch.cat([o[j] for o in out]) for j in range(3))


def device_events(ev):
    return lm.DeviceEvents(ev[0].to(torch.int16), ev[1].to(torch.int16), ev[2])


def model_args(case, rho):
    return dict(n=case["n"], pixel_cm=case["pixel_cm"], n_angles=case["n_angles"],
                n_bins=case["n_bins"], rho=rho, knot_keV=KNOTS, mu_water_cm=MU_WATER,
                scatter_n=case["scatter_n"], line_keV=LINES, yields=YIELDS,
                windows=WINDOWS[case["windows"]], fwhm_frac=FWHM_FRAC, e_ref_keV=E_REF,
                coll_fwhm0_cm=COLL_FWHM0, coll_fwhm_slope=COLL_SLOPE,
                n_subsets=case.get("subsets", 1))


def make_params(seed):
    """Xavier-uniform network parameters (float32, the library's order)."""
    rng = np.random.default_rng(seed)

    def xavier(rows, cols):
        lim = math.sqrt(6.0 / (rows + cols))
        return rng.uniform(-lim, lim, rows * cols)

    def bias():
        return rng.uniform(-0.1, 0.1, 128)

    p = [xavier(128, 32), bias(), xavier(128, 128), bias(), xavier(128, 128), bias(),
         xavier(1, 128), np.array([-10.0])]
    return np.concatenate(p).astype(np.float32)


def make_rows(rows, seed):
    """Network inputs in their ranges: geometry, energy, line, optical depths."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((rows, 32), generator=g, device="cuda") * 2.0 - 1.0
    line = torch.randint(0, 3, (rows,), generator=g, device="cuda")
    x[:, 6:9] = torch.nn.functional.one_hot(line, 3).float()
    x[:, 9:17] = x[:, 9:17].abs()
    x[:, 29:32] = 0.0
    return x


def prepare(case, seed):
    op = case["op"]
    st = {"case": case}
    if op in ("net_forward", "net_gradient"):
        st["net"] = lm.Surrogate(0)
        st["net"].set_params(make_params(seed))
        st["x"] = make_rows(case["rows"], seed)
        if op == "net_gradient":
            g = torch.Generator(device="cuda").manual_seed(seed + 1)
            st["target"] = -10.0 + 3.0 * torch.randn(case["rows"], generator=g, device="cuda")
            st["weight"] = torch.rand(case["rows"], generator=g, device="cuda") + 0.5
        return st
    rho, act = make_object(case, seed)
    if op == "model":
        st["args"] = model_args(case, rho)
        return st
    st["model"] = lm.Model(**model_args(case, rho))
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    body = torch.from_numpy((rho.reshape(-1) > 0).astype(np.float32)).cuda()
    if op == "batch":
        sizes = np.random.default_rng(seed).integers(
            int(0.8 * case["events"]), int(1.2 * case["events"]) + 1, size=case["realisations"])
        ev = make_events(case, act, int(sizes.sum()), seed)
        off = np.concatenate([[0], np.cumsum(sizes)])
        st["events"] = [device_events(tuple(t[off[i]:off[i + 1]] for t in ev))
                        for i in range(len(sizes))]
        st["image"] = body.repeat(len(sizes), 1).contiguous()
        return st
    st["events"] = device_events(make_events(case, act, case["events"], seed))
    if op == "forward":
        st["image"] = body * (0.2 + 2.8 * torch.rand(body.numel(), generator=g, device="cuda"))
    elif op == "backproject":
        st["weight"] = 0.1 + 0.9 * torch.rand(case["events"], generator=g, device="cuda")
    else:
        st["image"] = body
    if op == "osem_learned":
        st["net"] = lm.Surrogate(0)
        st["net"].set_params(make_params(seed))
        st["model"].set_coarse_stride(case["stride"])
        st["model"].set_scatter_model("surrogate_coarse", st["net"])
    return st


# ------------------------------------------------------------------- a pass
def run(state):
    case = state["case"]
    op = case["op"]
    if op == "net_forward":
        return state["net"].forward(state["x"])
    if op == "net_gradient":
        grad, loss = state["net"].gradient(state["x"], state["target"], state["weight"])
        return {"grad": grad, "loss": loss}
    if op == "model":
        m = lm.Model(**state["args"])
        out = {"all": m.sensitivity(-1), "last": m.sensitivity(case["subsets"] - 1)}
        m.close()
        return out
    m = state["model"]
    if op == "forward":
        return m.forward(state["events"], state["image"])
    if op == "backproject":
        return m.backproject(state["events"], state["weight"])
    img = state["image"].clone()
    if op == "batch":
        return m.osem_batch(state["events"], img, case["subsets"], case["iters"])
    if case.get("loglik"):
        ll = torch.zeros(case["iters"] * case["subsets"], dtype=torch.float64, device="cuda")
        m.osem(state["events"], img, case["subsets"], case["iters"], loglik=ll)
        return {"image": img, "loglik": ll}
    return m.osem(state["events"], img, case["subsets"], case["iters"])


def support_size(case):
    rho, _ = make_object(case, 0)
    return int((rho > 0).sum())


def work(case):
    op = case["op"]
    if op in ("net_forward", "net_gradient"):
        # multiply-adds of the four layers; the gradient takes them three times
        flops = 2.0 * case["rows"] * (32 * 128 + 2 * 128 * 128 + 128)
        if op == "net_forward":
            return {"bytes": case["rows"] * 4.0 * 33, "flops": flops}
        return {"bytes": case["rows"] * 4.0 * 34 + 37_377 * 8.0, "flops": 3.0 * flops}
    pix, nq = case["n"] ** 2, support_size(case)
    if op == "model":
        # one attenuation map in, two sensitivity images out; every path (voxel,
        # scatter cell of the body, angle, line) enters the sensitivity once
        cells = nq * (case["scatter_n"] / case["n"]) ** 2
        return {"bytes": pix * 4.0 + pix * 16.0,
                "flops": 2.0 * case["n_angles"] * len(LINES) * nq * cells}
    ev = case["events"] * case.get("realisations", 1)
    # an event (8 bytes) read once; every (event, support voxel) pair enters a
    # projection with one multiply-add
    if op in ("forward", "backproject"):
        return {"bytes": ev * 12.0 + pix * 4.0, "flops": 2.0 * ev * nq}
    return {"bytes": ev * 8.0 + pix * 8.0 * case.get("realisations", 1),
            "flops": 4.0 * ev * nq * case["iters"]}


# ------------------------------------------- the same, plainly, in 64 bits
class Plain:
    """The path model in plain torch, double precision: line integrals through
    the density map, path weights, rows and sensitivities."""

    def __init__(self, case, rho):
        self.case = case
        n, self.h, self.A, self.B = case["n"], case["pixel_cm"], case["n_angles"], case["n_bins"]
        self.n, self.S = n, case["scatter_n"]
        dev = self.dev = torch.device("cuda")
        self.rho = torch.from_numpy(rho).to(dev).double()
        self.pix = torch.nonzero(self.rho.reshape(-1) > 0).reshape(-1)
        self.qx, self.qy = (self.pix % n) + 0.5, torch.div(self.pix, n, rounding_mode="floor") + 0.5
        f = n // self.S
        cells = self.rho.reshape(self.S, f, self.S, f).mean(dim=(1, 3)).reshape(-1)
        cell = torch.nonzero(cells > 0).reshape(-1)
        self.p_rho = cells[cell]
        self.px = ((cell % self.S) + 0.5) * f
        self.py = (torch.div(cell, self.S, rounding_mode="floor") + 0.5) * f
        own = torch.div(torch.floor(self.qy), f, rounding_mode="floor") * self.S + torch.div(
            torch.floor(self.qx), f, rounding_mode="floor")
        self.own = own[:, None] == cell[None, :]
        # float32 parameters, as the library takes them
        f32 = lambda v: float(np.float32(v))  # noqa: E731
        self.h = f32(self.h)
        self.lines, self.yields = [f32(v) for v in LINES], [f32(v) for v in YIELDS]
        self.mu_k, self.e_k = [f32(v) for v in MU_WATER], [f32(v) for v in KNOTS]
        self.frac, self.f0, self.slope = f32(FWHM_FRAC), f32(COLL_FWHM0), f32(COLL_SLOPE)
        self.win = WINDOWS[case["windows"]]
        self.half = 0.5 * n * self.h
        self.area = (f * self.h) ** 2
        nq, npt = self.qx.numel(), self.px.numel()
        i = torch.arange(nq, device=dev).repeat_interleave(npt)
        j = torch.arange(npt, device=dev).repeat(nq)
        self.g_qp = (self.h * self.line(self.qx[i].double(), self.qy[i].double(), self.px[j].double(),
                                        self.py[j].double())).reshape(nq, npt)
        self.dx = (self.px[None, :] - self.qx[:, None]).double() * self.h
        self.dy = (self.py[None, :] - self.qy[:, None]).double() * self.h
        self.d = torch.sqrt(self.dx ** 2 + self.dy ** 2)
        self.kn_norm = [self.plane_norm(e) for e in self.lines]

    def line(self, x0, y0, x1, y1):
        """Density integral along segments, pixel units: cut at every grid
        line, each piece taken at its midpoint (a piece on a grid line: the
        mean of its two sides)."""
        out, n = torch.empty_like(x0), self.n
        grid = torch.arange(n + 1, device=self.dev, dtype=torch.float64)
        pad = torch.zeros((n + 2, n + 2), dtype=torch.float64, device=self.dev)
        pad[1:-1, 1:-1] = self.rho
        flat = pad.reshape(-1)
        for s in range(0, x0.numel(), 1 << 18):
            sl = slice(s, s + (1 << 18))
            a, b, c, d = x0[sl, None], y0[sl, None], x1[sl, None], y1[sl, None]
            inf = torch.full_like(a, 2.0)
            tx = torch.where(c != a, (grid - a) / torch.where(c != a, c - a, 1.0), inf)
            ty = torch.where(d != b, (grid - b) / torch.where(d != b, d - b, 1.0), inf)
            t = torch.cat([torch.zeros_like(a), tx, ty, torch.ones_like(a)], 1).clamp(0.0, 1.0)
            t = t.sort(dim=1).values
            dt, tm = t[:, 1:] - t[:, :-1], 0.5 * (t[:, 1:] + t[:, :-1])
            xm, ym = a + tm * (c - a), b + tm * (d - b)
            acc = 0.0
            for e in (-1e-9, 1e-9):
                ix = torch.floor(xm + e).long().clamp(-1, n) + 1
                iy = torch.floor(ym + e).long().clamp(-1, n) + 1
                acc = acc + 0.5 * flat[iy * (n + 2) + ix]
            out[sl] = (acc * dt).sum(1) * torch.sqrt((c - a) ** 2 + (d - b) ** 2)[:, 0]
        return out

    def mu(self, e):
        k, m = self.e_k, self.mu_k
        s0, s1 = (m[1] - m[0]) / (k[1] - k[0]), (m[2] - m[1]) / (k[2] - k[1])
        return torch.where(e < k[1], m[0] + (e - k[0]) * s0, m[1] + (e - k[1]) * s1)

    def plane_norm(self, e):
        th = (torch.arange(1 << 14, dtype=torch.float64, device=self.dev) + 0.5) * (
            2.0 * math.pi / (1 << 14))
        return float(self.kn(torch.cos(th), e).mean() * 2.0 * math.pi)

    @staticmethod
    def kn(c, e):
        r = 1.0 / (1.0 + (e / ME_C2) * (1.0 - c))
        return r * r * (r + 1.0 / r - (1.0 - c * c))

    def sigma(self, e):
        return self.frac * torch.sqrt(e * E_REF) * TO_SIGMA

    @staticmethod
    def mass(lo, hi, mean, sg):
        a, b = (lo - mean) / (math.sqrt(2.0) * sg), (hi - mean) / (math.sqrt(2.0) * sg)
        up = 0.5 * (torch.special.erfc(a) - torch.special.erfc(b))
        dn = 0.5 * (torch.special.erfc(-b) - torch.special.erfc(-a))
        return torch.where(a + b > 0, up, dn)

    def direction(self, a):
        if (4 * a) % self.A == 0:
            k = (4 * a) // self.A
            return (1.0, 0.0, -1.0, 0.0)[k], (0.0, 1.0, 0.0, -1.0)[k]
        t = 2.0 * math.pi * a / self.A
        return math.cos(t), math.sin(t)

    def angle(self, a):
        """Everything of one detector angle: blur of voxels and points (u,
        sigma), primary weights [W, nq], scatter weights and energies [W, nq, np]."""
        c, s = self.direction(a)
        far = 4.0 * self.n + 8.0

        def seen(x, y):
            x, y = x.double(), y.double()
            xc, yc = (x - 0.5 * self.n) * self.h, (y - 0.5 * self.n) * self.h
            g = self.h * self.line(x, y, x + far * c, y + far * s)
            dep = self.half - (xc * c + yc * s)
            return g, -xc * s + yc * c, (self.f0 + self.slope * dep) * TO_SIGMA

        gq, uq, sq = seen(self.qx, self.qy)
        gp, up, sp = seen(self.px, self.py)
        cos_t = (self.dx * c + self.dy * s) / self.d.clamp(min=1e-30)
        prim, wgt, en = [], [], []
        for e0, al, kn in zip(self.lines, self.yields, self.kn_norm):
            e0t = torch.tensor(e0, dtype=torch.float64, device=self.dev)
            mu0 = self.mu(e0t)
            prim.append(al * torch.exp(-mu0 * gq))
            e1 = e0 / (1.0 + (e0 / ME_C2) * (1.0 - cos_t))
            w = al * torch.exp(-mu0 * self.g_qp - self.mu(e1) * gp[None, :]) * (
                mu0 * self.p_rho[None, :] * self.area / self.d.clamp(min=1e-30)) * self.kn(cos_t, e0) / kn
            wgt.append(torch.where(self.own, torch.zeros_like(w), w))
            en.append(e1)
        return (uq, sq), (up, sp), torch.stack(prim), torch.stack(wgt), torch.stack(en)

    def rows(self, ev, sink):
        """Rows a_j[q] of the events, angle by angle and bin by bin, handed to
        sink(index, rows)."""
        w = 2.0 * self.half / self.B
        lines = torch.tensor(self.lines, dtype=torch.float64, device=self.dev)
        sl = self.sigma(lines)
        key = ev[0].long() * self.B + ev[1].long()
        order = torch.argsort(key, stable=True)
        start = torch.searchsorted(key[order], torch.arange(self.A * self.B + 1, device=self.dev)).tolist()
        for a in range(self.A):
            if start[a * self.B] == start[(a + 1) * self.B]:
                continue
            (uq, sq), (up, sp), prim, wgt, en = self.angle(a)
            sg = self.sigma(en)
            amp, inv = wgt / (math.sqrt(2.0 * math.pi) * sg), math.sqrt(0.5) / sg
            for b in range(self.B):
                i = order[start[a * self.B + b]:start[a * self.B + b + 1]]
                if not i.numel():
                    continue
                lo = -self.half + b * w
                cq, cp = self.mass(lo, lo + w, uq, sq), self.mass(lo, lo + w, up, sp)
                p = torch.nonzero(cp > 1e-13 * cp.max()).reshape(-1)
                ap, ip, ep = amp[:, :, p] * cp[p], inv[:, :, p], en[:, :, p]
                for k in range(0, i.numel(), 64):
                    j = i[k:k + 64]
                    e = ev[2][j].double()
                    gl = torch.exp(-0.5 * ((e[:, None] - lines) / sl) ** 2) / (math.sqrt(2.0 * math.pi) * sl)
                    r = (gl @ prim) * cq
                    for m in range(len(self.lines)):
                        t = (e[:, None, None] - ep[m]).mul_(ip[m])
                        r += t.square_().neg_().exp_().mul_(ap[m]).sum(-1)
                    sink(j, r)

    def sensitivity(self, subset, parts):
        out = torch.zeros(self.qx.numel(), dtype=torch.float64, device=self.dev)
        for a in range(self.A) if subset < 0 else range(subset, self.A, parts):
            (uq, sq), (up, sp), prim, wgt, en = self.angle(a)
            oq, op = self.mass(-self.half, self.half, uq, sq), self.mass(-self.half, self.half, up, sp)
            lines = torch.tensor(self.lines, dtype=torch.float64, device=self.dev)
            for lo, hi in self.win:
                out += oq * (self.mass(lo, hi, lines, self.sigma(lines)) @ prim)
                out += (wgt * self.mass(lo, hi, en, self.sigma(en))).sum(0) @ op
        return out

    def image(self, v):
        out = torch.zeros(self.n * self.n, dtype=torch.float64, device=self.dev)
        out[self.pix] = v
        return out


def plain_net(p, x):
    """(output, hidden activations) of the network in double precision."""
    p, x = torch.from_numpy(p).cuda().double(), x.double()
    k = [128 * 32, 128, 128 * 128, 128, 128 * 128, 128, 128, 1]
    w1, b1, w2, b2, w3, b3, w4, b4 = torch.split(p, k)
    v = [w1.reshape(128, 32), b1, w2.reshape(128, 128), b2, w3.reshape(128, 128), b3,
         w4.reshape(1, 128), b4]
    v = [t.clone().requires_grad_(True) for t in v]
    for i in range(0, 6, 2):
        x = torch.nn.functional.gelu(x @ v[i].T + v[i + 1], approximate="tanh")
    return (x @ v[6].T + v[7]).reshape(-1), v


def exact(case, seed):
    op = case["op"]
    if op == "net_forward":
        with torch.no_grad():
            return plain_net(make_params(seed), make_rows(case["rows"], seed))[0]
    if op == "net_gradient":
        st = prepare(case, seed)
        out, v = plain_net(make_params(seed), st["x"])
        loss = (st["weight"].double() * (out - st["target"].double()) ** 2).mean()
        loss.backward()
        return {"grad": torch.cat([t.grad.reshape(-1) for t in v]), "loss": float(loss.detach())}
    if op == "osem_learned":
        return None
    nq = support_size(case)
    cells = nq * (case["scatter_n"] / case["n"]) ** 2
    ev_n = case["events"] * case.get("realisations", 1)
    if 3.0 * nq * cells * (0.3 * ev_n + 4.0 * case["n_angles"]) > 2.2e11:
        return None
    rho, act = make_object(case, seed)
    ref = Plain(case, rho)
    if op == "model":
        s = case["subsets"]
        return {"all": ref.image(ref.sensitivity(-1, s)), "last": ref.image(ref.sensitivity(s - 1, s))}
    st = prepare(case, seed)
    lists = st["events"] if op == "batch" else [st["events"]]
    ev = tuple(torch.cat([getattr(e, k) for e in lists]) for k in ("angle", "bin", "energy"))
    if op == "forward":
        lam = st["image"].double()[ref.pix]
        y = torch.empty(ev_n, dtype=torch.float64, device="cuda")
        ref.rows(ev, lambda j, r: y.__setitem__(j, r @ lam))
        return y
    if op == "backproject":
        acc = torch.zeros(nq, dtype=torch.float64, device="cuda")
        wt = st["weight"].double()
        ref.rows(ev, lambda j, r: acc.add_(wt[j] @ r))
        return ref.image(acc)
    a = torch.empty((ev[0].numel(), nq), dtype=torch.float64, device="cuda")
    ref.rows(ev, lambda j, r: a.__setitem__(j, r))
    parts, lo, images, lls = case["subsets"], 0, [], []
    sens = [ref.sensitivity(s, parts) for s in range(parts)]
    for e in lists:
        lam = torch.ones(nq, dtype=torch.float64, device="cuda")
        sub = (e.angle.long() % parts)
        rows = a[lo:lo + len(e)]
        lo += len(e)
        for _ in range(case["iters"]):
            for s in range(parts):
                r = rows[sub == s]
                y = r @ lam
                lls.append(torch.log(y[y > 0]).sum() - (lam * sens[s]).sum())
                num = torch.where(y > 0, 1.0 / y, torch.zeros_like(y)) @ r
                lam = torch.where(sens[s] > 0, lam * num / sens[s], torch.zeros_like(lam))
        images.append(ref.image(lam))
    if op == "batch":
        return torch.stack(images)
    return {"image": images[0], "loglik": torch.stack(lls)} if case.get("loglik") else images[0]
