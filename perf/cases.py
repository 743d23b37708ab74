"""The work this framework is used for, as cases that can be timed and checked.

A case is a dict of plain values: a telescope with its sensors, layers and mirrors, and what is
done with it.  `prepare` makes a user's inputs and the handle a user's program keeps, `run` is one
pass through the public entry points, `exact` the same result in 64 bits by plain torch.

Inputs: von Karman layers (r0 = 0.157 m, L0 = 25 m) in frozen flow at 1 kHz and the slopes every
sensor would measure of them plus its noise; a frame's warm start is what the frames before it left.
"""

import math

import torch

from paper_2202_11945_gb300 import Batch, Reconstructor, autograd

ARCSEC = math.pi / (180.0 * 3600.0)
FOV = 60.0 * ARCSEC
SODIUM = 90e3
BEHIND = 3          # frames that a case's state has behind it
R0, L0 = 0.157, 25.0
MAORY_HEIGHTS = (0.0, 140.0, 280.0, 560.0, 1100.0, 2300.0, 4500.0, 9000.0, 18000.0)
DM_HEIGHTS = (0.0, 4000.0, 12700.0)

# One laser-tomography telescope of the ELT class: 6 laser stars on 80 x 80 subapertures, three
# coarse natural stars, nine layers, three mirrors.
MAORY = dict(nsub=80, d=0.4875, obs=0.28, lgs=6, ngs=3, coarse=True, heights=",".join("%g" % h for h in MAORY_HEIGHTS),
             twice_above=4500.0, levels=0, dms=3, elongated=False, iters=4, precision=32)
# The 37 m, three-layer geometry with spot elongation of the method's own simulations.
PAPER = dict(nsub=74, d=0.5, obs=0.33166, lgs=6, ngs=3, coarse=True, heights="0,4000,12700", twice_above=3000.0,
             levels=0, dms=3, elongated=True, iters=2, precision=32)
# A single-conjugate 8 m telescope with one natural star, two layers and one mirror.
SCAO = dict(nsub=16, d=0.5, obs=0.0, lgs=0, ngs=1, coarse=False, heights="0,8000", twice_above=4500.0, levels=3,
            dms=1, elongated=False, iters=4, precision=32)


def listed():
    return [
        # the smallest call: one frame of an 8 m system, all latency
        dict(SCAO, name="frame_8m", kind="frame"),
        # the same system as its control computer runs it: slopes from host memory frame after
        # frame, commands back to it
        dict(SCAO, name="loop_8m", kind="loop", frames=16),
        # the paper's geometry at its own two iterations, spot elongation on
        dict(PAPER, name="frame_paper", kind="frame"),
        # the framework's headline: one warm-started frame of the MAORY-size system
        dict(MAORY, name="frame_maory", kind="frame"),
        # the same frame in double precision (reference runs, simulations)
        dict(MAORY, name="frame_maory_fp64", kind="frame", precision=64),
        # the same system in closed loop: residual slopes in, integrated commands out
        dict(MAORY, name="closed_loop_maory", kind="frame", closed_loop=True),
        # three augmented iterations, which reach the residual of four plain ones
        dict(MAORY, name="augmented_maory", kind="frame", augmented=True, iters=3),
        # many telescopes at once (simulation campaigns): sixteen uneven instances, one batch
        dict(name="batch_uneven", kind="batch", instances=16, first=0, iters=4, precision=32),
        # training through the real-time frame: its commands and their gradient in the slopes
        dict(MAORY, name="grad_maory", kind="grad"),
        # the forward model and its adjoint, as an optimiser over layers calls them
        dict(MAORY, name="model_maory", kind="model"),
        # least-squares fitting of the mirrors over nine directions
        dict(PAPER, name="fit_paper", kind="fit", directions=3, spread=25.0, n_fit=74, eps=0.2),
        # the converged reconstruction and its gradient (calibration, learning of priors): the
        # longest call, thousands of iterations on a small system
        dict(SCAO, name="converged_8m", kind="converged", tol=1e-11),
    ]


def draw(rng):
    """One more case: another telescope, done one of the listed things with."""
    kind = rng.choice(["frame", "frame", "frame", "loop", "batch", "grad", "model", "fit", "converged"])
    if kind == "batch":
        return dict(kind=kind, instances=rng.randint(2, 16), first=rng.randint(1, 5000), iters=rng.randint(2, 5), precision=32)
    c = _draw_telescope(rng, 16 if kind == "converged" else 80)
    c["kind"] = kind
    if kind == "frame":
        c["precision"] = rng.choice([32, 32, 32, 64])
        c["augmented"] = rng.random() < 0.25
        c["closed_loop"] = rng.random() < 0.25
    elif kind == "loop":
        c["frames"] = rng.randint(4, 16)
    elif kind == "fit":
        c.update(directions=rng.choice([1, 2, 3]), spread=rng.uniform(5.0, 25.0), n_fit=c["nsub"], eps=0.2)
    elif kind == "converged":
        c.update(lgs=0, ngs=1, coarse=False, elongated=False, nsub=rng.randint(12, 16), obs=0.0, levels=3, d=0.5,
                 heights="0,%d" % rng.randint(7000, 9000), dms=1, tol=1e-10)
    return c


def _draw_telescope(rng, most):
    nsub = int(round(8 * (most / 8.0) ** rng.uniform(0.0, 1.0)))
    lgs = rng.randint(0, 6)
    count = rng.randint(2, 9)
    hs = [0.0] + sorted(rng.sample(MAORY_HEIGHTS[1:], count - 1))
    return dict(nsub=nsub, d=rng.choice([0.4875, 0.5]), obs=rng.choice([0.0, 0.2, 0.28]) if nsub > 12 else 0.0, lgs=lgs,
                ngs=rng.randint(1, 3) if lgs else 1, coarse=bool(lgs and nsub % 2 == 0), heights=",".join("%g" % h for h in hs),
                twice_above=4500.0, levels=rng.choice([0, 0, 3]), dms=rng.randint(1, 3), elongated=bool(lgs and rng.random() < 0.3),
                iters=rng.randint(2, 5), precision=32)


# ---------------------------------------------------------------- telescopes


def _ring(radius, count, start=0.0):
    return [(radius * math.cos(start + 2 * math.pi * k / count), radius * math.sin(start + 2 * math.pi * k / count)) for k in range(count)]


def workload(case):
    """The framework's workload description of a case's telescope."""
    nsub, d = case["nsub"], case["d"]
    D = nsub * d
    # a small telescope looks at a narrower field, so that its footprints stay on the layer grids
    field = min(1.0, D / 16.0)
    wfs = []
    for tx, ty in _ring(45.0 * ARCSEC * field, case["lgs"]) if case["lgs"] else []:
        w = dict(n_sub=nsub, nb=1, lgs=True, theta=(tx, ty), H=SODIUM, sigma=0.1)
        if case["elongated"]:
            az = math.atan2(ty, tx)
            w.update(launch=(0.5 * D * math.cos(az), 0.5 * D * math.sin(az)), na_fwhm=11.4e3, spot_fwhm=1.1 * ARCSEC)
        wfs.append(w)
    stars = [(0.0, 0.0)] if case["ngs"] == 1 else _ring(55.0 * ARCSEC * field, case["ngs"], math.pi / 3)
    for t in stars:
        if case["coarse"]:
            wfs.append(dict(n_sub=2, nb=nsub // 2, lgs=False, theta=t, H=0.0, sigma=0.02))
        else:
            wfs.append(dict(n_sub=nsub, nb=1, lgs=False, theta=t, H=0.0, sigma=0.05))
    hs = [float(h) for h in case["heights"].split(",")]
    ws = [math.exp(-h / 3000.0) for h in hs]
    dms = []
    for h, share in list(zip(DM_HEIGHTS, (1.0, 0.6, 0.5)))[: case["dms"]]:
        na = int(round(share * nsub)) + 1
        dms.append(dict(h=h, spacing=(D + h * FOV * field) / (na - 1), n_act=na))
    layers = []
    for h, w in zip(hs, ws):
        delta = d if h <= case["twice_above"] else 2 * d
        half = max([(1.0 - h / SODIUM if s["lgs"] else 1.0) * D / 2 + max(map(abs, s["theta"])) * h for s in wfs] +
                   [(m["n_act"] - 1) * m["spacing"] / 2 for m in dms] + [D / 2 + 25.0 * ARCSEC * field * h])
        n = 8
        while n / 2 < half / delta + 2:
            n *= 2
        full = n.bit_length() - 1
        layers.append(dict(h=h, w=w / sum(ws), delta=delta, n=n, levels=min(case["levels"], full) if case["levels"] else full))
    return dict(D=D, obs=case["obs"], wfs=wfs, layers=layers, dms=dms,
                params=dict(alpha=1.0, tau=0.0, gain=0.5 if case.get("closed_loop") else 1.0, iters=case["iters"], r0=R0, L0=L0,
                            alpha_eta=0.2 if case["elongated"] else 0.0))


def members(case):
    """The telescopes of a batch: sizes, stars, layers and mirrors differ."""
    import random
    out = []
    for k in range(case["instances"]):
        rng = random.Random(1000 * case["first"] + k)
        c = _draw_telescope(rng, 80)
        c.update(nsub=rng.choice([16, 32, 48, 80]), coarse=False, ngs=1, d=0.5, obs=0.0, iters=case["iters"], elongated=False, levels=0)
        out.append(c)
    return out


# ---------------------------------------------------------------- the model, in 64 bits


def _filters():
    s, q = math.sqrt(10.0), 16.0 * math.sqrt(2.0)
    r = math.sqrt(5.0 + 2.0 * s)
    h = [v / q for v in (1 + s + r, 5 + s + 3 * r, 10 - 2 * s + 2 * r, 10 - 2 * s - 2 * r, 5 + s - 3 * r, 1 + s - r)]
    return h, [(-1.0) ** m * h[5 - m] for m in range(6)]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _f64(x):
    return torch.as_tensor(x, dtype=torch.float64, device=_device())


def _hats(coord, n):
    """Linear interpolation on n unit-spaced nodes, zero outside them, as a matrix."""
    return (1.0 - (coord[:, None] - torch.arange(n, dtype=torch.float64, device=coord.device)[None, :]).abs()).clamp(min=0.0)


def _active(n, D, obs):
    c = -D / 2 + (torch.arange(n, dtype=torch.float64) + 0.5) * (D / n)
    r = torch.hypot(c[None, :], c[:, None])
    return ((r >= obs * D / 2) & (r <= D / 2)).to(_device())


class Model:
    """The reconstruction of one telescope as dense 1-D matrices, in 64 bits."""

    def __init__(self, wl):
        self.wl, self.p = wl, wl["params"]
        self.layers = wl["layers"]
        self.n_c = sum(L["n"] ** 2 for L in self.layers)
        D, taps = wl["D"], _filters()
        steps = {}
        for L in self.layers:
            for k in range(L["levels"]):
                m = L["n"] >> k
                if m not in steps:
                    A = torch.zeros(m, m, dtype=torch.float64)
                    for i in range(m // 2):
                        for t in range(6):
                            A[i, (2 * i + t) % m] += taps[0][t]
                            A[m // 2 + i, (2 * i + t) % m] += taps[1][t]
                    steps[m] = A.to(_device())
        self.steps = steps
        self.wfs = []
        for W in wl["wfs"]:
            N = W["n_sub"] * W["nb"]
            x = _f64([-D / 2 + k * (D / N) for k in range(N + 1)])
            mask = _active(N, D, wl["obs"])
            cmask = _active(W["n_sub"], D, wl["obs"])
            if W["nb"] > 1:
                mask = mask & cmask.repeat_interleave(W["nb"], 0).repeat_interleave(W["nb"], 1)

            def seen(h, spacing, centre, n):
                s = 1.0 - h / W["H"] if W["lgs"] else 1.0
                return [_hats((s * x + t * h) / spacing + centre, n) for t in (W["theta"][1], W["theta"][0])]

            w = dict(W, N=N, mask=mask, m=mask.double(), cmask=cmask, count=int((cmask if W["nb"] > 1 else mask).sum()),
                     P=[seen(L["h"], L["delta"], L["n"] / 2, L["n"]) for L in self.layers],
                     Q=[seen(m["h"], m["spacing"], (m["n_act"] - 1) / 2, m["n_act"]) for m in wl["dms"]], el=None)
            if W["lgs"] and self.p["alpha_eta"] > 0 and W.get("na_fwhm", 0) > 0:
                mid = x[:-1] + D / N / 2
                k, c = W["na_fwhm"] / W["H"] ** 2, (self.p["alpha_eta"] / W["spot_fwhm"]) ** 2
                b1 = (k * (mid - W["launch"][0]))[None, :].expand(N, N)
                b2 = (k * (mid - W["launch"][1]))[:, None].expand(N, N)
                w["el"] = (b1, b2, c / (1.0 + c * (b1 ** 2 + b2 ** 2)))
            self.wfs.append(w)
        # share of each layer in each mirror: linear in altitude between neighbouring mirrors
        hs = [m["h"] for m in wl["dms"]]
        self.F = []
        for i, m in enumerate(wl["dms"]):
            xa = (torch.arange(m["n_act"], dtype=torch.float64, device=_device()) - (m["n_act"] - 1) / 2) * m["spacing"]
            F = []
            for L in self.layers:
                h = min(max(L["h"], hs[0]), hs[-1])
                below, above = hs[max(i - 1, 0)], hs[min(i + 1, len(hs) - 1)]
                if h == hs[i]:
                    share = 1.0
                elif below < h < hs[i]:
                    share = (h - below) / (hs[i] - below)
                elif hs[i] < h < above:
                    share = (above - h) / (above - hs[i])
                else:
                    share = 0.0
                F.append((share, _hats(xa / L["delta"] + L["n"] / 2, L["n"])))
            self.F.append(F)

    # -- layers and coefficients --------------------------------------------------------
    def split(self, c):
        out, at = [], 0
        for L in self.layers:
            out.append(c[at:at + L["n"] ** 2].reshape(L["n"], L["n"]))
            at += L["n"] ** 2
        return out

    @staticmethod
    def join(xs):
        return torch.cat([x.reshape(-1) for x in xs])

    def dwt(self, phis):
        out = []
        for phi, L in zip(phis, self.layers):
            quads, x = [], phi
            for k in range(L["levels"]):
                m = L["n"] >> k
                y = self.steps[m] @ x @ self.steps[m].T
                quads.append(y)
                x = y[:m // 2, :m // 2]
            for y in reversed(quads):
                h = y.shape[0] // 2
                x = torch.cat([torch.cat([x, y[:h, h:]], 1), y[h:]], 0)
            out.append(x)
        return self.join(out)

    def idwt(self, c):
        out = []
        for x, L in zip(self.split(c), self.layers):
            y = x[:L["n"] >> L["levels"], :L["n"] >> L["levels"]]
            for k in reversed(range(L["levels"])):
                m = L["n"] >> k
                h = m // 2
                full = torch.cat([torch.cat([y, x[:h, h:m]], 1), x[h:m, :m]], 0)
                y = self.steps[m].T @ full @ self.steps[m]
            out.append(y)
        return out

    def unpiston(self, c):
        """c without the layers' pistons, which no slope sees (exact: the data term has none)."""
        keep = torch.ones_like(c)
        at = 0
        for L in self.layers:
            if 1 << L["levels"] == L["n"]:
                keep[at] = 0.0
            at += L["n"] ** 2
        return c * keep

    # -- sensors ------------------------------------------------------------------------
    @staticmethod
    def gamma(v):
        return 0.5 * ((v[:-1, 1:] - v[:-1, :-1]) + (v[1:, 1:] - v[1:, :-1])), 0.5 * ((v[1:, :-1] - v[:-1, :-1]) + (v[1:, 1:] - v[:-1, 1:]))

    @staticmethod
    def gamma_t(sx, sy):
        z = torch.nn.functional.pad
        return 0.5 * (z(sx, (1, 0, 0, 1)) - z(sx, (0, 1, 0, 1)) + z(sx, (1, 0, 1, 0)) - z(sx, (0, 1, 1, 0)) +
                      z(sy, (0, 1, 1, 0)) - z(sy, (0, 1, 0, 1)) + z(sy, (1, 0, 1, 0)) - z(sy, (1, 0, 0, 1)))

    def measure(self, W, v):
        sx, sy = self.gamma(v)
        if W["nb"] == 1:
            return torch.cat([sx[W["mask"]], sy[W["mask"]]])
        s, b = W["n_sub"], W["nb"]
        cut = lambda a: (a * W["m"]).reshape(s, b, s, b).sum((1, 3))[W["cmask"]] / b  # noqa: E731
        return torch.cat([cut(sx), cut(sy)])

    def measure_t(self, W, s):
        k = W["count"]
        grid = torch.zeros((2,) + tuple((W["mask"] if W["nb"] == 1 else W["cmask"]).shape), dtype=torch.float64, device=s.device)
        at = W["mask"] if W["nb"] == 1 else W["cmask"]
        gx, gy = grid[0].masked_scatter(at, s[:k]), grid[1].masked_scatter(at, s[k:])
        if W["nb"] > 1:
            gx, gy = [g.repeat_interleave(W["nb"], 0).repeat_interleave(W["nb"], 1) * W["m"] / W["nb"] for g in (gx, gy)]
        return self.gamma_t(gx, gy)

    def weigh(self, W, s):
        """The sensor's inverse noise, tip and tilt removed for a laser star."""
        if not W["lgs"]:
            return s / W["sigma"] ** 2
        k = W["count"]
        level = lambda v: torch.cat([v[:k] - v[:k].mean(), v[k:] - v[k:].mean()])  # noqa: E731
        u = level(s)
        if W["el"] is not None:
            b1, b2, g = (t[W["mask"]] for t in W["el"])
            bu = b1 * u[:k] + b2 * u[k:]
            u = level(torch.cat([u[:k] - g * b1 * bu, u[k:] - g * b2 * bu]))
        return u / W["sigma"] ** 2

    def forward(self, phis):
        return torch.cat([self.measure(W, sum(y @ phi @ x.T for (y, x), phi in zip(W["P"], phis))) for W in self.wfs])

    def forward_t(self, s, weigh=False):
        out, at = [0.0] * len(self.layers), 0
        for W in self.wfs:
            sg = s[at:at + 2 * W["count"]]
            at += 2 * W["count"]
            u = self.measure_t(W, self.weigh(W, sg) if weigh else sg)
            out = [o + y.T @ u @ x for o, (y, x) in zip(out, W["P"])]
        return out

    def mirror_slopes(self, a):
        out = []
        for W in self.wfs:
            v, at = 0.0, 0
            for (y, x), m in zip(W["Q"], self.wl["dms"]):
                k = m["n_act"]
                v = v + y @ a[at:at + k * k].reshape(k, k) @ x.T
                at += k * k
            out.append(self.measure(W, v))
        return torch.cat(out)

    def fit(self, phis):
        return torch.cat([sum(w * (R @ phi @ R.T) for (w, R), phi in zip(F, phis)).reshape(-1) for F in self.F])

    # -- the system ---------------------------------------------------------------------
    def diagonals(self):
        """The prior D and the inverse of the preconditioner's diagonal."""
        dev = _device()
        Ds, Js = [], []
        for li, L in enumerate(self.layers):
            n, lev = L["n"], L["levels"]
            dk = 1.0 / (n * L["delta"])
            k = torch.arange(-(n // 2), n // 2, dtype=torch.float64, device=dev)
            kap = dk * torch.hypot(k[None, :], k[:, None])
            var = (n * dk) ** 2 * L["w"] * 0.023 * self.p["r0"] ** (-5.0 / 3.0) * (kap ** 2 + self.p["L0"] ** -2) ** (-11.0 / 6.0)

            def box(m):
                inside = (k >= -m) & (k < m)
                return inside[None, :] & inside[:, None]

            Dl = torch.zeros(n, n, dtype=torch.float64, device=dev)
            Jl = torch.zeros(n, n, dtype=torch.float64, device=dev)
            low = torch.eye(n, dtype=torch.float64, device=dev)
            bands = []
            for j in range(1, lev + 1):
                h = n >> j
                step = self.steps[2 * h]
                high, low = low @ step[h:].T, low @ step[:h].T
                Dl[:2 * h, :2 * h] = 1.0 / var[box(n / 2 ** j) & ~box(n / 2 ** (j + 1))].mean()
                bands += [(low, high, 0, h), (high, low, h, 0), (high, high, h, h)]
            bands.append((low, low, 0, 0))
            h = n >> lev
            Dl[:h, :h] = 1.0 / var[box(n / 2 ** (lev + 1))].mean()
            for W in self.wfs:
                Ry, Rx = W["P"][li]
                for fy, fx, r, c in bands:
                    a, b = Ry @ fy, Rx @ fx
                    ya, yd = 0.5 * (a[:-1] + a[1:]), a[1:] - a[:-1]
                    xa, xd = 0.5 * (b[:-1] + b[1:]), b[1:] - b[:-1]
                    m = W["m"]
                    if W["nb"] == 1:
                        val = (ya ** 2).T @ m @ (xd ** 2) + (yd ** 2).T @ m @ (xa ** 2)
                        if W["lgs"]:
                            mx, my = ya.T @ m @ xd / W["count"], yd.T @ m @ xa / W["count"]
                            val = val - (mx ** 2 + my ** 2) * W["count"]
                            if W["el"] is not None:
                                b1, b2, g = W["el"]
                                G11, G12, G22 = m * g * b1 * b1, m * g * b1 * b2, m * g * b2 * b2
                                E = (ya ** 2).T @ G11 @ (xd ** 2) + 2 * (ya * yd).T @ G12 @ (xd * xa) + (yd ** 2).T @ G22 @ (xa ** 2)
                                e1, e2 = ya.T @ G11 @ xd + yd.T @ G12 @ xa, ya.T @ G12 @ xd + yd.T @ G22 @ xa
                                # the weighted slopes' square less their means, both without tip and tilt
                                val = val - (E - 2 * (mx * e1 + my * e2) + G11.sum() * mx ** 2 + 2 * G12.sum() * mx * my + G22.sum() * my ** 2)
                    else:
                        val = 0.0
                        for I in range(W["n_sub"]):
                            for J in range(W["n_sub"]):
                                if bool(W["cmask"][I, J]):
                                    rs, cs = slice(I * W["nb"], (I + 1) * W["nb"]), slice(J * W["nb"], (J + 1) * W["nb"])
                                    val = val + ((ya[rs].T @ m[rs, cs] @ xd[cs]) ** 2 + (yd[rs].T @ m[rs, cs] @ xa[cs]) ** 2) / W["nb"] ** 2
                    Jl[r:r + fy.shape[1], c:c + fx.shape[1]] += val / W["sigma"] ** 2
            Ds.append(Dl)
            Js.append(Jl)
        D = self.join(Ds)
        J = self.unpiston(self.join(Js)) + self.p["alpha"] * torch.clamp(D, min=self.p["tau"])
        return D, 1.0 / J

    def data(self, phis_or_slopes, weigh=True):
        return self.unpiston(self.dwt(self.forward_t(phis_or_slopes, weigh)))

    def apply(self, c, D):
        return self.data(self.forward(self.idwt(self.unpiston(c)))) + self.p["alpha"] * D * c

    def pcg(self, s, c, D, Jinv, prev=None):
        """The frame's iterations from c; `prev`: the frame before's directions (augmented)."""
        r = self.data(s) - self.apply(c, D)
        old = prev or []
        for p, q, pq in [(p, q, (p @ r) / pq) for p, q, pq in old]:
            c, r = c + pq * p, r - pq * q

        def conjugate(v):
            return v - sum((q @ v) / pq * p for p, q, pq in old) if old else v

        z = Jinv * r
        p, rz, kept = conjugate(z), r @ z, []
        for _ in range(self.p["iters"]):
            q = self.apply(p, D)
            pq = p @ q
            kept.append((p, q, pq))
            a = rz / pq
            c, r = c + a * p, r - a * q
            z = Jinv * r
            new = r @ z
            p, rz = conjugate(z) + (new / rz) * p, new
        return c, kept

    # -- inputs ---------------------------------------------------------------------------
    def layers_at(self, seed, times):
        """The layers in frozen flow at the given times in seconds."""
        gen = torch.Generator().manual_seed(int(seed))
        out = [[] for _ in times]
        for L in self.layers:
            n, delta = L["n"], L["delta"]
            f = torch.fft.fftfreq(n, d=delta, dtype=torch.float64)
            psd = 0.023 * R0 ** (-5.0 / 3.0) * L["w"] * (f[None, :] ** 2 + f[:, None] ** 2 + L0 ** -2) ** (-11.0 / 6.0)
            psd[0, 0] = 0.0
            noise = torch.randn(2, n, n, generator=gen, dtype=torch.float64)
            speed, angle = 5.0 + 25.0 * torch.rand(1, generator=gen).item(), 2 * math.pi * torch.rand(1, generator=gen).item()
            spec = (torch.complex(noise[0], noise[1]) * psd.sqrt() * (n * n / (n * delta))).to(_device())
            turn = (f[None, :] * math.cos(angle) + f[:, None] * math.sin(angle)).to(_device()) * (2 * math.pi * speed)
            for o, t in zip(out, times):
                o.append(torch.fft.ifft2(spec * torch.polar(torch.ones_like(turn), -turn * t)).real)
        return out

    def slopes_of(self, phis, seed):
        gen = torch.Generator().manual_seed(int(seed) + 7777)
        clean = self.forward(phis)
        sigma = torch.cat([torch.full((2 * W["count"],), W["sigma"], dtype=torch.float64) for W in self.wfs])
        return clean + (sigma * torch.randn(sigma.shape, generator=gen, dtype=torch.float64)).to(clean.device)


# ---------------------------------------------------------------- inputs of a case


def _type(case):
    return torch.float32 if case["precision"] == 32 else torch.float64


def inputs(case, seed, model):
    """What the case's pass reads, in its own type: by name."""
    t, kind = _type(case), case["kind"]
    if kind == "loop":
        phis = model.layers_at(seed, [0.001 * k for k in range(case["frames"])])
        return dict(s=torch.stack([model.slopes_of(p, seed + 31 * k).to(t) for k, p in enumerate(phis)]).cpu())
    if kind in ("frame", "grad"):
        # a loop that runs in earnest has frames behind it: its state is made by them
        phis = model.layers_at(seed, [0.001 * k for k in range(BEHIND + 1)])
        size = [0.4, 0.3, 0.2, 0.1] if case.get("closed_loop") else [1.0] * 4   # closed loop: residual slopes
        out = {"s%d" % k: (f * model.slopes_of(p, seed + 31 * k)).to(t) for k, (p, f) in enumerate(zip(phis, size))}
        out["s"] = out.pop("s%d" % BEHIND)
    else:
        now, later = model.layers_at(seed, [0.0, 0.2])
        out = dict(c=model.dwt(now).to(t), s=model.slopes_of(now, seed).to(t))
    if kind == "grad":
        # what a loss on the mirrors' shapes hands back: no mirror's piston, which no slope sees
        off, at = model.fit(model.layers_at(seed, [0.2])[0]), 0
        for m in model.wl["dms"]:
            k = m["n_act"] ** 2
            off[at:at + k] -= off[at:at + k].mean()
            at += k
        out["g"] = off.to(t)
    elif kind == "model":
        gen = torch.Generator().manual_seed(int(seed) + 99)
        out.update(phi=model.join(now).to(t), g=torch.randn(out["s"].numel(), generator=gen, dtype=torch.float64).to(_device(), t))
    elif kind == "converged":
        out["s_next"] = model.slopes_of(later, seed + 5).to(t)
        out["aim"], out["aim_next"] = model.fit(now).to(t), model.fit(later).to(t)
    return out


def fit_setup(case):
    """Directions and weights of a least-squares fit: a square of them, the centre weighs double."""
    k, a = case["directions"], case["spread"] * ARCSEC * min(1.0, case["nsub"] * case["d"] / 16.0)
    at = [0.0] if k == 1 else [a * (2.0 * i / (k - 1) - 1.0) for i in range(k)]
    dirs = [(x, y) for y in at for x in at]
    return dirs, [2.0 if x == 0.0 and y == 0.0 else 1.0 for x, y in dirs]


# ---------------------------------------------------------------- the measured path


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        recons, slopes = [], []
        for k, c in enumerate(members(case)):
            m = Model(workload(c))
            x = inputs(dict(c, kind="frame"), seed + 101 * k, m)
            r = Reconstructor(m.wl, precision=case["precision"])
            for j in range(BEHIND):
                r.reconstruct(x["s%d" % j])
            recons.append(r)
            slopes.append(x["s"])
        batch = Batch(recons)
        batch.config = dict(order=1, groups=4, vec_passes=4)
        return dict(kind=kind, batch=batch, s=slopes, dm=[torch.empty(r.n_act, dtype=r.dtype, device=r.device) for r in recons])
    model = Model(workload(case))
    st = dict(inputs(case, seed, model), kind=kind, case=case, turn=0)
    st["R"] = R = Reconstructor(model.wl, precision=case["precision"], augmented=bool(case.get("augmented")),
                                closed_loop=bool(case.get("closed_loop")))
    if kind in ("frame", "grad"):
        st["c"], st["dm"] = torch.zeros(R.n_coeffs, dtype=R.dtype, device=R.device), torch.empty(R.n_act, dtype=R.dtype, device=R.device)
        # one slope buffer, as a real-time computer has it
        now = st["s"].clone()
        for k in range(BEHIND):
            st["s"].copy_(st.pop("s%d" % k))
            R.reconstruct(st["s"], x_warm=st["c"], dm_out=st["dm"])
        st["s"].copy_(now)
        if kind == "grad":
            st["s"].requires_grad_(True)
    elif kind == "model":
        st["phi"].requires_grad_(True)
    elif kind == "converged":
        st["alpha"] = torch.tensor(model.p["alpha"], dtype=torch.float64)
        st["cn2"] = torch.tensor([L["w"] for L in model.layers], dtype=torch.float64)
        for n in ("s", "s_next"):
            st[n].requires_grad_(True)
    elif kind == "fit":
        st["dirs"], st["weights"] = fit_setup(case)
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        return st["batch"].reconstruct(st["s"], st["dm"])
    R = st["R"]
    if kind == "frame":
        R.reconstruct(st["s"], x_warm=st["c"], dm_out=st["dm"])
        return dict(dm=st["dm"], c=st["c"])
    if kind == "loop":
        return R.run_loop(st["s"], period_us=0.0)[0]
    if kind == "grad":
        dm = autograd.frame(R, st["s"], st["c"])
        return dict(dm=dm, grad=torch.autograd.grad(dm, st["s"], st["g"])[0])
    if kind == "model":
        s = autograd.forward_model(R, st["phi"])
        return dict(s=s, grad=torch.autograd.grad(s, st["phi"], st["g"])[0])
    if kind == "fit":
        c = st["case"]
        return R.fit_ls(st["c"], st["dirs"], st["weights"], c["n_fit"], c["eps"])[0]
    # a solve starts from the solution before: the two sets of slopes take turns
    s, aim = (st["s"], st["aim"]) if st["turn"] % 2 == 0 else (st["s_next"], st["aim_next"])
    st["turn"] += 1
    dm = autograd.reconstruct(R, s, st["alpha"], st["cn2"], tol=st["case"]["tol"], max_iters=60000)
    off = dm.detach() - aim
    return dict(dm=dm, grad=torch.autograd.grad(dm, s, 2.0 * (off - off.mean()))[0])


# ---------------------------------------------------------------- work and exact results


def _sizes(case):
    wl = workload(case)
    slopes = nodes = pairs = 0
    for W in wl["wfs"]:
        N = W["n_sub"] * W["nb"]
        slopes += 2 * int(_active(W["n_sub"], wl["D"], wl["obs"]).sum())
        nodes += (N + 1) ** 2
        pairs += len(wl["layers"]) * (N + 1) ** 2
    coeffs = sum(L["n"] ** 2 for L in wl["layers"])
    acts = sum(m["n_act"] ** 2 for m in wl["dms"])
    # one application of the system: two wavelet transforms (4/3 of 24 operations a value),
    # P and its transpose (9 a node and layer), slopes, weighting and back (30 a node)
    return dict(s=slopes, c=coeffs, a=acts, nodes=nodes, pairs=pairs, once=70 * coeffs + 18 * pairs + 30 * nodes)


def work(case):
    kind, b = case["kind"], case["precision"] // 8
    if kind == "batch":
        each = [work(dict(c, kind="frame")) for c in members(case)]
        return dict(bytes=sum(w["bytes"] for w in each), flops=sum(w["flops"] for w in each))
    n = _sizes(case)
    frame = (case["iters"] + 1) * n["once"] + case["iters"] * 14 * n["c"] + 12 * n["a"]
    if kind == "frame":
        kept = 4 * case["iters"] * n["c"] if case.get("augmented") else 0
        return dict(bytes=b * (n["s"] + 3 * n["c"] + 2 * n["a"] + kept), flops=frame + 4 * kept)
    if kind == "loop":
        return dict(bytes=b * case["frames"] * (n["s"] + 3 * n["c"] + 2 * n["a"]), flops=case["frames"] * frame)
    if kind == "grad":
        return dict(bytes=b * (2 * n["s"] + 2 * n["c"] + 2 * n["a"]), flops=3 * frame)
    if kind == "model":
        return dict(bytes=b * 2 * (n["s"] + n["c"]), flops=18 * n["pairs"] + 16 * n["nodes"])
    if kind == "fit":
        # some 80 steps, each the mirrors' shapes on the pupil in every direction and back
        return dict(bytes=b * (n["c"] + n["a"]), flops=80 * (20 * case["dms"] * case["directions"] ** 2 * (case["n_fit"] + 1) ** 2 + 14 * n["a"]))
    # two solves of some thousand iterations
    return dict(bytes=b * (2 * n["s"] + n["c"] + 2 * n["a"]), flops=2 * 6000 * (n["once"] + 14 * n["c"]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for k, c in enumerate(members(case)):
            c = dict(c, kind="frame")
            m = Model(workload(c))
            x = {n: v.double() for n, v in inputs(c, seed + 101 * k, m).items()}
            D, Jinv = m.diagonals()
            coeffs = torch.zeros_like(D)
            for name in [n for n in sorted(x) if n != "s"] + ["s"]:
                coeffs = m.pcg(x[name], coeffs, D, Jinv)[0]
            out.append(m.fit(m.idwt(coeffs)))
        return out
    m = Model(workload(case))
    x = {n: v.double().to(_device()) for n, v in inputs(case, seed, m).items()}
    if kind == "model":
        return dict(s=m.forward(m.split(x["phi"])), grad=m.join(m.forward_t(x["g"])))
    if kind == "fit":
        return _exact_fit(case, m, m.idwt(x["c"]))
    D, Jinv = m.diagonals()
    if kind == "grad":
        c = torch.zeros_like(D)
        for k in range(BEHIND):
            c = m.pcg(x["s%d" % k], c, D, Jinv)[0]
        s = x["s"].requires_grad_(True)
        dm = m.fit(m.idwt(m.pcg(s, c, D, Jinv)[0]))
        return dict(dm=dm.detach(), grad=torch.autograd.grad(dm, s, x["g"])[0])
    if kind == "converged":
        eye = torch.eye(m.n_c, dtype=torch.float64, device=D.device)
        M = torch.stack([m.apply(e, D) for e in eye])
        s = x["s"].requires_grad_(True)
        dm = m.fit(m.idwt(torch.linalg.solve(0.5 * (M + M.T), m.data(s))))
        off = dm.detach() - x["aim"]
        return dict(dm=dm.detach(), grad=torch.autograd.grad(dm, s, 2.0 * (off - off.mean()))[0])
    if kind == "loop":
        c, out = torch.zeros_like(D), []
        for s in x["s"]:
            c = m.pcg(s, c, D, Jinv)[0]
            out.append(m.fit(m.idwt(c)))
        return torch.stack(out)
    c, kept = torch.zeros_like(D), None
    a = old = torch.zeros(sum(k["n_act"] ** 2 for k in m.wl["dms"]), dtype=torch.float64, device=c.device)
    for name in ["s%d" % k for k in range(BEHIND)] + ["s"]:
        s = x[name] + m.mirror_slopes(old) if case.get("closed_loop") else x[name]
        c, new = m.pcg(s, c, D, Jinv, kept)
        kept = new if case.get("augmented") else None
        fit = m.fit(m.idwt(c))
        if case.get("closed_loop"):
            a, old = a + m.p["gain"] * (fit - old), a
        else:
            a = (1.0 - m.p["gain"]) * a + m.p["gain"] * fit
    return dict(dm=a, c=c)


def _exact_fit(case, m, phis):
    """The least-squares fit by conjugate gradients on its normal equations, to 1e-14."""
    dirs, weights = fit_setup(case)
    D, nf = m.wl["D"], case["n_fit"]
    x = torch.tensor([-D / 2 + k * (D / nf) for k in range(nf + 1)], dtype=torch.float64, device=_device())
    r = torch.hypot(x[None, :], x[:, None])
    pupil = ((r >= m.wl["obs"] * D / 2) & (r <= D / 2)).double()
    centre = lambda v: (v - (v * pupil).sum() / pupil.sum()) * pupil  # noqa: E731
    # the mirrors' matrices of all directions side by side: [directions, nodes, actuators]
    see = lambda h, spacing, mid, n: [torch.stack([_hats((x + t[i] * h) / spacing + mid, n) for t in dirs]) for i in (1, 0)]  # noqa: E731
    Q = [see(k["h"], k["spacing"], (k["n_act"] - 1) / 2, k["n_act"]) for k in m.wl["dms"]]
    w = torch.tensor(weights, dtype=torch.float64, device=_device())[:, None, None]
    mid = lambda v: (v - (v * pupil).sum((1, 2), keepdim=True) / pupil.sum()) * pupil  # noqa: E731

    def back(v):
        return torch.cat([(w * (y.transpose(1, 2) @ v @ z)).sum(0).reshape(-1) for y, z in Q])

    def shape(a):
        v, at = 0.0, 0
        for (y, z), k in zip(Q, m.wl["dms"]):
            n = k["n_act"]
            v, at = v + y @ a[at:at + n * n].reshape(n, n) @ z.transpose(1, 2), at + n * n
        return v

    seen = sum(y @ phi @ z.transpose(1, 2) for (y, z), phi in
               zip([see(L["h"], L["delta"], L["n"] / 2, L["n"]) for L in m.layers], phis))
    res = back(mid(seen))
    a, p, rr = torch.zeros_like(res), res, res @ res
    stop = float(rr) * 1e-28
    for k in range(4000):
        q = back(mid(shape(p))) + case["eps"] * p
        t = rr / (p @ q)
        a, res = a + t * p, res - t * q
        new = res @ res
        if k % 50 == 49 and float(new) <= stop:
            break
        p, rr = res + (new / rr) * p, new
    return a
