"""Timed cases of the MBIR library: what a user has it do, through ``paper_2202_09703_gb300.mbir``.

A scan is a layered medium, an image grid, transmitter positions, a receiver line and a record
length.  Its user keeps one ``Geometry`` per scan and applies A (``forward``) and its adjoint
(``backproject``), reconstructs (``reconstruct``), or hands many scans to an ``Engine``.  The cases
cover the apply pair from the 64 x 64 image to the 512 x 1024 one, the two storage forms (FP32 and
BF16), the stored (TAB) and on-the-fly (OTF) forms of A, and whole MAP reconstructions.

``exact`` evaluates the same operator (layered Snell travel times, attenuated pulse table read by
bilinear interpolation, apodised weights) and the same MAP iteration in FP64 with plain torch.
"""
import math

import numpy as np
import torch

from paper_2202_09703_gb300 import mbir, synth

DEV = "cuda"

CEMENTED = "water:20,steel:12,cement:40,rock:100"      # fluid-filled borehole, casing, cement, rock (mm)
PLATE = "water:10,steel:10"                            # immersed steel plate


def _case(name, op, form, stack, w, h, pitch, tx, tx_step, rx, samples, fs, fc, direct, iters=0, offset=0.0):
    return {"name": name, "op": op, "form": form, "stack": stack, "w": w, "h": h, "pitch_mm": pitch, "tx": tx,
            "tx_step_mm": tx_step, "tx_offset_mm": offset, "rx": rx, "rx_step_mm": 5.0, "samples": samples,
            "fs_mhz": fs, "fc_mhz": fc, "direct": direct, "iters": iters}


def listed():
    small = (PLATE, 64, 64, 0.5, 16, 2.0, 8, 512, 10.0, 1.0, False)
    middle = (CEMENTED, 256, 512, 0.5, 64, 2.0, 16, 2048, 20.0, 2.0, True)
    large = (CEMENTED, 512, 1024, 0.25, 128, 1.0, 32, 4096, 20.0, 2.0, True)
    ragged = (CEMENTED + ",steel:15", 203, 331, 0.5, 37, 2.0, 11, 1501, 20.0, 2.0, False)
    return [
        # one A x of a quick-look scan: launch and latency count
        _case("forward_64x64_fp32", "forward", "tab-fp32", *small),
        # the ordinary scan, A x and A^T r as any outer iteration of a user's own applies them
        _case("forward_256x512_fp32", "forward", "tab-fp32", *middle),
        _case("adjoint_256x512_fp32", "adjoint", "tab-fp32", *middle),
        # the largest scan (1.1e9 pairs)
        _case("forward_512x1024_fp32", "forward", "tab-fp32", *large),
        _case("adjoint_512x1024_fp32", "adjoint", "tab-fp32", *large),
        # the BF16 storage form: the largest scan, and one whose sizes are multiples of nothing
        _case("forward_512x1024_bf16", "forward", "tab-bf16", *large),
        _case("adjoint_203x331_bf16", "adjoint", "tab-bf16", *ragged),
        # travel times solved on every apply: geometries that are used once or change (no stored records)
        _case("forward_256x512_otf", "forward", "otf-fp32", *middle),
        _case("adjoint_256x512_otf", "adjoint", "otf-fp32", *middle),
        # a whole MAP reconstruction of the quick-look scan and of the ordinary one
        _case("reconstruct_64x64", "reconstruct", "tab-fp32", *small, iters=20),
        _case("reconstruct_256x512", "reconstruct", "tab-fp32", *middle, iters=20),
        # a burst of eight scans of uneven size handed to the batching engine at once
        _case("engine_8_uneven", "engine", "tab-fp32", CEMENTED, 256, 256, 0.5, 64, 2.0, 16, 2048, 20.0, 2.0, True,
              iters=10),
    ]


STACKS = [PLATE, CEMENTED, CEMENTED + ",steel:15", "water:15,cement:30,rock:60"]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    form = rng.choice(["tab-fp32", "tab-fp32", "tab-bf16", "otf-fp32"])
    op = rng.choice(["forward", "adjoint", "forward", "adjoint", "reconstruct", "engine"])
    if form != "tab-fp32" and op in ("reconstruct", "engine"):
        op = rng.choice(["forward", "adjoint"])
    otf = form == "otf-fp32"
    w, h = log(48, 256 if otf else 512), log(48, 400 if otf else 1024)
    tx, rx = log(6, 24 if otf else 128), log(4, 16 if otf else 32)
    samples = log(256, 4096)
    if op in ("reconstruct", "engine"):
        w, h, tx, rx, samples = min(w, 256), min(h, 512), min(tx, 64), min(rx, 16), min(samples, 2048)
    # on the pixel grid for the stored forms (a stepped scanner), anywhere for the on-the-fly one
    step, offset = (0.37 * rng.randint(2, 9), rng.uniform(-1.0, 1.0)) if otf else (0.5 * rng.randint(1, 5), 0.0)
    c = _case("", op, form, rng.choice(STACKS), w, h, 0.5, tx, round(step, 3), rx, samples, 20.0, 2.0,
              rng.random() < 0.5, {"reconstruct": 10, "engine": 5}.get(op, 0), round(offset, 3))
    del c["name"]
    return c


# ---- scenes ------------------------------------------------------------------------------------
def _scene(case):
    fc = case["fc_mhz"] * 1e6
    layers = [synth.material_layer(n, float(t) * 1e-3, fc) for n, t in (s.split(":") for s in case["stack"].split(","))]
    pitch = case["pitch_mm"] * 1e-3
    centre = case["w"] * pitch / 2 + case["tx_offset_mm"] * 1e-3
    return synth.Scene(
        name="scan", layers=layers, img_w=case["w"], img_h=case["h"], pitch=pitch, x0=0.0, z0=0.0,
        tx_x=synth.centred_positions(case["tx"], case["tx_step_mm"] * 1e-3, centre),
        rx_offset=synth.centred_positions(case["rx"], case["rx_step_mm"] * 1e-3),
        fs=case["fs_mhz"] * 1e6, n_samples=case["samples"], fc=fc, direct_arrival=case["direct"],
        prior=synth.Prior(m=0.1 if case["direct"] else 1.0))


def _scenes(case):
    """The scans of a case: one, or the engine's eight (sides and record lengths cut by halves and odd amounts)."""
    if case["op"] != "engine":
        return [_scene(case)]
    cuts = [(1, 1, 1), (2, 2, 2), (4, 4, 4), (1, 2, 1), (4, 4, 2), (2, 1, 2), (3, 3, 2), (4, 2, 3)]
    return [_scene(dict(case, w=max(16, case["w"] // a), h=max(16, case["h"] // b), tx=max(2, case["tx"] // a),
                        samples=max(128, case["samples"] // c))) for a, b, c in cuts]


def _image(scene, seed, dense):
    """A reflectivity image: interfaces and disc voids; `dense` adds the small values of an iterate between them."""
    x = torch.as_tensor(synth.phantom_layered(scene, seed), dtype=torch.float32, device=DEV).reshape(-1)
    if dense:
        gen = torch.Generator(DEV).manual_seed(seed + 7)
        x = x + 0.05 * torch.randn(scene.N, generator=gen, device=DEV)
    return x


def _residual(scene, seed, dtype):
    """A residual: noise whose level falls along the record, with a few coherent bursts."""
    gen = torch.Generator(DEV).manual_seed(seed + 9)
    n = torch.arange(scene.M, device=DEV, dtype=torch.float32)
    r = torch.randn(scene.K, scene.M, generator=gen, device=DEV) * torch.exp(-1.5 * n / scene.M)
    for _ in range(4):
        at = torch.rand(scene.K, 1, generator=gen, device=DEV) * scene.M
        r += 3.0 * torch.exp(-((n - at) / 9.0) ** 2) * torch.cos(2 * math.pi * scene.fc / scene.fs * (n - at))
    return r.reshape(-1).to(dtype)


def _record(scene, seed):
    """A-scans of a phantom with direct arrivals and 20 dB noise, as a 16-bit digitiser gives them, and its noise level."""
    x = _image(scene, seed, False).double()
    pix = torch.nonzero(x).reshape(-1)
    model = Model64(scene, pix)
    y = model.forward(x[pix])
    gen = torch.Generator(DEV).manual_seed(seed + 11)
    if scene.direct_arrival:
        gain = (0.5 + 0.5 * torch.rand(scene.K, generator=gen, device=DEV, dtype=torch.float64)) * y.abs().max()
        y = y + gain[:, None] * model.direct().repeat(scene.n_tx, 1)
    sigma = 0.1 * float(y.square().mean().sqrt())
    y = y + sigma * torch.randn(y.shape, generator=gen, device=DEV, dtype=torch.float64)
    lsb = float(y.abs().max()) / 32000
    return (torch.round(y / lsb) * lsb).float().reshape(-1), float("%.6g" % sigma)


# ---- prepare and run ---------------------------------------------------------------------------
def prepare(case, seed):
    op, (mode, precision) = case["op"], case["form"].split("-")
    scenes = _scenes(case)
    st = {"op": op, "iters": case["iters"], "scans": []}
    for i, s in enumerate(scenes):
        geo = mbir.Geometry(s, mode=mode, precision=precision)
        dtype = torch.bfloat16 if precision == "bf16" else torch.float32
        scan = {"geo": geo}
        if op == "forward":
            scan["x"], scan["y"] = _image(s, seed, True), torch.empty(s.K * s.M, dtype=dtype, device=DEV)
        elif op == "adjoint":
            scan["y"], scan["x"] = _residual(s, seed, dtype), torch.empty(s.N, device=DEV)
        else:
            scan["y"], scan["sigma"] = _record(s, seed + 101 * i)
            scan["x"], scan["g"] = torch.empty(s.N, device=DEV), torch.empty(s.K, device=DEV)
        st["scans"].append(scan)
    if op == "engine":
        st["engine"] = mbir.Engine(8 << 30)
    return st


def run(state):
    op, scans = state["op"], state["scans"]
    c = scans[0]
    if op == "forward":
        return c["geo"].forward(c["x"], c["y"])
    if op == "adjoint":
        return c["geo"].backproject(c["y"], c["x"])
    if op == "reconstruct":
        c["geo"].reconstruct(c["y"], c["sigma"], state["iters"], c["x"], g=c["g"])
        return c["x"], c["g"]
    for c in scans:
        state["engine"].submit(c["geo"], c["y"], c["sigma"], state["iters"], c["x"], g=c["g"])
    state["engine"].run_until_idle()
    return [(c["x"], c["g"]) for c in scans]


# ---- work --------------------------------------------------------------------------------------
_counts = {}


def work(case):
    """Image and A-scans once per apply.  The stored forms also read one entry of A per (pixel, A-scan) pair with a
    sample in the record: delay, weight and attenuation, 12 bytes, the operator the user keeps.  On the fly
    nothing is stored: each (pixel, transducer position) path is solved instead, about 40 operations per
    layer.  A pair costs two operations per bilinear corner; the table product is added once per sample of
    an A-scan, plane and tap (two neighbouring attenuation planes)."""
    op, (mode, precision) = case["op"], case["form"].split("-")
    tot_b = tot_f = 0.0
    for s in _scenes(case):
        key = repr(s)
        if key not in _counts:
            m = Model64(s)
            _counts[key] = (sum(m.pairs(i)[0].numel() for i in range(s.n_tx)), m.npos)
        pairs, npos = _counts[key]
        tw = math.ceil(8 * s.n_cycles / (2 * math.sqrt(2 * math.log(2)) * s.fc) * s.fs)
        b = 4 * s.N + (2 if precision == "bf16" else 4) * s.K * s.M
        f = 8.0 * pairs + 2.0 * s.K * s.M * 2 * (s.Q + 1) * tw
        if mode == "otf":
            f += 40.0 * len(s.layers) * npos * s.N
        else:
            b += 12 * pairs
        n = 1 if op in ("forward", "adjoint") else 2 * case["iters"] + 1
        tot_b += n * b
        tot_f += n * f
    return {"bytes": tot_b, "flops": tot_f}


# ---- the same operator and iteration in 64 bits -------------------------------------------------
class Model64:
    """A of a scene on all pixels, or on `pix` only, in FP64: plain torch, one transmitter position at a time."""

    def __init__(self, s, pix=None, keep=False):
        f64 = {"dtype": torch.float64, "device": DEV}
        self.s, self.keep, self.kept = s, keep, {}
        self.pix = torch.arange(s.N, device=DEV) if pix is None else pix
        self.row, self.col = self.pix // s.img_w, self.pix % s.img_w
        L = len(s.layers)
        eta, self.tau = np.zeros((s.img_h, L)), np.ones(s.img_h)
        for r in range(s.img_h):
            z, top = s.z0 + (r + 0.5) * s.pitch, 0.0
            for l in range(L):
                t = s.layers[l].thickness
                if l == L - 1 or z < top + t:
                    eta[r, l] = z - top
                    break
                eta[r, l] = t
                top += t
                z1, z2 = s.layers[l].density * s.layers[l].speed, s.layers[l + 1].density * s.layers[l + 1].speed
                self.tau[r] *= 4 * z1 * z2 / (z1 + z2) ** 2
        self.tau = torch.as_tensor(self.tau, **f64)
        # pulse: envelope of n_cycles periods FWHM, window of tw samples; its table over (attenuation, delay)
        sg = s.n_cycles / (2 * math.sqrt(2 * math.log(2)) * s.fc)
        self.tw = tw = math.ceil(8 * sg * s.fs)
        att = np.array([a.atten * 1e-6 for a in s.layers])
        gmax = s.gamma_max if s.gamma_max > 0 else 4 * float(eta[-1] @ att)
        self.G = s.G if gmax > 0 else 1
        self.gmax = gmax
        t0, sf = tw / s.fs, 1 / (2 * math.pi * sg)
        panels = math.ceil((s.fc + 16 * sf) / min(0.5 * sf, 0.25 / t0))
        pw = (s.fc + 16 * sf) / panels
        xn, wn = np.polynomial.legendre.leggauss(16)
        f = ((np.arange(panels)[:, None] + 0.5) * pw + 0.5 * pw * xn).reshape(-1)
        spec = sum(np.exp(-2 * (math.pi * sg * (f + d)) ** 2) for d in (-s.fc, s.fc))
        sw = np.tile(0.5 * pw * wn, panels) * sg * math.sqrt(2 * math.pi) * spec
        gam = np.arange(self.G) * (gmax / max(self.G - 1, 1))
        tau_q = np.arange(s.Q * tw + 1) / (s.fs * s.Q)
        tab = (sw * np.exp(-gam[:, None] * f)) @ np.cos(2 * math.pi * np.outer(f, tau_q - 0.5 * t0))
        self.line = tab[0]
        # T[plane * (Q + 1) + phase][tap]: every tap of a pair reads one phase
        q = np.arange(s.Q + 1)[:, None] + s.Q * np.arange(tw)[None, :]
        self.T = torch.as_tensor(tab[:, q].reshape(-1, tw), **f64)
        # paths from every distinct transducer position: one per row and distinct lateral distance
        pos = np.concatenate([s.tx_x] + [s.tx_x + o for o in s.rx_offset])
        pos = np.unique(np.round(pos * 1e12)) * 1e-12
        self.npos = len(pos)
        xc = s.x0 + (np.arange(s.img_w) + 0.5) * s.pitch
        self.lat = lambda u: np.round(np.abs(xc - u) * 1e12)
        dist = np.unique(np.concatenate([self.lat(u) for u in pos]))
        self.dist = dist
        h = torch.as_tensor(dist * 1e-12, **f64)
        c = torch.as_tensor([a.speed for a in s.layers], **f64)
        al = torch.as_tensor(att, **f64)
        self.leg = torch.empty(3, s.img_h, len(dist), **f64)          # time, attenuation, cos^beta of the angle sum
        rows = max(1, int(2e7) // max(1, len(dist)))
        for r0 in range(0, s.img_h, rows):
            e = torch.as_tensor(eta[r0:r0 + rows], **f64)
            live = e > 0
            hi = (1 / torch.where(live, c, torch.zeros_like(c)).amax(1))[:, None].expand(-1, len(dist)).clone()
            lo = torch.zeros_like(hi)
            used = [l for l in range(L) if bool(live[:, l].any())]
            for _ in range(64):                                        # ray parameter: lateral reach equals h
                mid = 0.5 * (lo + hi)
                reach = 0.0
                for l in used:
                    sn = mid * c[l]
                    reach = reach + torch.where(live[:, l:l + 1], e[:, l:l + 1] * sn / torch.sqrt(1 - sn * sn), 0.0)
                below = reach < h
                lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
            p = torch.where(h > 0, 0.5 * (lo + hi), 0.0)
            t, g, th = p * h, torch.zeros_like(p), torch.zeros_like(p)
            for l in used:
                sn, m = p * c[l], live[:, l:l + 1]
                cs = torch.sqrt(1 - sn * sn)
                t = t + torch.where(m, e[:, l:l + 1] * cs / c[l], 0.0)
                g = g + torch.where(m, al[l] * e[:, l:l + 1] / cs, 0.0)
                th = th + torch.where(m, torch.atan2(sn, cs), 0.0)
            self.leg[:, r0:r0 + rows] = torch.stack([t, g, torch.cos(th).clamp_min(0) ** s.beta])

    def _legs(self, us):
        at = np.stack([np.searchsorted(self.dist, self.lat(np.round(u * 1e12) * 1e-12) - 0.5) for u in us])
        hi = torch.as_tensor(at, device=DEV)[:, self.col]
        return self.leg[:, self.row[None, :], hi]

    def pairs(self, i):
        """Active pairs of transmitter i: slot of the pixel, receiver, first tap, table column, weights."""
        if i in self.kept:
            return self.kept[i]
        s = self.s
        tx, rx = self._legs([s.tx_x[i]]), self._legs([s.tx_x[i] + o for o in s.rx_offset])
        t, g, w = tx[0] + rx[0], tx[1] + rx[1], self.tau[self.row] * (tx[2] * rx[2])
        t = t * s.fs
        j, v = torch.nonzero((w != 0) & (torch.floor(t) + 1 < s.M), as_tuple=True)
        t, g, w = t[j, v], g[j, v], w[j, v]
        n0 = torch.floor(t)
        al = (t - n0) * s.Q
        ia = torch.floor(al).clamp_max(s.Q - 1)
        fa = al - ia
        b = (g / self.gmax * (self.G - 1)).clamp(0, self.G - 1) if self.G > 1 else torch.zeros_like(g)
        gi = torch.floor(b).clamp_max(max(self.G - 2, 0))
        out = (v, j, n0.long(), (gi * (s.Q + 1) + s.Q - 1 - ia).long(), fa, b - gi, w, t == n0)
        if self.keep:
            self.kept[i] = out
        return out

    def _corners(self, p):
        """(column, weight) of the four bilinear corners, and of the tap past the open window where there is one."""
        s, (v, j, n0, c, fa, psi, w, edge) = self.s, p
        up = s.Q + 1 if self.G > 1 else 0
        return [(c, w * fa * (1 - psi)), (c + up, w * fa * psi), (c + 1, w * (1 - fa) * (1 - psi)),
                (c + up + 1, w * (1 - fa) * psi)]

    def forward(self, x):
        s, tw = self.s, self.tw
        y = torch.zeros(s.n_tx, s.n_rx, s.M + tw + 1, dtype=torch.float64, device=DEV)
        nc = self.T.shape[0]
        for i in range(s.n_tx):
            p = self.pairs(i)
            v, j, n0, edge = p[0], p[1], p[2], p[7]
            S = torch.zeros(s.n_rx * s.M * nc, dtype=torch.float64, device=DEV)
            at, xv = (j * s.M + n0) * nc, x[v]
            for c, cw in self._corners(p):
                S.index_add_(0, at + c, cw * xv)
            U = (S.view(-1, nc) @ self.T).view(s.n_rx, s.M, tw)
            for m in range(tw):
                y[i, :, 1 + m:1 + m + s.M] += U[:, :, m]
            if bool(edge.any()):
                for c, cw in self._corners(p)[2:]:
                    off = (cw * xv * self.T[c, tw - 1])[edge]
                    y[i].view(-1).index_add_(0, (j * (s.M + tw + 1) + n0 + tw)[edge], -off)
        return y[:, :, :s.M].reshape(s.K, s.M)

    def adjoint(self, r):
        s, tw = self.s, self.tw
        e = torch.zeros(s.n_tx, s.n_rx, s.M + tw + 1, dtype=torch.float64, device=DEV)
        e[:, :, :s.M] = r.reshape(s.n_tx, s.n_rx, s.M)
        out = torch.zeros(self.pix.numel(), dtype=torch.float64, device=DEV)
        nc = self.T.shape[0]
        for i in range(s.n_tx):
            p = self.pairs(i)
            v, j, n0, edge = p[0], p[1], p[2], p[7]
            C = (e[i, :, 1:].unfold(1, tw, 1)[:, :s.M].reshape(-1, tw) @ self.T.t()).view(-1)
            at, val = (j * s.M + n0) * nc, 0.0
            for c, cw in self._corners(p):
                val = val + cw * C[at + c]
            if bool(edge.any()):
                past = e[i].reshape(-1)[j * (s.M + tw + 1) + n0 + tw]
                for c, cw in self._corners(p)[2:]:
                    val = val - torch.where(edge, cw * self.T[c, tw - 1] * past, 0.0)
            out.index_add_(0, v, val)
        return out

    def direct(self):
        """Direct-arrival column of every receiver: the unattenuated pulse after |offset| / c_1."""
        s = self.s
        u = (np.arange(s.M)[None, :] - np.abs(s.rx_offset)[:, None] / s.layers[0].speed * s.fs) * s.Q
        d = np.where((u > 0) & (u < s.Q * self.tw), np.interp(u, np.arange(len(self.line)), self.line), 0.0)
        return torch.as_tensor(d, device=DEV)

    def project(self, r):
        s = self.s
        if not s.direct_arrival:
            return r, torch.zeros(s.K, dtype=torch.float64, device=DEV)
        d = self.direct().repeat(s.n_tx, 1)
        dd = d.square().sum(1)
        g = torch.where(dd > 0, (d * r).sum(1) / dd, 0.0)
        return r - g[:, None] * d, g

    def reconstruct(self, y, sigma, iters):
        """Polak-Ribiere+ directions, each step the minimiser of the data term plus the prior's quadratic bound."""
        s, pr = self.s, self.s.prior
        z = torch.as_tensor(s.z0 + (np.arange(s.img_h) + 0.5) * s.pitch, device=DEV)
        ms = 1 + (pr.m - 1) * (z / z[-1]) ** pr.a
        edge = 1 / (4 + 4 / math.sqrt(2))

        def cliques(a):
            a = a.view(s.img_h, s.img_w)
            yield edge, ms[:, None], a[:, :-1], a[:, 1:]
            yield edge, (ms[:-1] * ms[1:]).sqrt()[:, None], a[:-1], a[1:]
            for u, w in ((a[:-1, 1:], a[1:, :-1]), (a[:-1, :-1], a[1:, 1:])):
                yield edge / math.sqrt(2), (ms[:-1] * ms[1:]).sqrt()[:, None], u, w

        def slope(dl, sg):
            ad = dl.abs()
            u = (ad / (pr.T * sg)) ** (pr.q - pr.p)
            k = ad ** (pr.p - 1) / sg ** pr.p * u / (1 + u) * (1 + (pr.q - pr.p) / (pr.p * (1 + u)))
            return torch.where(ad == 0, 0.0, torch.sign(dl) * k)

        def prior_grad(x):
            out = torch.zeros_like(x)
            o = list(cliques(out))
            for (b, sg, u, w), (_, _, ou, ow) in zip(cliques(x), o):
                d = b * slope(u - w, pr.sigma0 * sg)
                ou += d
                ow -= d
            return out

        def prior_curv(x, d):
            acc = 0.0
            for (b, sg, u, w), (_, _, du, dw) in zip(cliques(x), cliques(d)):
                dl, sg = u - w, pr.sigma0 * sg
                flat = 2 / (pr.p * sg ** 2 * pr.T ** (2 - pr.p))
                kappa = torch.where(dl == 0, flat.expand_as(dl), slope(dl, sg) / torch.where(dl == 0, 1.0, dl))
                acc = acc + (b * kappa * (du - dw) ** 2).sum()
            return acc

        s2 = sigma * sigma
        x = torch.zeros(s.N, dtype=torch.float64, device=DEV)
        e, _ = self.project(y)
        d, gprev, ggp = torch.zeros_like(x), torch.zeros_like(x), 0.0
        for it in range(iters):
            grad = prior_grad(x) - self.adjoint(e) / s2
            gg = float(grad @ grad)
            beta = max(0.0, (gg - float(grad @ gprev)) / ggp) if it and ggp > 0 else 0.0
            d = beta * d - grad
            gd = float(grad @ d)
            if not gd < 0:
                d, gd = -grad, -gg
            q, _ = self.project(self.forward(d))
            den = float(q.square().sum()) / s2 + float(prior_curv(x, d))
            alpha = -gd / den if den > 0 else 0.0
            x, e, gprev, ggp = x + alpha * d, e - alpha * q, grad, gg
        return x, self.project(y - self.forward(x))[1]


def exact(case, seed):
    op, (mode, precision) = case["op"], case["form"].split("-")
    dtype = torch.bfloat16 if precision == "bf16" else torch.float32
    outs = []
    for i, s in enumerate(_scenes(case)):
        if op == "forward":
            return Model64(s).forward(_image(s, seed, True).double()).reshape(-1)
        if op == "adjoint":
            return Model64(s).adjoint(_residual(s, seed, dtype).double())
        y, sigma = _record(s, seed + 101 * i)
        model = Model64(s, keep=True)
        outs.append(model.reconstruct(y.double().view(s.K, s.M), sigma, case["iters"]))
    return outs[0] if op == "reconstruct" else outs
