"""Workloads of the library over the range that it is used on, each through its public calls.

A case is a dict of plain values; ``prepare`` makes its inputs and plan, ``run`` is one pass as a user's program
makes it, ``exact`` the same results in 64-bit torch without the library.  The inputs come from the seed alone:
ellipsoid phantoms like those of ``phantom.py``, with counts drawn around the phantom's analytic line integrals, and
the listmode events of ``pet_phantom.py``.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2309_01977_gb300 import pet, pet_phantom, spect
from paper_2309_01977_gb300.autograd import poisson_loss

VOXEL_CM, SIGMA0, SLOPE, NSIGMA = 0.48, 0.5, 0.03, 3.0
SERVE_CLASSES = ((64, 60), (96, 96), (128, 120))  # (matrix size, angles)
RDP = {"beta": 0.3, "gamma": 2.0, "alpha0": 1.0}


def listed():
    return [
        # one iteration on a small ragged volume (a scout or a cropped organ): launches and latency
        {"name": "osem_40x36", "kind": "osem", "n": 40, "nz": 36, "angles": 24, "subsets": 4, "iters": 1},
        # the 64^3 clinical matrix, 64 angles, 2 iterations x 8 subsets
        {"name": "osem_64", "kind": "osem", "n": 64, "nz": 64, "angles": 64, "subsets": 8, "iters": 2},
        # the 128^3 x 120-angle matrix, one iteration of 8 subsets, FP32
        {"name": "osem_128", "kind": "osem", "n": 128, "nz": 128, "angles": 120, "subsets": 8, "iters": 1},
        # the same with the tensor-core PSF and FP64 attenuation sums
        {"name": "osem_128_bf16", "kind": "osem", "n": 128, "nz": 128, "angles": 120, "subsets": 8, "iters": 1,
         "bf16": True},
        # simulating an acquisition: every angle of a 128^3 volume
        {"name": "forward_128", "kind": "forward", "n": 128, "nz": 128, "angles": 120, "batch": 1},
        # back projection of a wide-body scan on a non-circular orbit with a shifted, masked detector
        {"name": "back_132x44", "kind": "back", "n": 132, "nz": 44, "angles": 60, "batch": 1, "orbit": True},
        # learned reconstruction: likelihood and gradient of a batch of 192^3 volumes
        {"name": "grad_192", "kind": "grad", "n": 192, "nz": 192, "angles": 128, "batch": 4},
        # MAP reconstruction: BSREM with the relative-difference prior
        {"name": "bsrem_128", "kind": "map", "n": 128, "nz": 128, "angles": 120, "subsets": 8, "iters": 1},
        # the next patient on a kept plan: new attenuation map, new sensitivities
        {"name": "set_mu_96", "kind": "set_mu", "n": 96, "nz": 96, "angles": 96, "subsets": 8},
        # listmode time-of-flight PET: one iteration of 3 subsets
        {"name": "pet_osem_tof", "kind": "pet_osem", "nx": 204, "nz": 154, "vox": 1.25, "events": 3000000,
         "subsets": 3, "tof": True},
        # listmode PET projector pair without time of flight (scatter and normalisation work)
        {"name": "pet_project", "kind": "pet_project", "nx": 128, "nz": 90, "vox": 2.0, "events": 1000000,
         "tof": False},
        # a reconstruction server under a burst of mixed requests
        {"name": "serve_mix", "kind": "serve", "requests": 12, "max_iters": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["osem", "osem", "osem", "osem", "forward", "back", "grad", "map", "set_mu", "pet_osem",
                       "pet_project", "serve"])
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(3, 12), "max_iters": rng.randint(2, 4)}
    if kind.startswith("pet"):
        c = {"kind": kind, "nx": rng.randint(64, 204), "nz": rng.randint(40, 154), "events": _log_int(rng, 5e4, 3e6),
             "tof": rng.random() < 0.5}
        c["vox"] = 255.0 / c["nx"]
        if kind == "pet_osem":
            c["subsets"] = rng.randint(1, 4)
        return c
    if kind == "grad":
        return {"kind": kind, "n": _log_int(rng, 40, 192), "nz": 4 * _log_int(rng, 8, 48), "angles": rng.randint(8, 96),
                "batch": rng.randint(1, 4)}
    bf16 = rng.random() < 0.35
    c = {"kind": kind, "n": 32 * rng.randint(2, 4) if bf16 else _log_int(rng, 32, 160),
         "nz": 8 * rng.randint(4, 16) if bf16 else 4 * _log_int(rng, 6, 40), "angles": _log_int(rng, 16, 120)}
    if bf16:
        c["bf16"] = True
    elif rng.random() < 0.25:
        c["orbit"] = True
    if kind in ("forward", "back"):
        c["batch"] = rng.randint(1, 3)
    else:
        c["subsets"] = rng.randint(2, 8)
        if kind != "set_mu":
            c["iters"] = rng.randint(1, 2)
    return c


# ---------------------------------------------------------------- inputs

def _f32(v):
    return float(np.float32(v))


def _phantom(n, nz, seed):
    """Activity, mu (float32, CUDA) and the ellipsoids behind the activity: a water cylinder with five ellipsoids
    of other activity (added, clamped at 0) and a bone insert."""
    rng = np.random.Generator(np.random.PCG64(seed))
    ax = [torch.arange(m, device="cuda", dtype=torch.float64) - 0.5 * (m - 1) for m in (n, n, nz)]
    x, y, z = ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]
    rad, half, scale = 0.4 * n, 0.4 * nz, min(n, nz) / 64.0
    body = (x * x + y * y <= rad * rad) & (z.abs() <= half)

    def ellipsoid():
        semi = rng.uniform(2.5, 10.0, size=3) * scale
        r, t = (rad - semi[:2].max()) * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi)
        cen = (r * math.cos(t), r * math.sin(t), rng.uniform(-0.7, 0.7) * max(half - semi[2], 0.0))
        ins = ((x - cen[0]) / semi[0]) ** 2 + ((y - cen[1]) / semi[1]) ** 2 + ((z - cen[2]) / semi[2]) ** 2 <= 1.0
        return cen, semi, ins

    f = body.double()
    blobs = []
    for _ in range(5):
        cen, semi, ins = ellipsoid()
        add = rng.uniform(-0.5, 4.0)
        f = f + add * ins
        blobs.append((cen, semi, add))
    mu = 0.15 * body
    mu = torch.where(ellipsoid()[2], torch.full_like(mu, 0.25), mu)
    return f.clamp_(min=0.0).float().contiguous(), mu.float().contiguous(), blobs


def _counts(n, nz, angles, blobs, per_bin, seed):
    """Poisson counts [angles][n][nz] (float32) around the phantom's line integrals, attenuated to its axis, and the
    constant scatter term (5 % of the mean bin)."""
    dev = "cuda"
    j = torch.arange(n, device=dev, dtype=torch.float64) - 0.5 * (n - 1)
    k = torch.arange(nz, device=dev, dtype=torch.float64) - 0.5 * (nz - 1)
    chord = 2.0 * torch.sqrt((0.16 * n * n - j * j).clamp(min=0.0))
    p = (chord[:, None] * (k.abs() <= 0.4 * nz)[None, :]).repeat(angles, 1, 1)
    for cen, semi, add in blobs:
        for a in range(angles):
            t = 2.0 * math.pi * a / angles
            c, s = math.cos(t), math.sin(t)
            off = -s * cen[0] + c * cen[1]
            w2, d2 = (s * semi[0]) ** 2 + (c * semi[1]) ** 2, (c * semi[0]) ** 2 + (s * semi[1]) ** 2
            q = 1.0 - ((j - off) ** 2 / w2)[:, None] - ((k - cen[2]) / semi[2])[None, :] ** 2
            p[a] += add * 2.0 * math.sqrt(d2) * torch.sqrt(q.clamp(min=0.0))
    p = p.clamp(min=0.0) * torch.exp(-0.15 * VOXEL_CM * 0.5 * chord)[None, :, None]
    p = p * (per_bin / p.mean())
    s = _f32(0.05 * per_bin)
    gen = torch.Generator(device=dev).manual_seed(seed)
    return torch.poisson((p + s).float(), generator=gen).contiguous(), s


def _orbit(c, seed):
    """Per-angle detector offsets (an elliptical orbit), shifts and a field-of-view band, or nothing."""
    if not c.get("orbit"):
        return {}
    rng = np.random.Generator(np.random.PCG64(seed + 3))
    na, n, nz = c["angles"], c["n"], c["nz"]
    t = 2.0 * np.pi * np.arange(na) / na
    shift = rng.uniform(-3.0, 3.0, size=na).astype(np.float32)
    j = np.arange(n) - 0.5 * (n - 1)
    fov = np.zeros((na, n, nz), dtype=np.float32)
    fov[np.abs(j[None, :] - shift[:, None]) <= 0.46 * n] = 1.0
    fov[:, :, :1] = 0.5
    return {"det_offsets": [_f32(v) for v in 4.0 + 4.0 * np.cos(t) ** 2], "det_shifts": [float(v) for v in shift],
            "fov_mask": fov}


def _geometry(c, seed):
    return spect.Geometry(n=c["n"], nz=c["nz"], n_angles=c["angles"], n_subsets=c.get("subsets", 1), voxel_cm=VOXEL_CM,
                          psf_sigma0=SIGMA0, psf_slope=SLOPE, psf_nsigma=NSIGMA, psf_bf16=bool(c.get("bf16")),
                          atten_f64=bool(c.get("bf16")), **_orbit(c, seed))


def _serve_requests(c, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    reqs = []
    for r in range(c["requests"]):
        n, na = SERVE_CLASSES[r % 3]
        _, mu, blobs = _phantom(n, n, seed * 1000 + r)
        per_bin = 10.0 ** rng.uniform(6.0, 7.0) / (na * n * n)
        y, s = _counts(n, n, na, blobs, per_bin, seed * 1000 + r)
        reqs.append({"n": n, "nz": n, "angles": na, "subsets": 8, "iters": 2 + (r // 3) % (c["max_iters"] - 1),
                     "mu": mu.cpu().numpy(), "y": y.cpu().numpy(), "s": s})
    return reqs


def _pet_inputs(c, seed):
    """Grid, events and images of a listmode PET case: the head phantom's events on the cylindrical scanner, the
    attenuation of each line through the head, a smooth sensitivity image."""
    wl = dataclasses.replace(pet_phantom.PET_WORKLOADS["petlm204tof"], shape=(c["nx"], c["nx"], c["nz"]),
                             voxel=(c["vox"],) * 3, prompts=c["events"], seed=seed, tof_bins=21 if c["tof"] else 0)
    act, mu, semi = pet_phantom.head_phantom(wl.shape, wl.voxel, wl.seed, device="cuda")
    lors, eta, s, _, tof = pet_phantom.draw_events(wl, act, semi, device="cuda")
    p1, p2 = lors[:, :3].double(), lors[:, 3:].double()
    d = (p2 - p1) / torch.linalg.norm(p2 - p1, dim=-1, keepdim=True)
    chord = pet_phantom._ellipsoid_chord(0.5 * (p1 + p2), d, semi)
    mult = (eta.double() * torch.exp(-pet_phantom.WATER_MU_MM * chord)).float().contiguous()
    ax = [torch.linspace(-1.0, 1.0, m, device="cuda", dtype=torch.float64) for m in wl.shape]
    r2 = ax[0][:, None, None] ** 2 + ax[1][None, :, None] ** 2
    sens = c["events"] / act.numel() * 40.0 * (1.0 - 0.3 * r2) * (1.05 - ax[2].abs())[None, None, :]
    g = pet.PetGeometry(wl.shape, wl.voxel, rr_sigma_mm=wl.rr_sigma_mm, n_subsets=c.get("subsets", 1),
                        n_tof_bins=wl.tof_bins, tof_bin_mm=wl.tof_bin_mm, tof_sigma_mm=wl.tof_sigma_mm)
    gen = torch.Generator(device="cuda").manual_seed(seed + 17)
    q = torch.rand(lors.shape[0], device="cuda", generator=gen)
    return g, {"act": act, "mu": mu, "lors": lors, "mult": mult, "s": s, "tof": tof, "q": q,
               "sens": sens.float().contiguous()}


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "serve":
        return {"kind": kind, "server": spect.Server(8 << 30, max_slots=8, n_streams=8),
                "reqs": [(spect.Geometry(n=r["n"], nz=r["nz"], n_angles=r["angles"], n_subsets=r["subsets"]), r)
                         for r in _serve_requests(c, seed)]}
    if kind.startswith("pet"):
        g, st = _pet_inputs(c, seed)
        st.update(kind=kind, subsets=c.get("subsets", 1), plan=pet.PetPlan(g, st["mu"]))
        return st
    n, nz = c["n"], c["nz"]
    f, mu, blobs = _phantom(n, nz, seed)
    plan = spect.Plan(_geometry(c, seed), mu)
    st = {"kind": kind, "plan": plan, "subsets": c.get("subsets", 1), "count": c.get("subsets", 1) * c.get("iters", 1)}
    if kind == "set_mu":
        st["mu"] = _phantom(n, nz, seed + 7)[1]
        return st
    y, s = _counts(n, nz, c["angles"], blobs, 5.0, seed)
    if kind == "forward":
        st["x"] = torch.stack([f * 2.0 ** b for b in range(c["batch"])])
    elif kind == "back":
        st["y"] = torch.stack([y * 2.0 ** b for b in range(c["batch"])])
    elif kind == "grad":
        st["x"] = torch.stack([0.1 * f + 0.05 * (b + 1) for b in range(c["batch"])])
        st.update(y=torch.stack([y] * c["batch"]), s=s)
    else:
        st.update(y=y, s=s, shape=(n, n, nz))
    return st


def run(state):
    st, kind = state, state["kind"]
    if kind == "serve":
        sv = st["server"]
        ids = [sv.submit(g, r["mu"], r["y"], r["s"], r["iters"]) for g, r in st["reqs"]]
        return [sv.wait(i)[0] for i in ids]
    plan = st["plan"]
    if kind == "pet_osem":
        x = torch.ones_like(st["sens"])
        plan.lm_osem(st["lors"], st["mult"], st["s"], st["sens"], x, 0, st["subsets"], tof_bin=st["tof"])
        return x
    if kind == "pet_project":
        return {"p": plan.forward(st["act"], st["lors"], st["mult"], tof_bin=st["tof"]),
                "b": plan.back(st["q"], st["lors"], st["mult"], tof_bin=st["tof"])}
    if kind == "set_mu":
        spect.spect_plan_set_mu(plan.handle, st["mu"])
        return [plan.sensitivity(m) for m in range(st["subsets"])]
    if kind == "forward":
        return plan.forward(st["x"])
    if kind == "back":
        return plan.back(st["y"])
    if kind == "grad":
        x = st["x"].clone().requires_grad_(True)
        loss = poisson_loss(x, st["y"], st["s"], plan)
        loss.backward()
        return {"loss": loss.detach().float(), "grad": x.grad}
    x = torch.ones(st["shape"], device="cuda")
    if kind == "map":
        plan.map(st["y"], st["s"], x, 0, st["count"], algorithm="bsrem", prior="rdp", **RDP)
    else:
        plan.osem(st["y"], st["s"], x, 0, st["count"])
    return x


# ---------------------------------------------------------------- work

def _radii(c, off=0.0):
    return [math.ceil(NSIGMA * (SIGMA0 + SLOPE * (c["n"] - i - 0.5 + off))) for i in range(c["n"])]


def _spect_work(c, sel, batch, both=False):
    """Bytes and operations of H or H^T (both: of the pair) over `sel` angles: the attenuation planes, the volume and
    the projections once; interpolation, attenuation and the two blur passes."""
    n, nz = c["n"], c["nz"]
    plane = n * nz
    flops = batch * sel * plane * sum(9.0 + 4.0 * (2 * r + 1) for r in _radii(c, 6.0 if c.get("orbit") else 0.0))
    return 4.0 * (sel * n * plane + batch * (n * plane + sel * plane)), flops * (2 if both else 1)


def work(case):
    c, kind = case, case["kind"]
    if kind == "serve":
        b = f = 0.0
        for r in range(c["requests"]):
            n, na = SERVE_CLASSES[r % 3]
            w = work({"kind": "osem", "n": n, "nz": n, "angles": na, "subsets": 8,
                      "iters": 2 + (r // 3) % (c["max_iters"] - 1)})
            b, f = b + w["bytes"], f + w["flops"]
        return {"bytes": b, "flops": f}
    if kind.startswith("pet"):
        vol = 4.0 * c["nx"] ** 2 * c["nz"]
        planes = (0.55 if c["tof"] else 0.85) * c["nx"]
        sub = c.get("subsets", 1)
        # 24 + 4 + 4 (+ 4) bytes an event; the image read, accumulated and blurred once a subiteration; about 30
        # operations a sample each way
        return {"bytes": c["events"] * 36.0 + 4.0 * vol * sub, "flops": c["events"] * planes * 60.0}
    if kind in ("forward", "back"):
        b, f = _spect_work(c, c["angles"], c["batch"])
    elif kind == "grad":
        b, f = _spect_work(c, c["angles"], c["batch"], True)
    elif kind == "set_mu":
        vol = 4.0 * c["n"] ** 2 * c["nz"]
        b, f = vol * (1 + c["angles"] + c["subsets"]), c["angles"] * vol / 4.0 * 30.0
    else:
        b, f = _spect_work(c, c["angles"], 1, True)
        b, f = b * c["iters"], f * c["iters"]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same in 64 bits

class _Spect64:
    """H and H^T of the parallel-hole model in float64, one angle at a time."""

    def __init__(self, c, mu, orbit):
        self.n, self.nz, self.na = c["n"], c["nz"], c["angles"]
        self.mu = mu.double()
        self.orbit = orbit
        self.tables = {}
        fov = orbit.get("fov_mask")
        self.fov = None if fov is None else torch.from_numpy(fov).cuda().double()

    def _taps(self, a):
        n, nz = self.n, self.nz
        c = 0.5 * (n - 1)
        t = 2.0 * math.pi * a / self.na
        ct, s = math.cos(t), math.sin(t)
        if (4 * a) % self.na == 0:
            ct, s = ((1.0, 0.0), (0.0, 1.0), (-1.0, 0.0), (0.0, -1.0))[4 * a // self.na]
        cj = c + (self.orbit["det_shifts"][a] if self.orbit else 0.0)
        g = torch.arange(n, device="cuda", dtype=torch.float64)
        i, j = g[:, None] - c, g[None, :] - cj
        u, v = c + ct * i - s * j, c + s * i + ct * j
        x0, y0 = torch.floor(u), torch.floor(v)
        ax, ay = u - x0, v - y0
        out = []
        for dx, wx in ((0, 1 - ax), (1, ax)):
            for dy, wy in ((0, 1 - ay), (1, ay)):
                x, y = (x0 + dx).long(), (y0 + dy).long()
                ok = (x >= 0) & (x < n) & (y >= 0) & (y < n)
                out.append(((x.clamp(0, n - 1) * n + y.clamp(0, n - 1)).reshape(-1),
                            (wx * wy * ok).reshape(-1, 1)))
        return out

    def _blur(self, a):
        off = self.orbit["det_offsets"][a] if self.orbit else 0.0
        if off not in self.tables:
            n = self.n
            sig = _f32(SIGMA0) + _f32(SLOPE) * (n - np.arange(n) - 0.5 + off)
            t = np.arange(-40, 41)
            w = np.exp(-t[None, :] ** 2 / (2 * sig[:, None] ** 2)) * (np.abs(t)[None, :] <= np.ceil(NSIGMA * sig)[:, None])
            w = torch.from_numpy(w / w.sum(1, keepdims=True)).cuda()

            def band(m):
                d = torch.arange(m, device="cuda")
                d = (d[:, None] - d[None, :]).clamp(-40, 40)
                return w[:, d + 40] * (d.abs() < 40)
            if len(self.tables) > 2:
                self.tables.clear()
            self.tables[off] = band(self.n), band(self.nz)
        return self.tables[off]

    def _rot(self, f, taps):
        flat = f.reshape(self.n * self.n, self.nz)
        return sum(w * flat[idx] for idx, w in taps).reshape(self.n, self.n, self.nz)

    def _angle(self, a):
        taps = self._taps(a)
        tau = _f32(VOXEL_CM) * self._rot(self.mu, taps)
        tail = torch.flip(torch.cumsum(torch.flip(tau, (0,)), 0), (0,)) - tau
        return taps, torch.exp(-(tail + 0.5 * tau)), *self._blur(a)

    def forward(self, vols, sel):
        out = torch.empty(len(vols), len(sel), self.n, self.nz, device="cuda", dtype=torch.float64)
        for q, a in enumerate(sel):
            taps, att, ty, tz = self._angle(a)
            for b, f in enumerate(vols):
                out[b, q] = torch.bmm(ty, torch.bmm(self._rot(f, taps) * att, tz)).sum(0)
                if self.fov is not None:
                    out[b, q] *= self.fov[a]
        return out

    def back(self, projs, sel):
        out = torch.zeros(len(projs), self.n * self.n, self.nz, device="cuda", dtype=torch.float64)
        for q, a in enumerate(sel):
            taps, att, ty, tz = self._angle(a)
            for b, p in enumerate(projs):
                r = p[q] if self.fov is None else p[q] * self.fov[a]
                v = (torch.bmm(ty, torch.matmul(r, tz)) * att).reshape(-1, self.nz)
                for idx, w in taps:
                    out[b].index_add_(0, idx, w * v)
        return out.reshape(len(projs), self.n, self.n, self.nz)

    def subset(self, m, M):
        return list(range(m, self.na, M))


def _ratio(a, b):
    return torch.where(b > 0, a / torch.where(b > 0, b, torch.ones_like(b)), torch.zeros_like(a))


def _osem64(h, y, s, M, count):
    x = torch.ones(h.n, h.n, h.nz, device="cuda", dtype=torch.float64)
    sens = {}
    for t in range(count):
        sel = h.subset(t % M, M)
        if t % M not in sens:
            sens[t % M] = h.back(torch.ones(1, len(sel), h.n, h.nz, device="cuda", dtype=torch.float64), sel)[0]
        r = _ratio(y[sel].double(), h.forward([x], sel)[0] + s)
        sm = sens[t % M]
        x = torch.where(sm > 0, x * _ratio(h.back([r], sel)[0], sm), x)
    return x


def _rdp_grad(x, gamma):
    g = torch.zeros_like(x)
    n0, n1, n2 = x.shape
    for di in (-1, 0, 1):
        for dj in (-1, 0, 1):
            for dk in (-1, 0, 1):
                if not (di or dj or dk):
                    continue
                here = tuple(slice(max(0, -d), m - max(0, d)) for d, m in ((di, n0), (dj, n1), (dk, n2)))
                there = tuple(slice(max(0, d), m - max(0, -d)) for d, m in ((di, n0), (dj, n1), (dk, n2)))
                a, b = x[here], x[there]
                d = a - b
                den = (a + b + gamma * d.abs()) ** 2
                g[here] += 2.0 / math.sqrt(di * di + dj * dj + dk * dk) * _ratio(d * (a + 3 * b + gamma * d.abs()), den)
    return g


def _bsrem64(h, y, s, M, count):
    x = torch.ones(h.n, h.n, h.nz, device="cuda", dtype=torch.float64)
    ones = torch.ones(1, 1, h.n, h.nz, device="cuda", dtype=torch.float64)
    sens = [h.back(ones.expand(1, len(h.subset(m, M)), -1, -1), h.subset(m, M))[0] for m in range(M)]
    total = sum(sens)
    for t in range(count):
        sel = h.subset(t % M, M)
        bp = h.back([_ratio(y[sel].double(), h.forward([x], sel)[0] + s)], sel)[0]
        step = RDP["alpha0"] / (1 + t // M) * M
        v = x + step * _ratio(x, total) * ((bp - sens[t % M]) - _f32(RDP["beta"]) / M * _rdp_grad(x, RDP["gamma"]))
        x = torch.where(total > 0, v.clamp(min=0.0), x)
    return x


class _Pet64:
    """Joseph line integrals of listmode lines (with time-of-flight bins when given) and their transpose in float64.
    The walk's integers, the principal axis and the first and last plane, are decided in float32 as the model
    defines them for float32 line ends."""

    def __init__(self, g):
        self.g, self.shape, self.v = g, g.shape, [_f32(v) for v in g.voxel]

    def walk(self, lors, tof, fn):
        """fn(line indices, flat voxel indices, weights) for every sample and tap of the lines."""
        p1, p2 = lors[:, :3], lors[:, 3:]
        vt = torch.tensor(self.v, dtype=torch.float32, device="cuda")
        sc = (p2 - p1).abs() / vt
        axis = torch.where(sc[:, 1] > sc[:, 0], 1, 0)
        axis = torch.where(sc[:, 2] > sc.gather(1, axis[:, None])[:, 0], torch.full_like(axis, 2), axis)
        stride = (self.shape[1] * self.shape[2], self.shape[2], 1)
        for a in range(3):
            ids = torch.nonzero(axis == a)[:, 0]
            if not len(ids):
                continue
            b, c = (1, 2) if a == 0 else (0, 2) if a == 1 else (0, 1)
            e1, e2 = p1[ids], p2[ids]
            half = torch.tensor(0.5 * (self.shape[a] - 1), dtype=torch.float32, device="cuda")
            org = -(half * vt[a])
            s1, s2 = (e1[:, a] - org) / vt[a], (e2[:, a] - org) / vt[a]
            lo = torch.ceil(torch.minimum(s1, s2)).clamp(min=0.0).double()
            hi = torch.floor(torch.maximum(s1, s2)).clamp(max=float(self.shape[a] - 1)).double()
            e1, e2 = e1.double(), e2.double()
            length = torch.linalg.norm(e2 - e1, dim=1)
            i1 = [(e1[:, k] + 0.5 * (self.shape[k] - 1) * self.v[k]) / self.v[k] for k in range(3)]
            i2 = [(e2[:, k] + 0.5 * (self.shape[k] - 1) * self.v[k]) / self.v[k] for k in range(3)]
            da = i2[a] - i1[a]
            step = self.v[a] * length / (e2[:, a] - e1[:, a]).abs()
            if tof is not None:
                g = self.g
                w, sig = _f32(g.tof_bin_mm), _f32(g.tof_sigma_mm)
                cen = (tof[ids].double() - 0.5 * (g.n_tof_bins - 1)) * w
                win = _f32(g.tof_nsigma) * sig + 0.5 * w
            for q in range(self.shape[a]):
                t = (q - i1[a]) / da
                ok = (q >= lo) & (q <= hi)
                wt = step
                if tof is not None:
                    x = (t - 0.5) * length - cen
                    ok &= x.abs() <= win
                    r = math.sqrt(2.0) * sig
                    wt = step * 0.5 * (torch.erf((x + 0.5 * w) / r) - torch.erf((x - 0.5 * w) / r))
                u, z = i1[b] + t * (i2[b] - i1[b]), i1[c] + t * (i2[c] - i1[c])
                fu, fz = torch.floor(u), torch.floor(z)
                for du, wu in ((0, 1 - (u - fu)), (1, u - fu)):
                    for dz, wz in ((0, 1 - (z - fz)), (1, z - fz)):
                        iu, iz = fu + du, fz + dz
                        m = ok & (iu >= 0) & (iu < self.shape[b]) & (iz >= 0) & (iz < self.shape[c])
                        flat = q * stride[a] + iu.long() * stride[b] + iz.long() * stride[c]
                        fn(ids, torch.where(m, flat, torch.zeros_like(flat)), wt * wu * wz * m)

    def forward(self, img, lors, tof):
        out, flat = torch.zeros(len(lors), device="cuda", dtype=torch.float64), img.reshape(-1)
        self.walk(lors, tof, lambda ids, idx, w: out.index_add_(0, ids, w * flat[idx]))
        return out

    def back(self, q, lors, tof):
        out = torch.zeros(math.prod(self.shape), device="cuda", dtype=torch.float64)
        self.walk(lors, tof, lambda ids, idx, w: out.index_add_(0, idx, w * q[ids]))
        return out.reshape(self.shape)

    def blur(self, img):
        for ax in range(3):
            s = _f32(self.g.rr_sigma_mm) / self.v[ax]
            r = math.ceil(_f32(self.g.rr_nsigma) * s)
            w = torch.exp(-torch.arange(-r, r + 1, dtype=torch.float64) ** 2 / (2 * s * s))
            w = (w / w.sum()).tolist()
            m = img.shape[ax]
            pad = torch.zeros_like(img)
            for t in range(-r, r + 1):
                if abs(t) < m:
                    pad.narrow(ax, max(0, t), m - abs(t)).add_(img.narrow(ax, max(0, -t), m - abs(t)), alpha=w[t + r])
            img = pad
        return img


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "serve":
        out = []
        for r in _serve_requests(c, seed):
            h = _Spect64(r, torch.from_numpy(r["mu"]).cuda(), {})
            out.append(_osem64(h, torch.from_numpy(r["y"]).cuda(), r["s"], 8, 8 * r["iters"]))
        return out
    if kind.startswith("pet"):
        g, st = _pet_inputs(c, seed)
        h, tof = _Pet64(g), st["tof"]
        mult = st["mult"].double()
        if kind == "pet_project":
            return {"p": mult * h.forward(h.blur(st["act"].double()), st["lors"], tof),
                    "b": h.blur(h.back(mult * st["q"].double(), st["lors"], tof))}
        x, M = torch.ones_like(st["sens"]).double(), c["subsets"]
        for m in range(M):
            lors, mu, s = st["lors"][m::M], mult[m::M], st["s"][m::M].double()
            sub = None if tof is None else tof[m::M]
            bp = h.blur(h.back(_ratio(mu, mu * h.forward(h.blur(x), lors, sub) + s), lors, sub))
            x = x * bp / (st["sens"].double() / M)
        return x
    n, nz = c["n"], c["nz"]
    f, mu, blobs = _phantom(n, nz, seed)
    M = c.get("subsets", 1)
    if kind == "set_mu":
        mu = _phantom(n, nz, seed + 7)[1]
    h = _Spect64(c, mu, _orbit(c, seed))
    every = list(range(c["angles"]))
    if kind == "set_mu":
        one = torch.ones(1, 1, n, nz, device="cuda", dtype=torch.float64)
        return [h.back(one.expand(1, len(h.subset(m, M)), -1, -1), h.subset(m, M))[0] for m in range(M)]
    y, s = _counts(n, nz, c["angles"], blobs, 5.0, seed)
    if kind == "forward":
        return h.forward([f.double() * 2.0 ** b for b in range(c["batch"])], every)
    if kind == "back":
        return h.back([y.double() * 2.0 ** b for b in range(c["batch"])], every)
    if kind == "grad":
        vols = [(0.1 * f + 0.05 * (b + 1)).double() for b in range(c["batch"])]
        lam = h.forward(vols, every) + s
        yy = y.double()
        loss = (yy * torch.log(lam) - lam).sum()
        return {"loss": loss.reshape(()), "grad": h.back(_ratio(yy.expand_as(lam), lam) - 1.0, every)}
    if kind == "map":
        return _bsrem64(h, y, s, M, M * c["iters"])
    return _osem64(h, y, s, M, M * c["iters"])
