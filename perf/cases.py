"""Timed cases of the library: what a program that inverts seismic data has
it do, through the public Python entry points.

A program of that kind keeps one Model handle per grid (its working fields
live in it) and gives it a new medium before each call, so a pass of the
wave-propagation cases is set_model plus one forward, misfit or gradient
call.  Media are smooth random fields with velocity growing with depth,
observed data are direct and reflected arrivals along straight rays; both
come from the seed, the acquisition geometry from the case.

Kinds of case:
  forward   ckfwi.Model.forward_shot: simulated data of one shot
  misfit    ckfwi.Model.misfit: what a line search evaluates
  gradient  ckfwi.Model.adjoint_gradient: misfit and gradient of one shot
  fwi       autograd.misfit and its backward over several shots: one
            iteration of an inversion, batched adjoint
  windows   ckfwi.batch_gradient_models: shots with uneven apertures
  codec     codec_compress + codec_decompress of one field (fixed accuracy)
  rate      codec_compress_rate + codec_decompress (fixed rate)
"""
import functools
import math

import numpy as np
import torch

from paper_1810_05268_gb300 import autograd as A
from paper_1810_05268_gb300 import ckfwi as C

NBL = 40          # damping layer [cells] of the full-size grids


def _wave(name, kind, shape, so, nt, h, dt, vmin, vmax, f0, nrec, **kw):
    c = {"name": name, "kind": kind, "nz": shape[0], "ny": shape[1] if len(shape) == 3 else 1, "nx": shape[-1],
         "dims": len(shape), "so": so, "nt": nt, "h": h, "dt": dt, "vmin": vmin, "vmax": vmax, "f0": f0,
         "nrec": nrec, "nbl": NBL, "time_order": 2, "store": "fp32", "slots": 0, "graph": False}
    c.update(kw)
    return c


def listed():
    return [
        # one shot modelled on a small 2D section: many short steps
        _wave("forward_2d_281", "forward", (281, 281), 4, 500, 10.0, 1.0, 1.5, 2.5, 0.010, 101),
        # the same section's gradient with 20 checkpoints, replayed as a graph
        _wave("gradient_2d_281", "gradient", (281, 281), 4, 500, 10.0, 1.0, 1.5, 2.5, 0.010, 101, slots=20,
              graph=True),
        # one trial of a line search on a 2D line of survey size
        _wave("misfit_2d_464x1104", "misfit", (464, 1104), 8, 2000, 10.0, 1.0, 1.5, 4.5, 0.010, 512),
        # one inversion iteration on that line: misfits, then the batched
        # adjoint with codec checkpoints
        _wave("fwi_2d_464x1104_codec", "fwi", (464, 1104), 8, 2000, 10.0, 1.0, 1.5, 4.5, 0.010, 512, slots=16,
              store="codec", tol=3e-3, shots=8),
        # the benchmark's gradient at the memory of 20 FP32 states
        _wave("gradient_3d_208_fp32", "gradient", (208, 208, 208), 8, 1000, 15.0, 1.0, 1.5, 4.5, 0.008, 64,
              slots=20, graph=True),
        # the same with block-codec checkpoints
        _wave("gradient_3d_208_codec", "gradient", (208, 208, 208), 8, 500, 15.0, 1.0, 1.5, 4.5, 0.008, 64,
              slots=116, store="codec", tol=1e-4, graph=True),
        # 16-bit checkpoints on a grid whose sides divide by no tile
        _wave("gradient_3d_ragged_fp16", "gradient", (187, 213, 229), 8, 300, 15.0, 1.0, 1.5, 4.5, 0.008, 41,
              slots=39, store="fp16"),
        # fourth order in time
        _wave("gradient_3d_208_ot4", "gradient", (208, 208, 208), 8, 200, 15.0, 1.0, 1.5, 4.5, 0.008, 64, slots=10,
              graph=True, time_order=4),
        # the largest grid, order 16, few checkpoints
        _wave("gradient_3d_300x600x600_so16", "gradient", (300, 600, 600), 16, 64, 25.0, 1.5, 1.5, 6.0, 0.005, 64,
              slots=8),
        # shots with uneven apertures in one batch
        _wave("windows_3d_fp32", "windows", (256, 288, 304), 8, 200, 15.0, 1.0, 1.5, 4.5, 0.008, 32, slots=16,
              shots=6, smallest=120),
        # one field through each mode of the standalone codec
        {"name": "codec_field_208", "kind": "codec", "nz": 208, "ny": 208, "nx": 208, "dims": 3, "tol": 1e-4},
        {"name": "rate_field_ragged", "kind": "rate", "nz": 187, "ny": 213, "nx": 229, "dims": 3, "rate": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "misfit", "gradient", "gradient", "gradient", "fwi", "windows", "codec", "rate"])
    if kind in ("codec", "rate"):
        if rng.random() < 0.3:
            c = {"kind": kind, "nz": _log(rng, 64, 2048), "ny": 1, "nx": _log(rng, 64, 4096), "dims": 2}
        else:
            c = {"kind": kind, "nz": _log(rng, 24, 256), "ny": _log(rng, 24, 256), "nx": _log(rng, 24, 256),
                 "dims": 3}
        if kind == "codec":
            c["tol"] = rng.choice([1e-2, 1e-3, 1e-4, 1e-5])
        else:
            c["rate"] = rng.choice([4, 8, 12, 16, 24])
        return c
    so = rng.choice([2, 4, 8, 8, 8, 16])
    slow, fast = rng.choice([(1.5, 3.0), (1.5, 4.5)])
    store = rng.choice(["fp32", "fp32", "fp16", "bf16", "codec", "rate"])
    kw = {"slots": _log(rng, 4, 60), "store": store, "tol": 1e-3, "rate": 16, "graph": rng.random() < 0.5,
          "nbl": rng.choice([10, 20, 40])}
    if kind == "windows":
        kw.update(shots=rng.randint(2, 5), smallest=rng.randint(90, 130))
        shape = tuple(rng.randint(150, 224) for _ in range(3))
        return _drawn(kind, shape, rng.choice([4, 8]), rng.randint(40, 150), slow, fast, 24, kw)
    if kind == "fwi" or rng.random() < 0.4:
        shape = (_log(rng, 100, 800), _log(rng, 100, 1600))
        nt = _log(rng, 100, 1500)
        if kind == "fwi":
            kw["shots"] = rng.randint(2, 8)
            nt = min(nt, 800)
    else:
        shape = tuple(_log(rng, 90, 260) for _ in range(3))
        nt = _log(rng, 20, 250)
        if kind == "gradient" and rng.random() < 0.25:
            kw["time_order"] = 4
            nt = min(nt, 120)
        if rng.random() < 0.2:
            kw["slots"] = nt          # every state kept
    return _drawn(kind, shape, so, nt, slow, fast, rng.randint(16, 64), kw)


def _drawn(kind, shape, so, nt, slow, fast, nrec, kw):
    h = 15.0 if fast > 4.0 else 10.0
    c = _wave("", kind, shape, so, nt, h, 1.0, slow, fast, 0.08 / h, nrec, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if case["dims"] == 3 else (case["nz"], case["nx"])


def _smooth(shape, cells, seed):
    """Smooth random field on the device, values about -1 .. 1: noise on a
    coarse grid of `cells` points a node, interpolated."""
    g = torch.Generator().manual_seed(seed)
    coarse = torch.randn((1, 1) + tuple(max(2, n // cells + 2) for n in shape), generator=g)
    mode = "trilinear" if len(shape) == 3 else "bilinear"
    f = torch.nn.functional.interpolate(coarse.cuda(), size=tuple(shape), mode=mode, align_corners=True)
    return (f[0, 0] / 3.0).clamp_(-1.0, 1.0)


def _medium(shape, vmin, vmax, seed):
    z = torch.linspace(0.0, 1.0, shape[0], device="cuda").reshape((-1,) + (1,) * (len(shape) - 1))
    f = (0.5 * z + 0.25 + 0.6 * _smooth(shape, 12, seed)).clamp_(0.0, 1.0)
    return (vmin + (vmax - vmin) * f).float().contiguous()


def _geometry(case, shape, shot=0, shots=1):
    """Source and receivers [m] from the first interior point: the source at
    two cells' depth, receivers on a line (2D) or a square grid (3D)."""
    h = case["h"]
    ext = [(n - 2 * case["nbl"] - 1) * h for n in shape]
    at = (shot + 0.5) / shots
    n = case["nrec"]
    if case["dims"] == 3:
        yy, xx = np.meshgrid(np.linspace(0.0, ext[1], n), np.linspace(0.0, ext[2], n), indexing="ij")
        rec = np.stack([np.full(yy.size, 2.0 * h), yy.ravel(), xx.ravel()], axis=1)
        return (2.0 * h, 0.47 * ext[1], at * ext[2]), rec
    xs = np.linspace(0.0, ext[1], n)
    return (2.0 * h, 0.0, at * ext[1]), np.stack([np.full(n, 2.0 * h), np.zeros(n), xs], axis=1)


def _observed(case, src, rec, seed):
    """Recorded data [nt + 1][nrec]: a direct and a reflected arrival with the
    seed's velocity, depth and reflectivity."""
    g = np.random.default_rng(seed)
    v = case["vmin"] + (case["vmax"] - case["vmin"]) * g.uniform(0.2, 0.5)
    depth, refl = case["h"] * g.uniform(20.0, 60.0), g.uniform(0.2, 0.5)
    h, f0 = case["h"], case["f0"]
    r = torch.from_numpy(np.asarray(rec) - np.asarray(src)).cuda()
    t = torch.arange(case["nt"] + 1, dtype=torch.float64, device="cuda")[:, None] * case["dt"] - 1.5 / f0
    d = torch.zeros(case["nt"] + 1, r.shape[0], dtype=torch.float64, device="cuda")
    for drop, amp in ((0.0, 1.0), (2.0 * depth, refl)):
        dist = (r.square().sum(1) + drop * drop + 4.0 * h * h).sqrt()
        a = (math.pi * f0) ** 2 * (t - dist / v) ** 2
        if case["dims"] == 3:
            scale = h ** 3 / (4.0 * math.pi * dist)
        else:
            scale = 0.25 * h * h * (v / (math.pi ** 2 * f0 * dist)).sqrt()
        d += amp * scale * (1.0 - 2.0 * a) * torch.exp(-a)
    d[0] = 0.0
    return d.float()


def _windows(case):
    """Sizes and offsets (total grid) of the shots' apertures."""
    g = np.random.default_rng(1813)
    survey, k, out = _shape(case), case["shots"], []
    for i in range(k):
        size = [int(round(min(s, case["smallest"]) + (s - min(s, case["smallest"])) * 0.8 * i / max(1, k - 1)))
                for s in survey]
        out.append((tuple(size), tuple(int(g.integers(0, s - n + 1)) for s, n in zip(survey, size))))
    return out


@functools.lru_cache(maxsize=1)
def _models(dims, shapes, nbl, h, so, dt, nt, vmax, time_order):
    """The handles a program keeps for its grids."""
    return [C.Model(C.GridSpec(dims, s, nbl, h, so, dt, nt, vmax, time_order)) for s in shapes]


def _handles(case, shapes):
    return _models(case["dims"], tuple(shapes), case["nbl"], case["h"], case["so"], case["dt"], case["nt"],
                   case["vmax"], case["time_order"])


def _wavefield(shape, seed):
    """A field like a wavefield in mid-propagation: a few spherical fronts
    in quiet surroundings."""
    g = np.random.default_rng(seed)
    axes = [torch.arange(n, dtype=torch.float32, device="cuda").reshape([-1 if i == a else 1 for i in range(len(shape))])
            for a, n in enumerate(shape)]
    f = torch.zeros(shape, device="cuda")
    for _ in range(4):
        r = sum((x - float(g.uniform(0.1, 0.9)) * n).square() for x, n in zip(axes, shape)).sqrt()
        front, width = float(g.uniform(0.1, 0.6)) * max(shape), float(g.uniform(4.0, 9.0))
        a = ((r - front) / width).square()
        f += float(g.uniform(0.2, 1.0)) * (1.0 - 2.0 * a) * torch.exp(-a) / (1.0 + 0.02 * r)
    return (0.2 * f * (1.0 + 0.1 * _smooth(shape, 8, seed))).contiguous()


def _options(case):
    o = {}
    if case["kind"] in ("gradient", "fwi", "windows"):
        o = {"store_mode": case["store"], "use_graph": case["graph"]}
        if case["store"] == "codec":
            o["tol"] = case["tol"]
            # a share of the FP32 states' bytes large enough for any field
            o["pool_bytes"] = case["slots"] * 2 * case["nz"] * case["ny"] * case["nx"] * 4
        elif case["store"] == "rate":
            o["rate"] = case["rate"]
    return o


def prepare(case, seed):
    kind, shape = case["kind"], _shape(case)
    if kind in ("codec", "rate"):
        # the archive's slab a stream goes into (no stream is longer than its field)
        return {"case": case, "x": _wavefield(shape, seed),
                "slab": torch.zeros(case["nz"] * case["ny"] * case["nx"] + 1024, dtype=torch.int32, device="cuda")}
    st = {"case": case, "opts": _options(case)}
    if kind == "windows":
        wins = _windows(case)
        st["models"] = _handles(case, [w[0] for w in wins])
        st["offsets"] = [w[1] for w in wins]
        vel = _medium(shape, case["vmin"], case["vmax"], seed)
        st["media"] = [vel[tuple(slice(o, o + n) for o, n in zip(off, size))].contiguous() for size, off in wins]
        geo = [_geometry(case, size) for size, _ in wins]
    else:
        st["model"] = _handles(case, [shape])[0]
        vel = _medium(shape, case["vmin"], case["vmax"], seed)
        st["medium"] = (1.0 / vel.double().square()).float() if kind == "fwi" else vel
        n = case.get("shots", 1)
        geo = [_geometry(case, shape, i, n) for i in range(n)]
    st["shots"] = [C.ShotSpec(src=s, rec=r, f0=case["f0"]) for s, r in geo]
    st["dobs"] = [_observed(case, s, r, seed + 7919 * i) for i, (s, r) in enumerate(geo)]
    return st


# --------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("codec", "rate"):
        if kind == "codec":
            words, _ = C.codec_compress(state["x"], case["tol"])
        else:
            words, _ = C.codec_compress_rate(state["x"], case["rate"])
        state["slab"][:words.numel()].copy_(words)
        return {"words": words.numel(), "slab": state["slab"], "field": C.codec_decompress(words, _shape(case))}
    if kind == "windows":
        for m, c in zip(state["models"], state["media"]):
            m.set_model(c)
        phi, grad, _ = C.batch_gradient_models(state["models"], state["shots"], state["dobs"], state["offsets"],
                                               _shape(case), case["slots"], **state["opts"])
        return {"phi": phi, "grad": grad}
    model = state["model"]
    if kind == "fwi":
        m = state["medium"].clone().requires_grad_(True)
        phi = A.misfit(m, model, state["shots"], state["dobs"], case["slots"], **state["opts"])
        (grad,) = torch.autograd.grad(phi, m)
        return {"phi": phi.detach(), "grad": grad}
    model.set_model(state["medium"])
    if kind == "forward":
        return {"d": model.forward_shot(state["shots"][0])}
    if kind == "misfit":
        d = torch.empty_like(state["dobs"][0])
        return {"phi": model.misfit(state["shots"][0], state["dobs"][0], d_sim=d), "d": d}
    phi, grad, _ = model.adjoint_gradient(state["shots"][0], state["dobs"][0], case["slots"], **state["opts"])
    return {"phi": phi, "grad": grad}


# -------------------------------------------------------------------- work
def _extra_steps(case):
    """Forward steps a checkpointed gradient needs beside its reverse steps."""
    if case["slots"] >= case["nt"]:
        return case["nt"]
    return C.revolve_schedule(case["nt"], case["slots"])[1][0] + 1


def work(case):
    npts = case["nz"] * case["ny"] * case["nx"]
    kind = case["kind"]
    if kind == "codec":      # the field in, about a tenth of it as stream out and in, the field out
        return {"bytes": 8.2 * npts, "flops": 0.0}
    if kind == "rate":
        return {"bytes": (8.0 + case["rate"] / 4.0) * npts, "flops": 0.0}
    shots = case.get("shots", 1)
    if kind == "windows":
        npts = sum(int(np.prod(s)) for s, _ in _windows(case)) / shots
    # a forward step reads u^n, u^{n-1}, w and writes u^{n+1}; a reverse step
    # reads two adjoint fields, u, w and g and writes one adjoint field and g
    lap = case["dims"] * (case["so"] // 2) * 4.0
    passes = 2.0 if case["time_order"] == 4 else 1.0
    fwd_b, rev_b = 16.0, 28.0
    fwd_f, rev_f = passes * lap + 8.0, 2.0 * passes * lap + 12.0
    steps_f, steps_r = {"forward": (case["nt"], 0), "misfit": (case["nt"], 0)}.get(kind, (0, case["nt"]))
    if kind in ("gradient", "fwi", "windows"):
        steps_f = _extra_steps(case) + (case["nt"] if kind == "fwi" else 0)
    n = npts * shots
    return {"bytes": n * (steps_f * fwd_b + steps_r * rev_b) + 8.0 * npts,
            "flops": n * (steps_f * fwd_f + steps_r * rev_f)}


# ------------------------------------------------------- the same in 64 bits
class _Wave64:
    """The acoustic recursion of one shot in torch float64: u^{n+1} from
    a u^{n+1} = 2 u^n - b u^{n-1} + w (A u^n + q^n), zero outside the grid."""

    def __init__(self, case, shape, vel, src, rec):
        self.k, self.h, self.dt, self.nt = case["so"] // 2, case["h"], case["dt"], case["nt"]
        self.shape, self.ot4 = shape, case["time_order"] == 4
        k = self.k
        self.coef = []
        for j in range(1, k + 1):
            c = 2.0 * math.factorial(k) ** 2 / (j * j * math.factorial(k - j) * math.factorial(k + j))
            self.coef.append((c if j % 2 else -c) / self.h ** 2)
        self.c2 = vel.double().square()
        length = case["nbl"] * self.h
        emax = 3.0 * case["vmax"] / (2.0 * length) * math.log(1000.0)
        eta = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for a, n in enumerate(shape):
            i = torch.arange(n, dtype=torch.float64, device="cuda")
            delta = torch.maximum(case["nbl"] - i, i - (n - 1 - case["nbl"])).clamp(min=0.0) * self.h
            eta += (emax * (delta / length) ** 2).reshape([-1 if b == a else 1 for b in range(len(shape))])
        e = eta * (self.dt / 2.0)
        self.ia, self.b = 1.0 / (1.0 + e), 1.0 - e
        del eta, e
        self.pad = torch.zeros([n + 2 * k for n in shape], dtype=torch.float64, device="cuda")
        self.tmp = torch.empty(shape, dtype=torch.float64, device="cuda")
        self.si, self.sw = self._points(np.asarray(src, dtype=np.float64).reshape(1, 3), case["nbl"])
        self.ri, self.rw = self._points(np.asarray(rec, dtype=np.float64), case["nbl"])
        t = torch.arange(self.nt, dtype=torch.float64, device="cuda") * self.dt - 1.5 / case["f0"]
        a = (math.pi * case["f0"]) ** 2 * t * t
        self.series = (1.0 - 2.0 * a) * torch.exp(-a)

    def _points(self, pos, nbl):
        """Flat indices and multilinear weights [points][corners]."""
        if len(self.shape) == 2:
            pos = pos[:, [0, 2]]
        g = nbl + pos / self.h
        base = np.minimum(np.floor(g), np.array(self.shape) - 2).astype(np.int64)
        fr = g - base
        idx, wt = [], []
        for corner in np.ndindex(*([2] * len(self.shape))):
            c = np.array(corner)
            idx.append(np.ravel_multi_index(tuple((base + c).T), self.shape))
            wt.append(np.prod(np.where(c == 1, fr, 1.0 - fr), axis=1))
        return (torch.from_numpy(np.stack(idx, 1)).cuda(), torch.from_numpy(np.stack(wt, 1)).cuda())

    def lap(self, u):
        k, mid = self.k, tuple(slice(self.k, self.k + n) for n in self.shape)
        self.pad[mid] = u
        out = u * (-2.0 * len(self.shape) * sum(self.coef))
        for a in range(len(self.shape)):
            for j in range(1, k + 1):
                up, dn = list(mid), list(mid)
                up[a] = slice(k + j, k + j + self.shape[a])
                dn[a] = slice(k - j, k - j + self.shape[a])
                torch.add(self.pad[tuple(up)], self.pad[tuple(dn)], out=self.tmp)
                out.add_(self.tmp, alpha=self.coef[j - 1])
        return out

    def space(self, u):
        """(A u, lap u)"""
        l0 = self.lap(u)
        if not self.ot4:
            return l0, l0
        return self.lap(self.c2 * l0).mul_(self.dt * self.dt / 12.0).add_(l0), l0

    def step(self, u, up, rhs):
        """Overwrites rhs with u^{n+1}."""
        return rhs.mul_(self.c2).mul_(self.dt * self.dt).add_(u, alpha=2.0).sub_(self.b * up).mul_(self.ia)

    def inject(self, f, idx, wt, values):
        f.view(-1).index_add_(0, idx.reshape(-1), (wt * values.reshape(-1, 1)).reshape(-1))

    def forward(self, keep=None):
        zero = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        u, up = zero, zero
        d = torch.zeros(self.nt + 1, self.ri.shape[0], dtype=torch.float64, device="cuda")
        for n in range(self.nt):
            if keep is not None:
                keep.append(u)
            rhs, _ = self.space(u)
            self.inject(rhs, self.si, self.sw, self.series[n:n + 1])
            u, up = self.step(u, up, rhs), u
            d[n + 1] = (u.view(-1)[self.ri] * self.rw).sum(1)
        return d

    def gradient(self, dobs):
        states = []
        r = self.forward(states) - dobs.double()
        phi = 0.5 * float(r[1:].square().sum())
        zero = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        lam, lnext, g = zero, zero, torch.zeros_like(zero)
        extra = None
        for j in range(self.nt, 0, -1):
            rhs, llap = self.space(lam)
            if extra is not None:
                g.addcmul_(extra, llap, value=self.dt * self.dt / 12.0)
            self.inject(rhs, self.ri, self.rw, -r[j])
            lam, lnext = self.step(lam, lnext, rhs), lam
            u = states.pop()
            image, ulap = self.space(u)
            if self.ot4:
                extra = self.c2 * ulap
            self.inject(image, self.si, self.sw, self.series[j - 1:j])
            g.addcmul_(lam, image)
            del u, image, ulap, rhs
        if self.ot4:
            g.addcmul_(extra, self.lap(lam), value=self.dt * self.dt / 12.0)
        return phi, g.mul_(self.c2)


def exact(case, seed):
    """What run returns, in 64 bits.  Lossy checkpoints have no such value."""
    kind, shape = case["kind"], _shape(case)
    if kind in ("codec", "rate"):
        return None
    if kind in ("gradient", "fwi", "windows") and case["store"] != "fp32":
        return None
    vel = _medium(shape, case["vmin"], case["vmax"], seed)
    if kind == "windows":
        total, grad = 0.0, torch.zeros(shape, dtype=torch.float64, device="cuda")
        for i, (size, off) in enumerate(_windows(case)):
            at = tuple(slice(o, o + n) for o, n in zip(off, size))
            src, rec = _geometry(case, size)
            phi, g = _Wave64(case, size, vel[at], src, rec).gradient(_observed(case, src, rec, seed + 7919 * i))
            total += phi
            grad[at] += g
        return {"phi": total, "grad": grad}
    n = case.get("shots", 1)
    geo = [_geometry(case, shape, i, n) for i in range(n)]
    if kind == "fwi":
        m = (1.0 / vel.double().square()).float()
        c = 1.0 / m.double().sqrt()
        total, grad = 0.0, torch.zeros(shape, dtype=torch.float64, device="cuda")
        for i, (src, rec) in enumerate(geo):
            phi, g = _Wave64(case, shape, c, src, rec).gradient(_observed(case, src, rec, seed + 7919 * i))
            total += phi
            grad += g
        return {"phi": torch.tensor(total, dtype=torch.float64), "grad": grad}
    src, rec = geo[0]
    wave = _Wave64(case, shape, vel, src, rec)
    dobs = _observed(case, src, rec, seed)
    if kind == "forward":
        return {"d": wave.forward()}
    if kind == "misfit":
        d = wave.forward()
        return {"phi": 0.5 * float((d - dobs.double())[1:].square().sum()), "d": d}
    phi, g = wave.gradient(dobs)
    return {"phi": phi, "grad": g}
