"""The work this library is timed on: forwards, adjoints, differentiation, inversion, batches, equal-dimension
products and plan creation, each through the entry point that a program calls, over the mesh sizes it is used at.

A case is a dict of plain values:
  kind   "forward", "adjoint"      one call on a resident plan
         "vjp"                     a forward under autograd and its vector-Jacobian product
         "batch"                   BatchRunner.forward of `batch` models on one plan
         "cgls"                    `iters` iterations of the damped inversion loop
         "plan"                    plan creation, one forward, release
         "forward3d", "adjoint3d"  one call on a resident equal-dimension plan
  nx, ny, nz   cells per axis; dx, dy, dz, h  cell sizes and station height in metres
  comps        component mask; fp64  FP64 spectra and arithmetic
`exact` recomputes every result in 64 bits with torch's FFT and the closed forms written out here."""
import math

import numpy as np
import torch

from paper_2005_10160_gb300 import capi
from paper_2005_10160_gb300.batch import BatchRunner
from paper_2005_10160_gb300.inversion import cgls, forward_model
from paper_2005_10160_gb300.plan import Plan, Plan3D

GZ_GZZ = capi.GRAV_GZ | capi.GRAV_GZZ
VERTICAL = capi.GRAV_GZ | capi.GRAV_GXZ | capi.GRAV_GYZ | capi.GRAV_GZZ
NINE = "gz gxx gxy gxz gyy gyz gzz gx gy".split()


def _case(kind, size, cell, comps=capi.GRAV_ALL6, **more):
    nx, ny, nz = size
    dx, dy, dz, h = cell
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "dx": dx, "dy": dy, "dz": dz, "h": h, "comps": comps,
            "fp64": False, **more}


def listed():
    cube20 = (20.0, 20.0, 20.0, 10.0)
    survey = (50.0, 50.0, 25.0, 10.0)
    return [
        # the smallest of the served meshes: three short launches, latency counts
        _case("forward", (64, 64, 16), cube20, name="forward_64x64x16"),
        # a mid-size survey block with all six components, both directions (served mesh and boxes model)
        _case("forward", (256, 256, 32), (25.0, 25.0, 20.0, 5.0), name="forward_256x256x32"),
        _case("adjoint", (256, 256, 32), (25.0, 25.0, 20.0, 5.0), name="adjoint_256x256x32"),
        # sixteen requests on one resident plan in one call: a serving loop's batch
        _case("batch", (128, 128, 32), cube20, name="batch16_128x128x32", batch=16),
        # a ragged survey area inside a larger torch graph: forward, then the gradient with respect to the density
        _case("vjp", (301, 217, 45), (30.0, 25.0, 20.0, 15.0), VERTICAL, name="vjp_301x217x45"),
        # the inversion loop on gz + gzz data: one forward, one adjoint and the vector updates per iteration
        _case("cgls", (512, 512, 64), cube20, GZ_GZZ, name="cgls3_512x512x64", iters=3),
        # the headline mesh, both directions
        _case("forward", (1024, 1024, 100), survey, name="forward_1024x1024x100"),
        _case("adjoint", (1024, 1024, 100), survey, name="adjoint_1024x1024x100"),
        # reference-quality fields: the FP64 path that FP32 results are checked against
        _case("forward", (512, 512, 64), cube20, name="forward_fp64_512x512x64", fp64=True),
        # a station in every cell: the headline mesh forward, and a ragged mid-size block's adjoint
        _case("forward3d", (1024, 1024, 100), survey, name="forward3d_1024x1024x100"),
        _case("adjoint3d", (384, 320, 64), cube20, name="adjoint3d_384x320x64"),
        # a mesh or station height used once: generate the kernels and spectra, one forward, release
        _case("plan", (512, 512, 64), cube20, name="plan_512x512x64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any kind, sizes spread over the logarithm of 24 .. 1024 (x, y) and 4 .. 100
    (z), about half of them odd, components from one to seven, cell sizes of 10 .. 60 m."""
    kind = rng.choice(["forward", "forward", "adjoint", "adjoint", "batch", "vjp", "cgls", "plan", "forward3d", "adjoint3d"])
    fp64 = kind in ("forward", "adjoint", "vjp") and rng.random() < 0.2
    top = 512 if fp64 or kind in ("cgls", "plan", "adjoint3d", "forward3d") else 1024
    if kind == "batch":
        top = 256
    nx, ny = _log_int(rng, 24, top), _log_int(rng, 24, top)
    nz = _log_int(rng, 4, 64 if top < 1024 else 100)
    comps = rng.choice([capi.GRAV_ALL6, capi.GRAV_ALL6, capi.GRAV_GZ, GZ_GZZ, VERTICAL,
                        127 & ~capi.GRAV_GZ, 127, capi.GRAV_GZ | capi.GRAV_GX | capi.GRAV_GY])
    cell = (round(rng.uniform(10, 60), 1), round(rng.uniform(10, 60), 1), round(rng.uniform(10, 30), 1),
            round(rng.uniform(5, 40), 1))
    more = {}
    if kind == "batch":
        more["batch"] = rng.choice([2, 3, 4, 8, 16])
    if kind == "cgls":
        comps, more["iters"] = GZ_GZZ, rng.choice([1, 2, 3])
    return _case(kind, (nx, ny, nz), cell, comps, **{**more, "fp64": fp64})


def _slots(case):
    return capi.comp_list(case["comps"])


def _mesh(case):
    return tuple(case[k] for k in ("nx", "ny", "nz", "dx", "dy", "dz", "h"))


def _inputs(case, seed):
    """Densities: six boxes of +-300 kg/m^3 in noise of 20 (a body in a host rock).  Data-space vectors: white residuals
    over the standard deviations 0.1 mGal and 1 Eotvos, as a weighted misfit hands them to the adjoint.  Inversion data:
    a noisy smooth field of a few mGal and tens of Eotvos with the inverse standard deviations as weights."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    dtype = torch.float64 if case["fp64"] else torch.float32
    kind = case["kind"]
    first = np.array([NINE[c] in ("gz", "gx", "gy") for c in _slots(case)])
    sigma = torch.tensor(np.where(first, 1e-6, 1e-9), dtype=torch.float64, device="cuda")
    got = {}
    if kind in ("forward", "vjp", "batch", "plan", "forward3d"):
        shape = ((case["batch"],) if kind == "batch" else ()) + (nz, ny, nx)
        rho = torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, 20.0, generator=gen)
        for model in rho if kind == "batch" else (rho,):
            for _ in range(6):
                sl = []
                for n in (nz, ny, nx):
                    lo = int(rng.integers(0, n))
                    sl.append(slice(lo, lo + 1 + int(rng.integers(0, max(1, n // 4)))))
                model[tuple(sl)] += 300.0 if rng.random() < 0.5 else -300.0
        got["rho"] = rho
    if kind in ("adjoint", "vjp", "adjoint3d"):
        shape = (len(first),) + ((nz,) if kind == "adjoint3d" else ()) + (ny, nx)
        r = torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=gen)
        got["r"] = r.mul_((1e-6 / sigma).to(dtype).reshape((-1,) + (1,) * (len(shape) - 1)))
    if kind == "cgls":
        y = torch.linspace(-1, 1, ny, dtype=torch.float64, device="cuda")[:, None]
        x = torch.linspace(-1, 1, nx, dtype=torch.float64, device="cuda")[None, :]
        d = torch.zeros((len(first), ny, nx), dtype=torch.float64, device="cuda")
        for _ in range(4):
            cx, cy, s = rng.uniform(-0.7, 0.7), rng.uniform(-0.7, 0.7), rng.uniform(0.05, 0.3)
            a = rng.normal()
            d += a * torch.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2 * s * s))
        d = d * 30.0 + torch.empty_like(d).normal_(generator=gen)
        s = sigma[:, None, None]
        got["d"] = (d * s).to(dtype).contiguous()
        got["w"] = (1.0 / s).to(dtype)
        got["lam"] = 1.0
    return got


def prepare(case, seed):
    state = {"case": case, **_inputs(case, seed)}
    if case["kind"] != "plan":
        cls = Plan3D if case["kind"].endswith("3d") else Plan
        state["plan"] = cls(_mesh(case), case["comps"], fp64=case["fp64"])
    if case["kind"] == "batch":
        state["runner"] = BatchRunner(state["plan"], case["batch"])
    if case["kind"] == "vjp":
        state["rho"].requires_grad_(True)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("forward", "forward3d"):
        return state["plan"].forward(state["rho"])
    if kind in ("adjoint", "adjoint3d"):
        return state["plan"].adjoint(state["r"])
    if kind == "batch":
        return state["runner"].forward(state["rho"])
    if kind == "vjp":
        d = forward_model(state["rho"], state["plan"])
        return [d.detach(), torch.autograd.grad(d, state["rho"], state["r"])[0]]
    if kind == "cgls":
        res = cgls(state["plan"], state["d"], state["w"], state["lam"], iters=case["iters"])
        return {"m": res.m, "objectives": res.objectives}
    with Plan(_mesh(case), case["comps"], fp64=case["fp64"]) as plan:
        return plan.forward(state["rho"])


def work(case):
    """Bytes: the kernel spectra of the smallest even circulant, one real number per mirror pair of frequencies (what
    symmetry leaves of them), once per product, and each input and output once.  A plan reads no spectra: its kernels
    come from the mesh.  Operations: 5/2 P log2 P for each real transform of P = 2n points, 5 P log2 P for each complex
    one, and the products."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    kind, nc = case["kind"], len(_slots(case))
    elem = 8 if case["fp64"] else 4
    kx, px, py = nx + 1, 2 * nx, 2 * ny
    row = 2.5 * px * math.log2(px)
    col = 5.0 * py * math.log2(py)
    cells, stations = nz * ny * nx, ny * nx
    if kind.endswith("3d"):
        pz = 2 * nz
        layer = 5.0 * pz * math.log2(pz) if nz > 1 else 0.0
        flops = (1 + nc) * (nz * ny * row + kx * nz * col + kx * py * layer) + nc * kx * py * pz * 4.0
        return {"bytes": elem * (nc * kx * (ny + 1) * (nz + 1) + (1 + nc) * cells), "flops": flops}
    spectra = elem * nc * nz * kx * (ny + 1)
    once = (nz + nc) * (ny * row + kx * col) + nc * nz * kx * py * 4.0
    io = elem * (cells + nc * stations)
    if kind == "batch":
        return {"bytes": spectra + case["batch"] * io, "flops": case["batch"] * once}
    if kind == "vjp":
        return {"bytes": 2 * spectra + 2 * io, "flops": 2 * once}
    if kind == "cgls":
        products = 2 * case["iters"] + 1
        return {"bytes": products * spectra + io, "flops": products * once + case["iters"] * 20.0 * cells}
    if kind == "plan":
        # corner terms (about 60 operations each for a square root, arc tangents and hyperbolic sines), the
        # kernels' transforms, and the forward
        return {"bytes": io, "flops": once + nz * nc * (kx * (ny + 1) * 60.0 + ny * row + kx * col)}
    return {"bytes": spectra + io, "flops": once}


# ---- the same results in 64 bits, from the closed forms and torch's FFT ----

def _terms(c, x, y, z):
    """The corner term of component c, (x, y, z) the station minus the corner."""
    r = torch.sqrt(x * x + y * y + z * z)
    def log_x(): return torch.asinh(x / torch.sqrt(y * y + z * z))
    def log_y(): return torch.asinh(y / torch.sqrt(x * x + z * z))
    def log_z(): return torch.asinh(z / torch.sqrt(x * x + y * y))
    def at_x(): return torch.atan(y * z / (x * r))
    def at_y(): return torch.atan(x * z / (y * r))
    def at_z(): return torch.atan(x * y / (z * r))
    name = NINE[c]
    if name == "gz":
        return -(x * log_y() + y * log_x() - z * at_z())
    if name == "gx":
        return -(y * log_z() + z * log_y() - x * at_x())
    if name == "gy":
        return -(z * log_x() + x * log_z() - y * at_y())
    return {"gxx": at_x, "gyy": at_y, "gzz": at_z, "gxy": lambda: -log_z(), "gxz": lambda: -log_y(),
            "gyz": lambda: -log_x()}[name]()


def _embedded(case, c, tops, dev, px, py):
    """Kernel of component c for the layers whose top and bottom lie at the station-minus-corner depths tops[j] and
    tops[j] - dz, embedded in a py x px circulant: entry (-v mod py, -u mod px)."""
    nx, ny = case["nx"], case["ny"]
    f8 = dict(dtype=torch.float64, device=dev)
    x = (0.5 - torch.arange(nx + 1, **f8)) * case["dx"]
    y = (0.5 - torch.arange(ny + 1, **f8)) * case["dy"]
    out = torch.zeros((len(tops), py, px), **f8)
    su = -1.0 if NINE[c] in ("gx", "gxy", "gxz") else 1.0
    sv = -1.0 if NINE[c] in ("gy", "gxy", "gyz") else 1.0
    above, at = None, None
    for j, top in enumerate(tops):
        hi = above if at == top else _terms(c, x[None, :], y[:, None], torch.tensor(top, **f8))
        lo = _terms(c, x[None, :], y[:, None], torch.tensor(top - case["dz"], **f8))
        above, at = lo, top - case["dz"]
        d = lo - hi
        k = 6.672e-11 * ((d[:-1, :-1] - d[1:, :-1]) - (d[:-1, 1:] - d[1:, 1:]))
        if su < 0:
            k[:, 0] = 0.0
        if sv < 0:
            k[0, :] = 0.0
        out[j, :ny, :nx] = su * sv * k
        if nx > 1:
            out[j, :ny, px - nx + 1:] = sv * k[:, 1:].flip(1)
        if ny > 1:
            out[j, py - ny + 1:, :nx] = su * k[1:, :].flip(0)
        if nx > 1 and ny > 1:
            out[j, py - ny + 1:, px - nx + 1:] = k[1:, 1:].flip(0, 1)
    return out


def _pow2(n):
    p = 1
    while p < n:
        p *= 2
    return p


def _product(case, fields, transpose):
    """sum over layers of K rho (one plane per component), or its transpose, in 64 bits, for a batch of inputs."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    px, py = _pow2(2 * nx), _pow2(2 * ny)
    slots = _slots(case)
    dev = fields.device
    nb = fields.shape[0]
    kx = px // 2 + 1
    c16 = dict(dtype=torch.complex128, device=dev)
    if transpose:
        spec_r = torch.fft.rfft2(fields.double(), s=(py, px))
        out = torch.empty((nb, nz, ny, nx), dtype=torch.float64, device=dev)
    else:
        acc = torch.zeros((nb, len(slots), py, kx), **c16)
    for n in range(nz):
        top = [-case["h"] - n * case["dz"]]
        if transpose:
            acc = torch.zeros((nb, py, kx), **c16)
        else:
            spec = torch.fft.rfft2(fields[:, n].double(), s=(py, px))
        for i, c in enumerate(slots):
            e = torch.fft.rfft2(_embedded(case, c, top, dev, px, py)[0])
            if transpose:
                acc += e.conj() * spec_r[:, i]
            else:
                acc[:, i] += e * spec
        if transpose:
            out[:, n] = torch.fft.irfft2(acc, s=(py, px))[:, :ny, :nx]
    return out if transpose else torch.fft.irfft2(acc, s=(py, px))[..., :ny, :nx].contiguous()


def _product3d(case, field, transpose):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    px, py, pz = _pow2(2 * nx), _pow2(2 * ny), _pow2(2 * nz)
    slots = _slots(case)
    dev = field.device
    acc = None
    outs = []
    if not transpose:
        spec = torch.fft.rfftn(field.double(), s=(pz, py, px))
    for i, c in enumerate(slots):
        e = torch.zeros((pz, py, px), dtype=torch.float64, device=dev)
        for w0 in range(-(nz - 1), nz, 16):
            ws = list(range(w0, min(w0 + 16, nz)))
            part = _embedded(case, c, [(0.5 - w) * case["dz"] for w in ws], dev, px, py)
            for j, w in enumerate(ws):
                e[-w % pz] = part[j]
        e = torch.fft.rfftn(e)
        if transpose:
            term = e.conj_physical_().mul_(torch.fft.rfftn(field[i].double(), s=(pz, py, px)))
            acc = term if acc is None else acc.add_(term)
        else:
            outs.append(torch.fft.irfftn(e.mul_(spec), s=(pz, py, px))[:nz, :ny, :nx].clone())
        del e
    if transpose:
        return torch.fft.irfftn(acc, s=(pz, py, px))[:nz, :ny, :nx].contiguous()
    return torch.stack(outs)


def _cgls64(case, got):
    """Damped CGLS with depth weights in 64 bits (Hestenes and Stiefel's recurrence in x = W_m m)."""
    z = case["h"] + (torch.arange(case["nz"], dtype=torch.float64, device="cuda") + 0.5) * case["dz"]
    wm = (1.0 / z) / (1.0 / z).max()
    wm = wm[:, None, None]
    w, d, lam = got["w"].double(), got["d"].double(), got["lam"]
    def a(x): return w * _product(case, (x / wm)[None], False)[0]
    def at(r): return _product(case, (w * r)[None], True)[0] / wm
    r = w * d
    x = torch.zeros((case["nz"], case["ny"], case["nx"]), dtype=torch.float64, device="cuda")
    s = at(r)
    p, gamma = s.clone(), float((s * s).sum())
    js = [float((r * r).sum())]
    for _ in range(case["iters"]):
        q = a(p)
        alpha = gamma / float((q * q).sum() + lam * (p * p).sum())
        x += alpha * p
        r = r - alpha * q
        s = at(r) - lam * x
        new = float((s * s).sum())
        p = s + (new / gamma) * p
        gamma = new
        js.append(float((r * r).sum() + lam * (x * x).sum()))
    return {"m": x / wm, "objectives": js}


def exact(case, seed):
    got = _inputs(case, seed)
    kind = case["kind"]
    if kind in ("forward", "plan"):
        return _product(case, got["rho"][None], False)[0]
    if kind == "batch":
        return _product(case, got["rho"], False)
    if kind == "adjoint":
        return _product(case, got["r"][None], True)[0]
    if kind == "vjp":
        return [_product(case, got["rho"][None], False)[0], _product(case, got["r"][None], True)[0]]
    if kind == "cgls":
        return _cgls64(case, got)
    if kind == "forward3d":
        return _product3d(case, got["rho"], False)
    return _product3d(case, got["r"], True)
