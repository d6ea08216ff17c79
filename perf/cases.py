"""Workloads of the collapse-time library, through the calls a program makes.

A case is a dict of plain values; `prepare` makes the seeded linear field and
the plan a program keeps, `run` is one pass through the public entry points of
paper_1305_1505_gb300.pin, `work` what that pass cannot do without, and `exact`
the same outputs in 64 bits from plain torch.

Kinds
  collapse   a field on the device -> set_ic, collapse_times (and, on plans made
             with velocities, velocities): what every run of the method does,
             once per realisation; cubic and non-cubic grids, single
             realisations and batches, both input types, both correction modes
  noalloc    the same through pin_collapse_times_noalloc (callers that cannot
             allocate at call time; grids up to 64^3)
  host       the same from page-locked host input to page-locked host outputs
  request    a request of the server: radii, seeded field, collapse times,
             results in page-locked host memory
  fp64       the double-precision mode (checking runs)
  fragment   pin_fragment_order after a collapse call: particle order and
             collapsed-neighbour counts for the fragmentation
  fields     the real-space products of one field: the deformation tensor at
             one radius, first- and second-order displacements
"""
import math

import numpy as np
import torch

from paper_1305_1505_gb300 import pin

SIZES = (8, 16, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768)


def _case(name, kind, n, cell, radii, r_min, r_max, **more):
    nx, ny, nz = (n, n, n) if isinstance(n, int) else n
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "cell": cell, "radii": radii, "r_min": r_min, "r_max": r_max,
         "batch": 1, "velocities": False, "correction": 1, "dtype": "c64", "tiles": "", **more}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest useful call: a test-sized box through the entry point of
        # latency-critical callers, double-precision input
        _case("noalloc-32", "noalloc", 32, 2.0, 8, 2.0, 16.0, dtype="c128"),
        # the 64^3 x 20 parity workload (100 Mpc/h box): one small realisation
        _case("collapse-64", "collapse", 64, 100.0 / 64, 20, 1.5625, 15.0),
        # an ensemble of 64 realisations of 128^3 in one plan (256 Mpc/h, 25 radii)
        _case("ensemble-128", "collapse", 128, 2.0, 25, 2.0, 40.0, batch=64),
        # a medium single realisation (512 Mpc/h, 30 radii)
        _case("collapse-256", "collapse", 256, 2.0, 30, 2.0, 40.0),
        # a slab with unequal sides and radix-3 lengths, without the correction
        _case("slab-192x384x96", "collapse", (192, 384, 96), 3.0, 13, 3.0, 60.0, correction=0, dtype="c128"),
        # 4 Mpc/h cells with the velocities at R_max
        _case("velocities-384", "collapse", 384, 4.0, 40, 4.0, 120.0, velocities=True),
        # the headline run: 768^3 in a 3072 Mpc/h box, 40 radii, with the tile
        # widths and radix schedules that the tuner keeps for this shape
        _case("collapse-768", "collapse", 768, 4.0, 40, 4.0, 120.0, tiles="16 8 1 1"),
        # a medium realisation from host memory to host memory
        _case("host-192", "host", 192, 2.0, 24, 2.0, 40.0),
        # the largest request of the served mix
        _case("request-512", "request", 512, 2.0, 30, 2.0, 40.0),
        # the double-precision checking mode on the parity workload
        _case("fp64-64", "fp64", 64, 100.0 / 64, 20, 1.5625, 15.0),
        # the fragmentation front end of the headline grid
        _case("fragment-768", "fragment", 768, 4.0, 4, 4.0, 16.0),
        # tensor and displacements of a medium-large field
        _case("fields-384", "fields", 384, 4.0, 3, 4.0, 16.0),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["collapse"] * 8 + ["noalloc", "noalloc", "host", "request", "request", "fp64", "fragment",
                                          "fragment", "fields", "fields"])
    cell = round(rng.uniform(1.0, 5.0), 3)
    more = {"correction": 0 if rng.random() < 0.15 else 1, "dtype": "c128" if rng.random() < 0.25 else "c64"}
    radii = rng.randint(5, 40)
    cubic = kind in ("noalloc", "request") or rng.random() < 0.6
    sizes = {"noalloc": (16, 32, 48, 64), "request": (64, 128, 256, 512), "fp64": (16, 32, 48, 64),
             "fields": SIZES[2:-1], "fragment": SIZES[3:], "host": SIZES[3:-2], "collapse": SIZES[2:]}[kind]
    if cubic:
        n = (rng.choice(sizes),) * 3
    else:
        while True:
            n = tuple(rng.choice(sizes) for _ in range(3))
            if len(set(n)) > 1 and n[0] * n[1] * n[2] <= 512 ** 3:
                break
    n3 = n[0] * n[1] * n[2]
    if kind == "request":
        cell, more = 2.0, {}
        radii = rng.randint(20, 40)
    elif kind == "fp64":
        radii = max(3, min(radii, 20 * 64 ** 3 // n3))
    elif kind in ("fragment", "fields"):
        radii = rng.randint(2, 5)
    elif kind == "collapse":
        if rng.random() < 0.25 and n3 <= 384 ** 3:
            more["velocities"] = True
        elif max(n) <= 128 and rng.random() < 0.4:
            more["batch"] = max(2, int(_log_uniform(rng, 2, min(64, 64 * 128 ** 3 // n3))))
    # radii from about a cell up to at most a quarter of the shortest side
    r_min = cell * rng.uniform(0.8, 1.5)
    r_max = min(r_min * _log_uniform(rng, 5.0, 30.0), max(0.25 * cell * min(n), 2.0 * r_min))
    if kind == "request":
        r_min, r_max = 2.0, 40.0
    return _case(None, kind, n, cell, radii, round(r_min, 4), round(r_max, 4), **more)


def _radii(case):
    """Log-spaced radii, largest first."""
    s = np.arange(case["radii"], dtype=np.float64)
    r = case["r_min"] * (case["r_max"] / case["r_min"]) ** (s / max(1, case["radii"] - 1))
    return r[::-1].copy()


def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _wavenumbers(case, dtype):
    """k along each axis of the half-spectrum, broadcastable (Nyquist negative)."""
    nx, ny, nz = _shape(case)
    kf = 2.0 * math.pi / case["cell"]
    kx = torch.fft.fftfreq(nx, device="cuda", dtype=dtype) * kf
    ky = torch.fft.fftfreq(ny, device="cuda", dtype=dtype) * kf
    kz = torch.arange(nz // 2 + 1, device="cuda", dtype=dtype) * (kf / nz)
    return kx[:, None, None], ky[None, :, None], kz[None, None, :]


def _power(k, amplitude):
    """Linear power spectrum: index 0.96, BBKS transfer function with Gamma = 0.21."""
    xp = torch if isinstance(k, torch.Tensor) else np
    q = k / 0.21
    t = xp.log1p(2.34 * q) / (2.34 * q) * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25
    return amplitude * k ** 0.96 * t * t


def _amplitude():
    """Amplitude that gives sigma_8 = 0.8 under a top-hat of 8 Mpc/h."""
    lnk = np.linspace(math.log(1e-4), math.log(1e2), 20001)
    k = np.exp(lnk)
    x = 8.0 * k
    w = 3.0 * (np.sin(x) - x * np.cos(x)) / x ** 3
    f = k ** 3 * _power(k, 1.0) * w * w / (2.0 * math.pi ** 2)
    return 0.8 ** 2 / float(np.sum(0.5 * (f[1:] + f[:-1])) * (lnk[1] - lnk[0]))


def _field(case, seed):
    """Seeded Gaussian field delta(k) with the linear power spectrum: coloured
    white noise, a half-spectrum on the device (a stack of them for a batch)."""
    shape = _shape(case)
    dtype = torch.float64 if case["dtype"] == "c128" else torch.float32
    kx, ky, kz = _wavenumbers(case, dtype)
    k = torch.sqrt(kx * kx + ky * ky + kz * kz)
    k[0, 0, 0] = 1.0
    colour = torch.sqrt(_power(k, _amplitude() / case["cell"] ** 3))
    colour[0, 0, 0] = 0.0
    del k
    out = torch.empty((case["batch"],) + colour.shape, device="cuda",
                      dtype=torch.complex128 if dtype == torch.float64 else torch.complex64)
    for b in range(case["batch"]):
        g = torch.Generator(device="cuda").manual_seed(1000 * int(seed) + b)
        out[b] = torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda", dtype=dtype))
        out[b] *= colour
    return out[0] if case["batch"] == 1 else out


def _request_seed(seed):
    return 100003 * int(seed) + 17


def prepare(case, seed):
    shape, radii = _shape(case), _radii(case)
    box = case["cell"] * case["nx"]
    state = {"case": case, "radii": radii, "box": box}
    if case["kind"] == "request":
        state["plan"] = pin.Plan(shape, box, radii)
        state["seed"] = _request_seed(seed)
    else:
        state["delta"] = _field(case, seed)
    if case["kind"] == "noalloc":
        state["F"] = torch.empty(shape, dtype=torch.float32, device="cuda")
        state["idx"] = torch.empty(shape, dtype=torch.int32, device="cuda")
    elif case["kind"] == "fp64":
        state["plan"] = pin.Plan(shape, box, radii, correction=case["correction"], precision=pin.PIN_FP64)
    elif case["kind"] != "request":
        state["plan"] = pin.Plan(shape, box, radii, correction=case["correction"], batch=case["batch"],
                                 velocities=case["velocities"])
    if case["tiles"]:
        tx, ty, vx, vy = (int(v) for v in case["tiles"].split())
        state["plan"].set_radix(vx, vy)
        state["plan"].set_tiles(tx, ty)
    if case["kind"] in ("host", "request"):
        state["F"] = torch.empty(shape, dtype=torch.float32, pin_memory=True)
        state["idx"] = torch.empty(shape, dtype=torch.int32, pin_memory=True)
    if case["kind"] == "host":
        host = torch.empty(state["delta"].shape, dtype=state["delta"].dtype, pin_memory=True)
        host.copy_(state["delta"])
        state["delta"] = host
    if case["kind"] in ("fragment", "fields"):
        state["plan"].set_ic(state.pop("delta"))
    if case["kind"] == "fragment":
        state["plan"].collapse_times()
    return state


def run(state):
    case, plan = state["case"], state.get("plan")
    kind = case["kind"]
    if kind == "collapse":
        plan.set_ic(state["delta"])
        F, idx = plan.collapse_times()
        if case["velocities"]:
            return {"F": F, "idx": idx, "psi": plan.velocities()}
        return {"F": F, "idx": idx}
    if kind == "noalloc":
        d = state["delta"]
        pin.pin_collapse_times_noalloc(d.data_ptr(), pin.PIN_C128 if case["dtype"] == "c128" else pin.PIN_C64,
                                       case["nx"], state["box"], state["radii"], case["correction"],
                                       state["F"].data_ptr(), state["idx"].data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        return {"F": state["F"], "idx": state["idx"]}
    if kind == "host":
        plan.set_ic(state["delta"])
        F, idx = plan.collapse_times(state["F"], state["idx"])
        return {"F": F, "idx": idx}
    if kind == "request":
        plan.set_radii(state["radii"])
        plan.set_ic_seed(state["seed"])
        F, idx = plan.collapse_times(state["F"], state["idx"])
        return {"F": F, "idx": idx}
    if kind == "fp64":
        plan.set_ic(state["delta"])
        F, idx = plan.collapse_times_f64()
        return {"F": F, "idx": idx}
    if kind == "fragment":
        order, before = plan.fragment_order()
        return {"order": order, "before": before}
    return {"hessian": plan.hessian(1), "psi": plan.displacements(), "psi2": plan.displacements_2lpt()}


def work(case):
    nx, ny, nz = _shape(case)
    n3 = nx * ny * nz
    half = nx * ny * (nz // 2 + 1)
    spectrum = half * (16 if case["dtype"] == "c128" else 8)
    if case["kind"] == "fragment":
        return {"bytes": n3 * (4 + 4 + 1), "flops": 0}
    # one component: an inverse real transform; the filter of a separable
    # window leaves 3 transforms along x, 6 along y and 6 real ones along z
    line = [2.5 * math.log2(n) for n in (nx, ny, nz)]
    tensor = n3 * (3 * line[0] + 6 * line[1] + 6 * line[2] + 20)
    if case["kind"] == "fields":
        grad = n3 * (2 * line[0] + 3 * line[1] + 3 * line[2] + 10)
        return {"bytes": 3 * half * 8 + n3 * 4 * (6 + 3 + 3),
                "flops": 2 * tensor + 2 * grad + n3 * (sum(line) + 15)}
    b = case["batch"]
    out = 12 if case["kind"] == "fp64" else 8
    extra = 0.0
    if case["velocities"]:
        out += 12
        extra = n3 * (3 * line[2] + 10)
    read = 0 if case["kind"] == "request" else spectrum
    # eigenvalues (about 60) and the roots of the axis cubics (about 150)
    return {"bytes": b * (read + out * n3), "flops": b * case["radii"] * (tensor + extra + 210 * n3)}


# ------------------------------------------------------------------ 64 bits --

def _window(case, delta, radius):
    """delta(k) W(kR), the wavenumbers and 1/k^2 (0 at k = 0), in 64 bits."""
    kx, ky, kz = _wavenumbers(case, torch.float64)
    k2 = kx * kx + ky * ky + kz * kz
    d = delta.to(torch.complex128) * torch.exp(-0.5 * radius * radius * k2)
    k2[0, 0, 0] = 1.0
    d = d / k2
    d[0, 0, 0] = 0.0
    return d, (kx, ky, kz)


def _odd(case, k):
    """Wavenumbers with the Nyquist index zeroed (odd powers of k)."""
    out = []
    for n, v, axis in zip(_shape(case), k, range(3)):
        v = v.clone()
        v.select(axis, n // 2).zero_()
        out.append(v)
    return out


def _tensor(case, delta, radius):
    """Six components xx, yy, zz, xy, xz, yz of the smoothed deformation tensor."""
    phi, k = _window(case, delta, radius)
    o = _odd(case, k)
    pairs = [(k[0], k[0]), (k[1], k[1]), (k[2], k[2]), (o[0], o[1]), (o[0], o[2]), (o[1], o[2])]
    return [torch.fft.irfftn(phi * (a * b), s=_shape(case)) for a, b in pairs]


def _gradient(case, phi, k):
    return torch.stack([torch.fft.irfftn(1j * (phi * a), s=_shape(case)) for a in _odd(case, k)])


def _eigenvalues(h):
    xx, yy, zz, xy, xz, yz = h
    q = (xx + yy + zz) / 3
    a, b, c = xx - q, yy - q, zz - q
    p = torch.sqrt((a * a + b * b + c * c + 2 * (xy * xy + xz * xz + yz * yz)) / 6)
    det = a * (b * c - yz * yz) - xy * (xy * c - yz * xz) + xz * (xy * yz - b * xz)
    r = torch.where(p > 0, det / (2 * p ** 3).clamp_min(1e-300), torch.ones_like(p)).clamp_(-1, 1)
    phi = torch.acos(r) / 3
    l0 = q + 2 * p * torch.cos(phi)
    l2 = q + 2 * p * torch.cos(phi + 2 * math.pi / 3)
    return l0, 3 * q - l0 - l2, l2


def _largest_root(c1, c2, c3):
    """Largest real root of F^3 - c1 F^2 - c2 F - c3, at least 0."""
    s = c1 / 3
    p = -c2 - c1 * s
    hq = 0.5 * (-c3 - c2 * s - 2 * s ** 3)
    disc = hq * hq + (p / 3) ** 3
    m = torch.sqrt((-p / 3).clamp_min(0))
    three = 2 * m * torch.cos(torch.acos((-hq / (m ** 3).clamp_min(1e-300)).clamp_(-1, 1)) / 3)
    w = torch.where(hq >= 0, -1.0, 1.0) * (hq.abs() + torch.sqrt(disc.clamp_min(0)))
    u = torch.sign(w) * w.abs() ** (1.0 / 3.0)
    one = torch.where(u != 0, u - p / (3 * torch.where(u != 0, u, 1.0)), 0.0)
    x = torch.where(disc <= 0, three, one) + s
    for _ in range(2):
        g = ((x - c1) * x - c2) * x - c3
        dg = (3 * x - 2 * c1) * x - c2
        x = torch.where(dg != 0, x - g / torch.where(dg != 0, dg, 1.0), x)
    return x.clamp_min(0)


def _spherical_root():
    x = 2.0
    for _ in range(60):
        x -= (x / 3 + x * x / 21 + 23 * x ** 3 / 1701 - 1) / (1 / 3 + 2 * x / 21 + 69 * x * x / 1701)
    return x


def _collapse(case, lam):
    l = list(lam)
    mu1, mu3 = l[0] + l[1] + l[2], l[0] * l[1] * l[2]
    e = [0.5 * l[i] * (l[(i + 1) % 3] + l[(i + 2) % 3]) for i in range(3)]
    F = torch.zeros_like(mu1)
    for i in range(3):
        j, k = (i + 1) % 3, (i + 2) % 3
        F = torch.maximum(F, _largest_root(l[i], 3 / 7 * e[i],
                                           10 / 84 * (l[i] * (e[j] + e[k]) + e[i] * (l[j] + l[k])) - mu3 / 9))
    if case["correction"]:
        dcorr = 1 / (3 / 20 * (12 * math.pi) ** (2 / 3)) - 1 / _spherical_root()
        z = 10 * (l[0] - l[2]) / torch.where(mu1 > 0, mu1, 1.0)
        F = F + torch.where(mu1 > 0, mu1 * dcorr * torch.exp(-z * z), 0.0)
    return F


def _exact_fields(case, delta):
    h = _tensor(case, delta, _radii(case)[1])
    phi, k = _window(case, delta, 0.0)
    psi = _gradient(case, phi, k)
    t = _tensor(case, delta, 0.0)
    s = t[0] * t[1] + t[0] * t[2] + t[1] * t[2] - t[3] ** 2 - t[4] ** 2 - t[5] ** 2
    del t
    phi2, k = _window(case, torch.fft.rfftn(s), 0.0)
    return {"hessian": torch.stack(h), "psi": psi, "psi2": _gradient(case, phi2 * (3 / 7), k)}


def exact(case, seed):
    n3 = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] in ("request", "fragment") or n3 * case["radii"] * case["batch"] > 2.4e9:
        return None  # seeded by the library itself; whole numbers only; or over about 20 seconds
    delta = _field(case, seed)
    if case["kind"] == "fields":
        return _exact_fields(case, delta)
    deltas = [delta] if case["batch"] == 1 else delta
    if case["kind"] != "fp64" and case["dtype"] == "c128":
        deltas = [d.to(torch.complex64) for d in deltas]  # the type the path works in
    best, moved = [], []
    for d in deltas:
        F, psi = torch.zeros(_shape(case), dtype=torch.float64, device="cuda"), None
        for r in _radii(case):
            f = _collapse(case, _eigenvalues(_tensor(case, d, float(r))))
            up = f > F
            if case["velocities"]:
                v = _gradient(case, *_window(case, d, float(r)))
                psi = torch.where(up, v, torch.zeros_like(v) if psi is None else psi)
            F = torch.where(up, f, F)
        best.append(F)
        moved.append(psi)
    out = {"F": best[0] if case["batch"] == 1 else torch.stack(best), "idx": None}
    if case["velocities"]:
        out["psi"] = moved[0] if case["batch"] == 1 else torch.stack(moved, 1)
    return out
