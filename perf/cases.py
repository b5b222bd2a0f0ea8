"""Performance cases: what programs that use this framework have it do, through its public entry points.

A case is a dict of plain values.  Five kinds of program:

* solve   one cavity: load a state, take leapfrog steps, check the energy, read the state back.  Storage
          FP32 / FP16 / BF16, spatial order 2 / 4, medium vacuum (scalar coefficients), dielectric spheres
          (a few materials) or graded (per-position coefficients, a different value in nearly every cell).
          Fields on the device (torch) or on the host (numpy).  With currents and probes (an antenna run) the
          state starts at zero and the probe traces are read back too.
* batch   many independent cavities stepped together (a parameter sweep; with own step counts per member, as
          in a served stream): load each, join, step, leave, read each back.
* checks  the energy and the divergences of a loaded state (the invariants watched during a long run).
* slabs   one cavity cut into z-slabs that exchange ghost cells, stepped and read back slab by slab; a pass
          goes on from the state the previous one reached.

Every solve and batch pass loads its state anew, so passes on one state repeat the same work.  No tuning is
set: programs take the library's own choice of kernel and launch shape.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2504_09118_gb300 import Cavity
from paper_2504_09118_gb300 import binding as B
from paper_2504_09118_gb300.slab import SlabDomain

DT = 0.5 / math.sqrt(3.0)   # half the Courant bound (dx = 1), the step of the paper's cavity benchmark
VAC = float(np.float32(DT))
STORAGE = {"f32": B.FDTD_F32, "f16": B.FDTD_F16, "bf16": B.FDTD_BF16}
UNIT = {"f32": 2.0 ** -24, "f16": 2.0 ** -11, "bf16": 2.0 ** -8}
C1, C2 = 9.0 / 8.0, -1.0 / 24.0


# ------------------------------------------------------------------------------------------- the cases
def _solve(name, nx, ny, nz, steps, storage="f32", order=2, medium="spheres", host=False, sources=0, probes=0):
    return {"name": name, "kind": "solve", "nx": nx, "ny": ny, "nz": nz, "steps": steps, "storage": storage,
            "order": order, "medium": medium, "host": host, "sources": sources, "probes": probes}


def _batch(name, count, steps, storage, own_steps, lo=16, hi=96):
    return {"name": name, "kind": "batch", "count": count, "lo": lo, "hi": hi, "steps": steps, "storage": storage,
            "own_steps": own_steps, "sizes_seed": 5}


def listed():
    return [
        # the quick start on a toy cavity, numpy in and out: latency, launches and host work decide
        _solve("quickstart_24x20x17_f32_host", 24, 20, 17, 10, host=True),
        # a small ragged cavity with a few dielectric bodies: one launch does little work
        _solve("ragged_131x67x45_f32", 131, 67, 45, 100),
        # a mid-size empty cavity in half-size storage
        _solve("vacuum_200x131x120_bf16", 200, 131, 120, 64, storage="bf16", medium="vacuum"),
        # the headline benchmark: 512^3 cells, 32 spheres, 200 steps
        _solve("spheres_512_f32", 512, 512, 512, 200),
        # the precision study's cavity in FP16
        _solve("spheres_384_f16", 384, 384, 384, 100, storage="f16"),
        # the fourth-order scheme
        _solve("order4_256_f32", 256, 256, 256, 64, order=4),
        # an antenna run: point currents drive an empty state, probes record every step
        _solve("antenna_128x96x80_f32", 128, 96, 80, 200, sources=4, probes=16),
        # a graded-index medium: more distinct coefficients than a one-byte material id can name
        _solve("graded_160x150x140_f32", 160, 150, 140, 50, medium="graded"),
        # a parameter sweep over small cavities
        _batch("sweep_48_f32", 48, 100, "f32", False),
        # cavities with their own step counts, as in a served stream
        _batch("served_24_bf16", 24, 128, "bf16", True),
        # the invariants of a large state
        {"name": "checks_320_f32", "kind": "checks", "nx": 320, "ny": 320, "nz": 320, "storage": "f32",
         "medium": "spheres"},
        # domain decomposition on one GPU: four slabs, two ghost planes, an exchange before every two steps
        {"name": "slabs_4x256_f32", "kind": "slabs", "nx": 256, "ny": 256, "nz": 256, "steps": 32, "slabs": 4,
         "ghost": 2, "storage": "f32", "medium": "spheres"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges: sides 16..320 per axis (log-uniform, any parity), at most
    2.4e7 cells, 4..200 steps."""
    kind = rng.choice(["solve"] * 8 + ["batch"] * 2 + ["checks", "slabs"])
    if kind == "batch":
        lo = rng.randint(16, 32)
        return {"kind": "batch", "count": rng.randint(8, 48), "lo": lo, "hi": rng.randint(lo + 8, 96),
                "steps": _log_int(rng, 8, 128), "storage": rng.choice(["f32", "f32", "bf16", "f16"]),
                "own_steps": rng.random() < 0.5, "sizes_seed": rng.randint(0, 10 ** 6)}
    while True:
        n = [_log_int(rng, 16, 320) for _ in range(3)]
        if n[0] * n[1] * n[2] <= 24_000_000 and (kind != "slabs" or n[2] >= 32):
            break
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "storage": rng.choice(["f32", "f32", "f32", "f16", "bf16"]),
         "medium": rng.choice(["vacuum", "spheres", "spheres"])}
    if kind == "solve":
        c.update(steps=_log_int(rng, 4, 200), order=rng.choice([2, 2, 2, 4]), host=False, sources=0, probes=0)
        use = rng.choice(["plain", "plain", "plain", "antenna", "graded", "host"])
        if use == "antenna":
            c.update(storage="f32", sources=rng.randint(1, 8), probes=rng.randint(1, 32))
        elif use == "graded" and n[0] * n[1] * n[2] <= 8_000_000:
            c.update(medium="graded", storage="f32")
        elif use == "host":
            c.update(host=True)
        if c["storage"] == "bf16":
            c["steps"] = min(c["steps"], 100)   # about 1.6e-2 of the state, the most this storage is used for here
    elif kind == "slabs":
        c.update(steps=_log_int(rng, 4, 64), slabs=rng.randint(2, 4), ghost=rng.choice([2, 4]), storage="f32")
    return c


# ------------------------------------------------------------------------------------------- inputs
def _axes_ext(comp, nx, ny, nz):
    """Extent (z, y, x) of a component inside its canonical (nz+1, ny+1, nx+1) array."""
    x = nx if comp in (0, 4, 5) else nx + 1
    y = ny if comp in (1, 3, 5) else ny + 1
    z = nz if comp in (2, 3, 4) else nz + 1
    return z, y, x


def _fields(seed, nx, ny, nz):
    """Six canonical FP32 device tensors: uniform [-1, 1) inside each extent, tangential E zero on the walls."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    out = []
    for c in range(6):
        f = torch.rand((nz + 1, ny + 1, nx + 1), generator=g, device="cuda", dtype=torch.float32).mul_(2).sub_(1)
        z, y, x = _axes_ext(c, nx, ny, nz)
        f[z:].zero_()
        f[:, y:].zero_()
        f[:, :, x:].zero_()
        if c in (0, 2):
            f[:, 0].zero_()
            f[:, ny].zero_()
        if c in (0, 1):
            f[0].zero_()
            f[nz].zero_()
        if c in (1, 2):
            f[:, :, 0].zero_()
            f[:, :, nx].zero_()
        out.append(f)
    return out


def _ce(seed, nx, ny, nz, medium):
    """ce = dt / (eps_r dx) at the Ex, Ey, Ez positions as three FP32 device tensors, or None for vacuum."""
    if medium == "vacuum":
        return None
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 17])
    half = ((0.5, 0, 0), (0, 0.5, 0), (0, 0, 0.5))
    n = (nx, ny, nz)
    if medium == "graded":   # a smooth index profile, eps_r between 1 and 4
        a = [rng.uniform(0.5, 2.5) for _ in range(3)]
        out = []
        for o in half:
            p = [torch.cos(math.pi * a[q] * (torch.arange(n[q] + 1, device="cuda", dtype=torch.float64) + o[q]) / n[q])
                 for q in range(3)]
            eps = 2.5 + 0.5 * (p[2][:, None, None] + p[1][None, :, None] + p[0][None, None, :])
            out.append((DT / eps).to(torch.float32))
        return out
    m = min(n)
    spheres = [([rng.uniform(0, q) for q in n], rng.uniform(m / 16, m / 6), float(rng.choice([2.25, 4.0])))
               for _ in range(32 if m >= 128 else 6)]
    out = []
    for o in half:
        eps = torch.ones((nz + 1, ny + 1, nx + 1), device="cuda", dtype=torch.float32)
        for (c, r, e) in spheres:   # a later sphere wins
            lo = [max(0, math.floor(c[q] - o[q] - r)) for q in range(3)]
            hi = [min(n[q], math.ceil(c[q] - o[q] + r)) + 1 for q in range(3)]
            d = [(torch.arange(lo[q], hi[q], device="cuda", dtype=torch.float64) + (o[q] - c[q])).square()
                 for q in range(3)]
            inside = d[2][:, None, None] + d[1][None, :, None] + d[0][None, None, :] <= r * r
            eps[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]][inside] = e
        out.append((DT / eps.double()).to(torch.float32))
    return out


def _host(ce):
    return None if ce is None else [c.cpu().numpy() for c in ce]


def _antenna(seed, nx, ny, nz, nsrc, nprobe, steps):
    """Sources [(comp, i, j, k)], their wave (nsrc, steps) and probes [(comp, i, j, k)]."""
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 23])
    src = [(int(rng.integers(0, 3)), int(rng.integers(1, nx)), int(rng.integers(1, ny)), int(rng.integers(1, nz)))
           for _ in range(nsrc)]
    t = np.arange(steps)
    wave = np.stack([-(t - 12.0 - s) / 4.0 * np.exp(-((t - 12.0 - s) / 4.0) ** 2 / 2) for s in range(nsrc)])
    probes = [(int(rng.integers(0, 6)), int(rng.integers(0, nx)), int(rng.integers(0, ny)), int(rng.integers(0, nz)))
              for _ in range(nprobe)]
    return src, wave.astype(np.float32), probes


def _members(case, seed):
    """[(nx, ny, nz, steps, medium)] of a batch."""
    rng = np.random.default_rng(case["sizes_seed"])
    out = []
    for _ in range(case["count"]):
        n = [int(v) for v in rng.integers(case["lo"], case["hi"] + 1, size=3)]
        steps = int(rng.integers(max(1, case["steps"] // 2), case["steps"] + 1)) if case["own_steps"] else case["steps"]
        out.append((*n, steps, "spheres" if rng.random() < 0.5 else "vacuum"))
    return out


def _initial(case, seed, nx, ny, nz):
    if case.get("sources"):
        return [torch.zeros((nz + 1, ny + 1, nx + 1), device="cuda") for _ in range(6)]
    return _fields(seed, nx, ny, nz)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        st = STORAGE[case["storage"]]
        cavs = []
        for m, (nx, ny, nz, steps, medium) in enumerate(_members(case, seed)):
            cav = Cavity(nx, ny, nz, DT, 1.0, _host(_ce(seed + 1000 * m, nx, ny, nz, medium)), None, st)
            out = torch.zeros((6, nz + 1, ny + 1, nx + 1), device="cuda")
            cavs.append((cav, _fields(seed + 1000 * m, nx, ny, nz), out, steps))
        return {"kind": kind, "batch": B.fdtd_batch_create(st, None), "cavs": cavs, "steps": case["steps"],
                "own": case["own_steps"]}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    st = STORAGE[case["storage"]]
    ce = _host(_ce(seed, nx, ny, nz, case["medium"]))
    if kind == "slabs":
        dom = SlabDomain(nx, ny, nz, DT, 1.0, ce, None, st, nslabs=case["slabs"], ghost=case["ghost"])
        dom.set_fields([f.cpu().numpy() for f in _fields(seed, nx, ny, nz)])
        outs = []
        for (k0, k1), (lo, hi, g_lo, _) in zip(dom.ranges, dom.locals):
            outs.append((torch.zeros((6, hi - lo + 1, ny + 1, nx + 1), device="cuda"), g_lo,
                         g_lo + k1 - k0 + (1 if k1 == nz else 0), (nx, ny, hi - lo)))
        return {"kind": kind, "dom": dom, "outs": outs, "steps": case["steps"]}
    cav = Cavity(nx, ny, nz, DT, 1.0, ce, None, st, order=case.get("order", 2))
    f = _initial(case, seed, nx, ny, nz)
    if kind == "checks":
        cav.set_fields(f, on_device=True)
        return {"kind": kind, "cav": cav}
    host = case["host"]
    if host:
        f = [t.cpu().numpy() for t in f]
    s = {"kind": kind, "cav": cav, "fields": f, "host": host, "steps": case["steps"], "probes": case["probes"],
         "out": None if host else [torch.zeros((nz + 1, ny + 1, nx + 1), device="cuda") for _ in range(6)]}
    if case["sources"]:
        src, wave, probes = _antenna(seed, nx, ny, nz, case["sources"], case["probes"], case["steps"])
        cav.set_sources(src, wave)
        cav.set_probes(probes, case["steps"])
    return s


def run(s):
    if s["kind"] == "solve":
        cav = s["cav"]
        cav.set_fields(s["fields"], on_device=not s["host"])
        cav.step(s["steps"])
        out = {"energy": cav.energy(), "fields": cav.get_fields(s["out"], on_device=not s["host"])}
        if s["probes"]:
            out["probes"] = cav.get_probes()
        return out
    if s["kind"] == "batch":
        b = s["batch"]
        for cav, fields, _, steps in s["cavs"]:
            cav.set_fields(fields, on_device=True)
            B.fdtd_batch_add(b, cav.handle)
            if s["own"]:
                B.fdtd_batch_set_steps(b, cav.handle, steps)
        B.fdtd_batch_step(b, s["steps"])
        for cav, _, out, _ in s["cavs"]:
            B.fdtd_batch_remove(b, cav.handle)
            cav.get_fields([out[c] for c in range(6)], on_device=True)
        return [out for _, _, out, _ in s["cavs"]]
    if s["kind"] == "checks":
        de, dh = s["cav"].divergence()
        return np.array([s["cav"].energy(), de, dh])
    s["dom"].step(s["steps"])
    for h, (out, _, _, dims) in zip(s["dom"].handles, s["outs"]):
        B.fdtd_get_fields(h, [out[c] for c in range(6)], 1, dims=dims)
    return [out[:, a:b] for out, a, b, _ in s["outs"]]


# ------------------------------------------------------------------------------------------- work
def work(case):
    """What a pass cannot do without: each FP32 input field read once, each output field written once, the medium
    read once (one id byte, or three FP32 coefficients, per cell), and every step's arithmetic (per component three
    differences and a multiply-add; the fourth-order differences take four taps)."""
    coef = {"vacuum": 0, "spheres": 1, "graded": 12}
    if case["kind"] == "batch":
        b = f = 0
        for nx, ny, nz, steps, medium in _members(case, 0):
            cells = nx * ny * nz
            b, f = b + cells * (48 + coef[medium]), f + cells * steps * 30
        return {"bytes": b, "flops": f}
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "checks":   # energy and divergence are two calls: each reads the stored state
        es = 4 if case["storage"] == "f32" else 2
        return {"bytes": 2 * cells * (6 * es + coef[case["medium"]]), "flops": cells * (33 + 27)}
    return {"bytes": cells * (48 + coef[case["medium"]]),
            "flops": cells * case["steps"] * (30 if case.get("order", 2) == 2 else 90)}


# ------------------------------------------------------------------------------------------- results
def tolerance(case):
    """Relative error of another correct implementation at the same precision, about four times the error against
    exact() measured here."""
    if case["kind"] == "checks":   # compensated sums, rounded once (measured below 1e-12)
        return {"rel": 1e-10}
    # Rounding adds as a random walk over the steps, since the scheme conserves the energy norm.  FP32: 1.1e-7 after
    # 10 steps, 3.6e-7 after 100, 4.9e-7 after 200.  A 16-bit state is rounded once a step or less often: FP16 1.6e-3
    # after 100 steps, BF16 1.0e-2 after 64.
    n = max(1, case["steps"])
    if case["storage"] == "f32":
        return {"rel": 1.5e-7 * math.sqrt(n + 8)}
    rel = min(0.03, 2.0 * UNIT[case["storage"]] / math.sqrt(3.0) * math.sqrt(n + 1))
    return {"rel": rel, "max": min(1.0, 10 * rel)}


def _curl_e(f, nx, ny, nz, order):
    """-(curl E) at the Hx, Hy, Hz positions (FP64, extents only)."""
    n = (nz, ny, nx)

    def d(a, ax):   # difference of E along axis ax (0 z, 1 y, 2 x): n + 1 nodes -> n
        m = n[ax]
        first = a.narrow(ax, 1, m) - a.narrow(ax, 0, m)
        if order == 2:
            return first
        ext = torch.cat([-a.narrow(ax, 1, 1), a, -a.narrow(ax, m - 1, 1)], ax)   # tangential E is odd about a wall
        return C1 * first + C2 * (ext.narrow(ax, 3, m) - ext.narrow(ax, 0, m))

    ex, ey, ez = f[0], f[1], f[2]
    return (d(ey, 0) - d(ez, 1), d(ez, 2) - d(ex, 0), d(ex, 1) - d(ey, 2))


def _curl_h(f, nx, ny, nz, order):
    """curl H at the interior Ex, Ey, Ez positions (FP64, extents without the walls)."""
    n = (nz, ny, nx)

    def d(a, ax):   # difference of H along axis ax: n midpoints -> n - 1 interior nodes
        m = n[ax]
        first = a.narrow(ax, 1, m - 1) - a.narrow(ax, 0, m - 1)
        if order == 2:
            return first
        ext = torch.cat([a.narrow(ax, 0, 1), a, a.narrow(ax, m - 1, 1)], ax)     # tangential H is even about a wall
        return C1 * first + C2 * (ext.narrow(ax, 3, m - 1) - ext.narrow(ax, 0, m - 1))

    hx, hy, hz = f[3], f[4], f[5]
    i = slice(1, -1)
    return (d(hz, 1)[i] - d(hy, 0)[:, i], d(hx, 0)[:, :, i] - d(hz, 2)[i], d(hy, 2)[:, i] - d(hx, 1)[:, :, i])


def _exact_solve(fields, ce, nx, ny, nz, steps, order=2, src=(), wave=None, probes=()):
    """(fields, energy, probe traces) of a leapfrog run in FP64, plain torch."""
    f = [t[tuple(slice(0, e) for e in _axes_ext(c, nx, ny, nz))].double() for c, t in enumerate(fields)]
    ch = VAC
    c64 = [VAC] * 3 if ce is None else [c[tuple(slice(0, e) for e in _axes_ext(q, nx, ny, nz))].double()
                                        for q, c in enumerate(ce)]
    i, full = slice(1, -1), slice(None)
    inner = ((i, i, full), (i, full, i), (full, i, i))
    cin = [c if ce is None else c[inner[q]] for q, c in enumerate(c64)]
    trace = torch.zeros((len(probes), steps), dtype=torch.float64, device="cuda")
    for n in range(steps):
        for q, cu in enumerate(_curl_e(f, nx, ny, nz, order)):
            f[3 + q].add_(cu, alpha=ch)
        for q, cu in enumerate(_curl_h(f, nx, ny, nz, order)):
            f[q][inner[q]] += cin[q] * cu
        for s, (c, si, sj, sk) in enumerate(src):
            cc = c64[c] if ce is None else c64[c][sk, sj, si]
            f[c][sk, sj, si] -= cc * float(wave[s, n])
        for p, (c, pi, pj, pk) in enumerate(probes):
            trace[p, n] = f[c][pk, pj, pi]
    w = 0.0
    for q, cu in enumerate(_curl_e(f, nx, ny, nz, order)):
        w += float((f[q].square() / c64[q]).sum())
        w += float((f[3 + q].square() / ch).sum() + (f[3 + q] * cu).sum())
    out = []
    for c in range(6):
        full_a = torch.zeros((nz + 1, ny + 1, nx + 1), dtype=torch.float64, device="cuda")
        full_a[tuple(slice(0, e) for e in _axes_ext(c, nx, ny, nz))] = f[c]
        out.append(full_a)
    return out, 0.5 * DT * w, trace


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for m, (nx, ny, nz, steps, medium) in enumerate(_members(case, seed)):
            s = seed + 1000 * m
            out.append(torch.stack(_exact_solve(_fields(s, nx, ny, nz), _ce(s, nx, ny, nz, medium), nx, ny, nz, steps)[0]))
        return out
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ce = _ce(seed, nx, ny, nz, case["medium"])
    f = _initial(case, seed, nx, ny, nz)
    if kind == "slabs":
        out = torch.stack(_exact_solve(f, ce, nx, ny, nz, case["steps"])[0])
        q, r = divmod(nz, case["slabs"])
        cuts = [0]
        for s in range(case["slabs"]):
            cuts.append(cuts[-1] + q + (1 if s < r else 0))
        return [out[:, a:b + (1 if b == nz else 0)] for a, b in zip(cuts[:-1], cuts[1:])]
    if kind == "checks":
        w = _exact_solve(f, ce, nx, ny, nz, 0)[1]
        dd = [a.double() / (VAC if ce is None else ce[q].double()) for q, a in enumerate(f[:3])]
        i = slice(1, -1)
        de = ((dd[0][i, i, 1:nx] - dd[0][i, i, 0:nx - 1]) + (dd[1][i, 1:ny, i] - dd[1][i, 0:ny - 1, i])
              + (dd[2][1:nz, i, i] - dd[2][0:nz - 1, i, i]))
        h = [a.double() / VAC for a in f[3:]]
        dh = ((h[0][:nz, :ny, 1:] - h[0][:nz, :ny, :-1]) + (h[1][:nz, 1:, :nx] - h[1][:nz, :-1, :nx])
              + (h[2][1:, :ny, :nx] - h[2][:-1, :ny, :nx]))
        return np.array([w, float(de.square().sum().sqrt()), float(dh.square().sum().sqrt())])
    src, wave, probes = ((), None, ())
    if case["sources"]:
        src, wave, probes = _antenna(seed, nx, ny, nz, case["sources"], case["probes"], case["steps"])
    out, w, trace = _exact_solve(f, ce, nx, ny, nz, case["steps"], case["order"], src, wave, probes)
    r = {"energy": w, "fields": out}
    if case["sources"]:
        r["probes"] = trace
    return r
