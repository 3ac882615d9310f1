"""What a program does with this library, as cases to be timed: each is one whole pass
through the public binding (``paper_2603_13618_gb300.kss``) from the caller's inputs to the
outputs that the caller reads.

  listed()             the fixed cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  the caller's inputs and its lattice, batch or adjoint handle
  run(state)           one pass: set the state, step, read the outputs back
  work(case)           bytes and operations one pass cannot do without
  exact(case, seed)    the outputs of run() in 64-bit torch arithmetic

Every pass starts by setting the state, so its outputs depend on the inputs alone.  Outputs
are what such a program reads: moments or populations of the new state, sensor fields,
flags, tile counts, tag counts, conservation sums, boxes, gradients.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2603_13618_gb300 import kss

CS = 1.0 / math.sqrt(3.0)
SENSORS = ("tau_ns", "c", "s", "e", "qh", "kn", "neq", "qe", "hr", "kl", "sigma_h", "sigma_kl",
           "alpha")
# refine / switch thresholds near which the sensors of these flows lie
THRESHOLD = {"tau_ns": 1e-3, "c": 1e-3, "s": 2e-3, "e": 1e-3, "qh": 1e-5, "kn": 1e-3,
             "neq": 1e-4, "qe": 1e-5, "hr": 1e-6, "kl": 1e-8, "sigma_h": 1e-6,
             "sigma_kl": 1e-8, "alpha": 1e-3}


def _lattice(name, nx, ny, precision="fp32", steps=1, calls=1, every=1, tau=0.6, aar=False,
             tile=16, refine="kn", switch="neq", record="kl", ask="", field="jump",
             start="fields", host=False, moments=True, stats=True, regrid=False):
    """One lattice: `calls` times kss_step(steps), then the reads.  record: sensors stored on
    output steps, all of them read; ask: a sensor evaluated on demand; start: the state is
    set from FP64 fields ("fields"), FP32 fields ("fields32") or populations
    ("populations", then read back too); host: fields and outputs live in host memory."""
    c = {"kind": "lattice", "nx": nx, "ny": ny, "precision": precision, "steps": steps,
         "calls": calls, "every": every, "tau": tau, "aar": aar, "tile": tile, "refine": refine,
         "switch": switch, "record": record, "ask": ask, "field": field, "start": start,
         "host": host, "moments": moments, "stats": stats, "regrid": regrid}
    return c if name is None else {"name": name, **c}


def listed():
    every13 = ",".join(SENSORS)
    return [
        # the FP64 correctness workload: a decaying shear wave, outputs every 10 steps
        _lattice("shear_128_fp64", 128, 128, "fp64", steps=100, every=10, tau=0.8,
                 record="kn,kl", field="shear", start="fields"),
        # the smallest call: one step of one patch of a refined level, tags back to the host
        _lattice("patch_64_host", 64, 64, steps=1, host=True, moments=False),
        # a patch advanced on its own with tags every step
        _lattice("patch_256", 256, 256, steps=50, field="smooth"),
        # an odd-sized domain in small tagging tiles
        _lattice("ragged_1021x517", 1021, 517, steps=20, tile=8, tau=0.53, record="kn,kl"),
        # the headline workload: the density step with all fused outputs every step
        _lattice("jump_4096", 4096, 4096, steps=20, start="fields32"),
        # a run resumed from a checkpoint, outputs now and then, checkpointed again
        _lattice("resume_2048", 2048, 2048, steps=20, every=10, start="populations"),
        # the largest lattice, populations stored as FP16 deviations
        _lattice("fp16dev_8192", 8192, 8192, "fp16dev", steps=8, start="fields32"),
        # adaptive algorithm refinement: the QE sensor switches the collision model
        _lattice("aar_1536x1200", 1536, 1200, steps=20, tau=0.55, aar=True, switch="qe",
                 record="kl,qe"),
        # a comparison of every sensor of the paper's Table 1
        _lattice("table1_1024", 1024, 1024, steps=4, tau=0.8, record=every13, field="smooth"),
        # the refinement cycle: tag on the strain sensor every 4 steps, cluster into boxes
        _lattice("regrid_3000x2000", 3000, 2000, steps=4, calls=3, every=4, refine="s",
                 switch="neq", record="s", regrid=True),
        # the patches of one level in one batch
        {"name": "batch_10", "kind": "batch", "members": 10, "largest": 1024, "smallest": 64,
         "square": True, "pick": 13618, "precision": "fp32", "steps": 25, "every": 1},
        # the gradient of the sensor objective in the initial density and the relaxation time
        {"name": "adjoint_512", "kind": "adjoint", "nx": 512, "ny": 512, "precision": "fp32",
         "steps": 200, "checkpoint": 20, "tau": 0.6, "weight": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice"] * 6 + ["batch", "adjoint"])
    if kind == "batch":
        return {"kind": "batch", "members": rng.randint(2, 10), "largest": _log(rng, 100, 1024),
                "smallest": rng.randint(33, 99), "square": rng.random() < 0.4,
                "pick": rng.randrange(1 << 20),
                "precision": rng.choice(["fp32", "fp32", "fp16dev", "fp64"]),
                "steps": rng.randint(2, 25), "every": rng.choice([1, 1, 1, 5])}
    if kind == "adjoint":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        top = 640 if precision == "fp32" else 200
        return {"kind": "adjoint", "nx": _log(rng, 40, top), "ny": _log(rng, 40, top),
                "precision": precision, "steps": _log(rng, 8, 200 if precision == "fp32" else 40),
                "checkpoint": rng.randint(4, 30), "tau": round(rng.uniform(0.52, 1.2), 3),
                "weight": rng.random() < 0.5}
    precision = rng.choice(["fp32", "fp32", "fp32", "fp16dev", "fp64"])
    cells = _log(rng, 4000, 600_000 if precision == "fp64" else 12_000_000)
    aspect = math.exp(rng.uniform(-0.9, 0.9))
    nx, ny = max(33, int(math.sqrt(cells * aspect))), max(33, int(math.sqrt(cells / aspect)))
    aar = rng.random() < 0.25
    few = rng.random() < 0.65  # the {Kn, KL, neq} set; else any sensors
    pool = ["kn", "kl", "neq"] if few else [s for s in SENSORS if aar or s != "qe"]
    record = ",".join(sorted(rng.sample(pool, rng.randint(1, min(4, len(pool))))))
    return _lattice(None, nx, ny, precision, steps=rng.randint(1, 20), calls=rng.randint(1, 2),
                    every=rng.choice([1, 1, 1, 2, 5]), tau=round(rng.uniform(0.52, 1.2), 3),
                    aar=aar, tile=rng.choice([8, 16, 16, 32, 64]), refine=rng.choice(pool),
                    switch="qe" if aar and rng.random() < 0.5 else rng.choice(pool),
                    record=record, ask=rng.choice(["", "", "kn", "sigma_kl"]),
                    field=rng.choice(["jump", "smooth"]),
                    start=rng.choice(["fields", "fields32", "populations"]),
                    host=nx * ny < 300_000 and rng.random() < 0.3,
                    moments=rng.random() < 0.8, stats=rng.random() < 0.8,
                    regrid=rng.random() < 0.2)


# ---------------------------------------------------------------- inputs ----


def _smooth(nx, ny, gen, kmax=8):
    """A random smooth periodic field [ny, nx] (FP64), scaled to max 1: Fourier modes up to
    kmax with Gaussian amplitudes / (1 + k^2) and uniform phases."""
    k = torch.arange(-kmax, kmax + 1, dtype=torch.float64)
    damp = 1.0 + k[:, None] ** 2 + k[None, :] ** 2
    n = 2 * kmax + 1
    amp = torch.randn(n, n, generator=gen, dtype=torch.float64) / damp
    phase = 2 * math.pi * torch.rand(n, n, generator=gen, dtype=torch.float64)
    amp[kmax, kmax] = 0.0
    co = torch.polar(amp.abs(), phase).cuda()
    k = k.cuda()
    x = 2j * math.pi * torch.outer(k, torch.arange(nx, device="cuda", dtype=torch.float64)) / nx
    y = 2j * math.pi * torch.outer(torch.arange(ny, device="cuda", dtype=torch.float64), k) / ny
    f = (torch.exp(y) @ co @ torch.exp(x)).real
    return f / f.abs().max()


def _fields(nx, ny, field, seed, mach=0.1, drho=1e-2):
    """(rho, ux, uy) [ny, nx] FP64 on the GPU: "shear" a shear wave along y and
    a weaker one along x, "smooth" smooth perturbations, "jump" the same on a 2:1 density step along x."""
    gen = torch.Generator().manual_seed(int(seed))
    if field == "shear":
        amp = 0.01 * (1.0 + 0.2 * torch.rand((), generator=gen).item())
        phase = 2 * math.pi * torch.rand((), generator=gen).item()
        y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
        x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
        ux = (amp * torch.sin(2 * math.pi * y / ny + phase)).expand(ny, nx).contiguous()
        uy = (0.3 * amp * torch.sin(2 * math.pi * x / nx)).expand(ny, nx).contiguous()
        return torch.ones_like(ux), ux, uy
    rho = 1.0 + drho * _smooth(nx, ny, gen)
    ux, uy = _smooth(nx, ny, gen), _smooth(nx, ny, gen)
    scale = mach * CS / torch.sqrt(ux * ux + uy * uy).max()
    if field == "jump":
        rho[:, : nx // 2] *= 2.0
    return rho.contiguous(), (scale * ux).contiguous(), (scale * uy).contiguous()


def _tau2(tau):
    return 0.5 + (3.0 / 16.0) / (tau - 0.5)


def _members(case):
    """[(nx, ny, tau, mach)] of a batch case."""
    rng = np.random.default_rng(case["pick"])
    lo, hi = case["smallest"], case["largest"]
    out = []
    for _ in range(case["members"]):
        if case["square"]:
            sizes = [s for s in (64, 128, 256, 512, 1024) if s <= max(hi, 64)]
            nx = ny = int(rng.choice(sizes))
        else:
            nx, ny = (int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
                      for _ in range(2))
        if case["precision"] == "fp64":
            nx, ny = min(nx, 300), min(ny, 300)
        out.append((nx, ny, round(float(rng.uniform(0.51, 1.5)), 3),
                    round(float(rng.uniform(0.01, 0.15)), 4)))
    return out


def _config(case):
    return {"precision": case["precision"], "tau": case["tau"], "refine_sensor": case["refine"],
            "refine_threshold": THRESHOLD[case["refine"]], "switch_sensor": case["switch"],
            "switch_threshold": THRESHOLD[case["switch"]],
            "record": tuple(case["record"].split(",")), "output_every": case["every"],
            "tile": case["tile"], "tau2": _tau2(case["tau"]) if case["aar"] else 0.0}


def _initial_populations(rho, ux, uy):
    return _equilibrium(rho, ux, uy).contiguous()


def prepare(case, seed):
    if case["kind"] == "lattice":
        f = _fields(case["nx"], case["ny"], case["field"], seed)
        if case["start"] == "populations":
            f = (_initial_populations(*f),)
        elif case["start"] == "fields32":
            f = tuple(a.float() for a in f)
        if case["host"]:
            f = tuple(a.cpu().numpy() for a in f)
        return case, kss.Lattice(case["nx"], case["ny"], **_config(case)), f
    if case["kind"] == "batch":
        specs = _members(case)
        batch = kss.Batch([{"nx": nx, "ny": ny, "tau": tau} for nx, ny, tau, _ in specs],
                          precision=case["precision"], output_every=case["every"])
        f = [_fields(nx, ny, "smooth", seed * 64 + k, mach=mach)
             for k, (nx, ny, _, mach) in enumerate(specs)]
        return case, batch, f
    f = _fields(case["nx"], case["ny"], "smooth", seed)
    w = 0.5 + torch.rand(case["ny"], case["nx"], device="cuda", dtype=torch.float64,
                         generator=torch.Generator("cuda").manual_seed(int(seed)))
    adj = kss.Adjoint(case["nx"], case["ny"], case["steps"], precision=case["precision"],
                      checkpoint_every=case["checkpoint"])
    return case, adj, (*f, w if case["weight"] else None)


# ---------------------------------------------------------------- one pass ----


MAX_BOXES = 4096  # rows of the box table a pass returns (the list itself has any length)


def run(state):
    case, handle, f = state
    if case["kind"] == "batch":
        for member, fields in zip(handle.members, f):
            member.set_fields(*fields)
        handle.step(case["steps"])
        out = []
        for member in handle.members:
            rho, ux, uy = member.read_moments(device=True)
            flags, _, counts = member.read_flags(device=True)
            out += [rho, ux, uy, member.read_sensor("kl", device=True), flags, counts]
        return out
    if case["kind"] == "adjoint":
        objective = handle.forward(f[0], f[1], f[2], case["tau"], f[3])
        grad_rho, grad_tau = handle.backward(device=True)
        return {"objective": objective, "rho": grad_rho, "tau": grad_tau}
    device = not case["host"]
    out = {}
    if case["start"] == "populations":
        handle.set_populations(f[0])
    else:
        handle.set_fields(*f)
    for call in range(case["calls"]):
        handle.step(case["steps"])
        if case["regrid"]:
            boxes, mask = handle.regrid(buffer=2, efficiency=0.98)
            rows = np.full((MAX_BOXES, 4), -1, dtype=np.int32)
            if boxes:
                rows[: min(len(boxes), MAX_BOXES)] = np.array(boxes[:MAX_BOXES], dtype=np.int32)
            out["boxes%d" % call], out["nboxes%d" % call] = rows, len(boxes)
            out["mask%d" % call] = mask
    flags, tiles, counts = handle.read_flags(device=device)
    out.update(flags=flags, tiles=tiles, counts=counts)
    for s in case["record"].split(","):
        out["sensor_" + s] = handle.read_sensor(s, device=device)
    if case["ask"]:
        out["asked"] = handle.read_sensor(case["ask"], device=device)
    if case["stats"]:
        out["sums"] = handle.read_stats()[0]
    if case["moments"]:
        out["moments"] = handle.read_moments(device=device)
    if case["start"] == "populations":
        out["populations"] = handle.get_populations(device=device)
    return out


# ---------------------------------------------------------------- work ----

L2_BYTES = 126e6  # a state above this cannot stay on the chip from step to step
ELEMENT = {"fp64": 8, "fp32": 4, "fp16dev": 2}


def _steps_work(cells, precision, steps, outputs, recorded, full):
    """Bytes and operations of `steps` steps, `outputs` of them with sensors and tags."""
    state = 9 * ELEMENT[precision] * cells
    sensor = 8 if precision == "fp64" else 4
    moved = 2 * state * steps if 2 * state > L2_BYTES else 0
    return (moved + outputs * cells * (sensor * recorded + 1),
            cells * (130.0 * steps + (900.0 if full else 140.0) * outputs))


def work(case):
    if case["kind"] == "batch":
        b = o = 0.0
        outputs = case["steps"] // case["every"]
        cells = sum(nx * ny for nx, ny, _, _ in _members(case))
        b, o = _steps_work(cells, case["precision"], case["steps"], outputs, 1, False)
        return {"bytes": b + cells * (24 + 24 + 8 + 1), "flops": o + 40.0 * cells}
    cells = case["nx"] * case["ny"]
    if case["kind"] == "adjoint":
        # forward states are produced once and read once by the reverse steps
        state = 9 * ELEMENT[case["precision"]] * cells
        return {"bytes": 24 * cells + 2.0 * case["steps"] * state + 8 * cells,
                "flops": 130.0 * case["steps"] * cells + 330.0 * case["steps"] * cells}
    total = case["steps"] * case["calls"]
    wanted = set(case["record"].split(",")) | {case["refine"], case["switch"]}
    full = bool(wanted - {"kn", "kl", "neq", "qe"})
    b, o = _steps_work(cells, case["precision"], total, total // case["every"],
                       len(case["record"].split(",")), full)
    b += cells * {"fields": 24, "fields32": 12, "populations": 144}[case["start"]]
    b += cells * (1 + 8 * len(case["record"].split(",")) + (8 if case["ask"] else 0)
                  + (24 if case["moments"] else 0))
    o += 40.0 * cells
    return {"bytes": float(b), "flops": float(o)}


# ---------------------------------------------------------------- 64 bits ----

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPPOSITE = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _equilibrium(rho, ux, uy):
    uu = 1.5 * (ux * ux + uy * uy)
    return torch.stack([w * rho * (1.0 + 3.0 * (cu := cx * ux + cy * uy) + 4.5 * cu * cu - uu)
                        for w, cx, cy in zip(W, CX, CY)])


def _stream(f):
    return torch.stack([torch.roll(f[q], (CY[q], CX[q]), (0, 1)) for q in range(9)])


def _moments(f):
    rho = f.sum(0)
    jx = (f[1] + f[5] + f[8]) - (f[3] + f[6] + f[7])
    jy = (f[2] + f[5] + f[6]) - (f[4] + f[7] + f[8])
    return rho, jx / rho, jy / rho


def _collide(f, tau, tau2=None, region=None):
    rho, ux, uy = _moments(f)
    d = f - _equilibrium(rho, ux, uy)
    new = f - d / tau
    if region is not None:
        a, b = 0.5 * (1 / tau + 1 / tau2), 0.5 * (1 / tau - 1 / tau2)
        other = f - a * d - b * d[list(OPPOSITE)]
        other[0] = new[0]
        new = torch.where(region, other, new)
    return new


def _sensor(f, name, tau, qe):
    """One sensor of Table 1 (single distribution) on the populations f."""
    rho, ux, uy = _moments(f)
    eq = _equilibrium(rho, ux, uy)
    d = f - eq
    x = d / eq
    if name == "neq":
        return d.abs().sum(0)
    if name == "qe":
        if not qe:
            return torch.zeros_like(rho)
        return 0.5 * (d - d[list(OPPOSITE)]).abs().sum(0)
    if name in ("tau_ns", "c", "s", "e", "qh"):
        diag = d[5] + d[6] + d[7] + d[8]
        pxx, pyy = d[1] + d[3] + diag, d[2] + d[4] + diag
        pxy = d[5] - d[6] + d[7] - d[8]
        mu = rho * tau / 3.0
        norm = torch.sqrt(pxx ** 2 + pyy ** 2 + 2 * pxy ** 2)
        if name == "tau_ns":
            return norm
        if name == "c":
            return math.sqrt(2.0) * (pxx + pyy).abs() / (2 * mu)
        if name == "s":
            return torch.sqrt(2.0 * ((0.5 * (pyy - pxx)) ** 2 + pxy ** 2)) / mu
        if name == "e":
            return norm / (2 * mu)
        return torch.sqrt((ux * pxx + uy * pxy) ** 2 + (ux * pxy + uy * pyy) ** 2)
    w = torch.tensor(W, device=f.device, dtype=f.dtype)[:, None, None]
    if name == "kn":
        out = x.abs().sum(0)
    elif name == "kl":
        out = (eq * ((1 + x) * torch.log1p(x) - x)).sum(0).abs()
    elif name == "sigma_kl":
        out = (d * torch.log1p(x)).sum(0) / tau
    elif name in ("hr", "sigma_h"):
        uu = 1.5 * (ux * ux + uy * uy)
        lin = torch.zeros_like(rho)
        for q in range(9):
            cu = CX[q] * ux + CY[q] * uy
            lin += d[q] * torch.log1p(3 * cu + 4.5 * cu * cu - uu)
        if name == "hr":
            out = (lin + (eq * ((1 + x) * torch.log1p(x) - x)).sum(0)).abs()
        else:
            out = (lin + (d * torch.log1p(x)).sum(0)) / tau
    else:  # alpha
        y = d / f
        a = [(-1.0) ** (n - 1) / (n * (n + 1)) * (d * y ** n).sum(0) for n in range(1, 5)]
        r2, r3, r4 = a[1] / a[0], a[2] / a[0], a[3] / a[0]
        out = (4 * r2 - 16 * r2 ** 2 + 8 * r3 - 80 * r2 * r3 + 80 * r2 ** 3 + 16 * r4).abs()
        out = torch.where(a[0] == 0, torch.zeros_like(out), out)
    bad = ((f <= 0) | (eq <= 0)).any(0)
    return torch.where(bad, torch.full_like(out, math.inf), out)


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    if case["kind"] == "batch":
        out = []
        for k, (nx, ny, tau, mach) in enumerate(_members(case)):
            f = _initial_populations(*_fields(nx, ny, "smooth", seed * 64 + k, mach=mach))
            pre = f
            for n in range(1, case["steps"] + 1):
                pre = _stream(f)
                f = _collide(pre, tau)
            out += [*_moments(f), _sensor(pre, "kl", tau, False), None, None]
        return out
    tau, tau2 = case["tau"], _tau2(case["tau"])
    fields = _fields(case["nx"], case["ny"], case["field"], seed)
    if case["start"] == "fields32":
        fields = tuple(a.float().double() for a in fields)
    f = _initial_populations(*fields)
    region = torch.zeros_like(f[0], dtype=torch.bool) if case["aar"] else None
    pre = f
    for n in range(1, case["steps"] * case["calls"] + 1):
        pre = _stream(f)
        f = _collide(pre, tau, tau2, region)
        if case["aar"] and n % case["every"] == 0:
            region = _sensor(pre, case["switch"], tau, True) > THRESHOLD[case["switch"]]
    out = {"flags": None, "tiles": None, "counts": None}
    for s in case["record"].split(","):
        out["sensor_" + s] = _sensor(pre, s, tau, case["aar"])
    if case["ask"]:
        out["asked"] = _sensor(pre, case["ask"], tau, case["aar"])
    if case["stats"]:
        rho = pre.sum(0)
        _, ux, uy = _moments(pre)
        out["sums"] = torch.stack([rho.sum(), (rho * ux).sum(), (rho * uy).sum()])
    if case["moments"]:
        out["moments"] = _moments(f)
    if case["start"] == "populations":
        out["populations"] = f
    return out


def _exact_adjoint(case, seed):
    rho, ux, uy = _fields(case["nx"], case["ny"], "smooth", seed)
    weight = 0.5 + torch.rand(case["ny"], case["nx"], device="cuda", dtype=torch.float64,
                              generator=torch.Generator("cuda").manual_seed(int(seed)))
    rho.requires_grad_(True)
    tau = torch.tensor(case["tau"], device="cuda", dtype=torch.float64, requires_grad=True)

    def segment(f, tau, n):
        for _ in range(n):
            f = _collide(_stream(f), tau)
        return f

    f, left = _equilibrium(rho, ux, uy), case["steps"] - 1
    while left > 0:
        n = min(10, left)
        f = torch.utils.checkpoint.checkpoint(segment, f, tau, n, use_reentrant=False)
        left -= n
    kl = _sensor(_stream(f), "kl", tau, False)
    objective = (kl * weight).sum() if case["weight"] else kl.sum()
    objective.backward()
    return {"objective": objective.detach(), "rho": rho.grad,
            "tau": tau.grad if tau.grad is not None else torch.zeros_like(rho[0, 0])}
