"""Performance cases of the two-beam BPM: what users of the library have it do.

A pass is what a program does with a plan it keeps: it sets a pulse (and, where
the case says so, a new deformed crystal), marches it to the exit and takes the
fields, the rocking curve and the time response; or it hands several plans to a
batch.  The physics is the common geometry of the repository's workloads
(C*(400) at 45 degrees, dx = 0.5 um in 2D, 1 um in 3D), drawn from a seed:
spectrum, beam, strain and incidence angle differ from seed to seed.

exact() marches the same inputs in complex128 with torch.fft.
"""
from __future__ import annotations

import math

import numpy as np
import torch

C_LIGHT = 299792458.0
THETA_B = math.radians(45.0)
LAMBDA_B = 1.26116e-10
D_HKL = LAMBDA_B / (2.0 * math.sin(THETA_B))
H = 4.0 * math.pi * math.sin(THETA_B) / LAMBDA_B
CHI0 = complex(-1.0e-5, 1.0e-8)
CHIH = complex(-4.0e-6, 0.5e-8)


def _plan2d(name, nx, nz, n_ch, order=1, strain="bump", shape="bragg", crystal="kept",
            time=True, tuned=False):
    return dict(name=name, path="plan", dims=2, nx=nx, ny=1, nz=nz, n_ch=n_ch, order=order,
                strain=strain, shape=shape, crystal=crystal, time=time, tuned=tuned)


def _plan3d(name, nx, ny, nz, n_ch, strain="bump", shape="bragg", tuned=False, time=False):
    return dict(name=name, path="plan", dims=3, nx=nx, ny=ny, nz=nz, n_ch=n_ch, order=1,
                strain=strain, shape=shape, crystal="kept", time=time, tuned=tuned)


def listed():
    return [
        # one rocking-curve probe: a single channel on a small grid, the shortest
        # request a program or the server makes; its latency is the user's wait
        _plan2d("probe", 512, 300, 1, strain="perfect", time=False),
        # the smallest whole pulse of the repository: perfect crystal, 64 channels
        _plan2d("tiny", 256, 200, 64, strain="perfect"),
        # a serving lane's round of short requests: 48 probes through the work queue
        dict(name="probe round", path="queue", nx=512, nz=300, plans=48),
        # a rocking curve of an odd number of points in a Laue slab, with its time
        # response; the crystal is kept and the pulse is new
        _plan2d("curve", 512, 400, 201, shape="laue"),
        # a deformed crystal at a channel count that fills no group and no power of two
        _plan2d("ragged", 1024, 600, 611, strain="random"),
        # an asymmetric cut, bent, Strang splitting, a third of a pulse's channels
        _plan2d("strang", 2048, 500, 300, order=2, strain="bent", shape="asymmetric"),
        # the repository's headline pulse: 1024 channels through a crystal deformed
        # anew for each pass, in the launch form that the tuner picked (as bench.py does)
        _plan2d("deformed", 4096, 2000, 1024, crystal="new", tuned=True),
        # fourth-order splitting on a crystal of any shape (a caller's mask)
        _plan2d("fourth order", 4096, 150, 256, order=4, shape="mask"),
        # the largest 2D transform
        _plan2d("wide", 8192, 500, 512, strain="random", tuned=True),
        # a small 3D problem, ragged channel count, unequal sides
        _plan3d("3D small", 256, 512, 100, 24, shape="asymmetric", time=True),
        # the repository's 3D pulse, a section of its march
        _plan3d("3D", 512, 512, 60, 128, tuned=True),
        # uneven instances in one captured batch (sizes and steps of the uneven batch)
        dict(name="uneven batch", path="graph", plans=10, steps=700, pick=3),
    ]


def draw(rng):
    """One more case of the same ranges; its march is never longer than the headline's."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["plan", "plan", "plan", "plan", "plan", "3d", "3d", "queue", "graph"])
    if kind == "queue":
        return dict(path="queue", nx=rng.choice([256, 512, 1024]), nz=rng.randint(100, 500),
                    plans=rng.randint(2, 64))
    if kind == "graph":
        return dict(path="graph", plans=rng.randint(2, 10), steps=rng.randint(100, 700),
                    pick=rng.randrange(1 << 20))
    strain = rng.choice(["perfect", "bump", "bent", "random"])
    shape = rng.choice(["bragg", "bragg", "asymmetric", "laue", "mask"])
    tuned = rng.random() < 0.4
    time = rng.random() < 0.5
    if kind == "3d":
        nx, ny = rng.choice([256, 512, 1024]), rng.choice([256, 512, 1024])
        n_ch = min(log_int(1, 128), (1 << 25) // (nx * ny))
        nz = max(20, min(rng.randint(20, 120), int(2.0e9 / (nx * ny * n_ch))))
        c = _plan3d("", nx, ny, nz, n_ch, strain, shape, tuned, time)
    else:
        nx = rng.choice([256, 512, 1024, 2048, 4096, 8192])
        order = rng.choice([1, 1, 1, 1, 2, 2, 4])
        n_ch = log_int(1, 700) if rng.random() < 0.7 else 1 << rng.randint(2, 10)
        nz = max(40, min(log_int(40, 2000), int(2.5e9 / (nx * n_ch * (3 if order == 4 else 1)))))
        c = _plan2d("", nx, nz, n_ch, order, strain, shape, rng.choice(["kept", "new"]), time,
                    tuned)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs (from the seed alone)
# ---------------------------------------------------------------------------
def _problem(c, seed):
    """Physical inputs of one plan: plain numbers and numpy arrays (u is made apart)."""
    r = np.random.default_rng([int(seed), c["nx"], c["nz"], c["n_ch"]])
    dims, nx, ny, nz, n_ch = c["dims"], c["nx"], c["ny"], c["nz"], c["n_ch"]
    dx = 0.5e-6 if dims == 2 else 1.0e-6
    dz = min(dx, nx * dx / (2.0 * nz)) if dims == 2 else 0.25e-6
    # +-5 Darwin widths around the reflection band, a Gaussian pulse with a random
    # centre and chirp; a single channel is a probe at a random angle instead
    eps_d = abs(CHIH) / math.sin(THETA_B) ** 2
    eps_c = -CHI0.real / (2.0 * math.sin(THETA_B) ** 2)
    off, chirp = r.uniform(-0.5, 0.5), r.uniform(-2.0, 2.0)
    i = np.arange(n_ch, dtype=np.float64)
    d = (i - n_ch // 2) * 10.0 / n_ch if n_ch > 1 else np.zeros(1)
    omega = 2.0 * math.pi * C_LIGHT / LAMBDA_B * (1.0 + eps_c + (d + off) * eps_d)
    S = np.exp(-(d ** 2) / (2.0 * 1.5 ** 2) + 1j * (chirp * d + r.uniform(0, 6.28)))
    first, cells = (nx // 5, nx // 10) if dims == 2 else (nx // 3, nx // 4)
    p = dict(c, dx=dx, dy=dx, dz=dz, omega=omega, S=S,
             theta_i=THETA_B + r.uniform(-1.0, 1.0) * eps_d,
             # the beam moves a step in x per step in z: it starts where it is well
             # into the crystal by the exit, also in a short march
             x0=first * dx - min(0.4 * first * dx, 0.2 * nz * dz),
             w0=max(8, nx // 60) * dx, zx=0.0, zR=1.0, x_surface=(first - 0.5) * dx,
             thickness=cells * dx, tan_psi=0.0, z_begin=-math.inf, z_end=math.inf)
    if c["shape"] == "asymmetric":
        p["tan_psi"] = math.tan(math.radians(r.uniform(2.0, 8.0))) * r.choice([-1.0, 1.0])
    elif c["shape"] == "laue":
        p["x_surface"], p["thickness"] = -nx * dx, 3 * nx * dx
        p["z_begin"], p["z_end"] = (nz // 6 - 0.5) * dz, (nz - nz // 6 - 0.5) * dz
    kind = c["strain"]
    if kind == "bump":
        p["u"] = dict(amp=r.uniform(0.1, 0.5) * D_HKL, wx=r.uniform(0.05, 0.25) * nx * dx,
                      wy=r.uniform(0.1, 0.4) * ny * dx)
    elif kind == "bent":
        p["u"] = dict(R=r.uniform(5.0, 50.0))
    elif kind == "random":
        p["u"] = dict(a=r.uniform(-0.5, 0.5, 8) * D_HKL, cx=r.uniform(0, cells * dx, 8),
                      cz=r.uniform(0, nz * dz, 8), wx=r.uniform(1 / 32, 1 / 4, 8) * nx * dx,
                      wz=r.uniform(1 / 32, 1 / 4, 8) * nx * dx)
    else:
        p["u"] = None
    return p


def _strain(p):
    """Displacement [nz][ny][nx] float64 on the GPU, or None for a perfect crystal."""
    if p["u"] is None:
        return None
    f = dict(dtype=torch.float64, device="cuda")
    x = (torch.arange(p["nx"], **f) * p["dx"] - p["x_surface"]).view(1, 1, -1)
    y = ((torch.arange(p["ny"], **f) - p["ny"] // 2) * p["dy"]).view(1, -1, 1)
    z = (torch.arange(p["nz"], **f) * p["dz"]).view(-1, 1, 1)
    Z, q = p["nz"] * p["dz"], p["u"]
    if p["strain"] == "bump":
        depth = x if p["shape"] != "laue" else x - p["nx"] * p["dx"]
        g = torch.exp(-(depth / q["wx"]) ** 2 - (y / q["wy"]) ** 2)
        return (q["amp"] * g * (z / Z) ** 2).contiguous()
    if p["strain"] == "bent":
        u = -((z - Z / 2) ** 2) / (2.0 * q["R"])
        return u.expand(p["nz"], p["ny"], p["nx"]).contiguous()
    u = torch.zeros(p["nz"], 1, p["nx"], **f)
    for a, cx, cz, wx, wz in zip(*(q[k] for k in ("a", "cx", "cz", "wx", "wz"))):
        u += a * torch.exp(-((z - cz) / wz) ** 2) * torch.exp(-((x - cx) / wx) ** 2)
    return u.expand(p["nz"], p["ny"], p["nx"]).contiguous()


def _mask(p):
    """A caller's crystal shape [nz][ny][nx] (bytes): a bulging slab with a void."""
    if p["shape"] != "mask":
        return None
    x = (torch.arange(p["nx"], device="cuda").double() / p["nx"]).view(1, 1, -1)
    y = (torch.arange(p["ny"], device="cuda").double() / p["ny"] - 0.5).view(1, -1, 1)
    z = (torch.arange(p["nz"], device="cuda").double() / p["nz"]).view(-1, 1, 1)
    front = 0.2 + 0.03 * torch.sin(3.0 * z) + 0.02 * y
    back = front + 0.12 + 0.02 * torch.cos(5.0 * z)
    void = ((x - 0.28) / 0.02) ** 2 + ((z - 0.5) / 0.2) ** 2 < 1.0
    m = (x >= front) & (x < back) & ~void
    return m.expand(p["nz"], p["ny"], p["nx"]).to(torch.uint8).contiguous()


def _members(c, seed):
    """The plans of a case: one, or those of a batch."""
    if c["path"] == "plan":
        return [_problem(c, seed)]
    if c["path"] == "queue":
        one = _plan2d("", c["nx"], c["nz"], 1, strain="perfect", time=False)
        return [_problem(one, 1000 * int(seed) + k) for k in range(c["plans"])]
    out = []
    r = np.random.default_rng([77, c["pick"]])  # shapes belong to the case, not to the seed
    for k in range(c["plans"]):
        nx = int(r.choice([1024, 2048, 4096, 8192]))
        nz = int(r.integers(max(40, c["steps"] // 8), c["steps"] + 1))
        one = _plan2d("", nx, nz, int(r.choice([128, 256, 512, 1024])),
                      strain=str(r.choice(["perfect", "bent", "random"])))
        out.append(_problem(one, 1000 * int(seed) + k))
    return out


# ---------------------------------------------------------------------------
# The framework's side
# ---------------------------------------------------------------------------
def _crystal(plan, p, u):
    plan.set_crystal(CHI0, CHIH, CHIH, THETA_B, LAMBDA_B, p["x_surface"], p["thickness"], u=u)


def _pulse(plan, p):
    plan.set_pulse(p["omega"], p["S"], p["theta_i"], p["x0"], p["w0"], p["zx"], p["zR"])


def _buffers(p):
    n, plane = p["n_ch"], p["nx"] * p["ny"]
    b = {k: torch.empty(n, plane, dtype=torch.complex64, device="cuda") for k in ("e0", "eh")}
    if p["time"]:
        b["eh_time"] = torch.empty(n, plane, dtype=torch.complex128, device="cuda")
    return b


def prepare(case, seed):
    from paper_2201_08500_gb300 import bpm

    bpm.tune_clear()
    s = dict(path=case["path"], members=_members(case, seed))
    p = s["members"][0]
    if case.get("tuned"):  # a program with many pulses of one shape tunes once
        bpm.tune(p["dims"], p["nx"], p["ny"], p["dx"], p["dy"], p["dz"], p["n_ch"],
                 split_order=p["order"], steps=48 if p["dims"] == 2 else 12)
    s["plans"], s["u"], s["out"] = [], [], []
    for p in s["members"]:
        plan = bpm.Plan(p["dims"], p["nx"], p["ny"], p["nz"], p["dx"], p["dy"], p["dz"],
                        p["n_ch"], split_order=p["order"])
        if p["shape"] in ("asymmetric", "laue"):
            plan.set_geometry(p["tan_psi"], p["z_begin"], p["z_end"])
        m = _mask(p)
        if m is not None:
            torch.cuda.synchronize()
            plan.set_crystal_shape(m)
            plan.sync() if p["crystal"] == "kept" else None
        u = _strain(p)
        torch.cuda.synchronize()
        _crystal(plan, p, u)
        _pulse(plan, p)
        plan.sync()
        s["plans"].append(plan)
        s["u"].append(u)
        s["out"].append(_buffers(p))
    if s["path"] != "plan":
        s["batch"] = bpm.Batch()
    if s["path"] == "graph":
        for plan in s["plans"]:
            s["batch"].submit(plan)
    bpm.tune_clear()
    return s


def _take(plan, out):
    from paper_2201_08500_gb300 import bpm

    plan.fetch(bpm.BPM_FIELD_E0, out["e0"])
    plan.fetch(bpm.BPM_FIELD_EH, out["eh"])
    if "eh_time" in out:
        plan.fetch(bpm.BPM_FIELD_EH_TIME, out["eh_time"])
    R, T, R_int = plan.reflectivity()
    return dict(out, R=R, T=T, R_int=R_int)


def run(state):
    plans, members, outs = state["plans"], state["members"], state["out"]
    if state["path"] == "plan":
        plan, p = plans[0], members[0]
        if p["crystal"] == "new":
            _crystal(plan, p, state["u"][0])
        _pulse(plan, p)
        plan.run()
        return _take(plan, outs[0])
    b = state["batch"]
    if state["path"] == "graph":
        b.run_graph()
        b.sync()
        return [_take(plan, out) for plan, out in zip(plans, outs)]
    tickets = []
    for plan, p in zip(plans, members):
        _pulse(plan, p)
        tickets.append(b.submit(plan))
    b.run()
    b.sync()
    got = []
    for ticket, plan in zip(tickets, plans):
        if not b.poll(ticket):
            raise RuntimeError("a synchronised batch left a ticket unfinished")
        got.append(plan.reflectivity())
    # one probe's answer is its rocking-curve point; the fields stay with the plans
    return dict(R=np.array([g[0][0] for g in got]), T=np.array([g[1][0] for g in got]),
                R_int=np.array([g[2] for g in got]))


# ---------------------------------------------------------------------------
# The least work of a pass, and its values in 64 bits
# ---------------------------------------------------------------------------
def work(case):
    nbytes = flops = 0.0
    for p in _members(case, 0):
        cells = float(p["nx"]) * p["ny"] * p["nz"]
        lg = math.log2(p["nx"] * p["ny"])
        props, couples = {1: (1, 1), 2: (1, 2), 4: (3, 4)}[p["order"]]
        # per cell-update: four transforms and two propagator products a propagation;
        # a coupling only where there is crystal (a tenth of a Bragg slab's grid)
        share = {"laue": 0.67, "mask": 0.12}.get(p["shape"], 0.1 if p["dims"] == 2 else 0.25)
        flops += cells * p["n_ch"] * (props * (20.0 * lg + 12.0) + couples * 40.0 * share)
        plane = float(p["nx"]) * p["ny"]
        nbytes += p["n_ch"] * (plane * 16.0 + 40.0)
        if p["u"] is not None and p["crystal"] == "new":
            nbytes += cells * 8.0
        if p["time"]:
            nbytes += p["n_ch"] * plane * 16.0
            flops += plane * 5.0 * p["n_ch"] * math.log2(max(2, p["n_ch"]))
    return {"bytes": nbytes, "flops": flops}


def _bessel(w2):
    """J0(w) and 2 J1(w) / w from the power series in w^2."""
    z, t0, t1, j0, g1 = -0.25 * w2, 1.0, 1.0, 1.0, 1.0
    for k in range(1, 30):
        t0 = t0 * z / (k * k)
        t1 = t1 * z / (k * (k + 1))
        j0, g1 = j0 + t0, g1 + t1
    return j0, g1


def _exact_plan(p):
    f = dict(dtype=torch.float64, device="cuda")
    dims3 = p["dims"] == 3
    om = torch.as_tensor(p["omega"], **f)
    k = (om / C_LIGHT).view(-1, 1, 1)
    qx = (2.0 * math.pi * torch.fft.fftfreq(p["nx"], p["dx"], **f)).view(1, 1, -1)
    qy = (2.0 * math.pi * torch.fft.fftfreq(p["ny"], p["dy"], **f)).view(1, -1, 1)
    cos_a = torch.sqrt(1.0 - (0.5 * H / k) ** 2)

    def propagator(sign, dz):
        q2 = (qx + sign * 0.5 * H) ** 2 + qy ** 2
        arg = k * k - q2
        ph = torch.where(arg >= 0, -dz * q2 / (torch.sqrt(arg.clamp(min=0)) + k), -dz * k)
        mag = torch.where(arg >= 0, torch.ones_like(ph),
                          torch.exp(-dz * torch.sqrt((-arg).clamp(min=0))))
        return torch.polar(mag, ph)

    def coupling(frac):
        kdz = frac * k * p["dz"]
        w2 = (kdz / cos_a) ** 2 * (CHIH * CHIH)
        ph = torch.exp(1j * CHI0 * (kdz / (2.0 * cos_a)))
        j0, g1 = _bessel(w2)
        b = 1j * g1 * ph * (CHIH * (kdz / (2.0 * cos_a)))
        return j0 * ph * torch.exp(0.125 * w2), b

    t4 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
    prop = {fr: (propagator(1.0, fr * p["dz"]), propagator(-1.0, fr * p["dz"]))
            for fr in ({4: (t4, 1.0 - 2.0 * t4)}.get(p["order"], (1.0,)))}
    x = torch.arange(p["nx"], **f) * p["dx"]
    y = (torch.arange(p["ny"], **f) - p["ny"] // 2) * p["dy"] * (1.0 if dims3 else 0.0)
    g = torch.exp(-(((x - p["x0"]) ** 2).view(1, -1) + (y ** 2).view(-1, 1)) / p["w0"] ** 2)
    dq = k * math.sin(p["theta_i"]) - 0.5 * H
    a = torch.as_tensor(p["S"], device="cuda").view(-1, 1, 1) * g * torch.exp(
        1j * dq * x.view(1, 1, -1))
    b = torch.zeros_like(a)
    inc = (a.abs() ** 2).sum((1, 2))
    u, mask = _strain(p), _mask(p)

    def cell(n):
        if mask is not None:
            pi = mask[n].bool()
        else:
            z = n * p["dz"]
            s = z * p["tan_psi"]
            inside = (x >= p["x_surface"] + s) & (x < p["x_surface"] + p["thickness"] + s)
            pi = (inside & (p["z_begin"] <= z < p["z_end"])).view(1, -1)
        ph = torch.zeros_like(pi, dtype=torch.float64) if u is None else H * u[n]
        return pi, torch.polar(torch.ones_like(ph), ph)

    dim = (1, 2) if dims3 else (2,)

    def propagate(fr):
        nonlocal a, b
        a = torch.fft.ifftn(torch.fft.fftn(a, dim=dim).mul_(prop[fr][0]), dim=dim)
        b = torch.fft.ifftn(torch.fft.fftn(b, dim=dim).mul_(prop[fr][1]), dim=dim)

    def couple(cf, pi, c):
        nonlocal a, b
        w = torch.nonzero(pi.any(0))[:, 0]
        if w.numel() == 0:
            return
        w = slice(int(w[0]), int(w[-1]) + 1)
        pi, c = pi[:, w], c[:, w]
        e, h = a[..., w], b[..., w]
        na, nb = cf[0] * e + cf[1] * c * h, cf[0] * h + cf[1] * c.conj() * e
        a[..., w], b[..., w] = torch.where(pi, na, e), torch.where(pi, nb, h)

    cfs = {fr: coupling(fr) for fr in {1: (1.0,), 2: (0.5,), 4: (0.5 * t4, 0.5 * (1 - t4))}[
        p["order"]]}
    for n in range(p["nz"]):
        pi, c = cell(n)
        if p["order"] == 1:
            propagate(1.0)
            couple(cfs[1.0], pi, c)
        elif p["order"] == 2:
            couple(cfs[0.5], pi, c)
            propagate(1.0)
            couple(cfs[0.5], pi, c)
        else:
            outer, inner = cfs[0.5 * t4], cfs[0.5 * (1 - t4)]
            for cf, fr in ((outer, t4), (inner, 1.0 - 2.0 * t4), (inner, t4)):
                couple(cf, pi, c)
                propagate(fr)
            couple(outer, pi, c)
    n = p["n_ch"]
    R = ((b.abs() ** 2).sum((1, 2)) / inc).cpu().numpy()
    T = ((a.abs() ** 2).sum((1, 2)) / inc).cpu().numpy()
    dom = float(p["omega"][1] - p["omega"][0]) if n > 1 else 1.0
    out = dict(e0=a.reshape(n, -1), eh=b.reshape(n, -1), R=R, T=T, R_int=dom * float(R.sum()))
    if p["time"]:
        j = torch.arange(n, device="cuda")
        turn = torch.polar(torch.ones(n, **f), 2.0 * math.pi * ((j * (n // 2)) % n).double() / n)
        out["eh_time"] = dom * turn.view(-1, 1) * torch.fft.fft(out["eh"], dim=0)
    return out


def exact(case, seed):
    got = [_exact_plan(p) for p in _members(case, seed)]
    if case["path"] == "plan":
        return got[0]
    if case["path"] == "graph":
        return got
    return dict(R=np.array([g["R"][0] for g in got]), T=np.array([g["T"][0] for g in got]),
                R_int=np.array([g["R_int"] for g in got]))
