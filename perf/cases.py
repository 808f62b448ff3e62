"""The work a user of this framework has it do, as cases that can be timed and compared.

Every case is one call (or one short chain of calls) of the public Python layer on a workload
description: fused traces of one simulation, one persistent launch over many simulations, the
gradient of the chi-squared loss, and the unfused component chain with stored packets.  Sizes,
samples, detectors and incident energies are those of the repository's own workloads
(`mcv_inputs`), its tests and its benchmark.  `exact` restates the method in 64-bit torch,
vectorised over neutrons, from the definitions in `include/mcv.h`.
"""
import dataclasses
import math

import numpy as np
import torch

import mcv_inputs as mi
from paper_1504_02776_gb300 import api, binding as B

# largest neutron count of a drawn case by (work, precision), so that none costs more than the
# largest listed ones; the smallest counts are single quick-look runs
_RANGES = {
    ("powder", 32): (1e5, 1e8), ("powder", 64): (1e4, 5e6),
    ("cylinder", 32): (1e4, 3e7), ("cylinder", 64): (1e4, 3e6),
    ("can", 32): (1e5, 2e7), ("can", 64): (1e4, 1e6),
    ("vanadium", 32): (1e5, 2e7), ("vanadium", 64): (1e4, 2e6),
    ("aluminium", 32): (1e5, 2e7), ("aluminium", 64): (1e4, 4e6),
    ("crystal", 32): (1e4, 4e6), ("crystal", 64): (5e3, 1e5),
}


def listed():
    return [
        # a test-sized run of the simplest sample, where the launch and the call count
        {"name": "cylinder-1e5-fp64", "kind": "trace", "sample": "cylinder", "fp": 64,
         "n": 100_000, "ei": 60.0, "orders": 1, "n_tof": 200, "estimator": "chain"},
        # a quick look at a powder on the whole tube system with coarse time bins
        {"name": "powder-1e6-fp32", "kind": "trace", "sample": "powder", "fp": 32,
         "n": 1_000_003, "ei": 100.0, "orders": 5, "n_tof": 100, "estimator": "chain"},
        # the paper's full powder run: 1e8 packets, 117,760 pixels x 1000 time bins
        {"name": "powder-1e8-fp32", "kind": "trace", "sample": "powder", "fp": 32,
         "n": 100_000_000, "ei": 100.0, "orders": 5, "n_tof": 1000, "estimator": "chain"},
        # the same run in the reference precision, as it is used to check a fast run
        {"name": "powder-5e6-fp64", "kind": "trace", "sample": "powder", "fp": 64,
         "n": 5_000_000, "ei": 100.0, "orders": 5, "n_tof": 1000, "estimator": "chain"},
        # vanadium-like calibration sample (incoherent phonon expansion)
        {"name": "vanadium-1e7-fp32", "kind": "trace", "sample": "vanadium", "fp": 32,
         "n": 10_000_000, "ei": 100.0, "orders": 5, "n_tof": 1000, "estimator": "chain"},
        # aluminium-like powder diffraction, reference precision
        {"name": "aluminium-2e6-fp64", "kind": "trace", "sample": "aluminium", "fp": 64,
         "n": 2_000_000, "ei": 100.0, "orders": 5, "n_tof": 200, "estimator": "chain"},
        # the paper's own recursive estimator, the fidelity mode
        {"name": "paper-powder-2e6-fp32", "kind": "trace", "sample": "powder", "fp": 32,
         "n": 2_000_000, "ei": 100.0, "orders": 5, "n_tof": 200, "estimator": "paper"},
        # one orientation of a single crystal in the reference precision
        {"name": "crystal-5e4-fp64", "kind": "trace", "sample": "crystal", "fp": 64,
         "n": 50_000, "ei": 50.0, "orders": 5, "n_tof": 100, "rot": 30.0, "estimator": "chain"},
        # a rotation scan of a single crystal: one simulation and histogram per orientation
        {"name": "crystal-scan-fp32", "kind": "batch", "sample": "crystal", "fp": 32,
         "n": 2_600_000, "sims": 13, "ei": 50.0, "orders": 5, "n_tof": 200},
        # an uneven incident-energy sweep, 10..500 meV, with the sample in its can
        {"name": "can-sweep-fp32", "kind": "batch", "sample": "can", "fp": 32,
         "n": 32_000_000, "sims": 32, "ei": 70.0, "orders": 5, "n_tof": 100},
        # one step of a fit: chi-squared loss and its gradient on the powder run
        {"name": "powder-grad-1e7-fp32", "kind": "grad", "sample": "powder", "fp": 32,
         "n": 10_000_000, "ei": 100.0, "orders": 5, "n_tof": 1000},
        # the components called one by one with packets stored in between
        {"name": "powder-chain-5e5-fp32", "kind": "chain", "sample": "powder", "fp": 32,
         "n": 500_001, "ei": 100.0, "orders": 5, "n_tof": 100},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["trace", "trace", "trace", "trace", "trace", "batch", "batch", "grad",
                       "chain"])
    fp = rng.choice([32, 32, 64])
    case = {"kind": kind, "fp": fp, "n_tof": rng.choice([40, 100, 199, 200, 500, 1000]),
            "orders": rng.choice([1, 2, 3, 5, 5, 5])}
    if kind == "trace":
        case["sample"] = rng.choice(["powder", "powder", "cylinder", "can", "vanadium",
                                     "aluminium", "crystal"])
        # the recursive estimator is the fidelity mode of the powder-like samples
        case["estimator"] = "paper" if (case["sample"] in ("powder", "cylinder", "can") and
                                        rng.random() < 0.25) else "chain"
    elif kind == "batch":
        case["sample"] = rng.choice(["can", "can", "powder", "crystal"])
        case["sims"] = rng.randint(2, 32)
        case["n_tof"] = min(case["n_tof"], 200)
    else:
        case["sample"] = "powder"
    lo, hi = _RANGES[(case["sample"], fp)]
    if case.get("estimator") == "paper":
        hi /= 12.0
    if kind == "chain":
        hi = min(hi, 4e6)
    if kind == "grad":
        hi /= 4.0
    case["n"] = int(_log_uniform(rng, lo, hi)) | 1
    if case["sample"] == "crystal":
        case["ei"] = round(rng.uniform(30.0, 70.0), 2)
        case["rot"] = float(rng.randint(0, 180))
    else:
        case["ei"] = round(_log_uniform(rng, 15.0, 300.0), 2)
    return case


# ---- inputs -------------------------------------------------------------------------------
_CTX = []


def _context():
    if not _CTX:
        _CTX.append(api.Context(torch.cuda.current_device()))
    return _CTX[0]


def _workload(case, seed, ei=None, rot=None, n=None, sim_id=0):
    """The workload of a case: one of the repository's descriptions at the case's energy,
    time bins, orders and count, with its random stream (and its S(Q,E)) from the seed."""
    ei = case["ei"] if ei is None else ei
    n = case["n"] if n is None else n
    rot = case.get("rot", 0.0) if rot is None else rot
    sample = case["sample"]
    make = {"cylinder": lambda: mi.config1(n=n),
            "powder": lambda: mi.config2(n=n, omega_scale=1.0 + 0.01 * (seed % 11 - 5)),
            "can": lambda: mi.powder_in_can(n=n, ei=ei),
            "vanadium": lambda: mi.vanadium_powder(n=n, ei=ei),
            "aluminium": lambda: mi.aluminium_powder(n=n, ei=ei),
            "crystal": lambda: mi.config3(rot_deg=rot, n=n)}[sample]
    wl = make()
    base = wl.detector
    if sample == "cylinder":
        f = math.sqrt(60.0 / ei)
        t0, t1 = 4.2e-3 * f, 4.4e-3 * f
    else:
        t0, t1 = mi.tof_window_for(ei)
    det = dataclasses.replace(base, tof_min_s=t0, tof_max_s=t1, n_tof=case["n_tof"])
    return wl.replace(beam=dataclasses.replace(wl.beam, ei_mev=ei), detector=det,
                      max_orders=case["orders"], seed=seed % (1 << 32), sim_id=sim_id)


def _sweep(case, seed):
    """The simulations of a batch: orientations of one crystal, or an energy sweep with
    log-uniform neutron counts, summing to about the case's n."""
    m = case["sims"]
    if case["sample"] == "crystal":
        return [_workload(case, seed, rot=180.0 * k / max(1, m - 1), n=case["n"] // m + k % 2,
                          sim_id=k) for k in range(m)]
    r = np.random.Generator(np.random.PCG64(seed))
    share = np.exp(r.uniform(math.log(1e-2), 0.0, m))
    n = np.maximum(1, (case["n"] * share / share.sum()).astype(np.int64))
    eis = np.geomspace(case["ei"] / 7.07, case["ei"] * 7.07, m)
    first = _workload(case, seed)
    return [_workload(case, seed, ei=float(eis[k]), n=int(n[k]), sim_id=k).replace(sqe=first.sqe)
            for k in range(m)]


def _target(det, seed):
    """A measured histogram with counting noise: an elastic line on a flat background, the
    line's height varying over the pixels; a few per cent of the bins hold counts."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    t = (torch.arange(det.n_tof, device="cuda", dtype=torch.float64) + 0.5) / det.n_tof
    line = torch.exp(-0.5 * ((t - 0.32) / 0.03) ** 2)
    height = 0.3 * torch.rand(det.n_pixels, 1, device="cuda", dtype=torch.float64, generator=gen)
    return torch.poisson((height * line + 0.004) * (1000.0 / det.n_tof), generator=gen).reshape(-1)


def prepare(case, seed):
    fp = B.FP32 if case["fp"] == 32 else B.FP64
    state = {"case": case, "ctx": _context(), "fp": fp}
    if case["kind"] == "batch":
        wls = _sweep(case, seed)
        # one block of memory for the histograms, so that they are cleared together
        bins = torch.zeros(len(wls), wls[0].detector.n_bins, dtype=torch.float64, device="cuda")
        tallies = torch.zeros(len(wls), B.MCV_NTALLY, dtype=torch.float64, device="cuda")
        state.update(bins=bins, tallies=tallies, batch=state["ctx"].batch(
            wls, fp_mode=fp, hists=[(bins[k], tallies[k]) for k in range(len(wls))]))
        return state
    wl = _workload(case, seed)
    state.update(wl=wl, table=state["ctx"].table(wl))
    if case["kind"] == "grad":
        state.update(target=_target(wl.detector, seed), scale=1e6 / case["n"])
    return state


# ---- one pass -----------------------------------------------------------------------------
def run(state):
    kind, ctx, fp = state["case"]["kind"], state["ctx"], state["fp"]
    if kind == "batch":
        state["bins"].zero_()
        state["tallies"].zero_()
        state["batch"].run()
        return {"hist": state["bins"], "tallies": state["tallies"]}
    wl, table = state["wl"], state["table"]
    if kind == "trace":
        est = B.EST_PAPER if state["case"]["estimator"] == "paper" else B.EST_CHAIN
        counts, tallies = ctx.trace(wl, fp_mode=fp, table=table, sync=False, estimator=est)
        return {"hist": counts, "tallies": tallies}
    if kind == "grad":
        out = ctx.grad(wl, state["target"], state["scale"], fp_mode=fp, table=table, sync=False)
        return {k: out[k] for k in ("loss", "dsqe", "dsig", "hist")}
    beam = ctx.beam(wl, fp_mode=fp, sync=False)
    packets = ctx.trace_packets(wl, fp_mode=fp, table=table, beam_in=beam, sync=False)
    counts, tallies, _ = ctx.detect(wl, packets, events=False, sync=False)
    # the packet slots of orders a neutron did not reach keep their other fields unwritten
    return {"beam": [beam.x, beam.y, beam.vx, beam.vy, beam.vz, beam.t],
            "id": packets.id, "order": packets.order, "hist": counts, "tallies": tallies}


# ---- the work a pass cannot do without ----------------------------------------------------
# arithmetic operations per incident neutron (floating point and integer, counted on an
# instrumented run of each workload; transcendentals as 8)
_OPS = {"powder": 1282.0, "cylinder": 1500.0, "can": 2200.0, "vanadium": 1926.0,
        "aluminium": 2322.0, "crystal": 3.0e4}


def work(case):
    n, sims = case["n"], case.get("sims", 1)
    pixels = 1024 if case["sample"] == "cylinder" else 117760
    hist = 8.0 * pixels * case["n_tof"] * sims
    table = 4.0 * 200 * 400 if case["sample"] in ("powder", "can") else 0.0
    flops = n * _OPS[case["sample"]] * (0.4 + 0.12 * case["orders"])
    nbytes = hist + table + 64.0 * sims
    if case.get("estimator") == "paper":
        flops *= 3.6
    if case["kind"] == "grad":       # the target and the table gradient as well
        nbytes += hist + 2 * table
        flops *= 2.0
    if case["kind"] == "chain":      # stored neutrons written and read, packets likewise
        real = case["fp"] // 8
        nbytes += 2.0 * n * (7 * real + 16) + 2.0 * n * 1.1 * (7 * real + 20)
        nbytes += n * (case["orders"] + 1) * 12.0
    return {"bytes": nbytes, "flops": flops}


# ---- the method in 64 bits ----------------------------------------------------------------
_MASK = 0xFFFFFFFF
_E_CHARGE, _HBAR, _MASS_N = 1.602176634e-19, 1.054571817e-34, 1.67492749804e-27
_E_PER_V2 = 0.5 * _MASS_N / (_E_CHARGE * 1e-3)
_K_PER_V = _MASS_N / _HBAR * 1e-10
_KT_PER_K = 1.380649e-23 / (_E_CHARGE * 1e-3)
_CHUNK = 500_000


def _uniforms(seed, sim, ids, c2, c3):
    """Philox4x32-10 at counters (id lo, id hi, c2, c3): two numbers of 53 bits in (0, 1)."""
    c0, c1 = ids & _MASK, (ids >> 32) & _MASK
    c2 = torch.zeros_like(ids) + c2
    c3 = torch.zeros_like(ids) + c3
    for r in range(10):
        k0, k1 = (seed + r * 0x9E3779B9) & _MASK, (sim + r * 0xBB67AE85) & _MASK
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2
        c0, c1, c2, c3 = (((p1 >> 32) & _MASK) ^ c1 ^ k0, p1 & _MASK,
                          ((p0 >> 32) & _MASK) ^ c3 ^ k1, p0 & _MASK)

    def unit(hi, lo):
        return ((hi << 21) | (lo >> 11)).double() * 2.0 ** -53 + 2.0 ** -54

    return unit(c0, c1), unit(c2, c3)


class _Rays:
    """Packets as equally long columns: x y z dx dy dz v t w id and whatever else is added."""

    def __init__(self, **cols):
        self.__dict__.update(cols)

    def take(self, m):
        return _Rays(**{k: v[m] for k, v in self.__dict__.items()})

    def but(self, **cols):
        return _Rays(**{**self.__dict__, **cols})


def _source(wl, ids):
    b = wl.beam
    u0, u1 = _uniforms(wl.seed, wl.sim_id, ids, 1, 0)
    x, y = (u0 - 0.5) * b.width_m, (u1 - 0.5) * b.height_m
    u0, u1 = _uniforms(wl.seed, wl.sim_id, ids, 2, 0)
    r = b.div_sigma_rad * torch.sqrt(-2.0 * torch.log(u0))
    tx, ty = torch.tan(r * torch.cos(2 * math.pi * u1)), torch.tan(r * torch.sin(2 * math.pi * u1))
    norm = torch.sqrt(1.0 + tx * tx + ty * ty)
    u0, u1 = _uniforms(wl.seed, wl.sim_id, ids, 0, 0)
    e = b.ei_mev * (1.0 + b.ei_rel_sigma * torch.sqrt(-2.0 * torch.log(u0)) *
                    torch.cos(2 * math.pi * u1))
    v = torch.sqrt(e / _E_PER_V2)
    one = torch.ones_like(x)
    rays = _Rays(x=x, y=y, z=-b.z0_m * one, dx=tx / norm, dy=ty / norm, dz=1.0 / norm, v=v,
                 t=(b.l1_m - b.z0_m) * norm / v, w=one, id=ids)
    return rays.take(e > 0)


def _cylinder(rad, r, cx=0.0):
    """Where rays cross the vertical cylinder of that radius: (hit, entry, exit)."""
    a = r.dx * r.dx + r.dz * r.dz
    mid = -(r.x * r.dx + r.z * r.dz) / a
    g = rad * rad - (r.x * r.dz - r.z * r.dx) ** 2 / a
    half = torch.sqrt(torch.clamp(g, min=0.0) / a)
    return g > 0, mid - half, mid + half


def _slab(half, p, d):
    a, b = (-half - p) / d, (half - p) / d
    return torch.minimum(a, b), torch.maximum(a, b)


def _segments(wl, r, s0):
    """The material ahead of each ray beyond distance s0, sorted by entry: entry, exit and
    scatterer, [rays, slots]; empty slots enter at infinity and have no length."""
    inf = torch.full_like(r.x, math.inf)
    entry, leave, which = [], [], []

    def put(j, ok, a, b):
        a = torch.maximum(a, s0)
        ok = ok & (b > a)
        entry.append(torch.where(ok, a, inf))
        leave.append(torch.where(ok, b, inf))
        which.append(torch.full_like(r.id, j))

    for j, s in enumerate(wl.scatterers):
        if s.kind == mi.BLOCK:
            c, q = math.cos(s.rot_y), math.sin(s.rot_y)
            spans = [_slab(0.5 * s.dims[0], c * r.x - q * r.z, c * r.dx - q * r.dz),
                     _slab(0.5 * s.dims[1], r.y, r.dy),
                     _slab(0.5 * s.dims[2], q * r.x + c * r.z, q * r.dx + c * r.dz)]
            a = torch.stack([p[0] for p in spans]).amax(0)
            b = torch.stack([p[1] for p in spans]).amin(0)
            put(j, b > a, a, b)
            continue
        hollow = s.kind == mi.HOLLOW_CYL
        ok, a, b = _cylinder(s.dims[1] if hollow else s.dims[0], r)
        ya, yb = _slab(0.5 * s.dims[-1], r.y, r.dy)
        a = torch.where(r.dy == 0, a, torch.maximum(a, ya))
        b = torch.where(r.dy == 0, b, torch.minimum(b, yb))
        ok = ok & (b > a) & ((r.dy != 0) | (r.y.abs() < 0.5 * s.dims[-1]))
        if not hollow:
            put(j, ok, a, b)
            continue
        inner, ia, ib = _cylinder(s.dims[0], r)
        put(j, ok, a, torch.where(inner, torch.minimum(b, ia), b))
        put(j, ok & inner, torch.maximum(a, ib), b)
    a, order = torch.sort(torch.stack(entry, 1), dim=1, stable=True)
    b, j = (torch.stack(c, 1).gather(1, order) for c in (leave, which))
    return a, b, j, torch.where(torch.isfinite(a), b - a, torch.zeros_like(a))


def _turn(r, m, c2t, s2t, u):
    """The directions of rays m turned by the angle (c2t, s2t) with azimuth 2 pi u."""
    x, y, z = r.dx[m], r.dy[m], r.dz[m]
    near = z.abs() < 0.9
    zero = torch.zeros_like(x)
    e1 = torch.stack([torch.where(near, -y, zero), torch.where(near, x, -z),
                      torch.where(near, zero, y)])
    e1 = e1 / torch.sqrt((e1 * e1).sum(0))
    d = torch.stack([x, y, z])
    e2 = torch.linalg.cross(d, e1, dim=0)
    d = d * c2t + (e1 * torch.cos(2 * math.pi * u) + e2 * torch.sin(2 * math.pi * u)) * s2t
    return d[0], d[1], d[2]


def _isotropic(u0, u1):
    st = 2.0 * torch.sqrt(u0 * (1.0 - u0))
    return st * torch.cos(2 * math.pi * u1), st * torch.sin(2 * math.pi * u1), 2.0 * u0 - 1.0


def _angle(ki, kf, q, below, above):
    """cos and sin of the angle at which |ki - kf| = q, from the offsets of q from the ends."""
    den = 2.0 * ki * kf
    one_m, one_p = below * (q + (ki - kf).abs()) / den, above * (ki + kf + q) / den
    c = torch.where(one_m <= one_p, 1.0 - one_m, one_p - 1.0).clamp(-1.0, 1.0)
    return c, torch.sqrt(torch.clamp(one_m * one_p, min=0.0))


class _Kernels:
    """The scattering kernels of a workload: each draws from `rand(block)` for the rays m of r
    and gives (scatters, dx, dy, dz, speed, weight factor without S, S, table entry)."""

    def __init__(self, wl, table):
        self.wl, self.table = wl, table
        if wl.phonon is not None:
            self._phonon_tables(wl.phonon)

    def _phonon_tables(self, ph):
        J, N, de = len(ph.z), ph.nmax, ph.de
        kt = _KT_PER_K * ph.temperature_K
        e = de * np.arange(1, J + 1)
        z = np.asarray(ph.z, dtype=np.float64) / np.sum(ph.z)
        gamma0 = np.sum(z / (e * np.tanh(e / (2 * kt))))
        nb = 1.0 / np.expm1(e / kt)
        a1 = np.concatenate([(z * nb / (e * gamma0))[::-1], [0.0], z * (nb + 1) / (e * gamma0)])
        rows, cur = [], a1
        for n in range(2, N + 1):
            cur = np.convolve(cur, a1)
            rows.append(np.pad(cur, (N - n) * J))
        b = sum(rows) / (N - 1)
        dev = lambda v: torch.as_tensor(np.ascontiguousarray(v), device="cuda")  # noqa: E731
        self.cdf1, self.cdfb, self.mix = dev(np.cumsum(a1)), dev(np.cumsum(b)), dev(b)
        self.rows, self.J = dev(np.stack(rows)), J
        hb2m = _HBAR ** 2 / (2 * ph.mass_u * 1.66053906660e-27) * 1e20 / (_E_CHARGE * 1e-3)
        self.cw = hb2m * gamma0

    def iso(self, r, rand, sc, sig):
        one = torch.ones_like(r.x)
        dx, dy, dz = _isotropic(*rand(1))
        return one > 0, dx, dy, dz, r.v, one, one, torch.full_like(r.id, -1)

    def sqe(self, r, rand, sc, sig):
        g = self.wl.sqe
        ei, ki = _E_PER_V2 * r.v * r.v, _K_PER_V * r.v
        top = torch.clamp(ei, max=g.e_max)
        (u0, u1), (u2, _) = rand(1), rand(2)
        de = top - g.e_min
        e = g.e_min + u0 * de
        ef = torch.where(top == ei, (1.0 - u0) * de, ei - e)
        ok = (de > 0) & (ef > 0)
        v = torch.sqrt(torch.clamp(ef, min=1e-300) / _E_PER_V2)
        kf = _K_PER_V * v
        q_lo, q_hi = (ki - kf).abs(), torch.clamp(ki + kf, max=g.q_max)
        dq = q_hi - q_lo
        q = q_lo + u1 * dq
        c, s = _angle(ki, kf, q, u1 * dq,
                      torch.where(q_hi == ki + kf, (1.0 - u1) * dq, (ki + kf) - q))
        iq = torch.floor(q / (g.q_max / g.nq)).long()
        ie = torch.floor((e - g.e_min) / ((g.e_max - g.e_min) / g.ne)).long()
        ok = ok & (dq > 0) & (iq >= 0) & (iq < g.nq) & (ie >= 0) & (ie < g.ne)
        entry = torch.where(ok, iq * g.ne + ie, torch.zeros_like(iq))
        dx, dy, dz = _turn(r, slice(None), c, s, u2)
        return ok, dx, dy, dz, v, q * de * dq / (2.0 * ki * ki), self.table[entry], entry

    def phonon(self, r, rand, sc, sig):
        ph, J, N = self.wl.phonon, self.J, self.wl.phonon.nmax
        p0, p1, p2 = ph.p
        ei, ki = _E_PER_V2 * r.v * r.v, _K_PER_V * r.v
        (u0, u1), (u2, u3) = rand(1), rand(2)
        elastic, single = u0 < p0, (u0 >= p0) & (u0 < p0 + p1)
        ex, ey, ez = _isotropic(u2, u3)
        q2 = ki * ki * ((r.dx - ex) ** 2 + (r.dy - ey) ** 2 + (r.dz - ez) ** 2)
        f_el = torch.exp(-self.cw * q2) / p0
        pc = torch.where(single, torch.full_like(u0, p1), torch.full_like(u0, p2))
        ue = (u0 - torch.where(single, torch.full_like(u0, p0),
                               torch.full_like(u0, p0 + p1))) / pc
        find = lambda cdf: torch.searchsorted(cdf, ue * cdf[-1], right=True).clamp(  # noqa: E731
            max=cdf.numel() - 1)
        i1, ib = find(self.cdf1), find(self.cdfb)
        i = torch.where(single, i1 - J, ib - N * J)
        e = (i.double() + (u1 - 0.5)) * ph.de
        ef = ei - e
        v = torch.sqrt(torch.clamp(ef, min=1e-300) / _E_PER_V2)
        kf = _K_PER_V * v
        q_lo = (ki - kf).abs()
        dq = ki + kf - q_lo
        q = q_lo + u2 * dq
        c, s = _angle(ki, kf, q, u2 * dq, (1.0 - u2) * dq)
        w2 = self.cw * q * q
        g = (i + N * J).clamp(0, 2 * N * J)
        many = sum(w2 ** n / math.factorial(n) * self.rows[n - 2][g] for n in range(2, N + 1))
        ratio = torch.where(single, w2, many / self.mix[ib]) * torch.exp(-w2)
        dx, dy, dz = _turn(r, slice(None), c, s, u3)
        pick = lambda a, b: torch.where(elastic, a, b)  # noqa: E731
        return (elastic | (ef > 0), pick(ex, dx), pick(ey, dy), pick(ez, dz), pick(r.v, v),
                pick(f_el, ratio * q * dq / (2.0 * ki * ki) / pc), torch.ones_like(u0),
                torch.full_like(r.id, -1))

    def bragg(self, r, rand, sc, sig):
        d = torch.as_tensor(np.sort(self.wl.bragg.d)[::-1].copy(), device="cuda")
        order = np.argsort(-self.wl.bragg.d, kind="stable")
        cum = torch.as_tensor(np.cumsum(self.wl.bragg.w[order] * self.wl.bragg.d[order]),
                              device="cuda")
        ki = _K_PER_V * r.v
        lam = 2.0 * math.pi / ki
        allowed = (lam[:, None] < 2.0 * d[None, :]).sum(1)
        total = cum[(allowed - 1).clamp(min=0)]
        u0, u1 = rand(1)
        pick = torch.searchsorted(cum, u0 * total, right=True)
        pick = torch.minimum(pick, (allowed - 1).clamp(min=0))
        s = (lam / (2.0 * d[pick])).clamp(max=1.0)
        dx, dy, dz = _turn(r, slice(None), 1.0 - 2.0 * s * s,
                           2.0 * s * torch.sqrt((1.0 - s) * (1.0 + s)), u1)
        return (allowed > 0, dx, dy, dz, r.v, 0.5 * lam * lam * total / sig,
                torch.ones_like(u0), torch.full_like(r.id, -1))

    _BONDS = ((1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1))

    def _crystal_q(self, sc, r, df, ef):
        """Q in the crystal frame, and dQ/dEf."""
        c, s = math.cos(sc.rot_y), math.sin(sc.rot_y)
        ki, kf = _K_PER_V * r.v, _K_PER_V * torch.sqrt(torch.clamp(ef, min=0.0) / _E_PER_V2)
        turn = lambda x, y, z: (s * x + c * z, c * x - s * z, y)  # noqa: E731
        q = turn(r.dx * ki - df[0] * kf, r.dy * ki - df[1] * kf, r.dz * ki - df[2] * kf)
        return q, turn(*df), kf

    def _dynamical(self, q):
        half = 0.25 * self.wl.bvk.a_A
        D = [torch.zeros_like(q[0]) for _ in range(6)]
        for n in self._BONDS:
            f = 2.0 * torch.sin(half * (q[0] * n[0] + q[1] * n[1] + q[2] * n[2])) ** 2
            for k, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
                D[k] = D[k] + f * (n[i] * n[j])
        return D

    def bvk(self, r, rand, sc, sig):
        b = self.wl.bvk
        mass = b.mass_u * 1.66053906660e-27
        unit = _HBAR * math.sqrt(b.phi_Nm / mass) / (_E_CHARGE * 1e-3)
        top = _HBAR * math.sqrt(24.0 * b.phi_Nm / mass) / (_E_CHARGE * 1e-3)
        (u0, u1), (u2, u3) = rand(1), rand(2)
        df = _isotropic(u0, u1)
        mode = torch.floor(6.0 * u2).clamp(0, 5)
        branch, sign = mode % 3, torch.where(mode < 3, 1.0, -1.0).double()
        ei, ki = _E_PER_V2 * r.v * r.v, _K_PER_V * r.v
        lo = torch.where(sign > 0, torch.zeros_like(ei), ei)
        step = torch.where(sign > 0, ei, torch.full_like(ei, top)) / 32.0

        def positive(ef):
            """Ei - Ef - sign hw(Q(Ef)) > 0: from how many eigenvalues lie below the square
            of the energy transfer (the signs of the leading minors of D - lambda)."""
            q, _, _ = self._crystal_q(sc, r, df, ef)
            D = self._dynamical(q)
            x = sign * (ei - ef) / unit
            lam = x * x
            p, qq, s = D[0] - lam, D[1] - lam, D[2] - lam
            m2 = p * qq - D[3] ** 2
            m3 = (p * (qq * s - D[5] ** 2) - D[3] * (D[3] * s - D[5] * D[4]) +
                  D[4] * (D[3] * D[5] - qq * D[4]))
            below = ((p < 0).int() + ((m2 < 0) != (p < 0)).int() + ((m3 < 0) != (m2 < 0)).int())
            more = (x > 0) & (below > branch)   # hw < the (positive) energy transfer
            return torch.where(sign > 0, more, ~more)

        grid = torch.stack([positive(lo + k * step) for k in range(33)])
        change = grid[1:] != grid[:-1]
        roots = change.sum(0)
        pick = torch.floor(u3 * roots).long().clamp(min=0)
        pick = torch.minimum(pick, (roots - 1).clamp(min=0))
        at = (torch.cumsum(change.int(), 0) == pick + 1).int().argmax(0)
        first = grid.gather(0, at[None])[0]
        ea, eb = lo + at * step, lo + (at + 1) * step
        for _ in range(50):
            mid = 0.5 * (ea + eb)
            same = positive(mid) == first
            ea, eb = torch.where(same, mid, ea), torch.where(same, eb, mid)
        ef = 0.5 * (ea + eb)
        q, dirs, kf = self._crystal_q(sc, r, df, ef)
        D = self._dynamical(q)
        full = torch.stack([D[0], D[3], D[4], D[3], D[1], D[5], D[4], D[5], D[2]], 1)
        # LAPACK on the host: the device's batched solver is slow for many small matrices
        val, vec = torch.linalg.eigh(full.reshape(-1, 3, 3).cpu())
        k = branch.long()
        lam = val.to(ei.device).gather(1, k[:, None])[:, 0].clamp(min=0.0)
        e = vec.to(ei.device).gather(2, k[:, None, None].expand(-1, 3, 1))[:, :, 0].T
        hw = unit * torch.sqrt(lam)
        dk = -kf / (2.0 * ef)
        slope = torch.zeros_like(ef)
        for n in self._BONDS:
            ph = 0.5 * b.a_A * (q[0] * n[0] + q[1] * n[1] + q[2] * n[2])
            dph = 0.5 * b.a_A * dk * (dirs[0] * n[0] + dirs[1] * n[1] + dirs[2] * n[2])
            slope = slope + torch.sin(ph) * dph * (e[0] * n[0] + e[1] * n[1] + e[2] * n[2]) ** 2
        gp = -1.0 - sign * unit * slope / (2.0 * torch.sqrt(lam))
        nb = 1.0 / torch.expm1(hw / (_KT_PER_K * b.temperature_K))
        hb2m = _HBAR ** 2 / (2 * mass) * 1e20 / (_E_CHARGE * 1e-3)
        q2 = q[0] ** 2 + q[1] ** 2 + q[2] ** 2
        qe = q[0] * e[0] + q[1] * e[1] + q[2] * e[2]
        f = (6.0 * roots * (kf / ki) * torch.exp(-q2 * b.msd_A2 / 3.0) * hb2m * qe * qe / hw *
             torch.where(sign > 0, nb + 1.0, nb) / gp.abs())
        ok = (roots > 0) & (ef > 0) & (hw >= 1e-3)
        return (ok, *df, torch.sqrt(torch.clamp(ef, min=0.0) / _E_PER_V2), f,
                torch.ones_like(ef), torch.full_like(r.id, -1))

    def scatter(self, r, j, rand, u_k):
        """The kernels of the rays' scatterers j, picked by u_k in proportion to their cross
        sections, applied to all rays."""
        out = None
        for s, sc in enumerate(self.wl.scatterers):
            total = sum(sig for _, sig in sc.kernels)
            for k, (kind, sig) in enumerate(sc.kernels):
                name = {mi.K_ISO: "iso", mi.K_SQE: "sqe", mi.K_BVK: "bvk",
                        mi.K_PHONON: "phonon", mi.K_BRAGG: "bragg"}[kind]
                mine = (j == s)
                if len(sc.kernels) == 2:
                    mine = mine & ((u_k * total < sc.kernels[0][1]) == (k == 0))
                got = getattr(self, name)(r, rand, sc, sig)
                out = got if out is None else tuple(torch.where(mine, a, b)
                                                    for a, b in zip(got, out))
        return out


def _detect(det, r, u):
    """First tube met (or the ideal surface): (hit, bin or -2, probability absorbed)."""
    hit, _, s = _cylinder(det.radius_m, r)
    hit = hit & (s > 0) & torch.isfinite(s)
    y, phi = r.y + s * r.dy, torch.atan2(r.x + s * r.dx, r.z + s * r.dz)
    if det.kind == mi.DET_SURFACE:
        half = 0.5 * det.height_m
        hit = hit & (y >= -half) & (y < half)
        ip = torch.floor((phi + math.pi) / (2 * math.pi) * det.n_phi).long().clamp(0, det.n_phi - 1)
        iy = torch.floor((y + half) / det.height_m * det.n_y).long().clamp(0, det.n_y - 1)
        return hit, _bin(det, ip * det.n_y + iy, r.t + s / r.v), torch.ones_like(s)
    row = torch.full_like(r.id, -1)
    for i in reversed(range(det.n_rows)):
        row = torch.where((y - det.row_y_m[i]).abs() <= 0.5 * det.tube_len_m, i, row)
    hit = hit & (row >= 0)
    at = row.clamp(min=0)
    packs = torch.tensor(det.packs[:det.n_rows], device=r.x.device)
    offset = torch.cumsum(packs, 0) - packs
    tpp = det.tubes_per_pack
    period = tpp * det.tube_pitch_m + det.pack_gap_m
    arc = (phi - det.phi0_rad) * det.radius_m
    p = torch.floor(arc / period)
    k = torch.floor((arc - p * period) / det.tube_pitch_m).clamp(max=tpp - 1)
    near = (p * tpp + k).long()
    y_row = torch.tensor(det.row_y_m[:det.n_rows], device=r.x.device, dtype=torch.float64)[at]
    ya, yb = _slab(0.5 * det.tube_len_m, r.y - y_row, r.dy)
    best = torch.full_like(s, math.inf)
    tube, out = torch.zeros_like(near), torch.zeros_like(s)
    for c in (near - 1, near, near + 1):
        pc = torch.floor(c.double() / tpp)
        mid = det.phi0_rad + (pc * period + (c - pc * tpp + 0.5) * det.tube_pitch_m) / det.radius_m
        ux, uz = torch.sin(mid), torch.cos(mid)
        o_r, o_t = r.x * ux + r.z * uz - det.radius_m, r.x * uz - r.z * ux
        d_r, d_t = r.dx * ux + r.dz * uz, r.dx * uz - r.dz * ux
        a = r.dx * r.dx + r.dz * r.dz
        g = det.tube_r_m ** 2 - (o_r * d_t - o_t * d_r) ** 2 / a
        half = torch.sqrt(torch.clamp(g, min=0.0) / a)
        m = -(o_r * d_r + o_t * d_t) / a
        s_in = torch.maximum(torch.maximum(m - half, ya), torch.zeros_like(m))
        s_out = torch.minimum(m + half, yb)
        ok = (c >= 0) & (c < packs[at] * tpp) & (g > 0) & (s_out > s_in) & (s_in < best)
        tube, out, best = (torch.where(ok, n, o) for n, o in ((c, tube), (s_out, out), (s_in, best)))
    hit = hit & torch.isfinite(best)
    best = torch.where(hit, best, torch.zeros_like(best))
    mu = 100.0 * det.he3_n_per_A3 * det.he3_sig_abs_b * 2200.0 / r.v
    absorbed = -torch.expm1(-mu * torch.where(hit, out - best, torch.zeros_like(best)))
    s_abs = best - torch.log1p(-u * absorbed) / mu
    y_abs = r.y + s_abs * r.dy - (y_row - 0.5 * det.tube_len_m)
    iy = torch.floor(y_abs / (det.tube_len_m / det.pixels_per_tube)).long()
    pixel = (offset[at] * tpp + tube) * det.pixels_per_tube + iy.clamp(0, det.pixels_per_tube - 1)
    return hit, _bin(det, pixel, r.t + s_abs / r.v), absorbed


def _bin(det, pixel, tof):
    b = torch.floor((tof - det.tof_min_s) / ((det.tof_max_s - det.tof_min_s) / det.n_tof))
    return torch.where((b >= 0) & (b < det.n_tof), pixel * det.n_tof + b.long(), -2)


def _mu(wl, j, v):
    """Attenuation and scattering coefficients (1/m) of scatterers j at speed v."""
    n = torch.tensor([100.0 * s.n_per_A3 for s in wl.scatterers], device=v.device,
                     dtype=torch.float64)
    sig = torch.tensor([sum(k[1] for k in s.kernels) for s in wl.scatterers], device=v.device,
                       dtype=torch.float64)
    sab = torch.tensor([s.sig_abs_b * 2200.0 for s in wl.scatterers], device=v.device,
                       dtype=torch.float64)
    vv = v.reshape(-1, *([1] * (j.dim() - 1)))
    return n[j] * (sig[j] + sab[j] / vv), (n * sig)[j]


def _tally_detected(hist, tallies, hit, b, w):
    inside, out = hit & (b >= 0), hit & (b < 0)
    if hist is not None:
        hist.index_add_(0, b[inside], w[inside])
    for k, v in ((1, w[inside].sum()), (2, w[out].sum()), (3, inside.sum()), (4, out.sum()),
                 (5, (~hit).sum()), (7, torch.tensor(hit.numel()))):
        tallies[k] += v


def _chain(wl, table, hist, tallies, grad=None):
    """The bounded chain over all neutrons of wl.  grad: (dchi2/dI, dS, dsig) to add the
    derivatives along the same paths to instead of the histogram."""
    kernels = _Kernels(wl, table)
    sc0 = wl.scatterers[0]
    n0, sig0 = 100.0 * sc0.n_per_A3, sum(k[1] for k in sc0.kernels)
    for first in range(0, wl.n, _CHUNK):
        ids = torch.arange(first, min(wl.n, first + _CHUNK), device="cuda")
        r = _source(wl, ids)
        hist_s = []          # per order: (scattering factor without S, S, entry) of the rays
        d_abs = torch.zeros_like(r.x)
        d_sig = torch.zeros_like(r.x)
        for o in range(wl.max_orders + 1):
            a, b, j, length = _segments(wl, r, torch.zeros_like(r.x))
            mu, _ = _mu(wl, j, r.v)
            total, atten = length.sum(1), torch.exp(-(mu * length).sum(1))
            we = r.w * atten
            if o == 0:
                tallies[0] += we.sum()
                tallies[6] += (total > 0).sum()
            elif grad is None or grad[0] is not None:
                u = _uniforms(wl.seed, wl.sim_id, r.id, 4 * (o + 1) + 3, 0)[0]
                hit, bins, absorbed = _detect(wl.detector, r, u)
                if grad is None:
                    _tally_detected(hist, tallies, hit, bins, we * absorbed)
                else:
                    g, ds, dsig = grad
                    m = hit & (bins >= 0)
                    gb, per = g[bins[m]], (atten * absorbed)[m]
                    w = we[m] * absorbed[m] * gb
                    dsig[0] += (w * (d_abs[m] - n0 * 2200.0 / r.v[m] * total[m])).sum()
                    dsig[1] += (w * (d_sig[m] - n0 * total[m])).sum()
                    for k in range(o):
                        prod = gb * per
                        for q, (fac, s, _) in enumerate(hist_s):
                            prod = prod * fac[m] * (s[m] if q != k else 1.0)
                        ds.index_add_(0, hist_s[k][2][m], prod)
            if o == wl.max_orders:
                break
            live = total > 0
            r, a, j, length, mu, total = (r.take(live), a[live], j[live], length[live], mu[live],
                                          total[live])
            u_pt, u_k = _uniforms(wl.seed, wl.sim_id, r.id, 4 * (o + 1), 0)
            ell = u_pt * total
            ends = torch.cumsum(length, 1)
            last = ((length > 0).sum(1) - 1).clamp(min=0)
            seg = torch.minimum((ell[:, None] >= ends).sum(1), last)
            col = lambda v: v.gather(1, seg[:, None])[:, 0]  # noqa: E731
            part = ell - (col(ends) - col(length))
            before = torch.arange(length.shape[1], device="cuda")[None, :] < seg[:, None]
            tau = (mu * length * before).sum(1) + col(mu) * part
            s = col(a) + part
            js = col(j)
            fac = _mu(wl, js, r.v)[1] * total * torch.exp(-tau)
            v_in, through = r.v, (length * before).sum(1) + part
            r = r.but(x=r.x + s * r.dx, y=r.y + s * r.dy, z=r.z + s * r.dz, t=r.t + s / r.v)
            ok, dx, dy, dz, v, rest, sv, entry = kernels.scatter(
                r, js, lambda block: _uniforms(wl.seed, wl.sim_id, r.id, 4 * (o + 1) + block, 0),
                u_k)
            r = r.but(dx=dx, dy=dy, dz=dz, v=v, w=r.w * fac * rest * sv)
            keep = ok & ~(r.w < wl.min_prob)
            if grad is None:
                keep = keep & (r.w != 0)
            else:
                d_abs = (d_abs[live] - n0 * 2200.0 / v_in * through)[keep]
                d_sig = (d_sig[live] - n0 * through + 1.0 / sig0)[keep]
                hist_s = [tuple(c[live][keep] for c in h) for h in hist_s]
                hist_s.append(((fac * rest)[keep], sv[keep], entry[keep]))
            r = r.take(keep)
            if not r.x.numel():
                break


def _recursion(wl, table, hist, tallies):
    """The paper's recursion: every interaction of node x gives the transmitted packet 2x and
    the scattered packet 2x + 1; all packets of a chunk advance together."""
    kernels = _Kernels(wl, table)
    key = wl.sim_id ^ 0x80000000
    for first in range(0, wl.n, _CHUNK):
        r = _source(wl, torch.arange(first, min(wl.n, first + _CHUNK), device="cuda"))
        r = r.but(m=torch.zeros_like(r.id), node=torch.ones_like(r.id), s0=torch.zeros_like(r.x),
                  j=torch.full_like(r.id, -1))
        while r.x.numel():
            a, b, j, length = _segments(wl, r, r.s0)
            mu, _ = _mu(wl, j, r.v)
            tallies[6] += ((r.node == 1) & (length[:, 0] > 0)).sum()
            mine = (j == r.j[:, None]) & (length > 0)
            same = mine.any(1)
            leaves = ~same & ((length[:, 0] <= 0) | (r.m >= wl.max_orders))
            w = r.w * torch.exp(-(mu * length).sum(1))
            tallies[0] += w[leaves & (r.m == 0)].sum()
            out = leaves & (r.m > 0)
            gone = r.take(out)
            c2, c3 = (gone.node & 0x3FFFFFFF) << 2, gone.node >> 30
            hit, bins, absorbed = _detect(wl.detector, gone,
                                          _uniforms(wl.seed, key, gone.id, c2 + 3, c3)[0])
            _tally_detected(hist, tallies, hit, bins, w[out] * absorbed)
            on = ~leaves & ~(r.w < wl.min_prob)
            seg = torch.where(same, mine.int().argmax(1), torch.zeros_like(r.id))
            col = lambda v: v.gather(1, seg[:, None])[:, 0][on]  # noqa: E731
            a, b, j, length, mu = (col(c) for c in (a, b, j, length, mu))
            r = r.take(on)
            through = r.but(s0=b, w=r.w * torch.exp(-mu * length), node=2 * r.node,
                            j=torch.full_like(r.id, -1))
            rand = lambda block: _uniforms(wl.seed, key, r.id,  # noqa: E731
                                           ((r.node & 0x3FFFFFFF) << 2) + block, r.node >> 30)
            u_pt, u_k = rand(0)
            s = a + u_pt * length
            at = r.but(x=r.x + r.dx * s, y=r.y + r.dy * s, z=r.z + r.dz * s, t=r.t + s / r.v)
            ok, dx, dy, dz, v, rest, sv, _ = kernels.scatter(at, j, rand, u_k)
            w = r.w * _mu(wl, j, r.v)[1] * length * torch.exp(-mu * u_pt * length) * rest * sv
            to = at.but(dx=dx, dy=dy, dz=dz, v=v, w=w, m=r.m + 1, node=2 * r.node + 1,
                        s0=torch.zeros_like(s), j=torch.where(r.m + 1 < wl.max_orders, j, -1))
            to = to.take(ok)
            r = _Rays(**{k: torch.cat([getattr(through, k), getattr(to, k)])
                         for k in to.__dict__})


def exact(case, seed):
    """What `run` gives, in 64 bits.  The tallies of an FP32 run have no such value: FP32 ends
    the histories whose weight leaves its range, and the tallies count packets."""
    wls = _sweep(case, seed) if case["kind"] == "batch" else [_workload(case, seed)]
    nb = wls[0].detector.n_bins
    hist = torch.zeros(len(wls), nb, dtype=torch.float64, device="cuda")
    tallies = torch.zeros(len(wls), B.MCV_NTALLY, dtype=torch.float64, device="cuda")
    table = None
    if wls[0].sqe is not None:
        table = torch.as_tensor(wls[0].sqe.table, device="cuda").double().reshape(-1)
    trace = _recursion if case.get("estimator") == "paper" else _chain
    for k, wl in enumerate(wls):
        trace(wl, table, hist[k], tallies[k])
    if case["kind"] == "grad":
        target, scale = _target(wls[0].detector, seed), 1e6 / case["n"]
        den = target.clamp(min=1.0)
        diff = scale * hist[0] - target
        ds = torch.zeros_like(table)
        dsig = torch.zeros(2, dtype=torch.float64, device="cuda")
        _chain(wls[0], table, None, tallies[0], grad=(2.0 * scale * diff / den, ds, dsig))
        return {"loss": (diff * diff / den).sum().reshape(1), "dsqe": ds, "dsig": dsig,
                "hist": hist[0]}
    counted = tallies if case["fp"] == 64 else None
    if case["kind"] == "batch":
        return {"hist": hist, "tallies": counted}
    counted = counted[0] if counted is not None else None
    if case["kind"] == "trace":
        return {"hist": hist[0], "tallies": counted}
    if counted is not None:
        counted[6] = 0.0     # the detector does not see which neutrons met the sample
    r = _source(wls[0], torch.arange(case["n"], device="cuda"))
    return {"beam": [r.x, r.y, r.dx * r.v, r.dy * r.v, r.dz * r.v, r.t], "id": None,
            "order": None, "hist": hist[0], "tallies": counted}
