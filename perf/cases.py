"""Performance cases of the spherical Radon transform: what a program that
uses this package has it compute, from gradient-check volumes to the 256^3
workload.

A case names a geometry (volume edge and slabs, sensor columns, rings, radius
bins), the plan's options, a batch and the calls made: forward, adjoint, both,
the gradient of a data misfit, or the forward on host buffers.  `exact`
computes the same discrete operator in 64 bits with torch alone: every circle
is cut at the grid's lines and each arc goes to the cell that holds it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2402_15641_gb300.autograd import srt as differentiable_srt
from paper_2402_15641_gb300.srt import Geometry, Plan


def _case(name, call, ms, n_phi, n_ell, spacing, radius, mz=None, n_zs=None, dz=None, ring_shift=0.0,
          ring_pitch=1.0, phi0=0.0, batch=1, weights="fp32", rho_linear=False, voxel_linear=False):
    """ring_shift (in slabs) and ring_pitch (ring spacing over slab spacing)
    place the rings; 0 and 1 put them at the slab centres."""
    mz = ms if mz is None else mz
    c = dict(call=call, ms=ms, mz=mz, n_phi=n_phi, n_zs=mz if n_zs is None else n_zs, n_ell=n_ell,
             dxy=spacing, dz=spacing if dz is None else dz, radius=radius, ring_shift=ring_shift,
             ring_pitch=ring_pitch, phi0=phi0, batch=batch, weights=weights, rho_linear=rho_linear,
             voxel_linear=voxel_linear)
    return dict(c, name=name) if name else c


def _serving(name, call, edge, n_phi, **kw):
    """A request of the serving mix: 25.6 mm field, radius bins 4 per voxel."""
    return _case(name, call, edge, n_phi, 4 * edge, 25.6 / edge, 20.0, **kw)


def listed():
    return [
        # the gradient-check volume: a pair of calls so small that launches and latency are all there is
        _case("fd16_pair", "pair", 16, 32, 48, 0.5, 12.0),
        # the smallest parity workload, one interactive forward
        _case("ball32_forward", "forward", 32, 64, 96, 0.5, 12.0),
        # a batch that the serving loop forms from queued small requests
        _serving("serve64_batch8_forward", "forward", 64, 128, batch=8),
        # one small adjoint request as it arrives
        _serving("serve96_adjoint", "adjoint", 96, 256),
        # the serving mix's largest volume
        _serving("serve192_forward", "forward", 192, 256),
        # a scanner whose sizes are nobody's multiples and whose rings are not spaced like the slabs:
        # rows that are no whole float4s, A2 stored entry by entry, every sensor column stored
        _case("ragged_pair", "pair", 75, 90, 201, 0.3, 22.0, mz=53, n_zs=41, dz=0.37, ring_shift=0.3,
              ring_pitch=1.21, phi0=0.2),
        # one iteration of a least-squares reconstruction at the reconstruction size: value and gradient
        _case("lsq128_gradient", "gradient", 128, 256, 512, 0.2, 20.0),
        # the same operator held in 16-bit entries, both directions
        _case("bf16_128_pair", "pair", 128, 256, 512, 0.2, 20.0, weights="bf16"),
        # the smoother bases (bilinear voxels, intermediate linear in rho), both directions
        _case("linear128_pair", "pair", 128, 256, 512, 0.2, 20.0, rho_linear=True, voxel_linear=True),
        # an offline program whose data lie in pinned host memory: copies inside the call
        _case("host128_forward", "host_forward", 128, 256, 512, 0.2, 20.0),
        # the benchmark workload, each direction by itself
        _case("volume256_forward", "forward", 256, 256, 768, 0.1, 20.0),
        _case("volume256_adjoint", "adjoint", 256, 256, 768, 0.1, 20.0),
    ]


def draw(rng):
    """Any volume of 16 to 256 voxels an edge with 1 to 16 of them in a call,
    rings at the slab centres, shifted or spaced otherwise, the options
    above; redrawn while it costs more than the 256^3 forward."""
    most = work(listed()[-2])["flops"]
    while True:
        edge = round(math.exp(rng.uniform(math.log(16), math.log(256))))
        edge = edge if rng.random() < 0.35 else max(16, 4 * round(edge / 4))
        mz = edge if rng.random() < 0.5 else max(8, round(edge * rng.uniform(0.5, 1.3)))
        n_phi = rng.choice([32, 64, 96, 128, 192, 256, 256, round(rng.uniform(24, 256))])
        n_ell = round(edge * rng.uniform(2.5, 4.0))
        field = rng.uniform(8.0, 25.6)
        spacing = field / edge
        rings = rng.choice(["centres", "centres", "centres", "shifted", "other"])
        n_zs = mz if rings == "centres" else max(4, round(mz * rng.uniform(0.6, 1.2)))
        call = rng.choice(["forward", "adjoint", "pair", "gradient", "host_forward"])
        batch = rng.choice([1, 1, 1, 1, 2, 3, 4, 8, 16]) if call in ("forward", "adjoint") else 1
        c = _case(None, call, edge, n_phi, n_ell, spacing, rng.uniform(0.8, 0.95) * field, mz=mz,
                  n_zs=n_zs, dz=spacing * rng.choice([1.0, 1.0, rng.uniform(0.7, 1.5)]),
                  ring_shift=0.0 if rings == "centres" else rng.uniform(-3.0, 3.0),
                  ring_pitch=rng.uniform(0.8, 1.3) if rings == "other" else 1.0,
                  phi0=rng.choice([0.0, 0.0, 0.0, rng.uniform(0.0, 1.0)]), batch=batch,
                  weights=rng.choice(["fp32", "fp32", "fp32", "bf16"]), rho_linear=rng.random() < 0.2,
                  voxel_linear=rng.random() < 0.2)
        if work(c)["flops"] <= most:
            return c


# ------------------------------------------------------------------ geometry
def _rings(c):
    """zs_lo, zs_hi of the case's rings; at the slab centres they span the volume."""
    pitch = c["ring_pitch"] * c["dz"]
    mid, half = c["ring_shift"] * c["dz"], 0.5 * c["n_zs"] * pitch
    if c["n_zs"] == c["mz"] and c["ring_shift"] == 0.0 and c["ring_pitch"] == 1.0:
        half = 0.5 * (c["mz"] * c["dz"])
    return mid - half, mid + half


def _radii(c):
    """ell_lo, ell_hi: the in-plane half diagonal on both sides of the radius."""
    r = c["ms"] * c["dxy"] / math.sqrt(2.0)
    return c["radius"] - r, c["radius"] + r


def _geometry(c):
    (z0, z1), (l0, l1) = _rings(c), _radii(c)
    return Geometry(c["ms"], c["mz"], c["dxy"], c["dz"], c["radius"], c["n_phi"], c["phi0"], c["n_zs"],
                    z0, z1, c["n_ell"], l0, l1, weight_dtype=c["weights"], rho_linear=c["rho_linear"],
                    voxel_linear=c["voxel_linear"])


# -------------------------------------------------------------------- inputs
def _volume(c, seed, device):
    """Balls and vessel-like blobs of random place, size and amplitude."""
    g = np.random.default_rng(seed)
    x = (torch.arange(c["ms"], device=device) - (c["ms"] - 1) / 2) * c["dxy"]
    z = (torch.arange(c["mz"], device=device) - (c["mz"] - 1) / 2) * c["dz"]
    hx, hz = 0.5 * c["ms"] * c["dxy"], 0.5 * c["mz"] * c["dz"]
    f = torch.zeros((c["batch"], c["ms"], c["ms"], c["mz"]), device=device)
    for b in range(c["batch"]):
        for _ in range(12):
            a = g.uniform(0.1, 0.35) * min(hx, hz)
            p = [g.uniform(a - h, h - a) for h in (hx, hx, hz)]
            d = torch.sqrt((x[:, None, None] - p[0]) ** 2 + (x[None, :, None] - p[1]) ** 2
                           + (z[None, None, :] - p[2]) ** 2)
            f[b] += g.uniform(0.2, 1.0) * torch.clamp((a - d) / c["dxy"] + 0.5, 0.0, 1.0)
        for _ in range(24):
            s = g.uniform(0.02, 0.06) * hx + 0.5 * c["dxy"]
            p = [g.uniform(-0.9, 0.9) * h for h in (hx, hx, hz)]
            e = [torch.exp(-0.5 * ((t - q) / s) ** 2) for t, q in zip((x, x, z), p)]
            f[b] += g.uniform(0.2, 1.0) * e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :]
    return f


def _noise(c, seed, device):
    """N(0, 1) of measurement shape."""
    gen = torch.Generator(device=device).manual_seed(seed)
    return torch.randn((c["batch"], c["n_phi"], c["n_zs"], c["n_ell"]), generator=gen, device=device)


def _inputs(c, seed, device):
    """The call's inputs, one item where the batch is one."""
    f = None if c["call"] == "adjoint" else _volume(c, seed, device)
    p = _noise(c, seed, device) if c["call"] in ("adjoint", "pair", "gradient") else None
    if c["batch"] == 1:
        f, p = (t if t is None else t[0] for t in (f, p))
    return f, p


def prepare(case, seed):
    plan = Plan(_geometry(case))
    f, p = _inputs(case, seed, plan.device)
    s = dict(plan=plan, call=case["call"], f=f, p=p)
    if case["call"] == "host_forward":
        s["f"] = f.cpu().pin_memory()
        s["out"] = torch.empty(plan.geom.p_shape, dtype=torch.float32).pin_memory()
    if case["call"] == "gradient":
        s["f"] = f.requires_grad_(True)
    return s


def run(state):
    plan, call, f, p = state["plan"], state["call"], state["f"], state["p"]
    if call == "forward":
        return plan.forward(f)
    if call == "adjoint":
        return plan.adjoint(p)
    if call == "pair":
        return {"p": plan.forward(f), "f": plan.adjoint(p)}
    if call == "host_forward":
        return plan.forward_host(f, state["out"])
    # gradient of 1/2 ||A f - p||^2 through autograd: forward, then the adjoint of the residual
    q = differentiable_srt(f, plan)
    r = q - p
    (grad,) = torch.autograd.grad(0.5 * (r * r).sum(), f)
    return {"p": q.detach(), "gradient": grad}


# ---------------------------------------------------------------------- work
def _entries(c):
    """Entries of A1 and A2, from the mean number of grid lines that a unit
    of arc crosses (no entry is enumerated)."""
    l0, l1 = _radii(c)
    dl, side = (l1 - l0) / c["n_ell"], c["ms"] * c["dxy"]
    n1 = c["n_phi"] * side * side / dl * (4.0 / math.pi) / c["dxy"]
    z0, z1 = _rings(c)
    h = z0 + (np.linspace(0.02, 0.98, 16)) * (z1 - z0)
    l = l0 + np.linspace(0.01, 0.99, 48) * (l1 - l0)
    t = (np.arange(512) + 0.5) * math.pi / 512
    z = h[:, None, None] + l[None, :, None] * np.cos(t)
    rho = l[:, None] * np.sin(t)
    inside = (np.abs(z) <= 0.5 * c["mz"] * c["dz"]) & (rho >= l0) & (rho <= l1)
    lines = l[:, None] * (np.sin(t) / c["dz"] + np.abs(np.cos(t)) / dl) * math.pi / 512
    n2 = c["n_zs"] * c["n_ell"] * float((inside * lines).sum(-1).mean())
    return n1 * (2.0 if c["voxel_linear"] else 1.0), n2 * (1.5 if c["rho_linear"] else 1.0)


def work(case):
    n1, n2 = _entries(case)
    b = case["batch"]
    f = 4 * b * case["ms"] ** 2 * case["mz"]
    p = 4 * b * case["n_phi"] * case["n_zs"] * case["n_ell"]
    one = 2.0 * b * (n1 * case["mz"] + n2 * case["n_phi"])
    twice = case["call"] in ("pair", "gradient")
    # gradient: p is the data read and the prediction returned, the residual stays inside
    return {"bytes": (2 if twice else 1) * (f + p), "flops": (2 if twice else 1) * one}


def tolerance(case):
    # 32-bit sums of a few hundred terms, in one order or another: against 64 bits 3e-8 to 2e-7 for
    # volumes (all terms of one sign) and up to 8e-7 for noise (the sums cancel); entries of 16 bits are
    # the same rounded numbers on both sides
    return {"rel": 3e-6}


# --------------------------------------------------------------------- exact
class _Triples:
    """(row, column, value) entries gathered chunk by chunk, equal places
    summed, as one sparse matrix in 64 bits."""

    def __init__(self, rows, cols):
        self.rows, self.cols, self.key, self.val = rows, cols, [], []

    def add(self, row, col, val, keep):
        self.key.append((row * self.cols + col)[keep])
        self.val.append(val[keep])

    def matrix(self, weights, transpose):
        key, val = torch.cat(self.key), torch.cat(self.val)
        self.key, self.val = [], []
        if transpose:
            key = key % self.cols * self.rows + torch.div(key, self.cols, rounding_mode="floor")
        rows, cols = (self.cols, self.rows) if transpose else (self.rows, self.cols)
        key, order = torch.sort(key)
        key, place = torch.unique_consecutive(key, return_inverse=True)
        val = torch.zeros(len(key), dtype=val.dtype, device=val.device).index_add_(0, place, val[order])
        if weights == "bf16":
            val = val.to(torch.bfloat16).to(val.dtype)
        row = torch.div(key, cols, rounding_mode="floor")
        start = torch.searchsorted(row, torch.arange(rows + 1, device=key.device))
        return torch.sparse_csr_tensor(start, key - row * cols, val, (rows, cols))


def _cell(x, lo, step, n):
    i = torch.floor((x - lo) / step).long()
    return i.clamp(0, n - 1), (i >= 0) & (i < n)


def _node(x, first, step, n):
    """The two nodes around x, with their hats as a + b x; beyond the outer
    nodes the outer one alone, at 1."""
    i = torch.floor((x - first) / step).long()
    inner = ((i >= 0) & (i < n - 1)).to(x.dtype)
    i0 = i.clamp(0, n - 1)
    i1 = torch.where(inner > 0, i0 + 1, i0).clamp(max=n - 1)
    b = inner / step
    b0 = b * (first + i0.to(x.dtype) * step)
    return (i0, 1.0 + b0, -b), (i1, -b0, b)


def _plane(c, dev):
    """A1: row (sensor column, radius), column (ix, iy)."""
    ms, d, n = c["ms"], c["dxy"], c["n_ell"]
    l0, l1 = _radii(c)
    half, dl = 0.5 * ms * d, (l1 - l0) / n
    phi = c["phi0"] + 2.0 * math.pi * torch.arange(c["n_phi"], dtype=torch.float64, device=dev) / c["n_phi"]
    cx = (c["radius"] * torch.cos(phi)).repeat_interleave(n)
    cy = (c["radius"] * torch.sin(phi)).repeat_interleave(n)
    r = (l0 + (torch.arange(n, dtype=torch.float64, device=dev) + 0.5) * dl).repeat(c["n_phi"])
    lines = -half + d * torch.arange(ms + 1, dtype=torch.float64, device=dev)
    if c["voxel_linear"]:
        lines = torch.cat([lines[:1], lines[:-1] + 0.5 * d, lines[-1:]])
    m = _Triples(c["n_phi"] * n, ms * ms)
    step = max(1, (1 << 25) // (4 * len(lines)))
    for a in range(0, len(r), step):
        x, y, q = (t[a:a + step, None] for t in (cx, cy, r))
        u = torch.acos(((lines - x) / q).clamp(-1.0, 1.0))
        v = torch.asin(((lines - y) / q).clamp(-1.0, 1.0))
        t = torch.cat([u, 2.0 * math.pi - u, v % (2.0 * math.pi), math.pi - v], 1).sort(1).values
        t = torch.cat([t, t[:, :1] + 2.0 * math.pi], 1)
        t0, t1 = t[:, :-1], t[:, 1:]
        mid = 0.5 * (t0 + t1)
        row = torch.arange(a, a + len(x), device=dev)[:, None].expand_as(mid)
        px, py = x + q * torch.cos(mid), y + q * torch.sin(mid)
        keep = (px.abs() < half) & (py.abs() < half) & (t1 - t0 > 1e-13)
        if not c["voxel_linear"]:
            ix, iy = _cell(px, -half, d, ms)[0], _cell(py, -half, d, ms)[0]
            m.add(row, ix * ms + iy, q * (t1 - t0), keep)
            continue
        x, y, q = (w.expand_as(mid)[keep] for w in (x, y, q))
        row, px, py, t0, t1 = row[keep], px[keep], py[keep], t0[keep], t1[keep]
        s, k = torch.sin(t1) - torch.sin(t0), torch.cos(t0) - torch.cos(t1)
        one = q * (t1 - t0)
        mx, my = x * one + q * q * s, y * one + q * q * k
        mxy = x * y * one + q * q * (x * k + y * s) + 0.5 * q ** 3 * (torch.sin(t1) ** 2 - torch.sin(t0) ** 2)
        first = -half + 0.5 * d
        for i, a0, b0 in _node(px, first, d, ms):
            for j, a1, b1 in _node(py, first, d, ms):
                w = a0 * a1 * one + b0 * a1 * mx + a0 * b1 * my + b0 * b1 * mxy
                m.add(row, i * ms + j, w, (a0 != 0) | (b0 != 0))
    return m


def _shell(c, dev):
    """A2: row (ring, shell radius), column (radius bin, slab)."""
    n, mz, dz = c["n_ell"], c["mz"], c["dz"]
    (l0, l1), (z0, z1) = _radii(c), _rings(c)
    dl, top = (l1 - l0) / n, 0.5 * mz * dz
    zr = (z0 + (torch.arange(c["n_zs"], dtype=torch.float64, device=dev) + 0.5) * (z1 - z0)
          / c["n_zs"]).repeat_interleave(n)
    nodes = l0 + (torch.arange(n, dtype=torch.float64, device=dev) + 0.5) * dl
    r = nodes.repeat(c["n_zs"])
    planes = -top + dz * torch.arange(mz + 1, dtype=torch.float64, device=dev)
    if c["rho_linear"]:
        edges = torch.cat([torch.tensor([l0, l1], dtype=torch.float64, device=dev), nodes])
    else:
        edges = l0 + dl * torch.arange(n + 1, dtype=torch.float64, device=dev)
    m = _Triples(c["n_zs"] * n, n * mz)
    step = max(1, (1 << 25) // (len(planes) + 2 * len(edges)))
    for a in range(0, len(r), step):
        z, q = zr[a:a + step, None], r[a:a + step, None]
        u = torch.acos(((planes - z) / q).clamp(-1.0, 1.0))
        v = torch.asin((edges / q).clamp(max=1.0))
        t = torch.cat([torch.zeros_like(q), u, v, math.pi - v, torch.full_like(q, math.pi)], 1).sort(1).values
        t0, t1 = t[:, :-1], t[:, 1:]
        mid = 0.5 * (t0 + t1)
        row = torch.arange(a, a + len(z), device=dev)[:, None].expand_as(mid)
        k, slab = _cell(z + q * torch.cos(mid), -top, dz, mz)
        rho = q * torch.sin(mid)
        keep = slab & (rho > l0) & (rho < l1) & (t1 - t0 > 1e-13)
        if not c["rho_linear"]:
            m.add(row, _cell(rho, l0, dl, n)[0] * mz + k, q * (t1 - t0), keep)
            continue
        q, row, k, rho, t0, t1 = q.expand_as(mid)[keep], row[keep], k[keep], rho[keep], t0[keep], t1[keep]
        one, first = q * (t1 - t0), q * q * (torch.cos(t0) - torch.cos(t1))
        for i, a0, b0 in _node(rho, l0 + 0.5 * dl, dl, n):
            m.add(row, i * mz + k, a0 * one + b0 * first, (a0 != 0) | (b0 != 0))
    return m


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    c, call, b = case, case["call"], case["batch"]
    f, p = _inputs(c, seed, dev)
    j, n, h, k, ms = c["n_phi"], c["n_ell"], c["n_zs"], c["mz"], c["ms"]

    def forward(f):
        y = m1 @ f.double().reshape(b, ms * ms, k).permute(1, 0, 2).reshape(ms * ms, b * k)
        y = y.reshape(j, n, b, k).permute(1, 3, 2, 0).reshape(n * k, b * j)
        q = (m2 @ y).reshape(h, n, b, j).permute(2, 3, 0, 1)
        return q.reshape(p_shape)

    def adjoint(p):
        y = t2 @ p.double().reshape(b, j, h, n).permute(2, 3, 0, 1).reshape(h * n, b * j)
        y = y.reshape(n, k, b, j).permute(3, 0, 2, 1).reshape(j * n, b * k)
        g = (t1 @ y).reshape(ms * ms, b, k).permute(1, 0, 2)
        return g.reshape(f_shape)

    lead = () if b == 1 else (b,)
    p_shape, f_shape = (*lead, j, h, n), (*lead, ms, ms, k)
    if call != "adjoint":
        m1, m2 = _plane(c, dev).matrix(c["weights"], False), _shell(c, dev).matrix(c["weights"], False)
        q = forward(f)
        if call in ("forward", "host_forward"):
            return q
        del m1, m2
    t1, t2 = _plane(c, dev).matrix(c["weights"], True), _shell(c, dev).matrix(c["weights"], True)
    if call == "adjoint":
        return adjoint(p)
    if call == "pair":
        return {"p": q, "f": adjoint(p)}
    return {"p": q, "gradient": adjoint(q - p.double())}
