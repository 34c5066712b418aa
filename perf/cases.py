"""The workloads whose time this library is measured by.

Each case is one call sequence of a Monte Carlo program that uses the Python
binding (``paper_1204_6192_gb300.hsg``), from the smallest lattice of the tests
to the benchmark's L = 128, over the storage formats, ragged system counts and
the calls a production run is made of: steps, single kinds of sweeps, the tile
schedule, energies and the replica measurements.

A case is a dict:

  op        step        n steps, then the spins
            loop        n steps and a measurement (energies, q, q(k), permutations),
                        then the spins: the inner loop of a production run
            or, hb      n over-relaxation or heat-bath sweeps, then the spins
            multihit    n steps of the tile schedule, then the spins
            energies    the energies of the present state
            overlaps    the pair and chiral overlaps of the present state
  sizes     lattice edges of the disorder samples, "L" or "LxCOUNT,LxCOUNT"
  temps, t_min, t_max, replicas, field    the geometric temperature ladder and the
            standard deviation of the random field (0: none)
  precision, j_fp16, n_hb, n_or           options of the context
  tile, rounds                            the tile schedule's

The spins come back as binary32 (x, y, z) in a device buffer the caller owns.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1204_6192_gb300 import hsg, inputs

DEFAULTS = dict(op="step", n=1, sizes="8", temps=8, t_min=0.1, t_max=0.4, replicas=2, field=0.1,
                precision="fp32", j_fp16=False, n_hb=1, n_or=5, tile=0, rounds=0)


def _case(**kw):
    return {**DEFAULTS, **kw}


def listed():
    return [
        # a single small lattice, stepped once per call: equilibration scripts and
        # checks; what counts is the latency of a call
        _case(name="step_L8", sizes="8", temps=8, t_min=0.15, t_max=0.6, field=0.0),
        # an odd shape: three replicas of eleven temperatures (33 systems, padded to
        # 40), an edge that is no power of two, FP16 spins beside binary32 couplings
        _case(name="step_L20_ragged", sizes="20", temps=11, t_min=0.12, t_max=0.5, replicas=3, field=0.05,
              precision="fp16"),
        # one L = 32 disorder sample in production: ten steps between measurements
        _case(name="loop_L32", op="loop", n=10, sizes="32", temps=32, field=0.05),
        # the disorder average: 512 small samples of four sizes advanced together
        _case(name="step_batch512", sizes="8x128,12x128,16x128,24x128", temps=16, t_max=0.5, field=0.05),
        # the medium production lattice in the default compressed form
        _case(name="step_L64_fp16", sizes="64", temps=32, precision="fp16", j_fp16=True),
        # the same lattice in the smallest storage form (two 16-bit coordinates a spin)
        _case(name="step_L64_oct16", sizes="64", temps=32, precision="oct16", j_fp16=True),
        # the largest production lattice, ten steps between measurements (the benchmark)
        _case(name="loop_L128_fp16", op="loop", n=10, sizes="128", temps=24, t_min=0.08, t_max=0.3,
              precision="fp16", j_fp16=True),
        # over-relaxation alone on that lattice in uncompressed form
        _case(name="or_L128_fp32", op="or", n=5, sizes="128", temps=24, t_min=0.08, t_max=0.3),
        # heat bath alone at high temperature: the paper's benchmark of 256 systems of
        # L = 32 at T = 100
        _case(name="hb_table1", op="hb", n=2, sizes="32", temps=1, t_min=100.0, t_max=100.0, replicas=256,
              field=0.0),
        # the paper's tile schedule on the same systems, ten rounds of ten
        # over-relaxation sweeps and one heat-bath sweep per tile load
        _case(name="multihit_table1", op="multihit", sizes="32", temps=1, t_min=100.0, t_max=100.0,
              replicas=256, field=0.0, tile=8, rounds=10, n_hb=1, n_or=10),
        # energies of a stored state (a restart, or a set of spins from elsewhere)
        _case(name="energies_L64_bf16", op="energies", sizes="64", temps=32, precision="bf16", j_fp16=True),
        # the four-replica and chiral overlaps that the susceptibilities are built from
        _case(name="overlaps_L48", op="overlaps", sizes="48", temps=16, replicas=4, precision="fp16",
              j_fp16=True),
    ]


def _spins(case):
    return sum(L ** 3 * k for L, k in _sizes(case)) * case["temps"] * case["replicas"]


def draw(rng):
    """One more case of the same ranges; at most the work of the largest listed one."""
    while True:
        op = rng.choices(["step", "loop", "or", "hb", "multihit", "energies", "overlaps"],
                         [30, 10, 12, 12, 12, 8, 16])[0]
        c = _case(op=op, temps=rng.randint(1, 32), replicas=rng.randint(1, 4),
                  t_min=round(rng.uniform(0.08, 0.3), 3), field=rng.choice([0.0, 0.05, 0.1, 1.0]),
                  precision=rng.choice(["fp32", "fp32", "fp16", "fp16", "bf16", "angle16", "oct16", "yx4"]),
                  j_fp16=rng.random() < 0.5)
        c["t_max"] = round(c["t_min"] * rng.uniform(1.5, 5.0), 3)
        L = 2 * round(math.exp(rng.uniform(math.log(4), math.log(128))) / 2)
        c["n"] = rng.randint(1, 4)
        if op in ("loop", "overlaps"):
            c["replicas"] = max(2, c["replicas"])
        if op in ("step", "loop"):
            c["n_hb"], c["n_or"] = rng.choice([(1, 5), (1, 5), (1, 10), (2, 3), (1, 1)])
        if op == "multihit":
            c["n"] = 1
            c["tile"] = rng.choice([4, 8])
            L = max(1, round(L / (2 * c["tile"]))) * 2 * c["tile"]
            c["rounds"] = rng.choice([1, 2, 10])
            c["n_or"] = rng.choice([5, 10])
        if L <= 24 and op != "multihit" and rng.random() < 0.5:
            Ls = sorted({L, max(4, L - 2 * rng.randint(1, 4))})
            c["sizes"] = ",".join("%dx%d" % (v, rng.randint(1, 96)) for v in Ls)
        else:
            c["sizes"] = "%d" % L
        sweeps = {"step": c["n"] * (c["n_hb"] + c["n_or"]), "loop": c["n"] * (c["n_hb"] + c["n_or"]),
                  "multihit": c["rounds"] * (c["n_hb"] + c["n_or"])}.get(op, c["n"])
        # the packed formats cost up to three times as much for an update
        cost = _spins(c) * sweeps * (3 if c["precision"] in ("angle16", "oct16", "yx4") else 1)
        if _spins(c) <= 50e6 and cost <= 3e9:
            return c


# -- inputs ---------------------------------------------------------------------

def _sizes(case):
    """[(L, number of samples)]"""
    return [(int(L), int(k or 1)) for L, _, k in (part.partition("x") for part in case["sizes"].split(","))]


def _disorder(case, seed):
    """Per sample (L, J [N, 3], H [N, 3] or None), Gaussian, on the GPU; and the spins, uniform on the
    sphere, as one flat binary32 tensor (samples, systems, sites, components)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W = case["temps"] * case["replicas"]
    samples, spins = [], []
    for L, count in _sizes(case):
        N = L ** 3
        J = torch.randn(count, N, 3, generator=g, device="cuda")
        H = torch.randn(count, N, 3, generator=g, device="cuda") * case["field"] if case["field"] else None
        samples += [(L, J[k], H[k] if H is not None else None) for k in range(count)]
        s = torch.randn(count, W, N, 3, generator=g, device="cuda")
        s /= s.norm(dim=-1, keepdim=True)
        spins.append(s.flatten())
    return samples, torch.cat(spins) if len(spins) > 1 else spins[0]


def _temps(case):
    return inputs.geometric_temperatures(case["t_min"], case["t_max"], case["temps"])


_streams = []


def _stream():
    """The stream all contexts of the program run on, so that the passes of several states follow
    each other as the steps of one chain do."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    samples, spins = _disorder(case, seed)
    host = []
    for L, count in _sizes(case):   # one copy to the host per lattice size
        part = samples[len(host):len(host) + count]
        J = torch.stack([p[1] for p in part]).cpu().numpy()
        H = torch.stack([p[2] for p in part]).cpu().numpy() if part[0][2] is not None else [None] * count
        host += [SimpleNamespace(L=L, J=J[k], H=H[k], temps=_temps(case)) for k in range(count)]
    ctx = hsg.Context(host, n_replicas=case["replicas"], seed=seed, precision=case["precision"],
                      j_fp16=case["j_fp16"], n_hb=case["n_hb"], n_or=case["n_or"],
                      stream=_stream().cuda_stream)
    torch.cuda.synchronize()
    ctx.set_spins_dev(spins.data_ptr())
    ctx.sync()
    # the spins' buffer is free again: the program reads the state back into it
    return {"ctx": ctx, "case": case, "spins": spins}


def run(state):
    ctx, case = state["ctx"], state["case"]
    op, n, spins = case["op"], case["n"], state["spins"]
    if op == "energies":
        return {"E": ctx.energies()}
    if op == "overlaps":
        return ctx.measure_overlaps()
    out = {}
    if op == "step":
        ctx.step(n)
    elif op == "loop":
        ctx.step(n)
        out.update(ctx.measure())
    elif op == "or":
        ctx.sweep_or(n)
    elif op == "hb":
        ctx.sweep_hb(n)
    else:
        ctx.step_multihit(n, tile=case["tile"], n_rounds=case["rounds"], n_or=case["n_or"], n_hb=case["n_hb"])
    ctx.get_spins_dev(spins.data_ptr())
    out["spins"] = spins
    return out


def work(case):
    """Bytes: the state and the disorder read once, the state written once in its storage form and
    the outputs written once (a measurement alone reads the state and writes a few numbers).
    Operations: binary32 multiplies, adds, divisions and roots of the moves, integer ones of the
    generator left out."""
    S = {"fp32": 12, "fp16": 6, "bf16": 6, "angle16": 4, "oct16": 4, "yx4": 8}[case["precision"]]
    sites, spins = sum(L ** 3 * k for L, k in _sizes(case)), _spins(case)
    disorder = sites * (6 if case["field"] else 3) * (2 if case["j_fp16"] else 4)
    field = 36 + (3 if case["field"] else 0)          # six bonds and the random field
    over_relaxation, heat_bath = field + 29, field + 75
    pairs = min(case["replicas"], 4) * (min(case["replicas"], 4) - 1) // 2
    op, n = case["op"], case["n"]
    if op == "energies":
        return {"bytes": spins * S + disorder, "flops": spins * (18 + 6)}
    if op == "overlaps":
        used = spins * min(case["replicas"], 4) // case["replicas"]
        return {"bytes": used * S, "flops": used * 42 + sites * case["temps"] * pairs * (5 + 3 + 4 * 13)}
    moves = {"step": (n * case["n_hb"], n * case["n_or"]), "loop": (n * case["n_hb"], n * case["n_or"]),
             "or": (0, n), "hb": (n, 0),
             "multihit": (n * case["rounds"] * case["n_hb"], n * case["rounds"] * case["n_or"])}[op]
    flops = spins * (moves[0] * heat_bath + moves[1] * over_relaxation)
    if op in ("step", "loop", "multihit"):
        flops += spins * n * 6
    if op == "loop":
        flops += sites * case["temps"] * (9 + 9 * 13)
    return {"bytes": spins * (2 * S + 12) + disorder, "flops": flops}


# -- the same in 64 bits, from the definitions (include/hsg.h) ---------------------

PI = math.pi


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors or ints holding 32-bit words."""
    k0, k1, mask = seed & 0xffffffff, (seed >> 32) & 0xffffffff, 0xffffffff
    c = [c0, c1, c2, c3]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _uniform(x):
    return (2 * (x >> 9) + 1) * 2.0 ** -24


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _stored(v, precision):
    """Unit vectors v [..., 3] as the storage form gives them back."""
    x, y, z = v.unbind(-1)
    if precision == "fp32":
        return v.float().double()
    if precision == "fp16":
        return v.half().double()
    if precision == "bf16":
        return v.bfloat16().double()
    sign = lambda t: torch.where(t >= 0, 1.0, -1.0)  # noqa: E731
    if precision == "yx4":
        sg = sign(z)
        y, x = y.float().double(), (x + 4 * sg).float().double() - 4 * sg
        return torch.stack([x, y, sg * (1 - x * x - y * y).clamp(min=0).sqrt()], -1)
    if precision == "angle16":
        t = torch.floor(torch.acos(z.clamp(-1, 1)) * 65535 / PI + 0.5).clamp(max=65535) * PI / 65535
        p = torch.remainder(torch.floor(torch.atan2(y, x) * 65536 / (2 * PI) + 0.5), 65536) * 2 * PI / 65536
        return torch.stack([t.sin() * p.cos(), t.sin() * p.sin(), t.cos()], -1)
    fold = lambda p, q: ((1 - q.abs()) * sign(p), (1 - p.abs()) * sign(q))  # noqa: E731  (oct16)
    l1 = x.abs() + y.abs() + z.abs()
    p, q = x / l1, y / l1
    fp, fq = fold(p, q)
    p, q = (torch.floor(torch.where(z < 0, f, o).clamp(-1, 1) * 32767 + 0.5) / 32767 for f, o in ((fp, p), (fq, q)))
    z = 1 - p.abs() - q.abs()
    fp, fq = fold(p, q)
    v = torch.stack([torch.where(z < 0, fp, p), torch.where(z < 0, fq, q), z], -1)
    return v / v.norm(dim=-1, keepdim=True)


class _Exact:
    """Systems w0 .. w0 + m of one sample, spins [m, z, y, x, 3] in binary64."""

    def __init__(self, case, seed, s, L, J, H, spins, w0):
        self.case, self.seed, self.L, self.sample = case, seed, L, s
        rounded = (lambda t: t.half().double()) if case["j_fp16"] else (lambda t: t.double())
        self.J = rounded(J).view(L, L, L, 3)
        self.H = rounded(H).view(L, L, L, 3) if H is not None else torch.zeros_like(self.J)
        self.s = _stored(spins.double().view(-1, L, L, L, 3), case["precision"])
        r = torch.arange(L, device="cuda")
        self.xyz = (r.view(1, 1, L), r.view(1, L, 1), r.view(L, 1, 1))
        self.parity = (self.xyz[0] + self.xyz[1] + self.xyz[2]) % 2
        self.site = (self.xyz[0] + L * (self.xyz[1] + L * self.xyz[2]))
        Wp = -(-case["temps"] * case["replicas"] // 8) * 8
        m = self.s.shape[0]
        w = w0 + torch.arange(m, device="cuda")
        self.gsys = (s * Wp + w).view(m, 1, 1, 1)
        T = torch.as_tensor(_temps(case), device="cuda")
        self.beta = 1 / T[w % case["temps"]].view(m, 1, 1, 1)

    def bonds(self):
        """sum of J s over the +x, +y, +z bonds, and over all six"""
        half, full = 0.0, 0.0
        for a, dim in ((0, 3), (1, 2), (2, 1)):
            Ja = self.J[..., a, None]
            up = Ja * self.s.roll(-1, dim)
            half = half + up
            full = full + up + Ja.roll(1, dim - 1) * self.s.roll(1, dim)
        return half, full

    def half_sweep(self, hb, sweep, where):
        h = self.bonds()[1] + self.H
        new = self.heat_bath(h, sweep) if hb else self.reflect(h)
        new = _stored(new / new.norm(dim=-1, keepdim=True), self.case["precision"])
        self.s = torch.where(where[..., None], new, self.s)

    def reflect(self, h):
        hh = _dot(h, h)
        return torch.where(hh > 0, 2 * _dot(self.s, h) / hh.clamp(min=1e-300) * h - self.s, self.s)

    def heat_bath(self, h, sweep):
        r = _philox(self.site, self.gsys >> 1, sweep, 1, self.seed)
        odd = (self.gsys & 1).bool()
        u1, u2 = _uniform(torch.where(odd, r[2], r[0])), _uniform(torch.where(odd, r[3], r[1]))
        hn = h.norm(dim=-1)
        a = self.beta * hn
        safe = a.clamp(min=1e-12)
        d = torch.where(a > 1e-12, -torch.log1p((1 - u1) * torch.expm1(-2 * safe)) / safe, 2 * (1 - u1))
        n = torch.where((hn > 0)[..., None], h / hn.clamp(min=1e-300)[..., None],
                        torch.tensor([0.0, 0.0, 1.0], device="cuda", dtype=h.dtype))
        x, y, z = n.unbind(-1)
        sg = torch.where(z >= 0, 1.0, -1.0)      # the frame of Duff et al., JCGT 2017
        A = -1 / (sg + z)
        B = x * y * A
        e1 = torch.stack([1 + sg * x * x * A, sg * B, -sg * x], -1)
        e2 = torch.stack([B, sg + y * y * A, -y], -1)
        st, phi = (d * (2 - d)).clamp(min=0).sqrt()[..., None], (2 * PI * u2)[..., None]
        return st * (phi.cos() * e1 + phi.sin() * e2) + (1 - d)[..., None] * n

    def sweep(self, hb, sweep, tiles=None):
        for p in (0, 1):
            where = self.parity == p
            self.half_sweep(hb, sweep, where if tiles is None else where & tiles)

    def energies(self):
        return -_dot(self.s, self.bonds()[0] + self.H).sum(dim=(1, 2, 3, 4))

    def modes(self, f):
        """(1/N) sum_i f_i e^{ik.R_i} for k = 0 and along x, y, z: f [m, z, y, x] to [m, 4, 2]"""
        out = [torch.stack([f.mean(dim=(1, 2, 3)), torch.zeros(f.shape[0], device="cuda").double()], -1)]
        for c in self.xyz:
            phase = 2 * PI * c.double() / self.L
            out.append(torch.stack([(f * phase.cos()).mean(dim=(1, 2, 3)), (f * phase.sin()).mean(dim=(1, 2, 3))], -1))
        return torch.stack(out, 1)

    def chirality(self):
        return [_dot(self.s.roll(-1, d), torch.cross(self.s, self.s.roll(1, d), dim=-1))[..., 0] for d in (3, 2, 1)]


def exact(case, seed):
    """What run() gives for a new state, in binary64.  None for runs of more than a few sweeps: the
    dynamics amplify any difference of rounding about tenfold in four sweeps, so the spins of such
    a run, and what is measured on them, have no 64-bit value to compare with."""
    op, n = case["op"], case["n"]
    sweeps = {"or": n, "hb": n, "step": n * (case["n_hb"] + case["n_or"]),
              "multihit": n * case["rounds"] * (case["n_hb"] + case["n_or"])}.get(op, 0)
    if op == "loop" or sweeps > 6 or (op == "step" and n > 1):
        return None
    samples, spins = _disorder(case, seed)
    W, R_T, at = case["temps"] * case["replicas"], case["temps"], 0
    E, D, C, out = [], [], [], []
    for s, (L, J, H) in enumerate(samples):
        N = L ** 3
        mine = spins[at:at + W * N * 3].view(W, N * 3)
        at += W * N * 3
        if op == "overlaps":     # all temperatures of the first four replicas, in slot order
            r = [_Exact(case, seed, s, L, J, H, mine[k * R_T:(k + 1) * R_T], k * R_T)
                 for k in range(min(4, case["replicas"]))]
            kappa = [x.chirality() for x in r]
            pairs = [(a, b) for b in range(1, len(r)) for a in range(b)]
            D.append(torch.stack([r[0].modes(_dot(r[a].s, r[b].s)[..., 0]) for a, b in pairs], 1))
            C.append(torch.stack([torch.stack([r[0].modes(kappa[a][d] * kappa[b][d]) for d in range(3)], 1)
                                  for a, b in pairs], 1))
            continue
        m = max(1, min(W, int(2e7 / N)))     # systems at a time
        for w0 in range(0, W, m):
            x = _Exact(case, seed, s, L, J, H, mine[w0:w0 + m], w0)
            if op == "energies":
                E.append(x.energies())
                continue
            if op == "multihit":
                T, per = case["tile"], case["n_hb"] + case["n_or"]
                colour = sum(c // T for c in x.xyz) % 2
                for k in (0, 1):
                    for j in range(case["rounds"] * per):
                        x.sweep(j % per >= case["n_or"], j, colour == k)
            else:
                n_hb = {"or": 0, "hb": n}.get(op, case["n_hb"])
                for j in range(sweeps):
                    x.sweep(j < n_hb, j)
            out.append(x.s.flatten())
    if op == "energies":
        return {"E": torch.cat(E).view(len(samples), W).cpu().numpy()}
    if op == "overlaps":
        return {"D": torch.stack(D).cpu().numpy(), "C": torch.stack(C).cpu().numpy()}
    return {"spins": torch.cat(out)}
