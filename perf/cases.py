"""Timed cases of the framework: what a program that evaluates leading-order
matrix elements has it do, each through the public entry points of
paper_2303_18244_gb300.mg.

The processes, energies and the larger batch sizes are the ones of bench.py
and of the GPU tests; the ranges reach from one small serving bucket (256
events) to the full batch of the paper's tables.  Momenta are flat RAMBO phase
space, drawn here from the seed, inside the cuts without which the cross
section of a process with final-state gluons does not exist (transverse
momentum and separation of every gluon).  The gg processes keep every helicity
(all of them contribute); e+e- and u u~ run with the filtered list, as bench.py
does.

A mode that computes its amplitudes in FP32 (MG_MIXED, MG_FLOAT) hands its
matrix elements on in FP32, the type that its values carry; the FP64 mode in
FP64.
"""
import itertools
import math

import numpy as np
import torch

from paper_2303_18244_gb300 import mg

MODES = {"fp64": mg.MG_FP64, "mixed": mg.MG_MIXED, "float": mg.MG_FLOAT}
SQRTS = {
    "e+ e- > mu+ mu-": 500.0,
    "u u~ > t t~": 1000.0,
    "u u~ > t t~ g": 1200.0,
    "g g > t t~": 1000.0,
    "g g > t t~ g": 1200.0,
    "g g > t t~ g g": 1500.0,
    "g g > t t~ g g g": 2000.0,
}
MT = 173.0

# (process, mode) -> the range of batch sizes of one mg.sigma call
SIGMA = {
    ("e+ e- > mu+ mu-", "mixed"): (256, 65536),
    ("g g > t t~", "mixed"): (4096, 524288),
    ("g g > t t~ g", "fp64"): (1024, 65536),
    ("g g > t t~ g g", "mixed"): (1024, 524288),
    ("g g > t t~ g g", "fp64"): (1024, 32768),
    ("g g > t t~ g g g", "mixed"): (512, 16384),
    ("g g > t t~ g g g", "fp64"): (256, 4096),
    ("u u~ > t t~ g", "float"): (4096, 524288),
}


def listed():
    return [
        # latency of the smallest serving bucket: launches and host path
        {"name": "ee_mumu_mixed_256", "op": "sigma", "proc": "e+ e- > mu+ mu-", "mode": "mixed", "n": 256},
        # the small QCD process of the paper's list, one full batch
        {"name": "ggtt_mixed_524288", "op": "sigma", "proc": "g g > t t~", "mode": "mixed", "n": 524288},
        # one extra gluon, double precision, the batch of the parity tests
        {"name": "ggttg_fp64_65536", "op": "sigma", "proc": "g g > t t~ g", "mode": "fp64", "n": 65536},
        # the headline batch (paper Tables 1-2) in the default fast mode
        {"name": "ggttgg_mixed_524288", "op": "sigma", "proc": "g g > t t~ g g", "mode": "mixed", "n": 524288},
        # a ragged batch of the headline process in double precision
        {"name": "ggttgg_fp64_32749", "op": "sigma", "proc": "g g > t t~ g g", "mode": "fp64", "n": 32749},
        # the largest process (paper Tables 3-4), a ragged mid-size batch
        {"name": "ggttggg_mixed_8229", "op": "sigma", "proc": "g g > t t~ g g g", "mode": "mixed", "n": 8229},
        # the largest process in double precision: a calibration-size batch
        {"name": "ggttggg_fp64_4096", "op": "sigma", "proc": "g g > t t~ g g g", "mode": "fp64", "n": 4096},
        # a quark-initiated process in the paper's all-float mode, ragged
        {"name": "uuttg_float_262147", "op": "sigma", "proc": "u u~ > t t~ g", "mode": "float", "n": 262147},
        # end to end from pinned host buffers: copy in, evaluate, copy out
        {"name": "ggttgg_host_mixed_65536", "op": "host", "proc": "g g > t t~ g g", "mode": "mixed", "n": 65536},
        # event generation: ME plus helicity and colour choice per event
        {"name": "ggttgg_select_fp64_8192", "op": "select", "proc": "g g > t t~ g g", "mode": "fp64", "n": 8192},
        # phase-space generation on the device for the headline batch
        {"name": "rambo_ggttgg_524288", "op": "rambo", "proc": "g g > t t~ g g", "mode": "fp64", "n": 524288},
        # hit-or-miss unweighting of a large accumulated sample
        {"name": "unweight_33554467", "op": "unweight", "proc": "", "mode": "fp64", "n": 33554467},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["sigma"] * 8 + ["host", "select", "rambo", "unweight"])
    if op == "sigma":
        (proc, mode), (lo, hi) = rng.choice(sorted(SIGMA.items()))
        return {"op": op, "proc": proc, "mode": mode, "n": _size(rng, lo, hi)}
    if op == "host":
        proc = rng.choice(["g g > t t~", "g g > t t~ g g"])
        return {"op": op, "proc": proc, "mode": "mixed", "n": _size(rng, 1024, 131072)}
    if op == "select":
        proc = rng.choice(["g g > t t~ g", "g g > t t~ g g"])
        return {"op": op, "proc": proc, "mode": "fp64", "n": _size(rng, 512, 16384)}
    if op == "rambo":
        proc = rng.choice(sorted(p for p in SQRTS))
        return {"op": op, "proc": proc, "mode": "fp64", "n": _size(rng, 4096, 524288)}
    return {"op": op, "proc": "", "mode": "fp64", "n": _size(rng, 1 << 16, 1 << 25)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _final_masses(proc):
    nf = len(proc.split(">")[1].split())
    return [0.0] * nf if proc.startswith("e+") else [MT, MT] + [0.0] * (nf - 2)


PT_MIN, DR_MIN = 20.0, 0.4  # of the final-state gluons, GeV


def _inside_cuts(p, masses):
    """Events whose final-state gluons are neither soft nor collinear."""
    g = p[:, 4:] if masses[0] else p[:, :0]
    pt = g[..., 1:3].norm(dim=2)
    ok = (pt > PT_MIN).all(1)
    eta, phi = torch.asinh(g[..., 3] / pt), torch.atan2(g[..., 2], g[..., 1])
    for i, j in itertools.combinations(range(g.shape[1]), 2):
        d = torch.remainder(phi[:, i] - phi[:, j] + math.pi, 2 * math.pi) - math.pi
        ok &= (eta[:, i] - eta[:, j]) ** 2 + d ** 2 > DR_MIN ** 2
    return ok


def _momenta(proc, n, seed):
    """The first n events inside the cuts of a stream of flat phase space."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    masses, got, have = _final_masses(proc), [], 0
    while have < n:
        p = _flat(proc, n - have + n // 2 + 64, g)
        got.append(p[_inside_cuts(p, masses)])
        have += got[-1].shape[0]
    return torch.cat(got)[:n].contiguous()


def _flat(proc, n, g):
    """Flat phase space at fixed sqrt(s) (RAMBO: Kleiss, Stirling, Ellis 1986)."""
    masses = torch.tensor(_final_masses(proc), dtype=torch.float64, device="cuda")
    nf, rs = masses.numel(), SQRTS[proc]
    u = torch.rand((n, nf, 4), dtype=torch.float64, device="cuda", generator=g).clamp_(min=2.0 ** -53)
    c, phi = 2.0 * u[..., 0] - 1.0, 2.0 * math.pi * u[..., 1]
    s = (1.0 - c * c).clamp(min=0.0).sqrt()
    e = -torch.log(u[..., 2] * u[..., 3]) + 1e-12
    q = torch.stack([e, e * s * torch.cos(phi), e * s * torch.sin(phi), e * c], -1)
    Q = q.sum(1)
    M = (Q[:, 0] ** 2 - (Q[:, 1:] ** 2).sum(1)).sqrt()[:, None]
    b, gamma = -Q[:, 1:] / M, Q[:, :1] / M
    bq = (b[:, None] * q[..., 1:]).sum(2)
    x = rs / M
    p3 = x[..., None] * (q[..., 1:] + b[:, None] * q[..., :1] + (bq / (1.0 + gamma))[..., None] * b[:, None])
    p3 = p3 - p3.mean(1, keepdim=True)
    k2 = (p3 ** 2).sum(2)
    xi = torch.full((n, 1), math.sqrt(1.0 - (float(masses.sum()) / rs) ** 2), dtype=torch.float64, device="cuda")
    for _ in range(12):
        en = (masses ** 2 + xi ** 2 * k2).sqrt()
        xi = xi - (en.sum(1, keepdim=True) - rs) / (xi * k2 / en).sum(1, keepdim=True)
    p = torch.zeros((n, nf + 2, 4), dtype=torch.float64, device="cuda")
    p[:, 0, 0] = p[:, 1, 0] = p[:, 0, 3] = 0.5 * rs
    p[:, 1, 3] = -0.5 * rs
    p[:, 2:, 1:] = p3 * xi[..., None]
    p[:, 2:, 0] = (masses ** 2 + xi ** 2 * k2).sqrt()
    return p


def _uniforms(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + (1 << 40))
    return torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)


def _weights(n, seed):
    """Event weights as flat phase space gives them: a long upper tail."""
    g = torch.Generator(device="cuda").manual_seed(seed + (1 << 41))
    return torch.exp(torch.randn((n,), dtype=torch.float64, device="cuda", generator=g))


def prepare(case, seed):
    op, proc, n = case["op"], case["proc"], case["n"]
    st = {"op": op, "n": n, "low": case["mode"] != "fp64", "seed": seed}
    if op == "unweight":
        st["w"], st["r"] = _weights(n, seed), _uniforms((n,), seed)
        st["wmax"] = 0.25 * float(st["w"].max())
        st["idx"] = torch.zeros((n,), dtype=torch.int64, device="cuda")
        st["kept"] = torch.zeros((1,), dtype=torch.int64, device="cuda")
        return st
    h = st["h"] = mg.Process(proc, precision=MODES[case["mode"]])
    st["rs"] = SQRTS[proc]
    if op == "rambo":
        st["mom"] = torch.empty((n, h.info.npar, 4), dtype=torch.float64, device="cuda")
        return st
    if not proc.startswith("g g"):
        mg.good_helicities(h, _momenta(proc, 1024, 1000003))
    st["mom"] = _momenta(proc, n, seed)
    st["me"] = torch.empty((n,), dtype=torch.float64, device="cuda")
    if op == "host":
        st["mom"] = st["mom"].cpu().pin_memory()
        st["me"] = torch.empty((n,), dtype=torch.float64).pin_memory()
    if op == "select":
        st["rnd"] = _uniforms((n, 2), seed)
        st["hel"] = torch.empty((n,), dtype=torch.int32, device="cuda")
        st["col"] = torch.empty((n,), dtype=torch.int32, device="cuda")
        st["colw"] = torch.empty((n, h.info.n_col), dtype=torch.float64, device="cuda")
    return st


def run(st):
    op = st["op"]
    if op == "unweight":
        mg.unweight(st["w"], st["r"], st["wmax"], st["idx"], st["kept"])
        return st["idx"], st["kept"]
    if op == "rambo":
        mg.rambo(st["h"], st["rs"], st["seed"], 0, st["mom"])
        return st["mom"]
    if op == "select":
        mg.sigma_select(st["h"], st["mom"], st["rnd"], st["me"], st["hel"], st["col"], st["colw"])
        return st["me"], st["hel"], st["col"], st["colw"]
    if op == "host":
        mg.sigma_host(st["h"], st["mom"], st["me"])
    else:
        mg.sigma(st["h"], st["mom"], st["me"])
    return st["me"].float() if st["low"] else st["me"]


# Floating-point operations per event that the matrix element cannot do
# without, from a colour-ordered recursion whose currents are shared between
# flows and helicities (currents, the closing contractions of every helicity
# and flow, the colour form block by block).
FLOPS = {"e+ e- > mu+ mu-": 1.5e3, "u u~ > t t~": 1.5e3, "u u~ > t t~ g": 1.2e4, "g g > t t~": 4e3, "g g > t t~ g": 3e4,
         "g g > t t~ g g": 3e5, "g g > t t~ g g g": 3e6}


def work(case):
    op, n = case["op"], case["n"]
    if op == "unweight":
        return {"bytes": 16.0 * n, "flops": 2.0 * n}
    npar = len(case["proc"].replace(">", " ").split())
    if op == "rambo":
        return {"bytes": 32.0 * npar * n, "flops": 250.0 * (npar - 2) * n}
    b, f = 32.0 * npar + 8, FLOPS[case["proc"]]
    if op == "select":
        b += 16 + 8 + 8 * math.factorial(npar - 2)
    return {"bytes": b * n, "flops": f * n}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the textbook formulas
# ---------------------------------------------------------------------------

_C = torch.complex128
ALPHA_S, GAMMA_T = 0.118, 1.4915
G2 = 4.0 * math.pi * ALPHA_S


def _dirac():
    s = np.zeros((4, 2, 2), complex)
    s[0], s[1], s[2], s[3] = np.eye(2), [[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]
    gam = np.zeros((4, 4, 4), complex)
    gam[0] = np.diag([1, 1, -1, -1])
    for k in (1, 2, 3):
        gam[k, :2, 2:], gam[k, 2:, :2] = s[k], -s[k]
    return torch.from_numpy(gam).cuda()


def _gell_mann():
    t = np.zeros((8, 3, 3), complex)
    t[0][0, 1] = t[0][1, 0] = 1
    t[1][0, 1], t[1][1, 0] = -1j, 1j
    t[2][0, 0], t[2][1, 1] = 1, -1
    t[3][0, 2] = t[3][2, 0] = 1
    t[4][0, 2], t[4][2, 0] = -1j, 1j
    t[5][1, 2] = t[5][2, 1] = 1
    t[6][1, 2], t[6][2, 1] = -1j, 1j
    t[7] = np.diag([1, 1, -2]) / math.sqrt(3)
    return t / 2


METRIC = torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=torch.float64)


def _slash(v, gam):
    return torch.einsum("...m,mab->...ab", v.to(_C) * METRIC.to(v.device), gam)


def _square(terms, m2=0.0):
    """(sum of the vectors)^2 - m2, the component sums and squares carried
    with their rounding errors, so that collinear sums keep their digits."""
    hi = torch.full_like(terms[0][..., 0], -m2)
    lo = torch.zeros_like(hi)

    def two(a, b):
        s = a + b
        bb = s - a
        return s, (a - (s - bb)) + (b - bb)

    for mu in range(4):
        c, cl = terms[0][..., mu], torch.zeros_like(hi)
        for t in terms[1:]:
            c, e = two(c, t[..., mu])
            cl = cl + e
        big = 134217729.0 * c
        h = big - (big - c)
        low = c - h
        sq = c * c
        er = ((h * h - sq) + 2.0 * h * low) + low * low + 2.0 * c * cl
        sg = 1.0 if mu == 0 else -1.0
        hi, e = two(hi, sg * sq)
        lo = lo + e + sg * er
    return hi + lo


def _spinors(p, m, gam, anti):
    """Two column spinors [n, 2, 4] with sum w wbar = pslash + m (or - m)."""
    sg = -1.0 if anti else 1.0
    basis = torch.zeros((2, 4), dtype=_C, device=p.device)
    for k in range(2):
        basis[k, k + (2 if anti else 0)] = 1.0
    num = _slash(p, gam) + sg * m * torch.eye(4, dtype=_C, device=p.device)
    w = torch.einsum("nab,kb->nka", num, basis) / (p[:, 0] + m).sqrt()[:, None, None]
    return sg * w


def _polarisations(k):
    """Two real transverse polarisations [n, 2, 4] of a light-like momentum."""
    d = k[:, 1:] / k[:, 1:].norm(dim=1, keepdim=True)
    a = torch.zeros_like(d)
    j = d.abs().argmin(1)
    a[torch.arange(d.shape[0], device=d.device), j] = 1.0
    e1 = torch.linalg.cross(d, a)
    e1 = e1 / e1.norm(dim=1, keepdim=True)
    e2 = torch.linalg.cross(d, e1)
    z = torch.zeros_like(e1[:, :1])
    return torch.stack([torch.cat([z, e1], 1), torch.cat([z, e2], 1)], 1).to(_C)


def _mdot(a, b):
    return (a * METRIC.to(a.device) * b).sum(-1)


def _bcast(x, ha, hb, left):
    """x [n, ha or hb, 4] -> [n, ha, hb, 4]."""
    return x[:, :, None].expand(-1, ha, hb, -1) if left else x[:, None].expand(-1, ha, hb, -1)


def _gg_flows(p, proc):
    """Colour-ordered amplitudes [n, n!, 2^n * 4] of g g -> t t~ + gluons (any
    helicity basis: only sums over it are used)."""
    n, dev = p.shape[1] - 2, p.device
    gam, g = _dirac(), math.sqrt(G2)
    slot = [0, 1] + list(range(4, n + 2))
    k = [p[:, s] if s < 2 else -p[:, s] for s in slot]  # incoming
    eps = [_polarisations(p[:, s]) for s in slot]
    ubar = torch.einsum("nka,ab->nkb", _spinors(p[:, 2], MT, gam, False).conj(), gam[0])
    v = _spinors(p[:, 3], MT, gam, True)
    J, K = {}, {}
    for m in range(1, n + 1):
        for w in itertools.permutations(range(n), m):
            K[w] = sum(k[i] for i in w)
            if m == 1:
                J[w] = eps[w[0]]
                continue
            H = 2 ** m
            acc = torch.zeros((p.shape[0], H, 4), dtype=_C, device=dev)
            for i in range(1, m):
                a, b = w[:i], w[i:]
                x = _bcast(J[a], 2 ** i, 2 ** (m - i), True)
                y = _bcast(J[b], 2 ** i, 2 ** (m - i), False)
                ka, kb = K[a].to(_C)[:, None, None], K[b].to(_C)[:, None, None]
                t = _mdot(x, y)[..., None] * (ka - kb) + y * _mdot(2 * kb + ka, x)[..., None] - x * _mdot(2 * ka + kb, y)[..., None]
                acc += -g * t.reshape(-1, H, 4)
            for i, j in itertools.combinations(range(1, m), 2):
                sh = (-1, 2 ** i, 2 ** (j - i), 2 ** (m - j), 4)
                x = J[w[:i]][:, :, None, None]
                y = J[w[i:j]][:, None, :, None]
                z = J[w[j:]][:, None, None, :]
                t = 2 * _mdot(x, z)[..., None] * y - _mdot(y, z)[..., None] * x - _mdot(x, y)[..., None] * z
                acc += G2 * t.expand(p.shape[0], *sh[1:]).reshape(-1, H, 4)
            inv = _square([k[i] for i in w]) if m < n else _square([p[:, 2], p[:, 3]])
            J[w] = acc / inv[:, None, None].to(_C)
    cols = {w: torch.einsum("nhab,nsb->nhsa", _slash(J[w], gam), v) for w in J}  # Jslash v
    rows = {(): ubar[:, None]}  # [n, hel, spin, 4]
    flows = []
    one = torch.eye(4, dtype=_C, device=dev)
    for m in range(1, n):
        for w in itertools.permutations(range(n), m):
            H = 2 ** m
            acc = torch.zeros((p.shape[0], H, 2, 4), dtype=_C, device=dev)
            for i in range(m):
                r, js = rows[w[:i]], _slash(J[w[i:]], gam)
                acc += torch.einsum("nxsa,nyab->nxysb", r, js).reshape(-1, H, 2, 4)
            D = _square([p[:, 2]] + [-k[i] for i in w], MT * MT).to(_C) + 1j * MT * GAMMA_T
            prop = (_slash(p[:, 2] - K[w], gam) + MT * one) * (-g / D)[:, None, None]
            rows[w] = torch.einsum("nhsa,nab->nhsb", acc, prop)
    for w in itertools.permutations(range(n)):
        a = torch.zeros((p.shape[0], 2 ** n, 2, 2), dtype=_C, device=dev)
        order = [w.index(i) for i in range(n)]
        for i in range(n):
            a += torch.einsum("nxsa,nyta->nxyst", rows[w[:i]], cols[w[i:]]).reshape(a.shape)
        # helicity axes of the word -> one common order
        a = a.reshape([-1] + [2] * n + [4]).permute([0] + [1 + o for o in order] + [n + 1])
        flows.append((1j * g * a).reshape(p.shape[0], -1))
    return torch.stack(flows, 1)


def _colour_strings(n):
    """C(identity, tau) for every ordering tau, by explicit index sums."""
    t = torch.from_numpy(_gell_mann()).cuda()
    w = t
    for _ in range(n - 1):  # w[a_1, ..., a_m] = T^{a_1} ... T^{a_m}
        w = torch.einsum("...ij,ajk->...aik", w, t)
    flat, row = w.reshape(-1).conj(), {}
    for tau in itertools.permutations(range(n)):
        # axis i of the string of tau carries the label of gluon i
        wt = w.permute([tau.index(i) for i in range(n)] + [n, n + 1]).reshape(-1)
        row[tau] = float((flat * wt).sum().real)
    return list(row), row


def _colour_matrix(n):
    words, row = _colour_strings(n)
    m = torch.empty((len(words), len(words)), dtype=torch.float64)
    for i, s in enumerate(words):
        for j, t in enumerate(words):
            # only the relative order matters: relabel so that s is the identity
            lab = {x: q for q, x in enumerate(s)}
            m[i, j] = row[tuple(lab[x] for x in t)]
    return m.cuda()


def _gg_exact(p, proc):
    """(ME [n], flow weights [n, n!]) of g g -> t t~ + gluons."""
    n = p.shape[1] - 2
    C = _colour_matrix(n)
    iden = 256.0 * math.factorial(n - 2)
    me, wk = [], []
    step = {2: 131072, 3: 65536, 4: 16384, 5: 2048}[n]
    for q in p.split(step):
        f = _gg_flows(q, proc)
        me.append((torch.einsum("nsh,st,nth->n", f.real, C, f.real) + torch.einsum("nsh,st,nth->n", f.imag, C, f.imag)) / iden)
        wk.append((f.abs() ** 2).sum(2))
    return torch.cat(me), torch.cat(wk)


def _dot(a, b):
    return a[:, 0] * b[:, 0] - (a[:, 1:] * b[:, 1:]).sum(1)


def _ee_exact(p):
    alpha, mz, wz, gf = 1.0 / 132.507, 91.188, 2.441404, 1.16639e-5
    e2 = 4 * math.pi * alpha
    mw2 = 0.5 * mz ** 2 + math.sqrt(0.25 * mz ** 4 - math.pi * alpha * mz ** 2 / (math.sqrt(2.0) * gf))
    sw2 = 1 - mw2 / mz ** 2
    gz2, gl, gr = e2 / (sw2 * (1 - sw2)), -0.5 + sw2, sw2
    s = 2 * _dot(p[:, 0], p[:, 1])
    # same-chirality amplitudes go with p(e-).p(mu+), opposite ones with p(e-).p(mu-)
    u, t = 2 * _dot(p[:, 1], p[:, 2]), 2 * _dot(p[:, 1], p[:, 3])
    z = 1.0 / torch.complex(s - mz * mz, torch.full_like(s, mz * wz))
    out = 0.0
    for a in (gl, gr):
        for b in (gl, gr):
            amp = (e2 / s + gz2 * a * b * z).abs() ** 2
            out = out + 4.0 * (u if a == b else t) ** 2 * amp
    return out / 4.0


def _uutt_exact(p):
    s = 2 * _dot(p[:, 0], p[:, 1])
    a, b = 2 * _dot(p[:, 0], p[:, 2]), 2 * _dot(p[:, 0], p[:, 3])  # m^2 - t, m^2 - u
    return 4.0 / 9.0 * G2 ** 2 * (a * a + b * b + 2 * MT * MT * s) / s ** 2


def _uuttg_exact(p):
    """u u~ -> t t~ g from its five diagrams, colour by explicit index sums."""
    gam, g, n = _dirac(), math.sqrt(G2), p.shape[0]
    pu, pub, pt, ptb, pg = (p[:, i] for i in range(5))
    one = torch.eye(4, dtype=_C, device=p.device)
    u = _spinors(pu, 0.0, gam, False)
    vb = torch.einsum("nka,ab->nkb", _spinors(pub, 0.0, gam, True).conj(), gam[0])
    ub = torch.einsum("nka,ab->nkb", _spinors(pt, MT, gam, False).conj(), gam[0])
    v = _spinors(ptb, MT, gam, True)
    eps = _polarisations(pg)
    es = _slash(eps, gam)
    met = METRIC.to(p.device).to(_C)

    def cur(a, M, b):  # abar gamma^mu M b with M between spinors given as a list
        return torch.einsum("nia,mab,njb->nijm", a, gam, b)

    def prop(q, m, terms, w):
        D = _square(terms, m * m).to(_C) + (1j * m * w)
        return (_slash(q, gam) + m * one) / D[:, None, None]

    s12, s34 = _square([pu, pub]).to(_C), _square([pt, ptb]).to(_C)
    L, Hc = cur(vb, None, u), cur(ub, None, v)  # [n,i(ub~),j(u),m], [n,k,l,m]
    sA = torch.einsum("nab,nhbc,njc->nhja", prop(pu - pg, 0.0, [pu, -pg], 0.0), es, u)
    sB = torch.einsum("nia,nhab,nbc->nhic", vb, es, prop(pg - pub, 0.0, [pg, -pub], 0.0))
    sC = torch.einsum("nka,nhab,nbc->nhkc", ub, es, prop(pt + pg, MT, [pt, pg], GAMMA_T))
    sD = torch.einsum("nab,nhbc,nlc->nhla", prop(-ptb - pg, MT, [ptb, pg], GAMMA_T), es, v)
    A = [torch.einsum("nia,mab,nhjb,m,nklm->nhijkl", vb, gam, sA, met, Hc) / s34[:, None, None, None, None, None],
         torch.einsum("nhia,mab,njb,m,nklm->nhijkl", sB, gam, u, met, Hc) / s34[:, None, None, None, None, None],
         torch.einsum("nhka,mab,nlb,m,nijm->nhijkl", sC, gam, v, met, L) / s12[:, None, None, None, None, None],
         torch.einsum("nka,mab,nhlb,m,nijm->nhijkl", ub, gam, sD, met, L) / s12[:, None, None, None, None, None]]
    q1, q2, q3 = pu + pub, -(pt + ptb), -pg  # incoming
    m3 = met
    LH = torch.einsum("nijm,m,nklm->nijkl", L, m3, Hc)
    Le, He = torch.einsum("nijm,m,nhm->nhij", L, m3, eps), torch.einsum("nklm,m,nhm->nhkl", Hc, m3, eps)

    def on(q, x):
        return torch.einsum("nm,m,n...m->n...", q.to(_C), m3, x)

    V = (torch.einsum("nijkl,nh->nhijkl", LH, on(q1 - q2, eps)) + torch.einsum("nhkl,nij->nhijkl", He, on(q2 - q3, L))
         + torch.einsum("nhij,nkl->nhijkl", Le, on(q3 - q1, Hc)))
    A.append(V / (s12 * s34)[:, None, None, None, None, None])
    # colour tensors over (j of u, i of u~, k of t, l of t~, a of g)
    T = torch.from_numpy(_gell_mann()).cuda()
    comm = torch.einsum("aij,bjk->abik", T, T) - torch.einsum("bij,ajk->abik", T, T)  # = i f^{abc} T^c
    f = (-2j * torch.einsum("abij,cji->abc", comm, T))
    col = [torch.einsum("bxy,ayj,bkl->xjkla", T, T, T), torch.einsum("axy,byj,bkl->xjkla", T, T, T),
           torch.einsum("bxj,aky,byl->xjkla", T, T, T), torch.einsum("bxj,bky,ayl->xjkla", T, T, T),
           torch.einsum("bca,bxj,ckl->xjkla", f, T, T)]
    # vertices i g gamma T and g f V, gluon propagators -i / q^2, quark propagators i / D
    ph = [(1j * g) ** 3 * -1j * 1j] * 4 + [(1j * g) ** 2 * g * (-1j) ** 2]
    out = 0.0
    for a in range(5):
        for b in range(5):
            c = complex((col[a] * col[b].conj()).sum()) * ph[a] * complex(ph[b]).conjugate()
            out = out + (c * (A[a] * A[b].conj()).flatten(1).sum(1)).real
    return out / 36.0


def _philox(ctr, seed):
    """Philox4x64-10 (Salmon et al. 2011) on uint64 arrays."""
    M, W, lo32 = (0xD2E7470EE14C6C93, 0xCA5A826395121157), (0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B), np.uint64(0xFFFFFFFF)

    def mul(a, b):
        bl, bh = np.uint64(b & 0xFFFFFFFF), np.uint64(b >> 32)
        al, ah = a & lo32, a >> np.uint64(32)
        mid = ((al * bl) >> np.uint64(32)) + ((ah * bl) & lo32) + al * bh
        return ah * bh + ((ah * bl) >> np.uint64(32)) + (mid >> np.uint64(32)), a * np.uint64(b)

    x, key = [c.copy() for c in ctr], [seed, 0]
    for _ in range(10):
        h0, l0 = mul(x[0], M[0])
        h1, l1 = mul(x[2], M[1])
        x = [h1 ^ x[1] ^ np.uint64(key[0]), l1, h0 ^ x[3] ^ np.uint64(key[1]), l0]
        key = [(key[0] + W[0]) % 2 ** 64, (key[1] + W[1]) % 2 ** 64]
    return x


def _rambo_exact(proc, n, seed):
    masses, rs = np.array(_final_masses(proc)), SQRTS[proc]
    nf = len(masses)
    ev, sl = np.meshgrid(np.arange(n, dtype=np.uint64), np.arange(nf, dtype=np.uint64), indexing="ij")
    z = np.zeros_like(ev)
    u = [((w >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53 for w in _philox([ev, sl, z, z], seed)]
    c, phi = 2 * u[0] - 1, 2 * math.pi * u[1]
    s, e = np.sqrt(np.maximum(0.0, 1 - c * c)), -np.log(u[2] * u[3])
    q = np.stack([e, e * s * np.cos(phi), e * s * np.sin(phi), e * c], -1)
    Q = q.sum(1)
    M = np.sqrt(Q[:, 0] ** 2 - (Q[:, 1:] ** 2).sum(1))[:, None]
    b, gamma = -Q[:, 1:] / M, Q[:, :1] / M
    bq = (b[:, None] * q[..., 1:]).sum(2)
    p3 = (rs / M)[..., None] * (q[..., 1:] + b[:, None] * q[..., :1] + (bq / (1 + gamma))[..., None] * b[:, None])
    p3 -= p3.mean(1, keepdims=True)
    k2 = (p3 ** 2).sum(2)
    xi = np.full((n, 1), math.sqrt(1 - (masses.sum() / rs) ** 2))
    for _ in range(30):
        en = np.sqrt(masses ** 2 + xi ** 2 * k2)
        xi = xi - (en.sum(1, keepdims=True) - rs) / (xi * k2 / en).sum(1, keepdims=True)
    p = np.zeros((n, nf + 2, 4))
    p[:, 0, 0] = p[:, 1, 0] = p[:, 0, 3] = 0.5 * rs
    p[:, 1, 3] = -0.5 * rs
    p[:, 2:, 1:] = p3 * xi[..., None]
    p[:, 2:, 0] = np.sqrt(masses ** 2 + xi ** 2 * k2)
    return p


def exact(case, seed):
    op, proc, n = case["op"], case["proc"], case["n"]
    if op == "unweight":
        return None  # whole numbers alone
    if op == "rambo":
        return _rambo_exact(proc, n, seed)
    p = _momenta(proc, n, seed)
    if proc.startswith("g g"):
        me, wk = _gg_exact(p, proc)
        return (me, None, None, wk) if op == "select" else me
    me = {"e+ e- > mu+ mu-": _ee_exact, "u u~ > t t~": _uutt_exact, "u u~ > t t~ g": _uuttg_exact}[proc](p)
    return me
