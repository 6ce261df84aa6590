"""The calls that a user of the library makes, at sizes over its whole range:
PM steps from a 32^3 box to the 512^3 / 1536^3 run and the filtered 768^3 /
1152^3 run, 2LPT set-ups, an ensemble replay, the outputs of a run (P(k),
multipoles, halos) and a training iteration of the learned correction.

Inputs are made with plain torch from the seed: a Gaussian field with a CDM-like
spectrum, its 2LPT displacements, and for the late states Lagrangian patches
collapsed into halos, so that positions cluster as they do at a ~ 0.5 while
neighbouring lattice sites stay neighbours.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1509_04685_gb300 as C

A_INIT, N_STEPS = 0.05, 40  # z = 19, 40 linearly spaced nodes
NODE = 20                   # a = 0.537: the node the late states sit at
MEMBERS = 101               # halos of more than 100 particles
OM, OL, OB, H, S8, NS, TCMB = 0.25, 0.75, 0.044, 0.7, 0.8, 0.95, 2.7255
DEV = "cuda"


def listed():
    return [
        # the smallest run (tests, quick looks): a step is launches and latency
        {"name": "step_32_96", "kind": "step", "nq": 32, "ng": 96, "box": 128.0, "flags": 0, "filter": False},
        # a mesh side picked for its physics (PM_grid = 2, 2^4 5^2), not a power-of-two family
        {"name": "step_200_400", "kind": "step", "nq": 200, "ng": 400, "box": 400.0, "flags": 0, "filter": False},
        # one production mock at PM_grid = 3, 3 Mpc/h spacing
        {"name": "step_256_768", "kind": "step", "nq": 256, "ng": 768, "box": 768.0, "flags": 0, "filter": False},
        # the benchmarked run: 512^3 particles, 1536^3 mesh, L = 1536 Mpc/h
        {"name": "step_512_1536", "kind": "step", "nq": 512, "ng": 1536, "box": 1536.0, "flags": 0, "filter": False},
        # the largest run in its learned form: 768^3 particles on a filtered 1.5x mesh
        {"name": "step_768_1152_filter", "kind": "step", "nq": 768, "ng": 1152, "box": 1536.0, "flags": 0,
         "filter": True},
        # uneven small realisations in one graph launch (covariance mocks): 2LPT + first nodes
        {"name": "ensemble_6", "kind": "ensemble", "members": 6, "nodes": 8, "streams": 4},
        # initial conditions of the 256^3 run, made once per seed
        {"name": "ic_256", "kind": "ic", "nq": 256, "ng": 256, "box": 768.0},
        # matter P(k) of the benchmarked particle count on a 1024^3 estimator mesh, closed-form corrections
        {"name": "pk_512_1024", "kind": "pk", "nq": 512, "ng_pk": 1024, "box": 1536.0, "flags": 3, "between": False},
        # the same statistic with the iterated aliasing correction, for a published spectrum
        {"name": "pk_iter_256_512", "kind": "pk", "nq": 256, "ng_pk": 512, "box": 768.0, "flags": 4,
         "between": False},
        # redshift-space multipoles at an output time between two nodes
        {"name": "multipoles_256_512", "kind": "multipoles", "nq": 256, "ng_pk": 512, "box": 768.0, "flags": 1,
         "between": True},
        # friends-of-friends halos of the benchmarked run
        {"name": "fof_512", "kind": "fof", "nq": 512, "box": 1536.0, "b": 0.2},
        # one training iteration (gradient + Adam) of the convolution net
        {"name": "train_128", "kind": "train", "nq": 128, "box": 256.0},
    ]


def _sides(lo, hi):
    """Even 2^a 3^b 5^c sides in [lo, hi]."""
    out = []
    for n in range(lo + lo % 2, hi + 1, 2):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def _pick(rng, lo, hi):
    """A side from the list, spread over the logarithm of the range."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_sides(lo, hi), key=lambda n: abs(n - x))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["ic", "pk", "pk", "multipoles", "fof", "train", "ensemble"])
    if kind == "step":
        while True:
            nq = _pick(rng, 32, 512)
            ng = min(_sides(nq, 1536), key=lambda n, t=nq * rng.choice([1.0, 1.5, 2.0, 3.0]): abs(n - t))
            if ng <= 1536:
                break
        filt = rng.random() < 0.25
        return {"kind": "step", "nq": nq, "ng": ng, "box": round(nq * rng.uniform(1.0, 4.0), 1),
                "flags": rng.choice([0, 0, C.FLAG_PM_ONLY, C.FLAG_MODIFIED_KDK]), "filter": filt}
    if kind == "ensemble":
        return {"kind": "ensemble", "members": rng.randint(2, 8), "nodes": rng.randint(2, 10),
                "streams": rng.randint(1, 8)}
    if kind == "ic":
        nq = _pick(rng, 32, 512)
        return {"kind": "ic", "nq": nq, "ng": nq, "box": round(nq * rng.uniform(1.0, 4.0), 1)}
    if kind in ("pk", "multipoles"):
        nq = _pick(rng, 32, 512)
        multi = kind == "multipoles"
        flags = rng.choice([0, 1, 3] if multi else [0, 1, 3, 3, 4])
        ng = _pick(rng, 48, 512 if flags == 4 else 1024)
        return {"kind": kind, "nq": nq, "ng_pk": ng, "box": round(nq * rng.uniform(1.0, 4.0), 1), "flags": flags,
                "between": rng.random() < 0.5}
    if kind == "fof":
        nq = _pick(rng, 32, 512)
        return {"kind": "fof", "nq": nq, "box": round(nq * rng.uniform(1.0, 4.0), 1),
                "b": round(rng.uniform(0.1, 0.3), 3)}
    nq = rng.choice([32, 48, 64, 80, 96, 128])
    return {"kind": "train", "nq": nq, "box": round(nq * rng.uniform(1.5, 3.0), 1)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _kgrids(n, box, dtype=torch.float32):
    k = torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=dtype) * (2 * math.pi / box)
    kz = torch.fft.rfftfreq(n, 1.0 / n, device=DEV, dtype=dtype) * (2 * math.pi / box)
    return k[:, None, None], k[None, :, None], kz[None, None, :]


def _lpt(nq, box, gen):
    """Psi1, Psi2 (3, nq^3) float32 of a Gaussian field with a CDM-like spectrum,
    Psi1 scaled to 4.5 Mpc/h rms per component."""
    ks = _kgrids(nq, box)
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    kk = k2.sqrt()
    q = kk / 0.17
    amp = kk.sqrt() * torch.log1p(2.34 * q) / (2.34 * q)
    amp = amp / (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** 0.25
    amp[0, 0, 0] = 0.0
    half = nq // 2  # the Nyquist planes carry no mode
    amp[half] = 0.0
    amp[:, half] = 0.0
    amp[:, :, half] = 0.0
    w = torch.randn((nq, nq, nq), generator=gen, device=DEV)
    phi = torch.fft.rfftn(w) * (amp / k2)
    del w, amp, q, kk
    shape = (nq, nq, nq)
    psi1 = torch.empty((3, nq**3), dtype=torch.float32, device=DEV)
    for a in range(3):
        psi1[a] = torch.fft.irfftn(1j * ks[a] * phi, s=shape).reshape(-1)
    scale = 4.5 / float(psi1[0].double().square().mean().sqrt())
    psi1 *= scale
    phi *= scale
    f = lambda a, b: torch.fft.irfftn(ks[a] * ks[b] * phi, s=shape)
    xx, yy = f(0, 0), f(1, 1)
    d2 = xx * yy
    xx += yy
    d2 += xx * f(2, 2)
    del xx, yy
    for a, b in ((0, 1), (0, 2), (1, 2)):
        d2 -= f(a, b).square_()
    phi = torch.fft.rfftn(d2) / k2
    del d2, k2
    phi[0, 0, 0] = 0.0
    phi[half] = 0.0
    phi[:, half] = 0.0
    phi[:, :, half] = 0.0
    psi2 = torch.empty_like(psi1)
    for a in range(3):
        psi2[a] = torch.fft.irfftn(-1j * ks[a] * phi, s=shape).reshape(-1)
    return psi1, psi2


def _late_state(nq, box, seed):
    """(d, v, psi1, psi2) at a ~ 0.5: 2LPT displacements, with a share of the
    Lagrangian patches of 4, 8 and 16 sites collapsed to a sixth of their size."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000003 * (seed + 1) % (2**31))
    psi1, psi2 = _lpt(nq, box, gen)
    D1 = 0.66
    d = D1 * psi1 + (-3.0 / 7.0 * D1 * D1) * psi2
    v = torch.randn((3, nq**3), generator=gen, device=DEV)
    v *= 0.1
    i = torch.arange(nq, device=DEV)
    spacing = box / nq
    for s, share in ((4, 0.06), (8, 0.02), (16, 0.003)):
        nb = -(-nq // s)
        hit = torch.rand((nb, nb, nb), generator=gen, device=DEV) < share
        b, mid = i // s, torch.clamp((i // s) * s + s // 2, max=nq - 1)
        m = hit[b][:, b][:, :, b].reshape(-1)
        for a in range(3):
            da = d[a].view(nq, nq, nq)
            centre = da[mid][:, mid][:, :, mid].reshape(-1)
            shape = [1, 1, 1]
            shape[a] = nq
            rel = ((i - mid).to(torch.float32) * spacing).view(shape).expand(nq, nq, nq).reshape(-1)
            noise = torch.randn(nq**3, generator=gen, device=DEV) * (0.04 * s * spacing)
            d[a] = torch.where(m, centre - (5.0 / 6.0) * rel + noise, d[a])
            v[a] = torch.where(m, v[a] * 10.0, v[a])
            del centre, rel, noise
    return d, v, psi1, psi2


def _filter(seed):
    """A fitted-looking transfer table: 8 scale-factor rows of 16 |k| nodes."""
    g = np.random.default_rng(seed)
    x = np.arange(16) / 15.0
    a = np.arange(8)[:, None] / 7.0
    t = 1.0 + (0.2 + 0.6 * a) * x**2 + 0.02 * g.standard_normal((8, 16))
    return torch.tensor(t, dtype=torch.float32, device=DEV)


def _a_of(node, n=N_STEPS):
    return A_INIT + node * (1.0 - A_INIT) / (n - 1)


def _members(count, seed):
    """(nq, ng, box, seed): 96^3, 128^3 and 160^3 particles, PM_grid 1, 2, 3, 1 Mpc/h spacing."""
    out = []
    for i in range(count):
        nq = (96, 128, 160)[(i // 2) % 3]
        out.append((nq, (1 + i % 3) * nq, float(nq), 7919 * (seed % 100003) + i))
    return out


def _between(case):
    return _a_of(NODE) + (0.4 * (1.0 - A_INIT) / (N_STEPS - 1) if case["between"] else 0.0)


def _train_inputs(case, seed):
    nq = case["nq"]
    d = _late_state(nq, case["box"], seed)[0]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(77 + seed)
    target = 0.5 * torch.randn((3, nq**3), generator=gen, device=DEV)
    g = torch.Generator().manual_seed(seed)
    p = torch.zeros(C.NET_NPARAMS, dtype=torch.float32)
    for k, (off, shape) in C.NET_OFFSETS.items():
        n = int(np.prod(shape))
        std = (2.0 / (shape[1] * 27)) ** 0.5 if k.startswith("W") else 0.05
        p[off: off + n] = torch.randn(n, generator=g) * (0.3 * std if k == "W3" else std)
    return d, target, p.to(DEV), _filter(seed)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        mem = _members(case["members"], seed)
        cfgs = [C.make_config(nq, ng, box, A_INIT, 1.0, N_STEPS) for nq, ng, box, _ in mem]
        sims = [C.Simulation(c) for c in cfgs]
        for s, m in zip(sims, mem):  # one uncaptured step sets the kernel attributes
            s.ic(m[3])
            s.step(0)
        ens = C.Ensemble(cfgs, [m[3] for m in mem], [s.state for s in sims], [s.ws for s in sims],
                         nstreams=case["streams"], step_from=0, step_to=case["nodes"])
        return {"kind": kind, "ens": ens, "sims": sims}
    nq, box = case["nq"], case["box"]
    if kind == "ic":
        sim = C.Simulation(C.make_config(nq, case["ng"], box, A_INIT, 1.0, N_STEPS))
        return {"kind": kind, "sim": sim, "seed": seed}
    if kind == "train":
        d, target, p, filt = _train_inputs(case, seed)
        wpack = torch.zeros(C.NET_NPACK, dtype=torch.bfloat16, device=DEV)
        net = C.make_net(p, wpack, filt)
        sim = C.Simulation(C.make_config(nq, nq, box, A_INIT, 1.0, N_STEPS, flags=C.FLAG_LEARNED, net=net))
        sim.init_tables()
        sim.d.copy_(d)
        C.cola_net_pack(net)
        z = torch.zeros_like
        return {"kind": kind, "sim": sim, "net": net, "p": p, "m": z(p), "v": z(p), "grad": z(p), "target": target,
                "loss": torch.zeros(1, dtype=torch.float64, device=DEV), "t": 0}
    ng = case["ng"] if kind == "step" else case.get("ng_pk", nq)
    flags, net = 0, None
    if kind == "step":
        flags = case["flags"]
        if case["filter"]:
            flags |= C.FLAG_LEARNED
            net = C.make_net(None, None, _filter(seed))
    sim = C.Simulation(C.make_config(nq, ng, box, A_INIT, 1.0, N_STEPS, flags=flags, net=net))
    sim.init_tables()
    sim.load_state(*_late_state(nq, box, seed))
    sim.node = NODE
    st = {"kind": kind, "sim": sim, "case": dict(case)}
    if kind == "step":
        st["d0"], st["v0"] = sim.d.clone(), sim.v.clone()
    if kind == "fof":
        i32 = lambda n: torch.zeros(n, dtype=torch.int32, device=DEV)
        cap = nq**3 // MEMBERS + 1
        st.update(group=i32(nq**3), roots=i32(cap), sizes=i32(cap),
                  count=torch.zeros(1, dtype=torch.int64, device=DEV),
                  fws=torch.empty(C.cola_fof_workspace_size(sim.cfg), dtype=torch.uint8, device=DEV))
    return st


def run(state):
    kind = state["kind"]
    if kind == "ensemble":
        state["ens"].launch()
        return [[s.d, s.v, s.psi1, s.psi2] for s in state["sims"]]
    sim = state["sim"]
    if kind == "ic":
        sim.ic(state["seed"])
        return [sim.d, sim.v, sim.psi1, sim.psi2]
    if kind == "train":
        state["t"] += 1
        C.cola_net_grad(sim.cfg, sim.state, _a_of(NODE), state["target"], state["grad"], state["loss"], sim.ws)
        C.cola_adam(state["p"], state["grad"], state["m"], state["v"], state["p"].numel(), state["t"], 1e-3)
        C.cola_net_pack(state["net"])
        return [state["grad"], state["p"], state["m"], state["v"], state["loss"]]
    case = state["case"]
    if kind == "step":
        # node after node to the end of the run, then the next run from the stored state
        if sim.node >= N_STEPS - 1:
            sim.d.copy_(state["d0"])
            sim.v.copy_(state["v0"])
            sim.node = NODE
        sim.step(sim.node)
        return [sim.d, sim.v]
    if kind == "pk":
        return list(sim.power(case["ng_pk"], a_out=_between(case), flags=case["flags"], node=NODE))
    if kind == "multipoles":
        return list(sim.multipoles(case["ng_pk"], a_out=_between(case), flags=case["flags"], node=NODE))
    C.cola_fof(sim.cfg, sim.state, case["b"], state["group"], state["fws"])
    C.cola_fof_halos(sim.cfg, state["group"], MEMBERS, state["roots"], state["sizes"], state["count"], state["fws"])
    return [state["group"], state["roots"], state["sizes"], state["count"]]


def work(case):
    """Inputs read once, outputs written once; transforms at 2.5 n log2 n per real
    mesh of n cells, CIC deposit or gather at about 50 flops per particle."""
    kind = case["kind"]
    fft = lambda n: 2.5 * n**3 * 3 * math.log2(n)
    if kind == "ensemble":
        b = f = 0.0
        for nq, ng, _, _ in _members(case["members"], 0):
            b += 48.0 * nq**3  # the set-up's four fields, updated in place by the nodes
            f += 14 * fft(nq) + case["nodes"] * (4 * fft(ng) + 150.0 * nq**3)
        return {"bytes": b, "flops": f}
    nq = case["nq"]
    n3 = float(nq) ** 3
    if kind == "step":
        return {"bytes": 72.0 * n3, "flops": 4 * fft(case["ng"]) + 150.0 * n3}
    if kind == "ic":
        return {"bytes": 48.0 * n3, "flops": 14 * fft(nq) + 200.0 * n3}
    if kind in ("pk", "multipoles"):
        ng = case["ng_pk"]
        read = 12.0 + (36.0 if case["between"] else (12.0 if kind == "multipoles" else 0.0))
        # iterated correction: 125 image terms for each of the ng^3 / 16 distinct modes, three times
        extra = 3 * 125 * 4 * ng**3 / 16.0 if case["flags"] == 4 else 0.0
        return {"bytes": read * n3, "flops": fft(ng) + 50.0 * n3 + 5.0 * ng**3 + extra}
    if kind == "fof":
        return {"bytes": 16.0 * n3, "flops": 200.0 * n3}
    # forward, weight and input gradients of the three layers (the first needs no input gradient)
    macs = 27.0 * (3 * 16 * 16 + 2 * 4 * 16 + 3 * 16 * 3)
    return {"bytes": 24.0 * n3, "flops": 2 * macs * n3 + 4 * fft(nq) + 300.0 * n3}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the method's definitions
# ---------------------------------------------------------------------------
def _E(a):
    return np.sqrt(OM / a**3 + (1 - OM - OL) / a**2 + OL)


def _growth(points):
    """{a: (D1, D2, dD1/da, dD2/da)} from the growth ODEs in ln a, D1(1) = 1, the
    Einstein-de Sitter modes D1 = a, D2 = -3/7 a^2 early on (u = D1/a, w = D2/a^2)."""
    def rhs(y, s):
        a = math.exp(y)
        E2 = OM / a**3 + (1 - OM - OL) / a**2 + OL
        oma = OM / a**3 / E2
        fr = 2.0 + (-3.0 * OM / a**3 - 2.0 * (1 - OM - OL) / a**2) / (2.0 * E2)
        u, up, w, wp = s
        return np.array([up, -(2 + fr) * up - (1 + fr - 1.5 * oma) * u,
                         wp, -(4 + fr) * wp - (4 + 2 * fr - 1.5 * oma) * w - 1.5 * oma * u * u])

    s, y, out = np.array([1.0, 0.0, -3.0 / 7.0, 0.0]), math.log(1e-5), {}
    for a in sorted(set(points) | {1.0}):
        y1 = math.log(a)
        n = max(1, math.ceil((y1 - y) / (1.0 / 256)))
        h = (y1 - y) / n
        for _ in range(n):
            k1 = rhs(y, s)
            k2 = rhs(y + h / 2, s + h / 2 * k1)
            k3 = rhs(y + h / 2, s + h / 2 * k2)
            k4 = rhs(y + h, s + h * k3)
            s = s + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
            y += h
        y = y1
        out[a] = (a * s[0], a * a * s[2], s[0] + s[1], a * (2 * s[2] + s[3]))
    n = out[1.0][0]
    return {a: (D1 / n, D2 / n**2, e1 / n, e2 / n**2) for a, (D1, D2, e1, e2) in out.items()}


def _quad(f, a, b):
    x, w = np.polynomial.legendre.leggauss(48)
    t = 0.5 * (b - a) * x + 0.5 * (a + b)
    return 0.5 * (b - a) * float(np.sum(w * f(t)))


def _row(j, flags):
    """The kick and drift coefficients of node j."""
    a = [_a_of(i) for i in range(N_STEPS)]
    g = _growth([a[j]] + ([a[j + 1]] if j + 1 < N_STEPS else []))
    lo = 0.5 * (a[j - 1] + a[j]) if j else a[0]
    hi = 0.5 * (a[j] + a[j + 1]) if j + 1 < N_STEPS else a[-1]
    last = j + 1 == N_STEPS
    kick = _quad(lambda t: 1 / (t * _E(t)), lo, hi)
    drift = 0.0 if last else _quad(lambda t: 1 / (t**3 * _E(t)), a[j], a[j + 1])
    if flags & C.FLAG_MODIFIED_KDK:
        n = -2.5
        kick = (hi**n - lo**n) / (n * a[j] ** n * _E(a[j]))
        drift = 0.0 if last else _quad(lambda t: t**n / (t**3 * _E(t)), a[j], a[j + 1]) / hi**n
    D1, D2 = g[a[j]][:2]
    green = 1.5 * OM / a[j]
    c1, c2, e1, e2 = green * D1, green * (D2 - D1 * D1), 0.0, 0.0
    if not last:
        e1, e2 = g[a[j + 1]][0] - D1, g[a[j + 1]][1] - D2
    if flags & C.FLAG_PM_ONLY:
        c1 = c2 = e1 = e2 = 0.0
    return green, c1, c2, kick, drift, e1, e2, last


def _cells(d, lo, hi, nq, ng, box):
    """CIC corners and weights of particles [lo, hi): 8 pairs (flat cell, weight)."""
    p = torch.arange(lo, hi, device=DEV)
    c0, c1, f = [], [], []
    for a, i in enumerate((p // (nq * nq), (p // nq) % nq, p % nq)):
        u = i.double() * (ng / nq) + 0.5 + d[a, lo:hi].double() * (ng / box)
        fl = torch.floor(u)
        f.append(u - fl)
        c = torch.remainder(fl.long(), ng)
        c0.append(c)
        c1.append(torch.remainder(c + 1, ng))
    for x, wx in ((c0[0], 1 - f[0]), (c1[0], f[0])):
        for y, wy in ((c0[1], 1 - f[1]), (c1[1], f[1])):
            for z, wz in ((c0[2], 1 - f[2]), (c1[2], f[2])):
                yield (x * ng + y) * ng + z, wx * wy * wz


CHUNK = 1 << 24


def _delta_k(d, nq, ng, box):
    rho = torch.zeros(ng**3, dtype=torch.float64, device=DEV)
    for lo in range(0, nq**3, CHUNK):
        hi = min(nq**3, lo + CHUNK)
        for cell, w in _cells(d, lo, hi, nq, ng, box):
            rho.scatter_add_(0, cell, w)
    rho *= (ng / nq) ** 3
    rho -= 1.0
    dk = torch.fft.rfftn(rho.view(ng, ng, ng))
    return dk


def _force(d, nq, ng, box, green, table=None):
    """The CIC-gathered force, component by component (a generator)."""
    phi = _delta_k(d, nq, ng, box)
    ks = _kgrids(ng, box, torch.float64)
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    phi /= k2
    phi[0, 0, 0] = 0.0
    if table is not None:
        step = math.sqrt(3.0) * math.pi * ng / box / (table.numel() - 1)
        t = table.double()
        for x in range(ng):
            u = k2[x].sqrt() / step
            b = u.long().clamp(max=table.numel() - 2)
            fr = (u - b).clamp(max=1.0)
            phi[x] *= (1 - fr) * t[b] + fr * t[b + 1]
    del k2
    phi *= green
    for a in range(3):
        k = ks[a].clone()
        k.view(-1)[ng // 2] = 0.0
        F = torch.fft.irfftn(phi * (1j * k), s=(ng, ng, ng)).view(-1)
        out = torch.empty(nq**3, dtype=torch.float64, device=DEV)
        for lo in range(0, nq**3, CHUNK):
            hi = min(nq**3, lo + CHUNK)
            acc = torch.zeros(hi - lo, dtype=torch.float64, device=DEV)
            for cell, w in _cells(d, lo, hi, nq, ng, box):
                acc += w * F[cell]
            out[lo:hi] = acc
        del F
        yield out


def _filter_row(table, a):
    r = int(math.floor((a - A_INIT) / (1.0 - A_INIT) * (table.shape[0] - 1) + 0.5))
    return table[min(max(r, 0), table.shape[0] - 1)]


def _step(d, v, psi1, psi2, j, nq, ng, box, flags, table=None):
    """One node on 64-bit fields; returns new (d, v)."""
    green, c1, c2, kick, drift, e1, e2, last = _row(j, flags)
    row = None if table is None else _filter_row(table, _a_of(j))
    nd, nv = torch.empty(3, nq**3, dtype=torch.float64, device=DEV), torch.empty(3, nq**3, dtype=torch.float64,
                                                                               device=DEV)
    for a, F in enumerate(_force(d, nq, ng, box, green, row)):
        s1, s2 = psi1[a].double(), psi2[a].double()
        nv[a] = v[a].double() + kick * (F - c1 * s1 - c2 * s2)
        nd[a] = d[a].double() if last else d[a].double() + drift * nv[a] + e1 * s1 + e2 * s2
    return nd, nv


def _noise(n, seed):
    """Philox-4x32-10 white noise of the n^3 cells (key = seed, counter = cell)."""
    mask = 0xFFFFFFFF
    out = torch.empty(n**3, dtype=torch.float64, device=DEV)

    def mul(m, x):  # the 64-bit product of two 32-bit values wraps into int64 exactly
        p = x * m
        return (p >> 32) & mask, p & mask

    for lo in range(0, n**3, CHUNK):
        i = torch.arange(lo, min(n**3, lo + CHUNK), device=DEV)
        c = [i & mask, i >> 32, torch.zeros_like(i), torch.zeros_like(i)]
        k0, k1 = seed & mask, (seed >> 32) & mask
        for r in range(10):
            if r:
                k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
            h0, l0 = mul(0xD2511F53, c[0])
            h1, l1 = mul(0xCD9E8D57, c[2])
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        u = lambda a, b: (((a >> 5) << 26) + (b >> 6) + 1).double() * 2.0**-53
        out[lo: lo + i.numel()] = torch.sqrt(-2.0 * torch.log(u(c[0], c[1]))) * torch.cos(2 * math.pi * u(c[2], c[3]))
    return out.view(n, n, n)


def _transfer(k, np_=torch):
    """Eisenstein & Hu (1998), no wiggles."""
    om, ob, fb = OM * H * H, OB * H * H, OB / OM
    s = 44.5 * math.log(9.83 / om) / math.sqrt(1 + 10 * ob**0.75)
    al = 1 - 0.328 * math.log(431 * om) * fb + 0.38 * math.log(22.3 * om) * fb * fb
    g = OM * H * (al + (1 - al) / (1 + (0.43 * k * H * s) ** 4))
    q = k * (TCMB / 2.7) ** 2 / g
    L0 = np_.log(2 * math.e + 1.8 * q)
    return L0 / (L0 + (14.2 + 731 / (1 + 62.5 * q)) * q * q)


def _amplitude():
    x = np.linspace(math.log(1e-7), math.log(250.0), (1 << 16) + 1)
    k = np.exp(x)
    y = 8 * k
    W = np.where(y < 0.1, 1 - y**2 / 10 + y**4 / 280 - y**6 / 15120, 3 * (np.sin(y) - y * np.cos(y)) / y**3)
    f = k ** (3 + NS) * _transfer(k, np) ** 2 * W * W
    w = np.ones(len(x))
    w[1:-1:2], w[2:-1:2] = 4, 2
    return S8**2 / (np.sum(w * f) * (x[1] - x[0]) / 3 / (2 * math.pi**2))


def _ic(seed, nq, box):
    ks = _kgrids(nq, box, torch.float64)
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    kk = k2.sqrt()
    amp = torch.sqrt(_amplitude() * kk**NS * _transfer(kk) ** 2 / (box / nq) ** 3)
    half = nq // 2
    amp[half] = 0.0
    amp[:, half] = 0.0
    amp[:, :, half] = 0.0
    amp[0, 0, 0] = 0.0
    phi = torch.fft.rfftn(_noise(nq, seed)) * (amp / k2)
    del amp, kk
    s = (nq, nq, nq)
    psi1 = torch.stack([torch.fft.irfftn(1j * ks[a] * phi, s=s).reshape(-1) for a in range(3)])
    f = lambda a, b: torch.fft.irfftn(ks[a] * ks[b] * phi, s=s)
    xx, yy, zz = f(0, 0), f(1, 1), f(2, 2)
    d2 = xx * yy + (xx + yy) * zz
    del xx, yy, zz
    for a, b in ((0, 1), (0, 2), (1, 2)):
        d2 -= f(a, b) ** 2
    phi = torch.fft.rfftn(d2) / k2
    phi[0, 0, 0] = 0.0
    phi[half] = 0.0
    phi[:, half] = 0.0
    phi[:, :, half] = 0.0
    psi2 = torch.stack([torch.fft.irfftn(-1j * ks[a] * phi, s=s).reshape(-1) for a in range(3)])
    D1, D2 = _growth([A_INIT])[A_INIT][:2]
    return D1 * psi1 + D2 * psi2, torch.zeros_like(psi1), psi1, psi2


def _jing(n, ng, lnk2, slope):
    """Image sum C of modes n (three index tensors) for power-law slopes `slope`."""
    xs = [[i.double() + ng * m for m in range(-2, 3)] for i in n]
    w = []
    for i, x in zip(n, xs):
        s4 = torch.sin(math.pi * i.double() / ng) ** 4
        w.append([torch.where(i == 0, torch.full_like(s4, float(m == 2)),
                              s4 / torch.where(i == 0, torch.ones_like(s4), math.pi * x[m] / ng) ** 4)
                  for m in range(5)])
    out = torch.zeros_like(lnk2)
    for a in range(5):
        for b in range(5):
            wab, rab = w[0][a] * w[1][b], xs[0][a] ** 2 + xs[1][b] ** 2
            for c in range(5):
                r2 = rab + xs[2][c] ** 2
                out += wab * w[2][c] * torch.exp(0.5 * slope * (torch.log(r2.clamp(min=0.25)) - lnk2))
    return out


def _spectrum(case, seed, multi):
    nq, ng, box, flags = case["nq"], case["ng_pk"], case["box"], case["flags"]
    d, v, psi1, psi2 = _late_state(nq, box, seed)
    a0, a1 = _a_of(NODE), _between(case)
    pos = d.double()
    g = _growth([a0, a1])
    if a1 != a0:
        pos += _quad(lambda t: 1 / (t**3 * _E(t)), a0, a1) * v
        pos += (g[a1][0] - g[a0][0]) * psi1 + (g[a1][1] - g[a0][1]) * psi2
    if multi:
        pos[2] += v[2].double() / (a1 * a1 * _E(a1)) + a1 * g[a1][2] * psi1[2] + a1 * g[a1][3] * psi2[2]
    del d, v, psi1, psi2
    dk = _delta_k(pos, nq, ng, box)
    del pos
    nb, half = ng // 2, ng // 2
    sums = torch.zeros(5, nb + 2, dtype=torch.float64, device=DEV)
    i = torch.fft.fftfreq(ng, 1.0 / ng, device=DEV, dtype=torch.float64)
    kz = torch.arange(half + 1, device=DEV, dtype=torch.float64)
    win = lambda n: torch.sinc(n / ng) ** 2
    jw = lambda n: 1 - 2.0 / 3.0 * torch.sin(math.pi * n / ng) ** 2
    weight = torch.full((half + 1,), 2.0, device=DEV, dtype=torch.float64)
    weight[0] = weight[half] = 1.0
    closed = 3 if flags == 4 else flags
    slabs = max(1, (1 << 24) // (ng * (half + 1)))
    for x0 in range(0, ng, slabs):
        nx = i[x0: x0 + slabs][:, None, None]
        n2 = nx**2 + i[None, :, None] ** 2 + kz[None, None, :] ** 2
        b = torch.floor(n2.sqrt() + 0.5).long()
        p = dk[x0: x0 + slabs].abs() ** 2 * (box**3 / float(ng) ** 6)
        if closed & 1:
            p /= (win(nx) * win(i)[None, :, None] * win(kz)) ** 2
        if closed & 2:
            p /= jw(nx) * jw(i)[None, :, None] * jw(kz)
        mu2 = kz**2 / n2.clamp(min=1.0)
        wt = weight.expand_as(n2)
        b = b.clamp(max=nb + 1).reshape(-1)
        l2, l4 = 1.5 * mu2 - 0.5, (35 * mu2**2 - 30 * mu2 + 3) / 8
        for q, val in enumerate((wt, wt * n2.sqrt(), wt * p, wt * p * l2, wt * p * l4)):
            sums[q].scatter_add_(0, b, val.reshape(-1))
    k = sums[1, 1: nb + 1] / sums[0, 1: nb + 1] * (2 * math.pi / box)
    n, pk = sums[0, 1: nb + 1], sums[2, 1: nb + 1] / sums[0, 1: nb + 1]
    if multi:
        return [k, pk, 5 * sums[3, 1: nb + 1] / n, 9 * sums[4, 1: nb + 1] / n, n]
    if flags != 4:
        return [k, pk, n]
    # C depends on the mode through |n_x|, |n_y|, n_z: fold the power onto one octant
    raw = dk.abs() ** 2 * (box**3 / float(ng) ** 6) * weight
    del dk
    for _ in range(2):
        fold = raw[: half + 1].clone()
        fold[1:half] += raw[half + 1:].flip(0)
        raw = fold.transpose(0, 1).contiguous()
    h = torch.arange(half + 1, device=DEV)
    for _ in range(3):
        lo = torch.clamp(torch.arange(nb, device=DEV) - 1, min=0)
        hi = torch.clamp(torch.arange(nb, device=DEV) + 1, max=nb - 1)
        sl = torch.where((pk[lo] > 0) & (pk[hi] > 0), torch.log(pk[hi] / pk[lo]) / torch.log(k[hi] / k[lo]),
                         torch.zeros_like(pk)).clamp(-4.0, 4.0)
        acc = torch.zeros(nb + 2, dtype=torch.float64, device=DEV)
        step = max(1, (1 << 23) // (half + 1) ** 2)
        for x0 in range(0, half + 1, step):
            nn = torch.meshgrid(h[x0: x0 + step], h, h, indexing="ij")
            n2 = (nn[0] ** 2 + nn[1] ** 2 + nn[2] ** 2).double()
            b = torch.floor(n2.sqrt() + 0.5).long()
            use = (b >= 1) & (b <= nb)
            m = [q[use] for q in nn]
            b = b[use]
            acc.scatter_add_(0, b, raw[x0: x0 + step][use] / _jing(m, ng, torch.log(n2[use]), sl[b - 1]))
        pk = acc[1: nb + 1] / n
    return [k, pk, n]


def _training(case, seed):
    """Gradient and Adam update of the net in 64 bits, by autograd."""
    nq, box = case["nq"], case["box"]
    d, target, p, table = _train_inputs(case, seed)
    a = _a_of(NODE)
    green = 1.5 * OM / a
    delta = torch.fft.irfftn(_delta_k(d, nq, nq, box), s=(nq, nq, nq))
    phi = torch.fft.rfftn(delta)
    ks = _kgrids(nq, box, torch.float64)
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    t = _filter_row(table, a).double()
    u = k2.sqrt() / (math.sqrt(3.0) * math.pi * nq / box / 15)
    b = u.long().clamp(max=14)
    fr = (u - b).clamp(max=1.0)
    phi *= green * ((1 - fr) * t[b] + fr * t[b + 1]) / k2
    phi[0, 0, 0] = 0.0
    F = []
    for e in range(3):
        k = ks[e].clone()
        k.view(-1)[nq // 2] = 0.0
        F.append(torch.fft.irfftn(phi * (1j * k), s=(nq, nq, nq)))
    x = torch.stack([delta] + [f / green for f in F])[None]
    w = p.double().requires_grad_(True)
    part = lambda name: w[C.NET_OFFSETS[name][0]: C.NET_OFFSETS[name][0] + int(np.prod(C.NET_OFFSETS[name][1]))]

    def layer(x, i):
        W = part(f"W{i}").view(*C.NET_OFFSETS[f"W{i}"][1][:2], 3, 3, 3)
        # 27 shifted products: no 64-bit convolution kernel is needed
        out = part(f"b{i}").view(1, -1, 1, 1, 1)
        for tx in range(3):
            for ty in range(3):
                for tz in range(3):
                    s = torch.roll(x, (1 - tx, 1 - ty, 1 - tz), (2, 3, 4))
                    out = out + torch.einsum("oc,bcxyz->boxyz", W[:, :, tx, ty, tz], s)
        return out

    y = layer(torch.relu(layer(torch.relu(layer(x, 1)), 2)), 3)[0]
    loss = 0.0
    cells = list(_cells(d, 0, nq**3, nq, nq, box))
    for e in range(3):
        m = (F[e] + green * y[e]).reshape(-1)
        f = sum(wt * m[cell] for cell, wt in cells)
        loss = loss + ((f - target[e].double()) ** 2).sum()
    loss = loss / (2 * nq**3)
    loss.backward()
    g = w.grad
    m, v = 0.1 * g, 0.001 * g * g
    q = p.double() - 1e-3 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    return [g, q, m, v, loss.detach().reshape(1)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "ic":
        return list(_ic(seed, case["nq"], case["box"]))
    if kind == "step":
        table = _filter(seed) if case["filter"] else None
        return list(_step(*_late_state(case["nq"], case["box"], seed), NODE, case["nq"], case["ng"], case["box"],
                          case["flags"], table))
    if kind == "ensemble":
        out = []
        for nq, ng, box, s in _members(case["members"], seed):
            d, v, psi1, psi2 = _ic(s, nq, box)
            for j in range(case["nodes"]):
                d, v = _step(d, v, psi1, psi2, j, nq, ng, box, 0)
            out.append([d, v, psi1, psi2])
        return out
    if kind in ("pk", "multipoles"):
        return _spectrum(case, seed, kind == "multipoles")
    if kind == "train":
        return _training(case, seed)
    return None  # labels and counts are whole numbers
