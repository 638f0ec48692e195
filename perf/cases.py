"""Measured cases of the framework: the calls that a program computing
Brillouin-zone bubbles makes, over the range of sizes, temperatures and options
it makes them in.

``listed()`` gives the fixed cases, ``draw(rng)`` further ones of the same
ranges; ``prepare`` builds what the program holds before the call (context,
transfer momenta, pairs, network), ``run`` is one pass through the public
entry points, ``work`` the traffic and arithmetic that no implementation of
the call can avoid, and ``exact`` the same outputs in plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_1610_09991_gb300 import paid as P
from paper_1610_09991_gb300 import proposal as PR
from paper_1610_09991_gb300 import workloads as W

#: shared partitions on the FP32 pipe, the options of the headline path
GROUP = dict(group_mode=1, rule_n=12, cover=1.0, eval_fp32=1)


def listed():
    """The fixed cases.  ``call``: multi (device tensors in and out), host
    (numpy in and out), learned (host call seeded by a trained network), traced
    (seeded from the level maps of an earlier run), flow (Omega-regulated kinds
    with the flow equations' products), train (the network)."""
    return [
        # one transfer momentum of a map that a program fills point by point:
        # the smallest call, all latency
        dict(name="one_momentum", call="multi", kinds="ph", q="path", n=1, nff=9, T=0.2,
             rel_tol=1e-6, **GROUP),
        # the 400-integral first-shell batch with the library's default options
        # (one FP64 partition per integral)
        dict(name="first_shell_default", call="multi", kinds="ph", q="quadrant", n=4, nff=5, T=0.5,
             rel_tol=1e-6, group_mode=0, rule_n=4, cover=0.5, eval_fp32=0),
        # one flow step, both channels, 93,312 integrals, device resident
        dict(name="flow_step", call="multi", kinds="ph+pp", q="zone", n=24, nff=9, T=0.05,
             rel_tol=1e-6, **GROUP),
        # the same size end to end from host arrays, its partition seeded by
        # the trained network
        dict(name="flow_step_learned_host", call="learned", kinds="ph+pp", q="zone", n=24, nff=9,
             T=0.07, rel_tol=1e-6, **GROUP),
        # a later flow step seeded from the partition its predecessor ended on
        dict(name="flow_step_traced_seed", call="traced", kinds="ph+pp", q="zone", n=16, nff=9,
             T=0.05, rel_tol=1e-6, **GROUP),
        # the precision study's regime: low temperature, deep partitions
        dict(name="low_temperature", call="multi", kinds="ph+pp", q="zone", n=12, nff=9, T=0.01,
             rel_tol=1e-6, **GROUP),
        # the temperature sweep in one call (16 batches, 331,776 integrals): the
        # largest
        dict(name="temperature_sweep", call="multi", kinds="ph+pp", q="zone", n=16, nff=9, T=1.0,
             T_lo=0.005, nT=8, rel_tol=1e-6, **GROUP),
        # Algorithm 2's global error along an odd number of points between the
        # zone's high-symmetry momenta, from host arrays, first shell only
        dict(name="path_global_host", call="host", kinds="ph+pp", q="path", n=301, nff=5, T=0.1,
             rel_tol=1e-6, group_mode=2, rule_n=12, cover=1.0, eval_fp32=1),
        # the Omega-regulated flow step with its three products
        dict(name="flow_omega_products", call="flow", kinds="flow", q="zone", n=10, nff=9, T=0.1,
             rel_tol=1e-6, **GROUP),
        # shared partitions held to FP64 arithmetic throughout
        dict(name="shared_fp64", call="multi", kinds="ph+pp", q="zone", n=12, nff=9, T=0.05,
             rel_tol=1e-6, group_mode=1, rule_n=12, cover=1.0, eval_fp32=0),
        # one partition per integral, mixed precision (FP32 with float-float
        # escalation), tuned rule
        dict(name="per_integral_fp32", call="multi", kinds="ph+pp", q="zone", n=5, nff=9, T=0.05,
             rel_tol=1e-6, group_mode=0, rule_n=6, cover=1.0, eval_fp32=1),
        # one epoch of the network's training on traced rows, then the maps of
        # a flow step from it
        dict(name="train_and_predict", call="train", rows=6912, batch=1024, predict=1152, lr=2e-3),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the listed ranges."""
    family = rng.choice(["group"] * 4 + ["host", "learned", "traced", "flow", "fp64", "single",
                                        "single", "train"])
    if family == "train":
        return dict(call="train", rows=int(_log_uniform(rng, 200, 6912)),
                    batch=rng.choice([256, 512, 777, 1024]),
                    predict=int(_log_uniform(rng, 1, 4000)), lr=2e-3)
    T = round(_log_uniform(rng, 0.01, 1.0), 4)
    kinds = rng.choice(["ph", "pp", "ph+pp", "ph+pp"])
    q = rng.choice(["path", "zone"])
    rel = rng.choice([1e-5, 1e-6, 1e-6])
    nff = rng.choice([5, 9, 9])
    opts = dict(GROUP)
    # microseconds per (kind, q) group or per integral, roughly, at T: the
    # lower the temperature the deeper the partitions
    cost = 7.0 * max(1.0, 0.05 / T) ** 1.5
    if family in ("host", "group"):
        opts["group_mode"] = rng.choice([1, 1, 2])
        opts["rule_n"] = rng.choice([12, 12, 12, 10, 8])
        cost *= {12: 1.0, 10: 1.3, 8: 2.5}[opts["rule_n"]]
    elif family == "fp64":
        opts["eval_fp32"] = 0
        cost *= 10.0
    elif family == "flow":
        T = round(_log_uniform(rng, 0.05, 1.0), 4)
        kinds, nff = "flow", 9
        cost = 200.0 * max(1.0, 0.1 / T)
    elif family == "single":
        T = round(_log_uniform(rng, 0.05, 1.0), 4)
        opts = dict(group_mode=0, rule_n=rng.choice([4, 6]), cover=rng.choice([0.5, 1.0]),
                    eval_fp32=rng.choice([0, 1]))
        cost = 160.0 * nff * nff * max(0.1, 0.05 / T)
    most = 60e3 / cost / (1 if kinds in ("ph", "pp") else 2)
    n = int(_log_uniform(rng, 1, max(1.0, min(600.0, most))))
    if q == "zone":
        n = max(1, math.isqrt(n))
    call = dict(host="host", learned="learned", traced="traced", flow="flow").get(family, "multi")
    return dict(call=call, kinds=kinds, q=q, n=n, nff=nff, T=T, rel_tol=rel, **opts)


def _momenta(case, rng):
    if case["q"] == "zone":
        return W.q_grid_bz(case["n"])
    if case["q"] == "quadrant":
        return W.q_grid_quadrant(case["n"])
    # points along Gamma - X - M - Gamma, from a seeded offset
    s = 3.0 * ((np.arange(case["n"]) + rng.uniform()) / case["n"])
    leg, f = np.minimum(s.astype(int), 2), s - np.minimum(s.astype(int), 2)
    qx = np.where(leg == 0, f, np.where(leg == 1, 1.0, 1.0 - f))
    qy = np.where(leg == 0, 0.0, np.where(leg == 1, f, 1.0 - f))
    return math.pi * np.stack([qx, qy], axis=1)


def _inputs(case, seed):
    """Lattice (t, t', mu), temperatures, momenta and pairs of a case: the
    lattice of the workloads, each parameter as a seed's own run would have it."""
    rng = np.random.default_rng(seed)
    t, tp, mu = W.LATTICE
    lattice = (t, tp + rng.uniform(-0.02, 0.02), mu + rng.uniform(-0.05, 0.05))
    f = math.exp(rng.uniform(-0.02, 0.02))
    if "nT" in case:
        Ts = [f * float(T) for T in W.log_temperatures(case["nT"], case["T"], case["T_lo"])]
    else:
        Ts = [f * case["T"]]
    kinds = {"ph": [W.PH], "pp": [W.PP], "ph+pp": [W.PH, W.PP],
             "flow": [W.FLOW_PH, W.FLOW_PP]}[case["kinds"]]
    return lattice, [(k, T) for T in Ts for k in kinds], _momenta(case, rng), W.all_pairs(case["nff"])


def _options(case):
    return {k: case[k] for k in ("group_mode", "rule_n", "cover", "eval_fp32")}


def _device_batches(case, channels, q, lm):
    qd = torch.as_tensor(q, device="cuda")
    lmd = torch.as_tensor(lm, dtype=torch.int32, device="cuda")
    return [dict(kind=k, T=T, q=qd, lm=lmd, rel_tol=case["rel_tol"]) for k, T in channels]


def _rows(n, seed):
    """n training rows: inputs as the library's feature kernel lays them out
    (sin / cos q, log10 T, mu, t', kind) and level maps shaped like traced
    ones."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((n, 6), generator=g, device="cuda")
    qx, qy = math.pi * (2 * u[:, 0] - 1), math.pi * (2 * u[:, 1] - 1)
    logT, mu, tp = math.log10(0.005) * u[:, 2], -1.4 * u[:, 3], -0.35 * u[:, 4]
    pp = (u[:, 5] < 0.5).float()
    x = torch.zeros((n, 32), device="cuda")
    x[:, :4] = torch.stack([qx.sin(), qx.cos(), qy.sin(), qy.cos()], 1)
    x[:, 22:27] = torch.stack([logT, mu, tp, 1 - pp, pp], 1)
    k = -math.pi + 2 * math.pi * (torch.arange(16, device="cuda") + 0.5) / 16
    kx, ky = k.repeat_interleave(16)[None], k.repeat(16)[None]

    def e(a, b):
        return -2 * (a.cos() + b.cos()) - 4 * tp[:, None] * a.cos() * b.cos() - mu[:, None]

    d = torch.minimum(e(kx, ky).abs(), e(kx + qx[:, None], ky + qy[:, None]).abs())
    target = (2 - 1.4 * logT[:, None] - 1.5 * d).clamp(2, 7).round()
    return x.to(torch.bfloat16), target.contiguous()


def prepare(case, seed):
    """What the program holds before the call, made from the seed."""
    if case["call"] == "train":
        x, target = _rows(case["rows"], seed)
        xp, _ = _rows(case["predict"], seed + 500_000)
        return dict(case=case, net=P.Proposal(seed=seed), x=x, target=target, xp=xp, seed=seed)
    lattice, channels, q, lm = _inputs(case, seed)
    ctx = P.Context(*lattice, ffset=case["nff"], **_options(case))
    s = dict(case=case, ctx=ctx)
    if case["call"] == "host":
        s["batches"] = [dict(kind=k, T=T, q=q, lm=lm, rel_tol=case["rel_tol"]) for k, T in channels]
    elif case["call"] == "learned":
        # a network trained on the traced partitions of two neighbouring
        # parameter points
        xs, ts = [], []
        for j in (0, 1):
            near, ch, qn, lmn = _inputs(dict(case, q="zone", n=8), 2 * seed + j)
            c = P.Context(*near, ffset=case["nff"], trace=1, **_options(case))
            bs = _device_batches(case, ch, qn, lmn)
            xs.append(PR.features(c, bs))
            ts.append(PR.traced_maps(c, bs))
            c.close()
        s["net"] = P.Proposal(seed=seed)
        s["net"].train(torch.cat(xs), torch.cat(ts), epochs=60, batch=256, lr=2e-3, seed=seed)
        s["policy"] = PR.MarginPolicy([0.5] * len(PR.T_BANDS))
        s["batches"] = [dict(kind=k, T=T, q=q, lm=lm, rel_tol=case["rel_tol"]) for k, T in channels]
    else:
        s["batches"] = _device_batches(case, channels, q, lm)
    if case["call"] == "traced":
        # the level maps of the step before, at a 5 % higher temperature
        c = P.Context(*lattice, ffset=case["nff"], trace=1, **_options(case))
        s["maps"] = PR.traced_maps(c, [dict(b, T=1.05 * b["T"]) for b in s["batches"]])
        c.close()
    if case["call"] == "flow":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["nff"]
        for b in s["batches"]:
            m = 1 if b["kind"] == W.FLOW_PP else 2
            b["tu_v"] = [torch.randn((len(q), n, n), generator=g, device="cuda", dtype=torch.float64)
                         for _ in range(m)]
            b["tu_out"] = [torch.empty_like(v) for v in b["tu_v"]]
    return s


def run(state):
    """One pass; every batch gives (values, errors, regions, status)."""
    case, call = state["case"], state["case"]["call"]
    if call == "train":
        net = state["net"]
        loss = net.train(state["x"], state["target"], epochs=1, batch=case["batch"], lr=case["lr"],
                         seed=state["seed"])
        return [net.params, net.m, net.v, loss, net.forward(state["xp"])]
    ctx, bs = state["ctx"], state["batches"]
    if call == "host":
        rs = ctx.integrate_host(bs)[0]
    elif call == "learned":
        rs = ctx.integrate_host(bs, proposal=state["net"], margin=state["policy"])[0]
    elif call == "traced":
        rs = ctx.integrate_multi_seeded(bs, state["maps"], 0.0)
    else:
        rs = ctx.integrate_multi(bs)
    out = [[r.values, r.errors, r.regions, r.status] for r in rs]
    if call == "flow":
        out += [b["tu_out"] for b in bs]
    return out


#: operations of the kernel F at one node (two exponentials, one quotient) and
#: of one weighted accumulation
_F_FLOPS, _ACC_FLOPS = 60, 2


def work(case):
    """Inputs read once and outputs written once; the arithmetic of the initial
    partition's fine rule, which every adaptive run evaluates (the refinement
    beyond it depends on the integrand)."""
    if case["call"] == "train":
        n, p, m = case["rows"], 271_616, 256
        weights = 32 * m + 4 * m * m
        steps = -(-n // case["batch"])
        return dict(bytes=n * (64 + 1024) + case["predict"] * (64 + 1024) + 24 * p,
                    flops=2 * weights * (3 * n + case["predict"]) + 12 * p * steps)
    nq = case["n"] if case["q"] == "path" else case["n"] ** 2
    batches = case.get("nT", 1) * (1 if case["kinds"] in ("ph", "pp") else 2)
    units, pairs = nq * batches, case["nff"] ** 2
    nodes = 16 * (2 * case["rule_n"] + 1) ** 2
    if case["group_mode"]:
        flops = units * nodes * (_F_FLOPS + 5 * _ACC_FLOPS)
    else:
        flops = units * (nodes * _F_FLOPS + pairs * nodes * 3 * _ACC_FLOPS)
    return dict(bytes=units * 16 + pairs * 8 + units * pairs * (8 + 8 + 8 + 4)
                + (units * 1024 if case["call"] == "traced" else 0)
                + (units * pairs * 24 if case["call"] == "flow" else 0), flops=flops)


# -- exact values ------------------------------------------------------------

def _form_factors(kx, ky, n):
    cx, sx, cy, sy = kx.cos(), kx.sin(), ky.cos(), ky.sin()
    r2 = math.sqrt(2.0)
    f = [torch.ones_like(cx), cx + cy, cx - cy, r2 * sx, r2 * sy, 2 * cx * cy, 2 * sx * sy,
         2 * sx * cy, 2 * cx * sy]
    return torch.stack(f[:n])


def _kernel(e1, e2, T):
    """[tanh(e1/2T) - tanh(e2/2T)] / (2 (e1 - e2))."""
    a, b = e1 / (2 * T), e2 / (2 * T)
    d = a - b
    va, vb = torch.exp(-a.abs()), torch.exp(-b.abs())
    sech = 4 * va * vb / ((1 + va * va) * (1 + vb * vb))
    small = d.abs() < 0.5
    ds = torch.where(small, d, torch.full_like(d, 0.5))
    shc = torch.where(ds.abs() < 1e-4, 1 + ds * ds / 6,
                      torch.sinh(ds) / torch.where(ds == 0, torch.ones_like(ds), ds))
    far = (a.tanh() - b.tanh()) / torch.where(small, torch.ones_like(d), d)
    return torch.where(small, sech * shc, far) / (4 * T)


#: nodes of the largest reference quadrature (about 20 s in FP64 on the device)
_MOST_NODES = 1.5e10


def _trapezoid_points(T):
    """Points per direction at which the periodic trapezoid has converged
    beyond 1e-10: the integrand is analytic within about pi T / 4 of the real
    momenta."""
    return 32 * math.ceil(34.0 / T / 32) if T < 0.25 else 160


def exact(case, seed):
    """The bubbles by the dense periodic trapezoid, or the training pass, in
    FP64; None for the Omega-regulated kinds (not analytic on the Fermi
    surface) and where the reference would take too long."""
    if case["call"] == "train":
        return _exact_train(case, seed)
    if case["call"] == "flow":
        return None
    (t, tp, mu), channels, q, lm = _inputs(case, seed)
    if sum(len(q) * _trapezoid_points(T) ** 2 for _, T in channels) > _MOST_NODES:
        return None
    out, n = [], case["nff"]
    for kind, T in channels:
        M = _trapezoid_points(T)
        k = -math.pi + 2 * math.pi * torch.arange(M, device="cuda", dtype=torch.float64) / M
        rows = max(1, min(M, 4_000_000 // M))
        vals = torch.zeros((len(q), n, n), device="cuda", dtype=torch.float64)
        for r0 in range(0, M, rows):
            kx, ky = (a.reshape(-1) for a in torch.meshgrid(k[r0:r0 + rows], k, indexing="ij"))

            def energy(x, y):
                cx, cy = x.cos(), y.cos()
                return -2 * t * (cx + cy) - 4 * tp * cx * cy - mu

            e1, fl = energy(kx, ky), _form_factors(kx, ky, n)
            for i, (qx, qy) in enumerate(q):
                x2, y2 = (qx - kx, qy - ky) if kind == W.PP else (kx + qx, ky + qy)
                e2 = energy(x2, y2)
                F = _kernel(e1, -e2 if kind == W.PP else e2, T)
                vals[i] += (fl * F) @ _form_factors(x2, y2, n).T
        out.append([(vals / M ** 2).reshape(-1), None, None, None])
    return out


def _exact_train(case, seed):
    s = prepare(case, seed)
    net = s["net"]
    shapes = [(32, 256)] + [(256, 256)] * 4

    def layers(p):
        o, ws = 0, []
        for k, m in shapes:
            ws.append((p[o:o + k * m].view(k, m), p[o + k * m:o + k * m + m]))
            o += k * m + m
        return ws

    def forward(p, x):
        ws = layers(p)
        for i, (w, b) in enumerate(ws):
            x = x @ w + b
            if i + 1 < len(ws):
                x = torch.nn.functional.gelu(x)
        return x

    decay = torch.cat([torch.cat([torch.ones(k * m), torch.zeros(m)]) for k, m in shapes])
    decay = decay.to("cuda", torch.float64)
    p, m, v = (a.double().clone() for a in (net.params, net.m, net.v))
    x, target = s["x"].double(), s["target"].double()
    rows, batch = case["rows"], min(case["rows"], case["batch"])
    # the seeded Fisher-Yates order of the epoch (splitmix64)
    order, z, mask = list(range(rows)), s["seed"], (1 << 64) - 1
    for i in range(rows - 1, 0, -1):
        z = (z + 0x9E3779B97F4A7C15) & mask
        r = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        r = ((r ^ (r >> 27)) * 0x94D049BB133111EB) & mask
        j = (r ^ (r >> 31)) % (i + 1)
        order[i], order[j] = order[j], order[i]
    order = torch.tensor(order, device="cuda")
    steps, losses = -(-rows // batch), []
    for k in range(steps):
        idx = order[k * batch:(k + 1) * batch]
        pk = p.requires_grad_(True)
        loss = (forward(pk, x[idx]) - target[idx]).square().mean()
        (g,) = torch.autograd.grad(loss, pk)
        p = p.detach()
        losses.append(float(loss.detach()))
        lr = case["lr"] * 0.5 * (1 + math.cos(math.pi * k / steps))
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        p = p - lr * (m / (1 - 0.9 ** (k + 1)) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
                      + 1e-4 * decay * p)
    return [p, m, v, [sum(losses) / len(losses)], forward(p, s["xp"].double())]
