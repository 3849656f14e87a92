"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is a plain dict.  `prepare` makes what a training program holds before a step
(network handle, parameters, collocation points, optimizer state), all from a seed and
on the GPU; `run` is one pass through the public Python API; `work` is what a pass
cannot do without; `exact` is the same result from plain torch in float64.
"""
import math
import random
from types import SimpleNamespace

import torch

from paper_2604_15645_gb300 import _lib, api

PDES = {"burgers": _lib.PINN_BURGERS_1D, "ns": _lib.PINN_NS_STEADY_2D, "maxwell": _lib.PINN_MAXWELL_TE_2D,
        "advection": _lib.PINN_ADVECTION_1D, "allen_cahn": _lib.PINN_ALLEN_CAHN_1D}
LR, STEP0 = 1e-3, 1000   # Adam's learning rate, and the step a training run is at


def net(name, pde, width, depth, precision, n_res, n_ic, n_bc, nu, call, **more):
    case = dict(name=name, kind="net", pde=pde, width=width, depth=depth, precision=precision, n_res=n_res, n_ic=n_ic,
                n_bc=n_bc, nu=nu, call=call, ff_m=0, ff_sigma=1.0, rwf=False, value_split=False, graph=False,
                segments=0)
    case.update(more)
    return case


def listed():
    cavity = dict(ff_m=128, ff_sigma=1.0, rwf=True)
    return [
        # the plain FP32 benchmark network, a whole training step as its program runs it: replayed graph, then Adam
        net("burgers_4x64_fp32_train", "burgers", 64, 4, "fp32", 4096, 256, 256, 0.01 / math.pi, "train", graph=True),
        # the smallest call: the narrowest and shortest member of the network family at its fewest points, launched
        # eagerly (the API's default), so latency and launches are most of it
        net("burgers_3x32_bf16_small", "burgers", 32, 3, "bf16", 1024, 256, 256, 0.01, "grad"),
        # advection with Fourier features, point counts as they come out of a sampler: no multiple of anything
        net("advection_4x128_bf16_ragged", "advection", 128, 4, "bf16", 10007, 331, 333, 10.0, "grad", ff_m=64),
        # Allen-Cahn with temporal causality, as the paper trains time-dependent problems
        net("allen_cahn_4x128_bf16_causal", "allen_cahn", 128, 4, "bf16", 16384, 512, 512, 1e-4, "train", graph=True,
            segments=16),
        # the headline workload: the lid-driven cavity in BF16, training step
        net("cavity_6x256_bf16_train", "ns", 256, 6, "bf16", 65536, 0, 4096, 0.01, "train", graph=True,
            value_split=True, **cavity),
        # its loss-balancing step (one gradient per loss term, then the weights) on a batch of another size
        net("cavity_6x256_bf16_balance", "ns", 256, 6, "bf16", 20000, 0, 1600, 0.01, "terms", value_split=True, **cavity),
        # validation: the loss alone (forward direction) over a large held-out set
        net("cavity_6x256_bf16_validate", "ns", 256, 6, "bf16", 262144, 0, 4096, 0.01, "loss", value_split=True,
            **cavity),
        # the same network where BF16 is too coarse: TF32 tensor cores, and FP32 for reference gradients
        net("cavity_6x256_tf32", "ns", 256, 6, "tf32", 65536, 0, 4096, 0.01, "grad", **cavity),
        net("cavity_6x256_fp32", "ns", 256, 6, "fp32", 16384, 0, 1024, 0.01, "grad", **cavity),
        # the electromagnetic workload: three inputs, wide layers, first-order rows
        net("maxwell_5x512_bf16_train", "maxwell", 512, 5, "bf16", 262144, 16384, 16384, 0.0, "train", graph=True,
            rwf=True),
        # many independent networks of uneven width, depth and point count in one training step
        dict(name="burgers_family_64_bf16", kind="family", nets=64, layout=5003, max_res=65536, n_ic=256, n_bc=256),
        # the largest: the cavity at scale, over a million points in one pass
        net("cavity_8x512_bf16_scale", "ns", 512, 8, "bf16", 1048576, 0, 16384, 0.01, "grad", graph=True,
            value_split=True, ff_m=256, ff_sigma=2.0, rwf=True),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case: small FP32 networks, BF16 networks up to 256 wide on 1-D and cavity
    problems, the wide ones, TF32 and FP32 cavities, and families of networks."""
    kind = rng.choice(["fp32_small", "bf16", "bf16", "bf16", "wide", "tf32", "fp32", "family"])
    pde1 = rng.choice(["burgers", "advection", "allen_cahn"])
    nu1 = {"burgers": 0.01, "advection": 10.0, "allen_cahn": 1e-4}[pde1]
    if kind == "fp32_small":   # 1-D problems on networks of the widths PINN papers use
        n = log_int(rng, 500, 16384)
        case = net("", pde1, rng.choice([20, 32, 40, 50, 64, 96, 100, 128]), rng.randint(2, 8), "fp32", n,
                   log_int(rng, 50, 512), log_int(rng, 50, 512), nu1, rng.choice(["grad", "train"]),
                   graph=rng.random() < 0.5)
    elif kind == "bf16":
        call = rng.choice(["grad", "train", "train", "loss", "terms"])
        width = rng.choice([32, 48, 64, 96, 100, 128, 160, 200, 256])
        n = log_int(rng, 1024, 131072)
        if rng.random() < 0.5:
            seg = rng.choice([0, 0, 8, 32]) if call != "terms" else 0
            case = net("", pde1, width, rng.randint(3, 6), "bf16", n, log_int(rng, 100, 2048), log_int(rng, 100, 2048),
                       nu1, call, ff_m=rng.choice([0, 0, 32, 64]), segments=seg, graph=rng.random() < 0.5)
        else:
            case = net("", "ns", width, rng.randint(3, 8), "bf16", n, 0, log_int(rng, 200, 8192), 0.01, call,
                       ff_m=rng.choice([64, 128]), rwf=True, value_split=rng.random() < 0.7, graph=rng.random() < 0.5)
    elif kind == "wide":
        n = log_int(rng, 16384, 393216)
        call = rng.choice(["grad", "train", "train", "loss"])
        if rng.random() < 0.5:
            case = net("", "maxwell", rng.choice([320, 384, 512]), rng.randint(3, 6), "bf16", n, log_int(rng, 500, 16384),
                       log_int(rng, 500, 16384), 0.0, call, rwf=True, graph=rng.random() < 0.5)
        else:
            case = net("", "ns", rng.choice([320, 384, 512]), rng.randint(4, 8), "bf16", n, 0, log_int(rng, 500, 16384),
                       0.01, call, ff_m=rng.choice([128, 256]), ff_sigma=2.0, rwf=True, value_split=True,
                       graph=rng.random() < 0.5)
    elif kind == "family":
        case = dict(kind="family", nets=rng.randint(8, 96), layout=rng.randint(1, 10000),
                    max_res=log_int(rng, 2048, 65536), n_ic=log_int(rng, 64, 512), n_bc=log_int(rng, 64, 512))
        return case
    else:
        n = log_int(rng, 2048, 65536 if kind == "tf32" else 24576)
        width = rng.choice([128, 192, 256]) if kind == "tf32" else rng.choice([80, 128, 200, 256])
        case = net("", "ns", width, rng.randint(3, 6), kind, n, 0, log_int(rng, 200, 4096), 0.01,
                   rng.choice(["grad", "train"]), ff_m=rng.choice([64, 128]), rwf=True, graph=rng.random() < 0.5)
    del case["name"]
    return case


# ---- inputs -------------------------------------------------------------------------------

def d_in_out(pde):
    return (3 if pde == "maxwell" else 2), (3 if pde in ("ns", "maxwell") else 1)


def layer_dims(case):
    d_in, d_out = d_in_out(case["pde"])
    first = 2 * case["ff_m"] if case["ff_m"] else d_in
    widths = [case["width"]] * case["depth"] + [d_out]
    return list(zip([first] + widths[:-1], widths))


def generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def init_params(case, g):
    """Xavier-normal weights, factorisation scales N(1, 0.1), biases as some training leaves them."""
    parts = []
    for fi, fo in layer_dims(case):
        parts.append(torch.randn(fo * fi, generator=g, device="cuda") * math.sqrt(2.0 / (fi + fo)))
        if case["rwf"]:
            parts.append(1.0 + 0.1 * torch.randn(fo, generator=g, device="cuda"))
        parts.append(0.1 * torch.randn(fo, generator=g, device="cuda"))
    return torch.cat(parts)


def points(case, g):
    """Collocation sets of the problem: uniform interior points, the initial state at t = 0, the walls."""
    pde, n_res, n_ic, n_bc = case["pde"], case["n_res"], case["n_ic"], case["n_bc"]
    u = lambda n: torch.rand(n, generator=g, device="cuda")
    zero = lambda n: torch.zeros(n, device="cuda")
    wall = lambda n, k: torch.arange(n, device="cuda") % k
    if pde == "ns":   # unit square; lid (y = 1) moving at u = 1; u and v constrained
        s, side = u(n_bc), wall(n_bc, 4)
        x = torch.where(side == 2, 0.0, torch.where(side == 3, 1.0, s))
        y = torch.where(side == 0, 0.0, torch.where(side == 1, 1.0, s))
        lid = (side == 1).float()
        return api.DeviceBatch(torch.stack([u(n_res), u(n_res)]), zero(0).reshape(2, 0), zero(0).reshape(3, 0), 0,
                               torch.stack([x, y]), torch.stack([lid, zero(n_bc), zero(n_bc)]), 3)
    if pde == "maxwell":   # unit cube; Gaussian pulse at t = 0; perfectly conducting walls (Ez = 0)
        xi, yi = u(n_ic), u(n_ic)
        ez = torch.exp(-((xi - 0.5) ** 2 + (yi - 0.5) ** 2) / (2 * 0.05 ** 2))
        s, side, tb = u(n_bc), wall(n_bc, 4), u(n_bc)
        x = torch.where(side == 0, 0.0, torch.where(side == 1, 1.0, s))
        y = torch.where(side == 2, 0.0, torch.where(side == 3, 1.0, s))
        return api.DeviceBatch(torch.stack([u(n_res), u(n_res), u(n_res)]), torch.stack([xi, yi, zero(n_ic)]),
                               torch.stack([ez, zero(n_ic), zero(n_ic)]), 7, torch.stack([x, y, tb]),
                               torch.zeros(3, n_bc, device="cuda"), 1)
    lo, hi = (0.0, 2 * math.pi) if pde == "advection" else (-1.0, 1.0)
    xi, tb = lo + (hi - lo) * u(n_ic), u(n_bc)
    xb = torch.where(wall(n_bc, 2) == 0, lo, hi)
    if pde == "burgers":
        g_ic, g_bc = -torch.sin(math.pi * xi), zero(n_bc)
    elif pde == "advection":
        g_ic, g_bc = torch.sin(xi), torch.sin(xb - case["nu"] * tb)
    else:
        g_ic, g_bc = xi ** 2 * torch.cos(math.pi * xi), zero(n_bc) - 1.0
    return api.DeviceBatch(torch.stack([lo + (hi - lo) * u(n_res), u(n_res)]), torch.stack([xi, zero(n_ic)]), g_ic[None],
                           1, torch.stack([xb, tb]), g_bc[None], 1)


def moments(n, g):
    """Adam's moments of a run that is on its way (no entry near zero)."""
    m = 1e-2 * torch.randn(n, generator=g, device="cuda")
    return m, 1e-4 * (0.5 + torch.rand(n, generator=g, device="cuda"))


def family(case):
    """The members of a family of Burgers networks: width, depth, viscosity and interior points of each."""
    rng = random.Random(case["layout"])
    out = []
    for _ in range(case["nets"]):
        width, depth = rng.choice([32, 64, 128, 256]), rng.randint(3, 6)
        out.append(net("", "burgers", width, depth, "bf16", log_int(rng, 1024, case["max_res"]), case["n_ic"],
                       case["n_bc"], 10.0 ** rng.uniform(-3, -1), "train"))
    return out


def spec_of(case):
    return SimpleNamespace(pde=PDES[case["pde"]], widths=[case["width"]] * case["depth"], ff_m=case["ff_m"],
                           rwf=case["rwf"])


def inputs(case, seed):
    """Parameters, Fourier matrix and points of a case, from the seed alone."""
    g = generator(seed)
    if case["kind"] == "family":
        members = family(case)
        params = torch.cat([init_params(c, g) for c in members])
        return members, params, None, [points(c, g) for c in members], *moments(params.numel(), g)
    params = init_params(case, g)
    B = None
    if case["ff_m"]:
        B = case["ff_sigma"] * torch.randn(d_in_out(case["pde"])[0], case["ff_m"], generator=g, device="cuda")
    return None, params, B, points(case, g), *moments(params.numel(), g)


def prepare(case, seed):
    members, params, B, batch, m, v = inputs(case, seed)
    s = SimpleNamespace(case=case, params=params, batch=batch, m=m, v=v, step=STEP0, grad=torch.empty_like(params))
    if case["kind"] == "family":
        s.net = api.PinnMulti([spec_of(c) for c in members], precision="bf16")
        s.net.set_inputs(batch, [api.make_problem(c["nu"]) for c in members])
        return s
    s.net = api.PinnNet.from_spec(spec_of(case), case["precision"], value_split=case["value_split"])
    if B is not None:
        s.net.set_ff_matrix(B)
    if case["segments"]:
        s.net.set_causal(case["segments"], 1.0)
    if case["graph"]:
        s.net.set_graph(True)
    s.problem = api.make_problem(case["nu"])
    if case["call"] == "terms":
        s.grads = torch.empty(3, params.numel(), device="cuda")
        s.weights = torch.ones(3, dtype=torch.float64, device="cuda")
    return s


def run(s):
    c = s.case
    if c["kind"] == "family":
        s.step += 1
        loss = s.net.train_step(s.params, s.grad, s.m, s.v, s.step, lr=LR)
        return {"loss": loss, "grad": s.grad, "params": s.params, "m": s.m, "v": s.v}
    if c["call"] == "loss":
        return {"loss": s.net.loss(s.params, s.batch, s.problem)}
    if c["call"] == "terms":
        terms, grads = s.net.loss_grad_terms(s.params, s.batch, s.problem, grads=s.grads)
        return {"loss": terms, "grads": grads, "weights": s.net.loss_balance(grads, s.weights)}
    terms, grad = s.net.loss_grad(s.params, s.batch, s.problem, grad=s.grad)
    if c["call"] == "grad":
        return {"loss": terms, "grad": grad}
    s.step += 1
    api.adam_step(s.params, grad, s.m, s.v, s.step, lr=LR)
    return {"loss": terms, "grad": grad, "params": s.params, "m": s.m, "v": s.v}


# ---- work ---------------------------------------------------------------------------------

def net_work(c):
    """Bytes: points, targets, parameters (and the optimizer's state) read once, results written once.
    FLOPs: the jet products W a of every layer (four rows per interior point, one per initial or
    boundary point), their adjoint and the weight gradients."""
    d_in, d_out = d_in_out(c["pde"])
    dims = layer_dims(c)
    rows = 4 * c["n_res"] + c["n_ic"] + c["n_bc"]
    mac = sum(fi * fo for fi, fo in dims)
    P = mac + sum(fo * (2 if c["rwf"] else 1) for _, fo in dims)
    n = 4 * (d_in * (c["n_res"] + c["n_ic"] + c["n_bc"]) + d_out * (c["n_ic"] + c["n_bc"])) + 4 * P + 64
    first = dims[0][0] * dims[0][1]   # no adjoint into the inputs
    sweeps = {"loss": 0, "terms": 3}.get(c["call"], 1)
    outs = {"loss": 0, "grad": 4 * P, "terms": 12 * P, "train": 4 * P * 6}[c["call"]]
    return n + outs, 2.0 * rows * (mac + sweeps * (2 * mac - first))


def work(case):
    parts = [net_work(c) for c in (family(case) if case["kind"] == "family" else [case])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ---- the same in float64, plain torch -------------------------------------------------------

def unpack(case, p):
    """(W, b) of every layer; W = diag(exp(s)) V with the weight factorisation."""
    out, at = [], 0
    for fi, fo in layer_dims(case):
        W = p[at:at + fo * fi].reshape(fo, fi)
        at += fo * fi
        if case["rwf"]:
            W = torch.exp(p[at:at + fo])[:, None] * W
            at += fo
        out.append((W, p[at:at + fo]))
        at += fo
    return out


def jets(case, layers, B, x, derivatives):
    """Output rows [r][n][d_out] at points x [n][d_in]: the value and, with `derivatives`, the first
    derivatives and the second-order row that the residual needs."""
    pde, (n, d) = case["pde"], x.shape
    second = [] if pde == "maxwell" else [0, 1] if pde == "ns" else [0]
    first = list(range(d)) if derivatives else []
    if B is not None:
        phi = x @ B
        co, si = torch.cos(phi), torch.sin(phi)
        a = [torch.cat([co, si], 1)] + [torch.cat([-si * B[k], co * B[k]], 1) for k in first]
        if derivatives and second:
            q = sum(B[k] ** 2 for k in second)
            a.append(torch.cat([-co * q, -si * q], 1))
    else:
        a = [x] + [torch.eye(d, dtype=x.dtype, device=x.device)[k].expand(n, d) for k in first]
        if derivatives and second:
            a.append(torch.zeros_like(x))
    a = torch.stack(a)
    for l, (W, b) in enumerate(layers):
        z = a @ W.T
        z = torch.cat([(z[0] + b)[None], z[1:]])
        if l == len(layers) - 1:
            return z
        t = torch.tanh(z[0])
        tp = 1 - t * t
        rows = [t] + [tp * z[1 + k] for k in first]
        if derivatives and second:
            rows.append(tp * z[1 + d] - 2 * t * tp * sum(z[1 + k] ** 2 for k in second))
        a = torch.stack(rows)


def squared_residuals(case, U):
    """Squared residual per equation, [n] each."""
    pde, nu = case["pde"], case["nu"]
    if pde == "ns":
        (u, v, _), (ux, vx, px), (uy, vy, py), (ul, vl, _) = (r.T for r in U)
        return [(u * ux + v * uy + px - nu * ul) ** 2, (u * vx + v * vy + py - nu * vl) ** 2, (ux + vy) ** 2]
    if pde == "maxwell":
        _, (ex, _, hyx), (ey, hxy, _), (et, hxt, hyt) = (r.T for r in U)
        return [(et - (hyx - hxy)) ** 2, (hxt + ey) ** 2, (hyt - ex) ** 2]
    u, ux, ut, uxx = (r[:, 0] for r in U)
    if pde == "burgers":
        return [(ut + u * ux - nu * uxx) ** 2]
    if pde == "advection":
        return [(ut + nu * ux) ** 2]
    return [(ut - nu * uxx + 5 * u ** 3 - 5 * u) ** 2]


def exact_net(case, params, B, batch, want="sum"):
    """Loss terms [8] and the gradient ("sum"), the gradient per term ("terms"), or no gradient (None)."""
    p = params.double().requires_grad_(want is not None)
    B = None if B is None else B.double()
    M, n_res = case["segments"], case["n_res"]
    sq = torch.zeros(3, dtype=torch.float64, device="cuda")
    grads = torch.zeros(3, p.numel(), dtype=torch.float64, device="cuda")

    def grad_of(term, loss):
        if want is not None:
            grads[term] += torch.autograd.grad(loss, p)[0]

    chunk = max(1024, (1 << 23) // max(case["width"], 2 * case["ff_m"]))
    weight = torch.full((n_res,), 1.0 / max(n_res, 1), dtype=torch.float64, device="cuda")
    passes = [True]
    if M:   # temporal causality: the segment losses first, then their weights, held constant in the gradient
        seg = torch.clamp(torch.floor(batch.x_res[1] * M), 0, M - 1).long()
        passes = [False, True]
        seg_sum = torch.zeros(M, dtype=torch.float64, device="cuda")
        count = torch.bincount(seg, minlength=M).double()
    for last in passes:
        if M and last:
            L = torch.where(count > 0, seg_sum / count.clamp(min=1), torch.zeros_like(count))
            omega = torch.exp(-1.0 * (torch.cumsum(L, 0) - L))
            weight = (omega / (M * count.clamp(min=1)))[seg]
        for s in range(0, n_res, chunk):
            e = min(n_res, s + chunk)
            with torch.set_grad_enabled(want is not None and last):
                r2 = squared_residuals(case, jets(case, unpack(case, p), B, batch.x_res[:, s:e].T.double(), True))
                if not last:
                    seg_sum.index_add_(0, seg[s:e], sum(r2).detach())
                    continue
                eq = torch.stack([(weight[s:e] * r).sum() for r in r2])
                sq[:len(r2)] += eq.detach()
                if want is not None:
                    grad_of(0, eq.sum())
    sets = []
    for term, (x, g, mask) in ((1, (batch.x_ic, batch.g_ic, batch.ic_mask)), (2, (batch.x_bc, batch.g_bc, batch.bc_mask))):
        if not mask or not x.shape[1]:
            sets.append(torch.zeros((), dtype=torch.float64, device="cuda"))
            continue
        with torch.set_grad_enabled(want is not None):
            u = jets(case, unpack(case, p), B, x.T.double(), False)[0]
            on = [k for k in range(u.shape[1]) if mask >> k & 1]
            loss = ((u[:, on] - g.T.double()[:, on]) ** 2).mean(0).sum()
            if want is not None:
                grad_of(term, loss)
        sets.append(loss.detach())
    pde = sq.sum()
    terms = torch.stack([pde + sets[0] + sets[1], pde, sq[0], sq[1], sq[2], sets[0], sets[1], torch.zeros_like(pde)])
    return terms, grads if want == "terms" else grads.sum(0)


def exact_adam(params, grad, m, v):
    t = STEP0 + 1
    m = 0.9 * m.double() + 0.1 * grad
    v = 0.999 * v.double() + 0.001 * grad ** 2
    p = params.double() - LR * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return {"params": p, "m": m, "v": v}


def exact(case, seed):
    if work(case)["flops"] > 1e13:   # more than about 20 seconds in float64
        return None
    members, params, B, batch, m, v = inputs(case, seed)
    if case["kind"] == "family":
        at, loss, grad = 0, [], []
        for c, b in zip(members, batch):
            n = init_params(c, generator(0)).numel()
            t, g = exact_net(c, params[at:at + n], None, b)
            loss.append(t)
            grad.append(g)
            at += n
        grad = torch.cat(grad)
        return {"loss": torch.stack(loss), "grad": grad, **exact_adam(params, grad, m, v)}
    call = case["call"]
    terms, grad = exact_net(case, params, B, batch, {"loss": None, "terms": "terms"}.get(call, "sum"))
    if call == "loss":
        return {"loss": terms}
    if call == "terms":   # one update of the balancing weights (alpha 0.9, eps 1e-9) from weights of one
        norm = grad.norm(dim=1)
        w = torch.where(norm > 0, 0.9 + 0.1 * norm.sum() / (norm + 1e-9), torch.ones_like(norm))
        return {"loss": terms, "grads": grad, "weights": w}
    out = {"loss": terms, "grad": grad}
    return out if call == "grad" else {**out, **exact_adam(params, grad, m, v)}
