"""The work that users of the library have it do, as timed cases.

Every case is one pass through the public Python binding on seeded synthetic
problems: minibatch steps and sweeps of the FP32 form in its ordered and
float-atomic updates, sweeps of the tensor-core (precision) form with both of
its matrix paths, sweeps with the learned coarse correction attached, sweeps
of a group of uneven reconstructions, the network's own forward and backward
pass, the per-window monitoring values, and the forward model.  Sizes follow
the workloads of `synth.WORKLOADS`, the batched workload of
`synth.make_batch` and the learned correction's network at those sizes.

A sweep starts from an object a few percent away from the truth: the state
that nearly all sweeps of a reconstruction begin from.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2504_10118_gb300 import learned, magpie, synth

ALPHA = 0.5    # the setting of the benchmark's convergence runs: the iteration contracts everywhere
PHOTONS = {256: 1e7}  # per pattern, by window side; 1e6 otherwise (as in the workloads)
TINY = 1e-30   # division rule of the method: a quotient with a smaller denominator is 0
ORDERS = 4     # permutations a state cycles through, one per sweep
DRIFT = 0.05   # distance of the start object from the truth, relative
PROPOSAL = 0.05  # scale of the network's last layer in learned sweeps


# ------------------------------------------------------------------- cases
def _scan(n, m, grid, levels, minibatch, **more):
    case = {"kind": "sweep", "n": n, "m": m, "grid": grid, "levels": levels, "minibatch": minibatch, "ordered": True,
            "precision": 0, "network": False}
    case.update(more)
    return case


def _sweep(name, *sizes, **more):
    return {"name": name, **_scan(*sizes, **more)}


def listed():
    return [
        # one small minibatch at a time, as a live acquisition loop calls it: launches and latency
        _sweep("step_small", 192, 64, 8, 2, 8, kind="step"),
        # the smallest complete problem: four short steps per sweep
        _sweep("sweep_tiny", 128, 32, 8, 2, 16),
        # the ordinary reconstruction, with the float-atomic update (the fast default of the benchmark) ...
        _sweep("sweep_mid", 512, 128, 30, 3, 64, ordered=False),
        # ... and with the ordered update, the binding's default (bitwise reproducible)
        _sweep("sweep_mid_ordered", 512, 128, 30, 3, 64),
        # the large problem, FP32 transforms
        _sweep("sweep_large", 1024, 256, 50, 4, 64),
        # the large problem with the tensor-core transforms, register fragments and tcgen05
        _sweep("sweep_large_mma", 1024, 256, 50, 4, 64, precision=1),
        _sweep("sweep_large_tcgen05", 1024, 256, 50, 4, 64, precision=2),
        # the ordinary reconstruction with the learned coarse correction attached
        _sweep("sweep_learned", 512, 128, 30, 3, 64, network=True),
        # training of that network: output and parameter gradient of one batch of windows
        {"name": "network_gradient", "kind": "network", "side": 32, "batch": 64},
        # a dozen independent reconstructions of uneven sizes advanced together
        {"name": "group_uneven", "kind": "group", "count": 12, "draw_seed": 5, "levels": 3, "minibatch": 64},
        # what a monitoring program reads every few sweeps: objective and per-window misfit and gradient norm
        _sweep("monitor_mid", 512, 128, 30, 3, 64, kind="monitor"),
        # simulated data of an ordinary scan
        _sweep("forward_mid", 512, 128, 30, 1, 1, kind="forward"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "sweep", "sweep", "sweep", "precision", "learned", "network", "group", "monitor",
                       "forward"])
    if kind == "network":
        return {"kind": "network", "side": rng.choice([8, 16, 32]), "batch": _log_int(rng, 5, 64)}
    if kind == "group":
        case = {"kind": "group", "count": rng.randint(3, 12), "draw_seed": rng.randrange(1, 1 << 20),
                "levels": rng.randint(1, 4), "minibatch": _log_int(rng, 40, 96)}
        most = max(work(c)["flops"] for c in listed() if c["kind"] == "group")
        while case["count"] > 1 and work(case)["flops"] > most:
            case["count"] -= 1
        return case
    m = rng.choice([64, 128, 256] if kind == "precision" else [64, 128] if kind == "learned" else
                   [16, 32, 64, 128, 256])
    n = _log_int(rng, m + 3, 1024)
    # 25 windows at least; at most the pixels, the windows and the steps of the listed cases
    grid = _log_int(rng, 5, 30 if kind == "learned" else 50 if m == 256 else 60)
    steps = 15 if kind == "learned" else 40
    minibatch = min(grid * grid, max(_log_int(rng, 5, 128), -(-grid * grid // steps)))
    log2m = int(math.log2(m))
    if kind == "learned":  # coarsest side 8, 16 or 32
        return _scan(n, m, grid, rng.randint(log2m - 4, log2m - 2), min(minibatch, 64), network=True)
    levels = 1 if kind == "forward" else rng.randint(1, min(log2m + 1, 5))
    if kind == "precision":
        return _scan(n, m, grid, levels, minibatch, precision=rng.choice([1, 2]))
    return _scan(n, m, grid, levels, minibatch, kind=kind, ordered=kind != "sweep" or rng.random() < 0.5)


def _batch(case):
    """The group's problems: (n, m, grid, levels, minibatch) each."""
    ws = synth.make_batch(count=case["count"], seed=case["draw_seed"], levels=case["levels"],
                          minibatch=case["minibatch"])
    return [(w.n, w.m, w.grid, w.levels, w.minibatch) for w in ws]


# ------------------------------------------------------------------ inputs
def _gen(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    return g


def _object(n, g, dev):
    """Amplitude U[0.8, 1], phase a Gaussian-blurred (sigma 4 px, periodic) white field in [-pi/2, pi/2]."""
    amp = 0.8 + 0.2 * torch.rand((n, n), generator=g, device=dev)
    white = torch.randn((n, n), generator=g, device=dev)
    f = torch.fft.fftfreq(n, device=dev)
    blur = torch.exp(-2.0 * (math.pi * 4.0) ** 2 * (f[:, None] ** 2 + f[None, :] ** 2))
    smooth = torch.fft.ifft2(torch.fft.fft2(white) * blur).real
    lo, hi = smooth.min(), smooth.max()
    return torch.polar(amp, (smooth - lo) / (hi - lo) * math.pi - math.pi / 2.0)


def _patches(z, pos, m):
    r = torch.arange(m, device=z.device)
    rows = pos[:, 0].long()[:, None] + r
    cols = pos[:, 1].long()[:, None] + r
    return z[rows[:, :, None], cols[:, None, :]]


def _problem(n, m, grid, seed, dev):
    """(start object, truth, probe, positions, intensities) of one seeded scan."""
    g = _gen(seed, dev)
    truth = _object(n, g, dev)
    probe = torch.from_numpy(synth.make_probe(m).astype(np.complex64)).to(dev)
    step = max(1, (n - m) // max(1, grid - 1))
    step = max(1, step - 1) if step > 2 else step
    pos = torch.from_numpy(synth.make_raster(n, m, grid, step, max(1, step // 8), seed=seed)).to(dev)
    N = grid * grid
    d = torch.empty((N, m, m), dtype=torch.float32, device=dev)
    chunk = max(1, (1 << 24) // (m * m))
    for i in range(0, N, chunk):
        d[i:i + chunk] = torch.fft.fft2(probe * _patches(truth, pos[i:i + chunk], m)).abs().square()
    eta = float(d.double().sum()) / N / PHOTONS.get(m, 1e6)
    for i in range(0, N, chunk):
        d[i:i + chunk] = eta * torch.poisson(d[i:i + chunk] / eta, generator=g)
    noise = torch.randn((n, n), dtype=torch.complex64, generator=g, device=dev)
    start = (truth * (1.0 + DRIFT * noise)).contiguous()
    return start, truth, probe, pos, d


def _orders(N, seed, dev):
    rng = np.random.default_rng(seed)
    return [torch.from_numpy(rng.permutation(N).astype(np.int32)).to(dev) for _ in range(ORDERS)]


def _params(seed, dev, last):
    theta = torch.from_numpy(synth.make_cnn_params(learned.LAYERS, seed=seed, zero_last=False)).to(dev)
    ci, co = learned.LAYERS[-1]
    theta[theta.numel() - co * 9 * ci - co:] *= last
    return theta


def _network_inputs(case, seed, dev):
    """Parameters, network input (coarse object, scaled coarse step) and output gradient of a batch."""
    h, b = case["side"], case["batch"]
    g = _gen(seed, dev)
    z = _object(2 * h, g, dev)
    corner = torch.randint(0, h + 1, (b, 2), generator=g, device=dev)
    x = torch.cat([torch.view_as_real(_patches(z, corner, h)),
                   math.sqrt(0.5) * torch.randn((b, h, h, 2), generator=g, device=dev)], dim=3).contiguous()
    dy = torch.randn((b, h, h, 2), generator=g, device=dev) / (2 * b * h * h)
    return _params(seed, dev, 1.0), x, dy


def _context(start, probe, pos, d, levels, minibatch, ordered=True):
    m = probe.shape[0]
    p = magpie.magpie_params_of(start.shape[0], start.shape[1], m, pos.shape[0], levels, minibatch, ALPHA,
                                deterministic=int(ordered))
    return magpie.magpie_create(p, start, probe, pos, d)


# ----------------------------------------------------------------- prepare
def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "network":
        theta, x, dy = _network_inputs(case, seed, dev)
        net = magpie.magpie_cnn_create(case["side"], case["batch"])
        magpie.magpie_cnn_set_params(net, theta)
        return {"kind": kind, "net": net, "x": x, "dy": dy, "y": torch.empty_like(dy), "grad": torch.empty_like(theta)}
    if kind == "group":
        ctxs, objects, orders = [], [], []
        for i, (n, m, grid, levels, minibatch) in enumerate(_batch(case)):
            start, _, probe, pos, d = _problem(n, m, grid, seed * 64 + i, dev)
            ctxs.append(_context(start, probe, pos, d, levels, minibatch))
            objects.append(start)
            orders.append(_orders(grid * grid, seed * 64 + i, dev))
        return {"kind": kind, "group": magpie.magpie_group_create(ctxs), "objects": objects,
                "orders": [list(o) for o in zip(*orders)], "next": 0}
    n, m, grid = case["n"], case["m"], case["grid"]
    start, truth, probe, pos, d = _problem(n, m, grid, seed, dev)
    if kind == "forward":
        return {"kind": kind, "object": truth, "probe": probe, "pos": pos, "m": m}
    ctx = _context(start, probe, pos, d, case["levels"], case["minibatch"], case["ordered"])
    if case["precision"]:
        magpie.magpie_set_precision(ctx, case["precision"])
    if case["network"]:
        net = magpie.magpie_cnn_create(learned.coarse_side(m, case["levels"]), case["minibatch"])
        magpie.magpie_cnn_set_params(net, _params(seed, dev, PROPOSAL))
        magpie.magpie_attach_cnn(ctx, net)
    orders = _orders(grid * grid, seed, dev)
    if kind == "step":
        orders = [o[:case["minibatch"]].contiguous() for o in orders]
    return {"kind": kind, "ctx": ctx, "object": start, "orders": orders, "next": 0}


def _next_order(state):
    order = state["orders"][state["next"] % ORDERS]
    state["next"] += 1
    return order


# --------------------------------------------------------------------- run
def run(state):
    kind = state["kind"]
    if kind == "step":
        magpie.magpie_step(state["ctx"], _next_order(state))
        return state["object"]
    if kind == "sweep":
        magpie.magpie_sweep(state["ctx"], _next_order(state))
        return state["object"]
    if kind == "group":
        magpie.magpie_group_sweep(state["group"], _next_order(state))
        return state["objects"]
    if kind == "network":
        magpie.magpie_cnn_forward(state["net"], state["x"], state["y"])
        magpie.magpie_cnn_backward(state["net"], state["dy"], state["grad"])
        return {"y": state["y"], "grad": state["grad"]}
    if kind == "monitor":
        # the misfit history and maps a program plots, kept in 32 bits
        phi = magpie.magpie_objective(state["ctx"])
        phi_k, gnorm_k = magpie.magpie_window_values(state["ctx"])
        return {"phi": torch.tensor([phi], dtype=torch.float32), "phi_k": phi_k.float(), "gnorm_k": gnorm_k.float()}
    return magpie.magpie_forward_intensities(state["object"], state["probe"], state["pos"], state["m"])


# -------------------------------------------------------------------- work
def _window_flops(m):
    """Two 2-D transforms and about 43 operations per pixel (exit wave, projection, gradient, V-cycle)."""
    return 10.0 * m * m * math.log2(m * m) + 43.0 * m * m


def _network_flops(side):
    return 2.0 * 9 * sum(ci * co * px for (ci, co), px in
                         zip(learned.LAYERS, (side ** 2, side ** 2 / 4, side ** 2 / 16, side ** 2 / 64,
                                              side ** 2 / 16, side ** 2)))


def work(case):
    kind = case["kind"]
    if kind == "network":
        h, b = case["side"], case["batch"]
        P = sum(co * 9 * ci + co for ci, co in learned.LAYERS)
        return {"bytes": 2 * 4 * P + 4 * b * h * h * (4 + 2 + 2), "flops": 3.0 * b * _network_flops(h)}
    problems = _batch(case) if kind == "group" else [(case["n"], case["m"], case["grid"], case["levels"],
                                                       case["minibatch"])]
    nbytes = flops = 0.0
    for n, m, grid, levels, minibatch in problems:
        N = minibatch if kind == "step" else grid * grid
        M = m * m
        if kind in ("forward", "monitor"):
            nbytes += 4.0 * N * M + 8.0 * n * n + 8.0 * M
            flops += N * (5.0 * M * math.log2(M) * (1 if kind == "forward" else 2) + (9.0 if kind == "forward" else 35.0) * M)
        else:
            nbytes += 4.0 * N * M + 16.0 * n * n + 8.0 * M
            flops += N * _window_flops(m)
            if case.get("network"):
                flops += N * _network_flops(learned.coarse_side(m, levels))
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------- the method in 64 bits
def _div(num, den):
    ok = den.abs() > TINY
    return torch.where(ok, num / torch.where(ok, den, torch.ones_like(den)), torch.zeros_like(num * den))


def _restrict(a):
    return 0.25 * (a[..., 0::2, 0::2] + a[..., 1::2, 0::2] + a[..., 0::2, 1::2] + a[..., 1::2, 1::2])


def _prolong(b):
    return b.repeat_interleave(2, dim=-2).repeat_interleave(2, dim=-1)


def _vcycle(z, Q, R, u, levels, propose=None):
    """The multigrid step of every window of a batch; `propose` may replace the coarsest correction."""
    a2 = Q.abs().square()
    step = _div(Q.conj(), (u + a2).to(Q.dtype))
    if levels == 1:
        e = step * (R - Q * z)
        return z + (propose(z, e) if propose else e)
    QH, S = _restrict(Q), _restrict(a2)
    Wz = _div(a2, _prolong(S))
    WR = _prolong(QH) * _div(Wz.to(Q.dtype), Q)
    zH = _restrict(Wz * z)
    uH = _div(QH.abs().square(), S) * _restrict(u)
    eH = _vcycle(zH, QH, _restrict(WR * R), uH, levels - 1, propose) - zH
    z = z + _prolong(eH)
    return z + step * (R - Q * z)


def _revised(psi, d):
    """The modulus projection of a batch of exit waves and the windows' misfits."""
    f = torch.fft.fft2(psi)
    a, mag = d.sqrt(), f.abs()
    unit = torch.where(mag > 0, f / torch.where(mag > 0, mag, torch.ones_like(mag)), torch.ones_like(f))
    m2 = psi.shape[-1] ** 2
    return torch.fft.ifft2(a * unit), 0.5 * (mag - a).square().sum(dim=(1, 2)) / m2


def _bf16(a):
    return a.float().bfloat16().double()


def _network(theta, x):
    """Output [b, h, h, 2] of the network in 64 bits, rounded to bfloat16 where its weights and
    activations are stored in it (the roundings passed straight through for gradients)."""
    a, o = _bf16(x).permute(0, 3, 1, 2), 0
    for i, ((ci, co), stride, up) in enumerate(zip(learned.LAYERS, (1, 2, 2, 2, 1, 1), (1, 1, 1, 1, 2, 4))):
        w = theta[o:o + co * 9 * ci].reshape(co, 3, 3, ci).permute(0, 3, 1, 2)
        o += co * 9 * ci
        bias = theta[o:o + co]
        o += co
        w = w + (_bf16(w.detach()) - w.detach())
        if up > 1:
            a = a.repeat_interleave(up, dim=2).repeat_interleave(up, dim=3)
        # the convolution as one matrix product (plain 64-bit arithmetic)
        cols = F.unfold(a, 3, padding=1, stride=stride)
        side = a.shape[-1] // stride
        y = (w.reshape(co, ci * 9) @ cols + bias[:, None]).reshape(a.shape[0], co, side, side)
        if i + 1 < len(learned.LAYERS):
            y = y.relu()
            y = y + (_bf16(y.detach()) - y.detach())
        a = y
    return a.permute(0, 2, 3, 1)


def _proposal(theta, kept):
    """Coarsest correction of the learned form: the plain one plus the network's, scaled by its RMS."""
    def propose(zH, e):
        s = e.abs().square().mean(dim=(1, 2), keepdim=True).sqrt()
        es = _div(e, s.to(e.dtype))
        y = _network(theta, torch.stack([zH.real, zH.imag, es.real, es.imag], dim=-1))
        kept.append((s > TINY).reshape(-1))
        return e + s * torch.complex(y[..., 0], y[..., 1])
    return propose


def _step64(z, Q, pos, d, u, levels, batch, theta=None):
    m = Q.shape[0]
    zk = _patches(z, pos[batch], m)
    R, _ = _revised(Q * zk, d[batch].double())
    zh = _vcycle(zk, Q, R, u, levels)
    if theta is not None:
        kept = []
        other = _vcycle(zk, Q, R, u, levels, _proposal(theta, kept))
        sur = [0.5 * (Q * v - R).abs().square().sum(dim=(1, 2)) for v in (zh, other)]
        zh = torch.where((kept[0] & (sur[0] - sur[1] >= 0))[:, None, None], other, zh)
    w = u + Q.abs().square()
    r = torch.arange(m, device=z.device)
    rows = pos[batch, 0].long()[:, None] + r
    cols = pos[batch, 1].long()[:, None] + r
    flat = (rows[:, :, None] * z.shape[1] + cols[:, None, :]).reshape(-1)
    num = torch.zeros(z.numel(), 2, dtype=torch.float64, device=z.device)
    den = torch.zeros(z.numel(), dtype=torch.float64, device=z.device)
    num.index_add_(0, flat, torch.view_as_real((w * (zh - zk)).contiguous()).reshape(-1, 2))
    den.index_add_(0, flat, w.expand(zk.shape).reshape(-1))
    num = torch.view_as_complex(num).reshape(z.shape)
    den = den.reshape(z.shape)
    return torch.where(den > 0, z + num / torch.where(den > 0, den, torch.ones_like(den)), z)


def _regulariser(Q):
    a2 = Q.abs().square()
    return float(np.float32(ALPHA)) * (a2.max() - a2)


def _sweep64(problem, levels, minibatch, order, theta=None):
    start, _, probe, pos, d = problem
    z, Q = start.to(torch.complex128), probe.to(torch.complex128)
    u = _regulariser(Q)
    for i in range(0, order.numel(), minibatch):
        z = _step64(z, Q, pos, d, u, levels, order[i:i + minibatch].long(), theta)
    return z


def exact(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "network":
        theta, x, dy = _network_inputs(case, seed, dev)
        t = theta.double().requires_grad_(True)
        y = _network(t, x)
        (grad,) = torch.autograd.grad(y, t, dy.double())
        return {"y": y.detach().contiguous(), "grad": grad}
    if kind == "group":
        out = []
        for i, (n, m, grid, levels, minibatch) in enumerate(_batch(case)):
            problem = _problem(n, m, grid, seed * 64 + i, dev)
            out.append(_sweep64(problem, levels, minibatch, _orders(grid * grid, seed * 64 + i, dev)[0]))
        return out
    n, m, grid = case["n"], case["m"], case["grid"]
    problem = _problem(n, m, grid, seed, dev)
    start, truth, probe, pos, d = problem
    if kind in ("forward", "monitor"):
        Q, N = probe.to(torch.complex128), grid * grid
        z = (truth if kind == "forward" else start).to(torch.complex128)
        chunk = max(1, (1 << 22) // (m * m))
        out, phi, gn = torch.empty((N, m, m) if kind == "forward" else 0, dtype=torch.float64, device=dev), [], []
        for i in range(0, N, chunk):
            psi = Q * _patches(z, pos[i:i + chunk], m)
            if kind == "forward":
                out[i:i + chunk] = torch.fft.fft2(psi).abs().square()
            else:
                R, p = _revised(psi, d[i:i + chunk].double())
                phi.append(p)
                gn.append((Q.conj() * (psi - R)).abs().square().sum(dim=(1, 2)).sqrt())
        if kind == "forward":
            return out
        phi, gn = torch.cat(phi), torch.cat(gn)
        return {"phi": phi.sum().reshape(1), "phi_k": phi, "gnorm_k": gn}
    theta = _params(seed, dev, PROPOSAL).double() if case["network"] else None
    order = _orders(grid * grid, seed, dev)[0]
    if kind == "step":
        order = order[:case["minibatch"]]
    return _sweep64(problem, case["levels"], case["minibatch"], order, theta)
