"""Performance cases of the Gray-Scott framework: what its users have it do.

The kinds, each through the Python binding's public entry points:

  grid    GrayScott: n steps of one L^3 grid in one step() call (FP32 or
          FP64, the four arithmetics of FP64 fields, periodic or held outer
          layer, with or without noise), result left on the GPU
  batch   GrayScottBatch: n steps of many grids of different sizes in one
          launch, then every grid read back into page-locked host memory
  apply   Surrogate.forward: one 16-step network application to N grids
  train   Surrogate.train_step: forward, every gradient and Adam for N pairs,
          and the gradients read back

Sizes come from the configurations, tests and benchmark of this repository
(L = 32 to 1024, batches of 32^3 to 128^3 grids, surrogate on 128^3 and
256^3) and from the ordinary spread between them: odd and ragged edges too.
Inputs are smooth random patterns, u in [0.3, 1] and v in [0, 0.35], the
range a run's own patterns have.
"""
import math

import numpy as np
import torch

from paper_2309_10292_gb300 import gs, inputs

DU, DV, DT = 0.2, 0.1, 1.0
ARITHS = {"ieee": gs.GS_ARITH_IEEE, "ds": gs.GS_ARITH_DS, "fx": gs.GS_ARITH_FX, "fxf": gs.GS_ARITH_FXF}
# floating-point operations of one cell and step (Eq. 1-3): 12 for the two
# neighbour sums' additions and centres, the rest reaction and update; the
# noise hash's integer operations are not counted
STENCIL_FLOPS = 31
CHANNELS = (4, 32, 32, 32, 32, 32, 2)
CONV_FLOPS = [2 * 27 * a * b for a, b in zip(CHANNELS[:-1], CHANNELS[1:])]


def _grid(L, steps, dtype="f32", noise=0.1, arith="ieee", held=False, tuned=False):
    return {"kind": "grid", "L": L, "steps": steps, "dtype": dtype, "noise": noise, "arith": arith, "held": held,
            "tuned": tuned}


def _batch(n, sizes, steps, noise=0.1):
    return {"kind": "batch", "n": n, "sizes": sizes, "steps": steps, "noise": noise}


def listed():
    return [
        # a small grid stepped one step at a time by a program that looks at the state between steps
        dict(_grid(32, 1), name="grid_f32_L32_1step"),
        # the accuracy workload: FP64, 64^3, 100 steps without noise
        dict(_grid(64, 100, dtype="f64", noise=0.0), name="grid_f64_L64"),
        # an ordinary exploratory run
        dict(_grid(128, 50), name="grid_f32_L128"),
        # an edge that is no multiple of the vector width
        dict(_grid(250, 20), name="grid_f32_L250_odd"),
        # the benchmark's grid, tuned as its program does
        dict(_grid(512, 20, tuned=True), name="grid_f32_L512_tuned"),
        # the largest production grid, as created
        dict(_grid(1024, 6), name="grid_f32_L1024"),
        # FP64 fields in the fast FP64 arithmetic
        dict(_grid(256, 20, dtype="f64", arith="fxf"), name="grid_f64_fxf_L256"),
        # the paper's own boundary: outer layer held
        dict(_grid(256, 20, held=True), name="grid_f32_held_L256"),
        # a parameter study: hundreds of uneven grids
        dict(_batch(256, "32,48,64,96,128", 100), name="batch_256"),
        # a small study: a few small grids, no noise
        dict(_batch(12, "32,48,64", 200, noise=0.0), name="batch_12_small"),
        # surrogate inference at its run size
        {"kind": "apply", "L": 256, "N": 1, "name": "apply_L256"},
        # surrogate training at its training size
        {"kind": "train", "L": 128, "N": 2, "name": "train_L128"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid"] * 6 + ["batch"] * 2 + ["apply", "train"])
    if kind == "grid":
        L = _log_int(rng, 16, 640)
        if rng.random() < 0.6:  # most edges are multiples of 8, the others are what they come out as
            L = max(16, L // 8 * 8)
        dtype = rng.choice(["f32", "f32", "f64"])
        arith = "ieee" if dtype == "f32" else rng.choice(["ieee", "fxf", "ds", "fx"])
        steps = max(1, min(_log_int(rng, 1, 100), int(1.5e9 / L ** 3)))
        return _grid(L, steps, dtype, rng.choice([0.0, 0.1, 0.1]), arith, rng.random() < 0.25)
    if kind == "batch":
        sizes = sorted(rng.sample([32, 48, 64, 96, 128], rng.randint(1, 5)))
        n = _log_int(rng, 4, 160)
        return _batch(n, ",".join(map(str, sizes)), _log_int(rng, 20, 100), rng.choice([0.0, 0.1]))
    if kind == "apply":
        L = 16 * rng.randint(2, 8)
        return {"kind": "apply", "L": L, "N": max(1, min(_log_int(rng, 1, 16), int(1.1e7 / L ** 3)))}
    L = 16 * rng.randint(2, 8)
    return {"kind": "train", "L": L, "N": max(1, min(_log_int(rng, 1, 8), int(2.2e6 / L ** 3)))}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _pattern(shape, seed):
    """Smooth random u, v on the GPU, float32 [n, L, L, L]."""
    n, L = shape
    g = torch.Generator(device="cuda").manual_seed(seed)
    m = max(2, L // 8)
    p = torch.rand((n, 1, m, m, m), generator=g, device="cuda")
    p = torch.nn.functional.interpolate(p, size=(L, L, L), mode="trilinear").squeeze(1)
    v = p.mul_(p).mul_(0.35)
    return 1 - 2 * v, v


def _batch_setup(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    sizes = [int(s) for s in case["sizes"].split(",")]
    L = [int(x) for x in rng.permutation(np.resize(sizes, case["n"]))]  # every size as often
    F = [float(x) for x in rng.uniform(0.01, 0.06, case["n"])]
    k = [float(x) for x in rng.uniform(0.04, 0.07, case["n"])]
    return L, F, k


def _surr_setup(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    params = inputs.surrogate_init_params(seed=seed, last_scale=0.1)
    u, v = _pattern((case["N"], case["L"]), seed)
    F = [float(x) for x in rng.uniform(0.01, 0.06, case["N"])]
    k = [float(x) for x in rng.uniform(0.04, 0.07, case["N"])]
    return params, u, v, F, k


def _targets(case, seed, u, v):
    a, b = _pattern((case["N"], case["L"]), seed + 1_000_003)
    return 0.9 * u + 0.1 * a, 0.9 * v + 0.1 * b


def prepare(case, seed):
    if case["kind"] == "grid":
        sim = gs.GrayScott(case["L"], Du=DU, Dv=DV, F=0.02, k=0.048, dt=DT, noise=case["noise"], seed=seed,
                           dtype=case["dtype"])
        u, v = _pattern((1, case["L"]), seed)
        for dst, src in zip(sim.tensors(), (u, v)):
            dst.copy_(src[0])
        if case["arith"] != "ieee":
            sim.arith = ARITHS[case["arith"]]
        if case["held"]:
            sim.boundary = gs.GS_BOUNDARY_HELD
        if case["tuned"]:
            sim.autotune()
        return {"case": case, "sim": sim}
    if case["kind"] == "batch":
        L, F, k = _batch_setup(case, seed)
        b = gs.GrayScottBatch(L, F, k, Du=DU, Dv=DV, dt=DT, noise=case["noise"], seed=seed)
        cells = [x ** 3 for x in L]
        host = [torch.empty(sum(cells), dtype=torch.float32, pin_memory=True) for _ in range(2)]
        at = np.concatenate([[0], np.cumsum(cells)])
        parts = [[h[int(lo):int(hi)] for lo, hi in zip(at[:-1], at[1:])] for h in host]
        return {"case": case, "batch": b, "host": host, "parts": parts}
    params, u, v, F, k = _surr_setup(case, seed)
    state = {"case": case, "net": gs.Surrogate(params), "u": u, "v": v, "F": F, "k": k}
    if case["kind"] == "train":
        state["ut"], state["vt"] = _targets(case, seed, u, v)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "grid":
        sim = state["sim"]
        sim.step(case["steps"])
        return sim.tensors()
    if case["kind"] == "batch":
        b = state["batch"]
        b.step(case["steps"])
        for field, parts in zip((gs.GS_U, gs.GS_V), state["parts"]):
            for i, dst in enumerate(parts):
                gs.gs_batch_read(b.handle, i, field, dst)
        return state["host"]
    if case["kind"] == "apply":
        return state["net"].forward(state["u"], state["v"], state["F"], state["k"])
    loss = state["net"].train_step(state["u"], state["v"], state["F"], state["k"], state["ut"], state["vt"], 1e-4)
    return loss, gs.gs_surr_get_grads(state["net"].handle)


# ---------------------------------------------------------------------------
# work: the state read once and written once per pass, and the operations
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] == "grid":
        cells = case["L"] ** 3
        esz = 4 if case["dtype"] == "f32" else 8
        return {"bytes": 4 * esz * cells, "flops": STENCIL_FLOPS * cells * case["steps"]}
    if case["kind"] == "batch":
        sizes = [int(s) for s in case["sizes"].split(",")]
        cells = sum(int(s) ** 3 for s in np.resize(sizes, case["n"]))
        # the state in and out, and its copy to the host
        return {"bytes": 24 * cells, "flops": STENCIL_FLOPS * cells * case["steps"]}
    cells = case["N"] * case["L"] ** 3
    weights = sum(27 * a * b + b for a, b in zip(CHANNELS[:-1], CHANNELS[1:]))
    if case["kind"] == "apply":
        return {"bytes": 16 * cells + 4 * weights, "flops": sum(CONV_FLOPS) * cells}
    # forward, weight gradients of all layers, data gradients of all but the first
    return {"bytes": 16 * cells + 5 * 4 * weights, "flops": (3 * sum(CONV_FLOPS) - CONV_FLOPS[0]) * cells}


# ---------------------------------------------------------------------------
# exact: the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _fmix(h):
    h = h ^ (h >> 16)
    h = (h * 0x85EBCA6B) & M32
    h = h ^ (h >> 13)
    h = (h * 0xC2B2AE35) & M32
    return h ^ (h >> 16)


def _keys(seed, t):
    k1 = _fmix((seed & M32) ^ _fmix((t & M32) ^ 0x9E3779B9))
    return k1, _fmix((seed >> 32) ^ _fmix(k1 ^ 0x7F4A7C15))


def _advance(u, v, steps, F, k, noise, seeds, held):
    """steps of n grids [n, L, L, L] (float64), each with its own F, k and noise seed."""
    n, L = u.shape[0], u.shape[1]
    col = lambda x, dt: torch.tensor(x, dtype=dt, device=u.device).view(n, 1, 1, 1)  # noqa: E731
    F, k = col(F, torch.float64), col(k, torch.float64)
    planes = max(1, min(L, int(6e7 / (n * L * L))))

    def lap(f, z, zs):
        c = f[:, zs]
        s = torch.roll(c, 1, 3) + torch.roll(c, -1, 3) + torch.roll(c, 1, 2) + torch.roll(c, -1, 2)
        s += f[:, (z - 1) % L] + f[:, (z + 1) % L]
        return (s - 6 * c) / 6

    for t in range(steps):
        un, vn = torch.empty_like(u), torch.empty_like(v)
        keys = [_keys(s, t) for s in seeds]
        k1, k2 = (col([x[i] for x in keys], torch.int64) for i in (0, 1))
        for z0 in range(0, L, planes):
            zs = slice(z0, min(L, z0 + planes))
            z = torch.arange(z0, min(L, z0 + planes), device=u.device)
            cu, cv = u[:, zs], v[:, zs]
            uvv = cu * cv * cv
            du = DU * lap(u, z, zs) - uvv + F * (1 - cu)
            if noise:
                c = torch.arange(z0 * L * L, (z0 + len(z)) * L * L, device=u.device).view(1, -1, L, L)
                m = _fmix(_fmix(c ^ k1) ^ k2) >> 8
                du += noise * ((2 * m + 1 - (1 << 24)).double() / (1 << 24))
            un[:, zs] = cu + DT * du
            vn[:, zs] = cv + DT * (DV * lap(v, z, zs) + uvv - (F + k) * cv)
        if held:
            for a, b in ((un, u), (vn, v)):
                for d in (1, 2, 3):
                    for e in (0, L - 1):
                        a.select(d, e).copy_(b.select(d, e))
        u, v = un, vn
    return u, v


def _shift(tap):
    """Roll that brings the neighbour of `tap` to its cell."""
    return -(tap // 9 - 1), -((tap // 3) % 3 - 1), -(tap % 3 - 1)


def _conv(h, w, b):
    """Circular 3x3x3 convolution of channels-last [n, L, L, L, cin]."""
    out = b.expand(h.numel() // h.shape[-1], b.shape[0]).clone()
    for tap in range(27):
        out.addmm_(torch.roll(h, _shift(tap), (1, 2, 3)).view(-1, h.shape[-1]), w[tap])
    return out.view(*h.shape[:-1], b.shape[0])


def _network(params, u, v, F, k):
    """(u, v) after 16 steps as the network has it, float64."""
    n, L = u.shape[0], u.shape[1]
    one = torch.ones((n, L, L, L), dtype=torch.float64, device=u.device)
    col = lambda x: torch.tensor(x, dtype=torch.float64, device=u.device).view(n, 1, 1, 1)  # noqa: E731
    h = torch.stack([u - 1, v, 20 * col(F) * one, 20 * col(k) * one], dim=-1)
    del one
    h = torch.relu(_conv(h, *params[0]))
    for l in range(1, 5):
        h = h + torch.relu(_conv(h, *params[l]))
    out = _conv(h, *params[5])
    return u + out[..., 0], v + out[..., 1]


class _ConvGrad(torch.autograd.Function):
    """The convolution with its two gradients, tap by tap, so that nothing but h is kept."""

    @staticmethod
    def forward(ctx, h, w, b):
        ctx.save_for_backward(h, w)
        return _conv(h, w.detach(), b.detach())

    @staticmethod
    def backward(ctx, g):
        h, w = ctx.saved_tensors
        flat = g.reshape(-1, g.shape[-1])
        gh, gw = torch.zeros_like(h), torch.zeros_like(w)
        for tap in range(27):
            d = _shift(tap)
            gw[tap] = torch.roll(h, d, (1, 2, 3)).reshape(-1, h.shape[-1]).T @ flat
            gh += torch.roll((flat @ w[tap].T).view_as(h), tuple(-x for x in d), (1, 2, 3))
        return gh, gw, flat.sum(0)


def exact(case, seed):
    if case["kind"] == "grid":
        u, v = _pattern((1, case["L"]), seed)
        u, v = _advance(u.double(), v.double(), case["steps"], [0.02], [0.048], case["noise"], [seed], case["held"])
        return u[0], v[0]
    if case["kind"] == "batch":
        L, F, k = _batch_setup(case, seed)
        out = [[None] * len(L), [None] * len(L)]
        for size in sorted(set(L)):
            at = [i for i, x in enumerate(L) if x == size]
            u = torch.ones((len(at), size, size, size), dtype=torch.float64, device="cuda")
            v = torch.zeros_like(u)
            c = slice(size // 2 - 3, size // 2 + 3)
            u[:, c, c, c], v[:, c, c, c] = 0.25, 0.33
            u, v = _advance(u, v, case["steps"], [F[i] for i in at], [k[i] for i in at], case["noise"],
                            [seed + i for i in at], False)
            for j, i in enumerate(at):
                out[0][i], out[1][i] = u[j].reshape(-1), v[j].reshape(-1)
        return [torch.cat(x) for x in out]
    params, u, v, F, k = _surr_setup(case, seed)
    p = [(torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda()) for w, b in params]
    if case["kind"] == "apply":
        return _network(p, u.double(), v.double(), F, k)
    ut, vt = _targets(case, seed, u, v)
    for w, b in p:
        w.requires_grad_(), b.requires_grad_()
    n, L = u.shape[0], u.shape[1]
    ones = torch.ones((n, L, L, L), dtype=torch.float64, device="cuda")
    fk = [torch.tensor(x, dtype=torch.float64, device="cuda").view(n, 1, 1, 1) * 20 * ones for x in (F, k)]
    h = torch.stack([u.double() - 1, v.double(), *fk], dim=-1)
    h = torch.relu(_ConvGrad.apply(h, *p[0]))
    for l in range(1, 5):
        h = h + torch.relu(_ConvGrad.apply(h, *p[l]))
    o = _ConvGrad.apply(h, *p[5])
    d = torch.stack([u.double() + o[..., 0] - ut.double(), v.double() + o[..., 1] - vt.double()], dim=-1)
    loss = (d * d).mean()
    loss.backward()
    return float(loss), torch.cat([x.grad.reshape(-1) for wb in p for x in wb]).cpu().numpy()
