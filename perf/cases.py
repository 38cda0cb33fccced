"""Performance cases of the holography library: what its users have it do, as calls.

Every case is one call sequence of a reconstruction program through the package's public
entry points: the gradient of F2 (or F1) of one chunk of angles with the probe set anew, as
every conjugate-gradient step does it, from the tiny to the large configuration; the simulation
of detector fields; the autograd function; the host-buffer call; the batch of uneven problems;
the propagation of one field; the vector operations of a step.

`listed` gives the cases, `draw` one more of the same ranges, `prepare` the inputs and the context
a program keeps, `run` one pass, `work` the bytes and flops a pass cannot do without, and `exact`
the outputs in 64 bits from plain torch.

The inputs are the synthetic ones of the configurations, made on the GPU with torch alone:
phase objects of random ellipses over fine layers, a striped Gaussian probe, sub-pixel sample
shifts, counting noise at 1e4 photons per pixel.  The evaluation point is a reconstruction that is
under way: the object at 60 % of its phase with 2 % noise, the probe with 10 % noise.
"""

import math
import random

import numpy as np
import torch

from paper_2407_20304_gb300 import Holo
from paper_2407_20304_gb300.autograd import holo_loss
from paper_2407_20304_gb300.batch import HoloBatch, Instance

WAVELENGTH, PIXEL, DIST_Z = 3.72e-11, 1.0e-8, 1.208
Z = (4.6e-4, 5.1e-4, 6.2e-4, 8.3e-4)
COUNTS = 1e4

# line lengths P of the padded grid that draw() takes (2^k and 3 * 2^k)
GRIDS = (64, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048, 3072, 4096)
BATCH_SIDES = (256, 384, 512, 1024)


def listed():
    return [
        # the tiny configuration, one step's gradient: launches and latency count
        {"name": "tiny_gradient", "kind": "gradient", "n": 128, "P": 256, "K": 8, "J": 4},
        # a problem of the batch configuration by itself: side 384, line length 3 * 256, odd count
        {"name": "ragged_gradient", "kind": "gradient", "n": 384, "P": 768, "K": 17, "J": 3},
        # the medium configuration, all its angles in one evaluation
        {"name": "medium_gradient", "kind": "gradient", "n": 512, "P": 1024, "K": 180, "J": 4},
        # a detector side that is not half the padded grid, and F1 (intensities as data)
        {"name": "wide_intensity", "kind": "gradient", "n": 1218, "P": 2048, "K": 24, "J": 3,
         "functional": "intensity"},
        # the large configuration, one chunk of its stream: the headline workload
        {"name": "large_gradient", "kind": "gradient", "n": 2048, "P": 4096, "K": 60, "J": 4},
        # probe shifts (the full-grid form of the passes)
        {"name": "probe_shift_gradient", "kind": "gradient", "n": 512, "P": 1024, "K": 40, "J": 4,
         "probe_shifts": True},
        # simulation of a data set: the detector fields of every plane
        {"name": "simulate_fields", "kind": "forward", "n": 1024, "P": 2048, "K": 30, "J": 4},
        # the autograd configuration: loss, then backward with the planes recomputed
        {"name": "autograd_recompute", "kind": "autograd", "n": 1024, "P": 2048, "K": 90, "J": 4},
        # a program that keeps its arrays in pinned host memory
        {"name": "host_buffers", "kind": "host", "n": 1024, "P": 2048, "K": 24, "J": 4},
        # independent reconstructions of uneven sizes, one graph launch
        {"name": "uneven_batch", "kind": "batch", "count": 8, "mix": 7},
        # one field moved by D_z on the largest grid
        {"name": "propagate_field", "kind": "propagate", "P": 4096},
        # the vector operations of one conjugate-gradient step on an object stack
        {"name": "step_vectors", "kind": "vectors", "n": 2048, "K": 16},
    ]


def _batch_problems(case):
    """The problems {n, P, K, J} of a batch case: sides of the batch configuration."""
    rng = random.Random(int(case["mix"]))
    out = []
    for _ in range(int(case["count"])):
        n = rng.choice(BATCH_SIDES)
        K = rng.randint(16, 64 if n < 1024 else 24)
        out.append({"n": n, "P": 2 * n, "K": K, "J": rng.randint(1, 4)})
    return out


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("gradient", "gradient", "gradient", "gradient", "forward", "autograd",
                       "host", "batch", "propagate", "vectors"))
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 8), "mix": rng.randint(0, 10 ** 6)}
    if kind == "propagate":
        return {"kind": kind, "P": rng.choice(GRIDS)}
    if kind == "vectors":
        n = 2 * _log_int(rng, 32, 1024)
        return {"kind": kind, "n": n, "K": max(1, _log_int(rng, 1, 16 * 2048 ** 2 // (n * n)))}
    P = rng.choice(GRIDS)
    # half of the problems at the default padding, the others at any even side
    n = P // 2 if rng.random() < 0.5 else 2 * rng.randint(max(8, P // 6), 3 * P // 8)
    J = rng.randint(1, 4)
    # planes: at most half of the large configuration's grid points, a quarter where probe shifts,
    # host copies or written fields cost more
    shifts = kind == "gradient" and rng.random() < 0.2
    cap = 240 * 4096 ** 2 // (P * P) // J
    cap = cap // 4 if shifts or kind in ("host", "forward") else cap // 2
    K = max(1, min(_log_int(rng, 2, max(2, min(cap, 240))), cap))
    case = {"kind": kind, "n": n, "P": P, "K": K, "J": J}
    if kind == "gradient" and rng.random() < 0.25:
        case["functional"] = "intensity"
    if shifts:
        case["probe_shifts"] = True
    return case


# ---------------------------------------------------------------- the model in plain torch

def _geometry(J):
    z = np.asarray(Z[:J])
    mt = z / z[0]
    omega = (z - z[0]) / mt
    zeta = z * (DIST_Z - z) / DIST_Z
    return mt, omega, zeta, zeta / mt ** 2


def _transfer(P, z, dtype):
    """exp(-i pi lambda z f^2) along one axis of the P grid."""
    k = torch.fft.fftfreq(P, d=1.0 / P, dtype=torch.float64, device="cuda")
    return torch.polar(torch.ones_like(k), -math.pi * WAVELENGTH * z * (k / (P * PIXEL)) ** 2).to(dtype)


def _shift_ramp(P, s):
    k = torch.fft.fftfreq(P, d=1.0 / P, dtype=torch.float64, device="cuda")
    return torch.polar(torch.ones_like(k), -2.0 * math.pi * k * s / P)


def _filter(x, hy, hx):
    f = torch.fft.fft2(x)
    f.mul_(hy[:, None]).mul_(hx[None, :])
    return torch.fft.ifft2(f)


def _axis(mt, t, n, P):
    """Bilinear taps along one axis: (first grid position, indices into psi with a zero border on
    either side, weight of the second tap) over the positions that reach psi."""
    X = torch.arange(P, dtype=torch.float64, device="cuda") - P // 2
    xi = mt * X - t + n // 2
    i0 = torch.floor(xi)
    on = torch.nonzero((i0 >= -1) & (i0 < n)).flatten()
    lo, hi = int(on[0]), int(on[-1]) + 1
    return lo, i0[lo:hi].long() + 1, (xi - i0)[lo:hi]


def _resample(psi, mt, t, P):
    """M_{1/m~} S_t psi on the P grid (1 outside psi) and its taps."""
    n = psi.shape[-1]
    ay, ax = _axis(mt, t[0], n, P), _axis(mt, t[1], n, P)
    real = torch.float64 if psi.dtype == torch.complex128 else torch.float32
    fy, fx = ay[2].to(real)[:, None], ax[2].to(real)[None, :]
    w = torch.zeros((n + 2, n + 2), dtype=psi.dtype, device=psi.device)
    w[1:-1, 1:-1] = psi - 1
    w = w[ay[1]] * (1 - fy) + w[ay[1] + 1] * fy
    w = w[:, ax[1]] * (1 - fx) + w[:, ax[1] + 1] * fx
    out = torch.ones((P, P), dtype=psi.dtype, device=psi.device)
    out[ay[0]:ay[0] + w.shape[0], ax[0]:ax[0] + w.shape[1]] += w
    return out, ay, ax


def _resample_transpose(g, ay, ax, n):
    """The transpose of the linear part of _resample."""
    g = g[ay[0]:ay[0] + len(ay[1]), ax[0]:ax[0] + len(ax[1])]
    fy, fx = ay[2][:, None], ax[2][None, :]

    def add(v, dim, idx, f):
        shape = [n + 2 if d == dim else v.shape[d] for d in (0, 1)] + [2]
        out = torch.zeros(shape, dtype=torch.float64, device=v.device)
        out.index_add_(dim, idx, torch.view_as_real(v * (1 - f)))
        out.index_add_(dim, idx + 1, torch.view_as_real(v * f))
        return torch.view_as_complex(out)

    return add(add(g, 0, ay[1], fy), 1, ax[1], fx)[1:-1, 1:-1]


def _crop(x, n):
    o = x.shape[-1] // 2 - n // 2
    return x[..., o:o + n, o:o + n]


def _embed(y, P):
    n = y.shape[-1]
    o = P // 2 - n // 2
    out = torch.zeros((P, P), dtype=y.dtype, device=y.device)
    out[o:o + n, o:o + n] = y
    return out


# ---------------------------------------------------------------- inputs

def _probe(P, n, gen):
    """The striped Gaussian probe of the configurations (sigma 0.3125 n)."""
    c = torch.arange(P, device="cuda", dtype=torch.float64) - P / 2

    def stripes():
        v = torch.rand(6, 3, generator=gen, device="cuda", dtype=torch.float64).cpu()
        acc = torch.zeros((P, P), device="cuda", dtype=torch.float64)
        for a, b, side in v.tolist():
            w = torch.sin(2 * math.pi * (c / (3 + 9 * a) + b))
            acc += w[:, None] if side < 0.5 else w[None, :]
        return acc

    r2 = c[:, None] ** 2 + c[None, :] ** 2
    amp = torch.exp(-r2 / (2 * (0.3125 * n) ** 2)) * (1 + 0.2 * stripes())
    return torch.polar(torch.ones_like(amp), 0.5 / 6 * stripes()).mul_(amp).to(torch.complex64)


def _noise(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=gen, device="cuda")) * math.sqrt(0.5)


def _phase(K, n, gen):
    """Phases in [-1.5, 0] of K objects: six ellipses each over layers of 2 .. 20 pixels."""
    v = torch.rand(6, 6, K, 1, 1, generator=gen, device="cuda")
    c = torch.arange(n, device="cuda", dtype=torch.float32) - n / 2
    y, x = c[None, :, None], c[None, None, :]
    phase = torch.zeros((K, n, n), device="cuda")
    for val, cy, cx, ay, ax, th in v:
        cos, sin = torch.cos(math.pi * th), torch.sin(math.pi * th)
        dy, dx = y - 0.6 * n * (cy - 0.5), x - 0.6 * n * (cx - 0.5)
        u = (dx * cos + dy * sin) / (n / 16 + 3 * n / 16 * ax)
        w = (dy * cos - dx * sin) / (n / 16 + 3 * n / 16 * ay)
        phase = torch.where(u * u + w * w <= 1, -val, phase)
    edges = torch.cumsum(torch.randint(2, 21, (n,), generator=gen, device="cuda"), 0)
    layer = torch.bucketize(torch.arange(n, device="cuda"), edges) % 2
    return phase - 0.5 * layer[None, :, None] * (phase < 0)


def _transmittance(phase):
    return torch.polar(torch.exp(phase / 50), phase)


def _inputs(case, seed):
    """Inputs of one reconstruction problem, from the seed alone."""
    n, P, K, J = case["n"], case["P"], case["K"], case["J"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    mt, omega, zeta, zhat = _geometry(J)
    intensity = case.get("functional") == "intensity"
    q = _probe(P, n, gen)
    phase = _phase(K, n, gen)
    t = (4 * torch.rand((K, J, 2), generator=gen, device="cuda") - 2).cpu()
    s = (4 * torch.rand((K, J, 2), generator=gen, device="cuda") - 2).cpu() if case.get("probe_shifts") else None

    def counted(u):
        # counting noise; F2's data are amplitudes, F1's intensities
        i = u.real ** 2 + u.imag ** 2
        c = COUNTS / i.mean()
        i = torch.poisson(c * i, generator=gen) / c
        return i if intensity else torch.sqrt(i)

    data = torch.empty((K, J, n, n), device="cuda")
    for j in range(J):
        p = _filter(q, *[_transfer(P, omega[j], q.dtype)] * 2) if j else q
        h = _transfer(P, zhat[j], q.dtype)
        for k in range(K):
            tk = t[k, j].double()
            hy = hx = h
            if s is not None:
                sk = s[k, j].double()
                tk = tk - mt[j] * sk
                hy, hx = (h * _shift_ramp(P, float(v)).to(q.dtype) for v in sk)
            r = _resample(_transmittance(phase[k]), mt[j], tk.tolist(), P)[0]
            data[k, j] = counted(_crop(_filter(p * r, hy, hx), n))
    dref = counted(_crop(_filter(q, *[_transfer(P, zeta[0], q.dtype)] * 2), n))
    psi = torch.empty((K, n, n), dtype=torch.complex64, device="cuda")
    for k in range(K):
        psi[k] = _transmittance(0.6 * phase[k]) + 0.02 * _noise((n, n), gen)
    q = q * (1 + 0.1 * _noise(q.shape, gen))
    return {"psi": psi, "q": q, "t": t, "s": s, "data": data, "dref": dref}


def _vector_inputs(case, seed):
    """Object, direction and two gradients of a step; the direction leans against them."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    shape = (case["K"], case["n"], case["n"])
    g = _noise(shape, gen)
    g_prev = 0.5 * g + _noise(shape, gen)
    eta = _noise(shape, gen) - 0.8 * g - 0.7 * g_prev
    return {"x": 1 + 0.1 * _noise(shape, gen), "eta": eta, "g": g, "g_prev": g_prev}


def _field(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    P = case["P"]
    return _probe(P, P // 2, gen) * (1 + 0.1 * _noise((P, P), gen))


# ---------------------------------------------------------------- prepare, run

BETA, GAMMA = 0.3, 1e-3


def _context(case, inp, chunk=0, data=True):
    h = Holo(case["n"], case["K"], case["J"], WAVELENGTH, PIXEL, DIST_Z, Z[:case["J"]], pad=case["P"],
             chunk=chunk)
    h.set_shifts(inp["t"].numpy())
    if inp["s"] is not None:
        h.set_probe_shifts(inp["s"].numpy())
    if case.get("functional"):
        h.set_functional(case["functional"])
    h.set_data(inp["data"] if data else None, inp["dref"])
    return h


def _pinned(x):
    return x.cpu().pin_memory().numpy()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "propagate":
        P = case["P"]
        x = _field(case, seed)
        h = Holo(P // 2, 1, 1, WAVELENGTH, PIXEL, DIST_Z, Z[:1], pad=P)
        return {"kind": kind, "h": h, "x": x, "out": torch.empty_like(x)}
    if kind == "vectors":
        h = Holo(case["n"], case["K"], 1, WAVELENGTH, PIXEL, DIST_Z, Z[:1], pad=_grid_for(case["n"]))
        return dict(_vector_inputs(case, seed), kind=kind, h=h)
    if kind == "batch":
        inst = []
        for i, p in enumerate(_batch_problems(case)):
            inp = _inputs(p, seed * 64 + i)
            inst.append(Instance(_context(p, inp, chunk=16), inp["psi"], inp["q"]))
        b = HoloBatch(inst)
        b.prepare_persistent("one")
        b.issue_persistent()    # the contexts' workspaces: nothing may be allocated while capturing
        b.capture_persistent()
        return {"kind": kind, "batch": b}
    inp = _inputs(case, seed)
    if kind == "host":
        h = _context(case, inp, data=False)
        return {"kind": kind, "h": h, "keep": inp["dref"], "psi": _pinned(inp["psi"]), "q": _pinned(inp["q"]),
                "data": _pinned(inp["data"]), "grad_psi": _pinned(torch.zeros_like(inp["psi"])),
                "grad_q": _pinned(torch.zeros_like(inp["q"]))}
    state = {"kind": kind, "h": _context(case, inp), "keep": inp["dref"], "psi": inp["psi"], "q": inp["q"]}
    if kind == "gradient":
        state["grad_psi"], state["grad_q"] = torch.empty_like(inp["psi"]), torch.empty_like(inp["q"])
    elif kind == "forward":
        state["u"] = torch.empty((case["K"], case["J"], case["n"], case["n"]), dtype=torch.complex64, device="cuda")
    return state


def _grid_for(n):
    return min(p for p in GRIDS if p >= n)


def run(state):
    kind = state["kind"]
    if kind == "propagate":
        return state["h"].propagate(state["x"], 3.1e-4, out=state["out"])
    if kind == "vectors":
        h = state["h"]
        dots = h.dy_dots(state["g"], state["g_prev"], state["eta"])
        h.direction_step(state["x"], state["eta"], state["g"], BETA, GAMMA)
        return list(dots) + [state["eta"], state["x"]]
    if kind == "batch":
        b = state["batch"]
        b.replay_persistent()
        return [list(b.losses())] + [[i.grad_psi, i.grad_q] for i in b.inst]
    h = state["h"]
    if kind == "host":
        return list(h.gradient_host(state["psi"], state["data"], state["q"], grad_psi=state["grad_psi"],
                                    grad_q=state["grad_q"]))
    if kind == "autograd":
        psi, q = state["psi"].requires_grad_(), state["q"].requires_grad_()
        psi.grad = q.grad = None
        loss = holo_loss(psi, q, h, recompute=True)
        loss.backward()
        return [float(loss), psi.grad, q.grad]
    h.set_probe(state["q"])
    if kind == "forward":
        return [h.forward(state["psi"], u_out=state["u"]), state["u"]]
    return list(h.gradient(state["psi"], grad_psi=state["grad_psi"], grad_q=state["grad_q"]))


# ---------------------------------------------------------------- work, exact

def _problem_work(case):
    """Bytes: object, probe and data read, gradients (or fields) written.  Flops: the line transforms
    (5 P log2 P each) of the rows that the object reaches and of the detector's columns, and those of
    the probe's planes and gradient."""
    n, P, K, J = case["n"], case["P"], case["K"], case["J"]
    fft = 5.0 * P * math.log2(P)
    mt = _geometry(J)[0]
    rows = [P if case.get("probe_shifts") else min(P, n / m + 3) for m in mt]
    probe = (2 * P * (J - 1) + P + n) * fft
    forward = sum(K * (2 * s + 2 * n) * fft for s in rows)
    reads = 8 * K * n * n + 8 * P * P + 4 * K * J * n * n + 4 * n * n
    if case["kind"] == "forward":
        return {"bytes": reads + 8 * K * J * n * n, "flops": probe + forward}
    back = (sum(min(P, s) for s in rows) + n + (J + 2) * P) * fft
    return {"bytes": reads + 8 * K * n * n + 8 * P * P,
            "flops": probe + (3 if case["kind"] == "autograd" else 2) * forward + back}


def work(case):
    kind = case["kind"]
    if kind == "propagate":
        P = case["P"]
        return {"bytes": 16 * P * P, "flops": 20.0 * P * P * math.log2(P)}
    if kind == "vectors":
        c = case["K"] * case["n"] ** 2
        return {"bytes": 8 * 6 * c, "flops": 20.0 * c}
    if kind == "batch":
        each = [_problem_work(dict(p, kind="gradient")) for p in _batch_problems(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    return _problem_work(case)


def _exact_problem(case, inp, fields=False):
    n, P, K, J = case["n"], case["P"], case["K"], case["J"]
    mt, omega, zeta, zhat = _geometry(J)
    c128 = torch.complex128
    q = inp["q"].detach().to(c128)
    intensity = case.get("functional") == "intensity"

    def residual(u, d):
        d = d.double()
        i2 = u.real ** 2 + u.imag ** 2
        if intensity:
            return ((i2 - d) ** 2).sum(), u * (2 * (i2 - d))
        mag = torch.sqrt(i2)
        return ((mag - d) ** 2).sum(), u * torch.where(mag > 0, 1 - d / mag.clamp_min(1e-300), 0.0)

    u_all = torch.empty((K, J, n, n), dtype=c128, device="cuda") if fields else None
    grad_psi = torch.zeros((K, n, n), dtype=c128, device="cuda")
    h0 = _transfer(P, zeta[0], c128)
    loss, r = residual(_crop(_filter(q, h0, h0), n), inp["dref"])
    grad_q = _filter(_embed(r, P), h0.conj(), h0.conj())
    for j in range(J):
        ho, hz = _transfer(P, omega[j], c128), _transfer(P, zhat[j], c128)
        p = _filter(q, ho, ho)
        gj = torch.zeros_like(q)
        for k in range(K):
            t, hy, hx = inp["t"][k, j].double(), hz, hz
            if inp["s"] is not None:
                s = inp["s"][k, j].double()
                t = t - mt[j] * s
                hy, hx = (hz * _shift_ramp(P, float(v)) for v in s)
            w, ay, ax = _resample(inp["psi"][k].detach().to(c128), mt[j], t.tolist(), P)
            u = _crop(_filter(p * w, hy, hx), n)
            lk, r = residual(u, inp["data"][k, j])
            loss = loss + lk
            if fields:
                u_all[k, j] = u
                continue
            v = _filter(_embed(r, P), hy.conj(), hx.conj())
            gj += w.conj() * v
            grad_psi[k] += 2 * _resample_transpose(p.conj() * v, ay, ax, n)
        if not fields:
            grad_q += _filter(gj, ho.conj(), ho.conj())
    return [float(loss), u_all] if fields else [float(loss), grad_psi, 2 * grad_q]


def exact(case, seed):
    kind = case["kind"]
    if kind == "propagate":
        h = _transfer(case["P"], 3.1e-4, torch.complex128)
        return _filter(_field(case, seed).to(torch.complex128), h, h)
    if kind == "vectors":
        v = {k: x.to(torch.complex128) for k, x in _vector_inputs(case, seed).items()}
        dots = [float((a.conj() * b).sum().real) for a, b in
                ((v["g"], v["g"]), (v["g"], v["eta"]), (v["g_prev"], v["eta"]))]
        eta = BETA * v["eta"] - v["g"]
        return dots + [eta, v["x"] + GAMMA * eta]
    if kind == "batch":
        each = [_exact_problem(p, _inputs(p, seed * 64 + i)) for i, p in enumerate(_batch_problems(case))]
        return [[e[0] for e in each]] + [e[1:] for e in each]
    return _exact_problem(case, _inputs(case, seed), fields=kind == "forward")
