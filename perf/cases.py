"""The performance cases of the phase-mask library: what a user has it do, through
its public entry points, from the smallest mask to the largest batch.

Targets are patterns of Gaussian spots (sigma 1.5 px, cut off at 6 px, centres at
least 7 px from the zero frequency), start phases are uniform in [0, 2 pi), and
everything follows from the seed. The gaps r and g are delivered in FP64 but are
sums of single-precision squares, so the cases keep them as a program's log would,
in single precision.
"""

import math

import numpy as np
import torch

from paper_1302_0120_gb300 import GerchbergSaxton, MixedGerchbergSaxton
from paper_1302_0120_gb300.differentiable import LossContext, intensity_loss, optimize_phase

SIZES = (256, 512, 1024)


def listed():
    return [
        # The smallest mask in use: five neurons on 64 x 64, a latency.
        {"name": "spots64", "kind": "gs", "nx": 64, "ny": 64, "batch": 1, "iters": 20, "spots": 5, "laser": False, "host": False},
        # One interactive request on a coarse grid.
        {"name": "request256", "kind": "gs", "nx": 256, "ny": 256, "batch": 1, "iters": 30, "spots": 25, "laser": False, "host": False},
        # What a serving lane launches: the requests that waited, 30 iterations each.
        {"name": "lane512x4", "kind": "gs", "nx": 512, "ny": 512, "batch": 4, "iters": 30, "spots": 50, "laser": False, "host": False},
        # The headline workload: one 1024 x 1024 mask, 100 iterations.
        {"name": "spots1024", "kind": "gs", "nx": 1024, "ny": 1024, "batch": 1, "iters": 100, "spots": 50, "laser": False, "host": False},
        # The same grid under a measured beam profile instead of a uniform one.
        {"name": "laser1024", "kind": "gs", "nx": 1024, "ny": 1024, "batch": 1, "iters": 50, "spots": 100, "laser": True, "host": False},
        # The paper's SLM and iteration count, from arrays in host memory to arrays in host memory.
        {"name": "slm800x600", "kind": "gs", "nx": 800, "ny": 600, "batch": 1, "iters": 25, "spots": 40, "laser": False, "host": True},
        # An SXGA SLM: a side that is neither a power of two nor one of the paper's.
        {"name": "sxga1280", "kind": "gs", "nx": 1280, "ny": 1024, "batch": 1, "iters": 30, "spots": 60, "laser": False, "host": False},
        # The largest grid: its field does not fit the L2 cache.
        {"name": "grid4096", "kind": "gs", "nx": 4096, "ny": 4096, "batch": 1, "iters": 10, "spots": 200, "laser": False, "host": False},
        # A planning run: 64 masks of three sizes in one launch, in single precision ...
        {"name": "mixed64", "kind": "mixed", "n256": 22, "n512": 21, "n1024": 21, "iters": 50, "tensor_core": False},
        # ... and in the reduced-precision form on the tensor cores.
        {"name": "mixed64_tc", "kind": "mixed", "n256": 22, "n512": 21, "n1024": 21, "iters": 50, "tensor_core": True},
        # One evaluation of the loss and its gradient inside a user's own optimiser.
        {"name": "loss512", "kind": "loss", "n": 512, "spots": 50},
        # The library's optimiser: 200 Adam steps on a 100-spot pattern.
        {"name": "adam1024", "kind": "adam", "n": 1024, "steps": 200, "spots": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _smooth(lo, hi):
    return sorted(2 ** a * 3 ** b * 5 ** c for a in range(12) for b in range(8) for c in range(6)
                  if lo <= 2 ** a * 3 ** b * 5 ** c <= hi)


def draw(rng):
    kind = rng.choices(["pow2", "general", "batch", "mixed", "loss", "adam"], [30, 25, 15, 12, 9, 9])[0]
    if kind == "mixed":
        while True:
            n = [rng.randint(0, 16) for _ in SIZES]
            if sum(n) >= 2:
                break
        return {"kind": "mixed", "n256": n[0], "n512": n[1], "n1024": n[2], "iters": _log(rng, 5, 50), "tensor_core": rng.random() < 0.4}
    if kind == "loss":
        n = 1 << rng.randint(6, 11)
        return {"kind": "loss", "n": n, "spots": _log(rng, 3, max(4, n // 8))}
    if kind == "adam":
        n = 1 << rng.randint(7, 11)
        return {"kind": "adam", "n": n, "steps": _log(rng, 10, 200 if n <= 1024 else 50), "spots": _log(rng, 5, n // 8)}
    batch = 1
    if kind == "general":
        sides = _smooth(48, 1536)
        nx = sides[min(range(len(sides)), key=lambda k: abs(sides[k] - _log(rng, 48, 1536)))]
        ny = rng.choice([s for s in sides if nx / 2 <= s <= 2 * nx])
    else:
        e = rng.randint(5, 11 if kind == "pow2" else 10)
        nx, ny = 1 << e, 1 << max(5, min(11, e + rng.choice([-1, 0, 0, 0, 1])))
        if kind == "batch":
            batch = _log(rng, 2, 16 if nx * ny > 8192 else 64)
    most = max(5, min(100, 200_000_000 // (nx * ny * batch)))
    return {"kind": "gs", "nx": nx, "ny": ny, "batch": batch, "iters": _log(rng, 5, most),
            "spots": _log(rng, 3, max(4, min(200, nx * ny // 3000))), "laser": rng.random() < 0.2,
            "host": batch == 1 and rng.random() < 0.2}


# -- inputs

def _targets(rng, count, ny, nx, spots, peaks=(0.5, 1.0)):
    """[count, ny, nx] spot patterns in DFT order; ``spots`` is a number, or a (least, most) pair."""
    d = np.arange(-6, 7)
    dy, dx = (a.ravel() for a in np.meshgrid(d, d, indexing="ij"))
    keep = dy * dy + dx * dx <= 36
    dy, dx = dy[keep], dx[keep]
    at, value = [], []
    for b in range(count):
        n = spots if isinstance(spots, int) else int(rng.integers(spots[0], spots[1] + 1))
        y, x = rng.integers(0, ny, 64 + 8 * n), rng.integers(0, nx, 64 + 8 * n)
        ty, tx = np.minimum(y, ny - y), np.minimum(x, nx - x)
        y, x = (a[ty * ty + tx * tx >= 49][:n] for a in (y, x))
        p = rng.uniform(*peaks, len(y))
        at.append((b * ny * nx + ((y[:, None] + dy) % ny) * nx + (x[:, None] + dx) % nx).ravel())
        value.append((p[:, None] * np.exp(-(dy * dy + dx * dx) / 4.5)).ravel())
    img = torch.zeros(count * ny * nx, device="cuda")
    at = torch.from_numpy(np.concatenate(at)).cuda()
    value = torch.from_numpy(np.concatenate(value).astype(np.float32)).cuda()
    return img.scatter_reduce_(0, at, value, "amax").view(count, ny, nx)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)

    def phases(*shape):
        return torch.rand(*shape, generator=gen, device="cuda") * (2 * math.pi)

    if case["kind"] == "mixed":
        n = {s: case["n%d" % s] for s in SIZES if case["n%d" % s] > 0}
        return {"target": {s: _targets(rng, k, s, s, (10, 200)) for s, k in n.items()},
                "phase": {s: phases(k, s, s) for s, k in n.items()}}
    if case["kind"] in ("loss", "adam"):
        n = case["n"]
        target = _targets(rng, 1, n, n, case["spots"])[0]
        return {"target": target * float(n * n / target.sum(dtype=torch.float64)), "phase": phases(n, n)}
    b, ny, nx = case["batch"], case["ny"], case["nx"]
    d = {"target": _targets(rng, b, ny, nx, case["spots"]), "phase": phases(b, ny, nx)}
    if case["laser"]:  # a Gaussian beam, a little off centre, on a floor
        y = (torch.arange(ny, device="cuda")[:, None] / ny - float(rng.uniform(0.45, 0.55))) / 0.45
        x = (torch.arange(nx, device="cuda")[None, :] / nx - float(rng.uniform(0.45, 0.55))) / 0.45
        d["laser"] = (torch.exp(-(x * x + y * y)) + 0.01).float().contiguous()
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    if case["kind"] == "mixed":
        d["gs"] = MixedGerchbergSaxton({s: t.shape[0] for s, t in d["target"].items()}, tensor_core=case["tensor_core"])
    elif case["kind"] == "loss":
        d["ctx"] = LossContext(case["n"])
        d["phase"].requires_grad_(True)
    elif case["kind"] == "adam":
        d["ctx"] = LossContext(case["n"])
    else:
        d["gs"] = GerchbergSaxton(case["nx"], case["ny"], max_batch=case["batch"])
        if case["laser"]:
            d["gs"].set_slm_amplitude(d["laser"])
        if case["batch"] == 1:
            d["target"], d["phase"] = d["target"][0], d["phase"][0]
        if case["host"]:
            d["target"], d["phase"] = d["target"].cpu().numpy(), d["phase"].cpu().numpy()
    d["case"] = dict(case)
    return d


def run(state):
    case = state["case"]
    if case["kind"] == "mixed":
        out = state["gs"].run(state["target"], state["phase"], case["iters"])
        return {str(n): {"phase": p, "r": r.float(), "g": g.float()} for n, (p, r, g) in out.items()}
    if case["kind"] == "loss":
        state["phase"].grad = None
        loss = intensity_loss(state["phase"], state["target"], state["ctx"])
        loss.backward()
        return {"loss": loss.detach().float(), "grad": state["phase"].grad}
    if case["kind"] == "adam":
        phase, losses = optimize_phase(state["target"], state["phase"], steps=case["steps"], lctx=state["ctx"])
        return {"phase": phase, "losses": losses.astype(np.float32)}
    gs, iters = state["gs"], case["iters"]
    if case["host"]:
        p, r, g = gs.run_host(state["target"], state["phase"], iters)
        return {"phase": p, "r": r.astype(np.float32), "g": g.astype(np.float32)}
    p, r, g = (gs.run if case["batch"] == 1 else gs.run_batched)(state["target"], state["phase"], iters)
    return {"phase": p, "r": r.float(), "g": g.float()}


def work(case):
    def fft2(n):  # one two-dimensional transform of n points
        return 5 * n * math.log2(n)

    if case["kind"] in ("loss", "adam"):
        n, steps = case["n"] ** 2, case.get("steps", 1)
        return {"bytes": 12 * n, "flops": steps * (2 * fft2(n) + 30 * n)}
    if case["kind"] == "mixed":
        masks = [(s * s, case["n%d" % s]) for s in SIZES]
    else:
        masks = [(case["nx"] * case["ny"], case["batch"])]
    k = case["iters"]
    return {"bytes": sum(12 * n * b for n, b in masks) + (4 * masks[0][0] if case.get("laser") else 0),
            "flops": sum(b * ((2 * k + 1) * fft2(n) + 20 * n * k) for n, b in masks)}


# -- the same in 64 bits

def _exact_gs(target, phase, p, iters):
    """Alternating projections of a batch in FP64: phase of u^K, r^0..r^K, g^0..g^{K-1}."""
    n = target.shape[-1] * target.shape[-2]
    p = torch.ones((), dtype=torch.float64, device="cuda") if p is None else p.double()
    energy = (p * p).expand(target.shape[1:]).sum()
    m = target.double().sqrt()
    m *= (energy / (m * m).sum((1, 2), keepdim=True)).sqrt()
    one = torch.ones((), dtype=torch.complex128, device="cuda")
    u = torch.polar(p.expand(target.shape).contiguous(), phase.double())
    r, g = [], []

    def gap(d):
        return (d.square().sum((1, 2)) / energy).sqrt()

    for k in range(iters + 1):
        y = torch.fft.fft2(u, norm="ortho")
        a = y.abs()
        r.append(gap(a - m))
        if k == iters:
            break
        v = torch.fft.ifft2(m * torch.where(a > 0, y / a, one), norm="ortho")
        a = v.abs()
        g.append(gap(a - p))
        u = p * torch.where(a > 0, v / a, one)
    return u.angle(), torch.stack(r, 1), torch.stack(g, 1)


def _exact_loss(target, phase):
    x = torch.polar(torch.ones_like(phase), phase)
    y = torch.fft.fft2(x)
    d = (y.real.square() + y.imag.square()) / phase.numel() - target
    return d.square().sum(), 4 * (x.conj() * torch.fft.ifft2(d * y)).imag


def exact(case, seed):
    d = _inputs(case, seed)
    if case["kind"] == "mixed":
        out = {}
        for s, t in d["target"].items():
            q = [_exact_gs(t[b:b + 1], d["phase"][s][b:b + 1], None, case["iters"]) for b in range(t.shape[0])]
            p, r, g = (torch.cat(a) for a in zip(*q))
            # the FP16 transforms leave the 64-bit trajectory; only their gaps follow it
            out[str(s)] = {"phase": None if case["tensor_core"] else p, "r": r, "g": g}
        return out
    if case["kind"] == "loss":
        loss, grad = _exact_loss(d["target"].double(), d["phase"].double())
        return {"loss": loss, "grad": grad}
    if case["kind"] == "adam":
        target, x = d["target"].double(), d["phase"].double()
        m, v, losses = torch.zeros_like(x), torch.zeros_like(x), []
        for k in range(1, case["steps"] + 1):
            loss, grad = _exact_loss(target, x)
            losses.append(loss)
            m = 0.9 * m + 0.1 * grad
            v = 0.999 * v + 0.001 * grad * grad
            x = x - (0.05 / (1 - 0.9 ** k)) * m / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
        losses.append(_exact_loss(target, x)[0])
        return {"phase": x, "losses": torch.stack(losses)}
    p, r, g = _exact_gs(d["target"], d["phase"], d.get("laser"), case["iters"])
    if case["batch"] == 1:
        p, r, g = p[0], r[0], g[0]
    return {"phase": p, "r": r, "g": g}
