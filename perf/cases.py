"""What the framework is used for, as timed cases: energies and forces of one frame in a
molecular-dynamics loop, forward + backward (Hessian-vector product) of force matching, batches
of uneven frames, point quadrupoles, host-resident callers, and the learned network's gradient.

Frames are molten-salt-like (32.35 cubic Angstrom per ion, charge-ordered, shortest separations
near 2.2 Angstrom, no ion in spatial order), made on the GPU from the seed. alpha, cutoffs, spline
orders and mesh spacings are those of the repository's workloads (alpha 0.30, 9-10 Angstrom,
orders 4-6, spacings of about 0.7-1 Angstrom).

Energies, virials and losses are float64 sums of the library's float32 per-ion, per-pair and
per-mode terms; a float32 training or dynamics program takes them as float32, and so do the cases.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2606_01598_gb300 as gb

ALPHA = 0.30
VOLUME_PER_ION = 32.35


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------

def listed():
    one = dict(order=6, rcut=9.0, tilt=False, virial=False, reuse=True)
    return [
        # the smallest frames a dynamics loop steps through: launches and latency are all of it
        dict(one, name="md_64", kind="forward", n=64, nx=16, ny=16, nz=16, order=4),
        # the rock-salt check configuration (512 ions, 32^3, order 4), outputs allocated per call
        dict(one, name="md_512", kind="forward", n=512, nx=32, ny=32, nz=32, order=4, rcut=10.0, reuse=False),
        # a constant-pressure step: triclinic cell, odd ion count, ragged 2,3,5-smooth mesh, virial
        dict(one, name="npt_9999", kind="forward", n=9999, nx=80, ny=81, nz=90, order=5, tilt=True, virial=True,
             reuse=False),
        # dynamics on the benchmark frame
        dict(one, name="md_32768", kind="forward", n=32768, nx=128, ny=128, nz=128),
        # force matching of a small odd frame on a general mesh
        dict(one, name="fm_1999", kind="step", n=1999, nx=48, ny=50, nz=54, order=5, tilt=True, reuse=False),
        # force matching through autograd's double backward, the training loop of one frame
        dict(one, name="autograd_4096", kind="autograd", n=4096, nx=64, ny=64, nz=64),
        # the benchmark's forward + backward
        dict(one, name="fm_32768", kind="step", n=32768, nx=128, ny=128, nz=128),
        # the largest frame
        dict(one, name="fm_262144", kind="step", n=262144, nx=256, ny=256, nz=256),
        # a caller whose arrays live in pinned host memory
        dict(one, name="host_32768", kind="host", n=32768, nx=128, ny=128, nz=128),
        # the uneven batch: 256 frames of 64-1024 ions, orders 4 and 6 alternating, forward + backward
        dict(name="batch_256", kind="batch", frames=256, n_lo=64, n_hi=1024, spacing=0.8, sizes=1002, rcut=9.0,
             backward=True),
        # point quadrupoles, forward + backward
        dict(name="quad_4096", kind="quad", n=4096, nx=64, ny=64, nz=64, order=6, rcut=9.0),
        # the learned network's force-matching gradient on its training batch
        dict(name="train_32x512", kind="train", frames=32, n=512, mesh=32, order=4, rcut=9.0),
    ]


def _smooth(target: int) -> int:
    m = target
    while True:
        r = m
        for f in (2, 3, 5):
            while r % f == 0:
                r //= f
        if r == 1:
            return m
        m += 1


def _edge(n: int) -> float:
    return (VOLUME_PER_ION * n) ** (1.0 / 3.0)


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh(rng, n: int, order: int):
    """Mesh sizes a program would take for this box: power-of-two, 2,3,5-smooth or the plain target."""
    h = rng.uniform(0.8, 1.0)
    rule = rng.choice(("power", "smooth", "smooth", "plain"))
    t = max(order + 2, int(math.ceil(_edge(n) / h)))
    out = []
    for a in range(3):
        ta = t + (rng.randrange(3) if rule == "plain" else 0)
        out.append(1 << (ta - 1).bit_length() if rule == "power" and t > 8 else ta if rule == "plain" else _smooth(ta))
    if max(out) > 256:
        out = [256, 256, 256]
    return out


def draw(rng: random.Random):
    kind = rng.choice(("forward", "forward", "step", "step", "autograd", "host", "batch", "quad", "train"))
    if kind == "batch":
        lo = _log_int(rng, 64, 512)
        return dict(kind=kind, frames=_log_int(rng, 4, 256), n_lo=lo, n_hi=rng.randint(lo, 1024),
                    spacing=round(rng.uniform(0.8, 1.0), 3), sizes=rng.randrange(1 << 30), rcut=9.0,
                    backward=rng.random() < 0.6)
    if kind == "train":
        return dict(kind=kind, frames=_log_int(rng, 2, 32), n=rng.randint(96, 512), mesh=rng.choice((24, 27, 30, 32)),
                    order=rng.choice((4, 4, 5)), rcut=9.0)
    top = {"quad": 32768, "autograd": 65536}.get(kind, 262144)
    n = _log_int(rng, 64, top)
    order = rng.choice((4, 5, 6, 6))
    nx, ny, nz = _mesh(rng, n, order)
    c = dict(kind=kind, n=n, nx=nx, ny=ny, nz=nz, order=order, rcut=rng.choice((8.0, 9.0, 10.0)))
    if kind == "quad":
        return c
    c.update(tilt=rng.random() < 0.3, reuse=rng.random() < 0.5, virial=kind == "forward" and rng.random() < 0.25)
    return c


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _generator(seed: int):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _box(n: int, tilt: bool) -> np.ndarray:
    L = _edge(n)
    if not tilt:
        return np.eye(3) * L
    return np.array([[L, 0.0, 0.0], [0.15 * L, L, 0.0], [-0.1 * L, 0.12 * L, L]])


def _frame(n: int, box: np.ndarray, g):
    """Positions, charges and dipoles (float32) of a molten-salt-like frame: a jittered, slowly
    strained and randomly placed lattice with alternating charges, ions in random order."""
    dev = _device()
    m = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
    a = _edge(n) / m
    site = torch.randperm(m ** 3, generator=g, device=dev)[:n]
    ijk = torch.stack([site // (m * m), (site // m) % m, site % m], 1)
    u = torch.rand((n + 3, 3), generator=g, device=dev, dtype=torch.float64)
    shift, phase, strain = u[n], u[n + 1], 0.015 * (0.5 + u[n + 2])
    s = (ijk + 0.5 + (2.0 * u[:n] - 1.0) * (0.5 * max(0.0, a - 2.2) / a)) / m
    s = s + strain * torch.sin(2.0 * math.pi * (s.roll(1, 1) + phase)) + shift
    pos = (s - torch.floor(s)) @ torch.as_tensor(box, dtype=torch.float64, device=dev)
    v = torch.randn((n, 4), generator=g, device=dev, dtype=torch.float64)
    q = 0.8 * (1.0 - 2.0 * (ijk.sum(1) % 2)) + 0.05 * v[:, 0]
    q = q - q.mean()
    return pos.float(), q.float(), (0.05 * v[:, 1:]).float().contiguous()


def _cotangents(n: int, g):
    v = torch.randn((n, 7), generator=g, device=_device())
    return v[:, :3].contiguous(), v[:, 3].contiguous(), v[:, 4:].contiguous()


def _batch_frames(case):
    """(n, box, mesh, order) of each frame of a batch: the same for every seed."""
    r = random.Random(case["sizes"])
    out = []
    for f in range(case["frames"]):
        n = r.randint(case["n_lo"], case["n_hi"])
        m = min(48, max(16, _smooth(int(math.ceil(_edge(n) / case["spacing"])))))
        out.append((n, _box(n, False), (m, m, m), (4, 6)[f % 2]))
    return out


_NET_BF16 = ("WA", "WB", "WU", "WY", "Wh")


def _net_params(g):
    """Gaussian initial parameters, sigma = 1/sqrt(fan_in), biases zero, mixing matrices in bfloat16."""
    from paper_2606_01598_gb300.net import PARAM_LAYOUT
    out = {}
    for name, shape in PARAM_LAYOUT:
        if name.startswith("b"):
            v = torch.zeros(shape, device=_device())
        else:
            v = torch.randn(shape, generator=g, device=_device()) / math.sqrt(shape[0])
            if name.startswith(_NET_BF16):
                v = v.bfloat16().float()
        out[name] = v
    return out


def _inputs(case, seed):
    """Everything of a case that comes from the seed (GPU tensors) and its frames."""
    g = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        frames = _batch_frames(case)
        parts = [_frame(n, box, g) for n, box, _, _ in frames]
        x = dict(zip(("pos", "q", "mu"), (torch.cat(t) for t in zip(*parts))))
        x["gf"], x["gphi"], x["gfield"] = _cotangents(len(x["q"]), g)
        x["ge"] = torch.randn(len(frames), generator=g, device=_device(), dtype=torch.float64)
    elif kind == "train":
        n, F, m = case["n"], case["frames"], case["mesh"]
        frames = [(n, _box(n, False), (m, m, m), case["order"])] * F
        x = dict(pos=torch.cat([_frame(n, box, g)[0] for n, box, _, _ in frames]))
        x["species"] = torch.randint(0, 2, (n * F,), generator=g, device=_device(), dtype=torch.int32)
        x["e_ref"] = n * torch.randn(F, generator=g, device=_device(), dtype=torch.float64)
        x["f_ref"] = torch.randn((n * F, 3), generator=g, device=_device())
        x["params"] = _net_params(g)
    else:
        frames = [(case["n"], _box(case["n"], case.get("tilt", False)), (case["nx"], case["ny"], case["nz"]),
                   case["order"])]
        x = dict(zip(("pos", "q", "mu"), _frame(case["n"], frames[0][1], g)))
        x["gf"], x["gphi"], x["gfield"] = _cotangents(case["n"], g)
        x["ge"] = torch.randn(1, generator=g, device=_device(), dtype=torch.float64)
        if kind == "quad":
            x["theta"] = 0.1 * torch.randn((case["n"], 6), generator=g, device=_device())
        if kind == "autograd":
            x["f_ref"] = 0.1 * torch.randn((case["n"], 3), generator=g, device=_device())
    return frames, x


def prepare(case, seed):
    frames, x = _inputs(case, seed)
    kind = case["kind"]
    s = dict(case=case, **x)
    if kind in ("batch", "train"):
        ns = np.array([f[0] for f in frames])
        offsets = np.concatenate([[0], np.cumsum(ns)])
        boxes = [f[1] for f in frames]
        s["plan"] = gb.BatchPlan(boxes, [f[2] for f in frames], [f[3] for f in frames], offsets, ALPHA, case["rcut"])
        if kind == "train":
            s["net"] = gb.Net(int(offsets[-1]), len(frames))
            s["net"].set_frames(offsets, boxes, x["species"].cpu().numpy())
            s["net"].set_params({k: v.cpu().numpy() for k, v in x["params"].items()})
        return s
    n, box, mesh, order = frames[0]
    s["plan"] = gb.Plan(box, mesh, order, ALPHA, case["rcut"], max_ions=n)
    if kind == "host":
        for k, v in x.items():
            s[k] = v.cpu().pin_memory()
    if kind == "host" or (kind in ("forward", "step") and case["reuse"]):
        new = lambda *shape, dtype=torch.float32: (  # noqa: E731
            torch.empty(shape, dtype=dtype, pin_memory=True) if kind == "host"
            else torch.empty(shape, dtype=dtype, device=_device()))
        s["out"] = dict(energy=new(1, dtype=torch.float64), force=new(n, 3), phi=new(n), field=new(n, 3))
        s["grads"] = (new(n, 3), new(n), new(n, 3))
    return s


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------

def _single(out):
    """The float64 energy (and virial) as a float32 program takes them."""
    return {k: v.float() if v.dtype == torch.float64 else v for k, v in out.items()}


def run(state):
    s, plan, kind = state, state["plan"], state["case"]["kind"]
    if kind == "forward":
        return _single(plan.forward(s["pos"], s["q"], s["mu"], virial=s["case"]["virial"], out=s.get("out")))
    if kind == "step":
        out = plan.forward(s["pos"], s["q"], s["mu"], out=s.get("out"))
        grads = plan.backward(s["pos"], s["q"], s["mu"], s["ge"], s["gf"], s["gphi"], s["gfield"], out=s.get("grads"))
        return dict(_single(out), grads=grads)
    if kind == "host":
        out = plan.forward(s["pos"], s["q"], s["mu"], out=s["out"], sync=False)
        grads = plan.backward(s["pos"], s["q"], s["mu"], s["ge"], s["gf"], s["gphi"], s["gfield"], out=s["grads"])
        return dict(_single(out), grads=grads)
    if kind == "autograd":
        x = [s[k].detach().requires_grad_(True) for k in ("pos", "q", "mu")]
        e = gb.pme_energy(plan, *x)
        force = -torch.autograd.grad(e, x[0], create_graph=True)[0]
        loss = ((force - s["f_ref"]) ** 2).mean()
        return dict(energy=e.detach().float(), force=force.detach(), grads=torch.autograd.grad(loss, x))
    if kind == "batch":
        out = _single(plan.forward(s["pos"], s["q"], s["mu"]))
        if s["case"]["backward"]:
            out["grads"] = plan.backward(s["pos"], s["q"], s["mu"], s["ge"], s["gf"], s["gphi"], s["gfield"])
        return out
    if kind == "quad":
        out = _single(plan.forward_quad(s["pos"], s["q"], s["mu"], s["theta"]))
        out["grads"] = plan.backward_quad(s["pos"], s["q"], s["mu"], s["theta"], s["ge"], s["gf"], s["gphi"],
                                          s["gfield"])
        return out
    loss, force, grad = s["net"].loss_grad(plan, s["pos"], s["e_ref"], s["f_ref"])
    return dict(loss=loss.float(), force=force, grad=grad)


def work(case):
    """Inputs read once, outputs written once; operations of the splines' separable sums, of the
    transforms and of the pairs inside the cutoff (80 a pair forward, 450 backward, 380 with
    quadrupoles), and of the network's products and messages."""
    kind = case["kind"]
    if kind == "batch":
        frames = _batch_frames(case)
    elif kind == "train":
        frames = [(case["n"], None, (case["mesh"],) * 3, case["order"])] * case["frames"]
    else:
        frames = [(case["n"], None, (case["nx"], case["ny"], case["nz"]), case["order"])]
    n = sum(f[0] for f in frames)
    pairs = n * 4.0 / 3.0 * math.pi * case["rcut"] ** 3 / VOLUME_PER_ION
    sten = sum(f[0] * f[3] ** 3 for f in frames)
    fft = sum(2 * 2.5 * math.prod(f[2]) * math.log2(math.prod(f[2])) for f in frames)
    forward, backward = 4 * sten + fft + 80 * pairs, 8 * sten + fft + 450 * pairs
    if kind == "quad":
        return dict(bytes=n * (52 + 52 + 80 + 52), flops=12 * sten + 2 * fft + (380 + 760) * pairs)
    if kind == "train":
        edges = n * 4.0 / 3.0 * math.pi * 5.0 ** 3 / VOLUME_PER_ION
        return dict(bytes=n * (12 + 12 + 12) + 2 * 4 * 13266,
                    flops=forward + backward + 6 * 2 * 13000 * 2 * n + 2 * 6 * 2 * 500 * edges)
    bwd = kind in ("step", "host", "autograd") or case.get("backward", False)
    return dict(bytes=n * (28 + 28 + (56 if bwd else 0)), flops=forward + (backward if bwd else 0))


# ------------------------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ------------------------------------------------------------------------------------------

F64 = torch.float64
SQRT_PI = math.sqrt(math.pi)


def _spline(p: int, f):
    """[W, W', W''] of the p stencil points (columns in mesh order) at fractional offsets f."""
    zero = torch.zeros_like(f)
    level = [torch.ones_like(f)]          # N_1(f + k)
    levels = {1: level}
    for m in range(2, p + 1):
        prev = [zero] + level + [zero]    # N_(m-1)(f + k - 1) at index k
        level = [((f + k) * prev[k + 1] + (m - f - k) * prev[k]) / (m - 1) for k in range(m)]
        levels[m] = level

    def derivative(m, order):
        if order == 0:
            return levels[m]
        if m == 1:
            return [zero]
        low = [zero] + derivative(m - 1, order - 1) + [zero]
        return [low[k + 1] - low[k] for k in range(m)]

    return [torch.stack(derivative(p, d)[::-1], 1) for d in range(3)]


def _pairs(pos, box, rcut):
    """Ordered pairs (i, j, integer shift) with |r_i - r_j + shift box| < rcut, every image."""
    dev, n = pos.device, len(pos)
    inv = torch.linalg.inv(box)
    s = pos @ inv
    widths = 1.0 / torch.linalg.norm(inv, dim=0)
    found = []
    if float(widths.min()) > 2.0 * rcut:
        for at in range(0, n, max(1, 200_000_000 // n)):
            d = s[at:at + max(1, 200_000_000 // n), None, :] - s[None, :, :]
            k = -torch.round(d)
            d += k
            r2 = ((d @ box) ** 2).sum(-1)
            i, j = torch.nonzero(r2 < rcut * rcut, as_tuple=True)
            keep = i + at != j
            i, j = i[keep], j[keep]
            found.append((i + at, j, k[i, j]))
    else:
        reach = [int(math.ceil(rcut / float(w))) + 1 for w in widths]
        images = torch.cartesian_prod(*[torch.arange(-r, r + 1, device=dev, dtype=F64) for r in reach])
        step = max(1, 100_000_000 // (n * len(images)))
        for at in range(0, n, step):
            d = (s[at:at + step, None, None, :] - s[None, :, None, :] + images) @ box
            i, j, k = torch.nonzero((d * d).sum(-1) < rcut * rcut, as_tuple=True)
            keep = (i + at != j) | (images[k] != 0).any(1)
            i, j, k = i[keep], j[keep], k[keep]
            found.append((i + at, j, images[k]))
    return [torch.cat(t) for t in zip(*found)]


class _Exact:
    """The energies of a list of frames (n, box, mesh, order), in torch operations."""

    def __init__(self, frames, rcut, pos):
        self.frames, dev = frames, pos.device
        self.start = np.concatenate([[0], np.cumsum([f[0] for f in frames])])
        self.boxes = [torch.as_tensor(f[1], dtype=F64, device=dev) for f in frames]
        self.of = torch.repeat_interleave(torch.arange(len(frames), device=dev),
                                          torch.tensor([f[0] for f in frames], device=dev))
        parts = []
        for f, box in enumerate(self.boxes):
            a = int(self.start[f])
            i, j, k = _pairs(pos[a:a + frames[f][0]], box, rcut)
            parts.append((i + a, j + a, k))
        self.i, self.j, self.k = [torch.cat(t) for t in zip(*parts)]

    def energy(self, pos, q, mu, theta=None, strain=None):
        """[F] energies; with strain, those of the cell and positions under r -> (1 + strain) r."""
        dev, frames = pos.device, self.frames
        boxes = self.boxes
        if strain is not None:
            grow = (torch.eye(3, dtype=F64, device=dev) + strain).T
            boxes, pos = [b @ grow for b in boxes], pos @ grow
        box = torch.stack(boxes)
        inv = torch.linalg.inv(box)
        size = torch.tensor([f[2] for f in frames], device=dev)
        points = [math.prod(f[2]) for f in frames]
        base = torch.tensor(np.concatenate([[0], np.cumsum(points)[:-1]]), device=dev)
        to_mesh = inv[self.of] * size[self.of][:, None, :]                       # columns scaled by N
        x = torch.einsum("na,nab->nb", pos, to_mesh)
        d = torch.einsum("na,nab->nb", mu, to_mesh)
        t = None if theta is None else torch.einsum("nka,nkl,nlb->nab", to_mesh, theta, to_mesh)
        orders = torch.tensor([f[3] for f in frames], device=dev)[self.of]
        rho = torch.zeros(sum(points), dtype=F64, device=dev)
        for p in sorted({f[3] for f in frames}):
            at = torch.nonzero(orders == p)[:, 0]
            xp = x[at]
            low = torch.floor(xp.detach() - 0.5 * p)
            w, w1, w2 = zip(*[_spline(p, xp[:, a] - 0.5 * p - low[:, a]) for a in range(3)])
            X, Y, Z = ([u[a] for u in (w, w1, w2)] for a in range(3))
            c, dm = q[at][:, None], d[at]
            zz = c * Z[0] + dm[:, 2:3] * Z[1]
            if t is not None:
                tt = t[at]
                zz = zz + tt[:, 2, 2, None] * Z[2]
                yz = dm[:, 1:2] * Z[0] + 2 * tt[:, 1, 2, None] * Z[1]
                xz = dm[:, 0:1] * Z[0] + 2 * tt[:, 0, 2, None] * Z[1]
                plane0 = Y[0][:, :, None] * zz[:, None, :] + Y[1][:, :, None] * yz[:, None, :] \
                    + Y[2][:, :, None] * (tt[:, 1, 1, None] * Z[0])[:, None, :]
                plane1 = Y[0][:, :, None] * xz[:, None, :] \
                    + Y[1][:, :, None] * (2 * tt[:, 0, 1, None] * Z[0])[:, None, :]
                plane2 = Y[0][:, :, None] * (tt[:, 0, 0, None] * Z[0])[:, None, :]
                val = X[0][:, :, None, None] * plane0[:, None] + X[1][:, :, None, None] * plane1[:, None] \
                    + X[2][:, :, None, None] * plane2[:, None]
            else:
                plane0 = Y[0][:, :, None] * zz[:, None, :] + Y[1][:, :, None] * (dm[:, 1:2] * Z[0])[:, None, :]
                plane1 = Y[0][:, :, None] * (dm[:, 0:1] * Z[0])[:, None, :]
                val = X[0][:, :, None, None] * plane0[:, None] + X[1][:, :, None, None] * plane1[:, None]
            N = size[self.of[at]]
            m = low.long()[:, :, None] + 1 + torch.arange(p, device=dev)
            m = torch.remainder(m, N[:, :, None])
            flat = (m[:, 0, :, None, None] * N[:, 1, None, None, None] + m[:, 1, None, :, None]) \
                * N[:, 2, None, None, None] + m[:, 2, None, None, :] + base[self.of[at]][:, None, None, None]
            rho = rho.scatter_add(0, flat.reshape(-1), val.reshape(-1))
        total = []
        for f, (n, _, mesh, p) in enumerate(frames):
            r = torch.fft.rfftn(rho[int(base[f]):int(base[f]) + points[f]].reshape(mesh))
            sig = [torch.fft.fftfreq(mesh[0], dtype=F64, device=dev) * mesh[0],
                   torch.fft.fftfreq(mesh[1], dtype=F64, device=dev) * mesh[1],
                   torch.arange(mesh[2] // 2 + 1, dtype=F64, device=dev)]
            G = 2 * math.pi * inv[f]
            kv = sig[0][:, None, None, None] * G[:, 0] + sig[1][:, None, None] * G[:, 1] + sig[2][:, None] * G[:, 2]
            k2 = (kv * kv).sum(-1)
            some = torch.ones_like(k2, dtype=torch.bool)
            some[0, 0, 0] = False
            k2 = torch.where(some, k2, torch.ones_like(k2))
            green = torch.where(some, 4 * math.pi * torch.exp(-k2 / (4 * ALPHA ** 2)) / k2, torch.zeros_like(k2))
            for a, shape in enumerate(((-1, 1, 1), (1, -1, 1), (1, 1, -1))):
                green = green / (torch.sinc(sig[a] / mesh[a]) ** (2 * p)).reshape(shape)
            twice = torch.full((mesh[2] // 2 + 1,), 2.0, dtype=F64, device=dev)
            twice[0] = 1.0
            if mesh[2] % 2 == 0:
                twice[-1] = 1.0
            V = torch.linalg.det(box[f]).abs()
            e = 0.5 / V * (green * twice * (r.real ** 2 + r.imag ** 2)).sum()
            Q = q[int(self.start[f]):int(self.start[f]) + n].sum()
            total.append(e - math.pi * Q * Q / (2 * V * ALPHA ** 2))
        own = -(ALPHA / SQRT_PI) * q * q - (2 * ALPHA ** 3 / (3 * SQRT_PI)) * (mu * mu).sum(1)
        if theta is not None:
            tr = torch.einsum("naa->n", theta)
            own = own - (ALPHA / SQRT_PI) * (-(4 * ALPHA ** 2 / 3) * q * tr + (4 * ALPHA ** 4 / 5)
                                             * (tr * tr + 2 * (theta * theta).sum((1, 2))))
        per = torch.zeros(len(frames), dtype=F64, device=dev).index_add(0, self.of, own)
        per = per.index_add(0, self.of[self.i], 0.5 * self._pair(pos, q, mu, theta, box))
        return torch.stack(total) + per

    def _pair(self, pos, q, mu, theta, box):
        i, j = self.i, self.j
        r = pos[i] - pos[j] + torch.einsum("pa,pab->pb", self.k, box[self.of[i]])
        r2 = (r * r).sum(1)
        d = torch.sqrt(r2)
        ex = torch.exp(-ALPHA * ALPHA * r2) / (ALPHA * SQRT_PI)
        B = [torch.special.erfc(ALPHA * d) / d]
        for l in range(1, 3 if theta is None else 5):
            B.append(((2 * l - 1) * B[-1] + (2 * ALPHA * ALPHA) ** l * ex) / r2)
        a, b = (mu[i] * r).sum(1), (mu[j] * r).sum(1)
        u = q[i] * q[j] * B[0] + (q[i] * b - q[j] * a + (mu[i] * mu[j]).sum(1)) * B[1] - a * b * B[2]
        if theta is None:
            return u
        Ti, Tj = theta[i], theta[j]
        ti, tj = torch.einsum("paa->p", Ti), torch.einsum("paa->p", Tj)
        vi, vj = torch.einsum("pab,pb->pa", Ti, r), torch.einsum("pab,pb->pa", Tj, r)
        si, sj = (vi * r).sum(1), (vj * r).sum(1)
        u = u + q[i] * (sj * B[2] - tj * B[1]) + q[j] * (si * B[2] - ti * B[1])
        u = u + (tj * a + 2 * (mu[i] * vj).sum(1)) * B[2] - sj * a * B[3]
        u = u - (ti * b + 2 * (mu[j] * vi).sum(1)) * B[2] + si * b * B[3]
        return u + (ti * tj + 2 * (Ti * Tj).sum((1, 2))) * B[2] \
            - (ti * sj + tj * si + 4 * (vi * vj).sum(1)) * B[3] + si * sj * B[4]


def _six(T):
    T = 0.5 * (T + T.transpose(1, 2))
    return torch.stack([T[:, 0, 0], T[:, 1, 1], T[:, 2, 2], T[:, 0, 1], T[:, 0, 2], T[:, 1, 2]], 1)


def _network(P, pos, species, offsets, boxes):
    """q, mu and per-frame short-range energies of the two-layer network (32 scalar and 16 vector
    channels, 8 Bessel functions, 5 Angstrom, messages over 16)."""
    S, V, rc = 32, 16, 5.0
    dev, n = pos.device, len(pos)
    I, J, D = [], [], []
    for f, box in enumerate(boxes):
        a, b = int(offsets[f]), int(offsets[f + 1])
        s = pos.detach()[a:b] @ torch.linalg.inv(box)
        d = s[None] - s[:, None]
        k = -torch.round(d)
        i, j = torch.nonzero((((d + k) @ box) ** 2).sum(-1) < rc * rc, as_tuple=True)
        keep = i != j
        i, j = i[keep], j[keep]
        I.append(i + a), J.append(j + a), D.append(k[i, j] @ box)
    i, j = torch.cat(I), torch.cat(J)
    d = pos[j] - pos[i] + torch.cat(D)
    r = torch.sqrt((d * d).sum(1))
    h = d / r[:, None]
    x = r / rc
    k = torch.arange(1, 9, dtype=F64, device=dev)
    e = math.sqrt(2 / rc) * torch.sin(k * math.pi * x[:, None]) / r[:, None] \
        * (1 - 21 * x ** 5 + 35 * x ** 6 - 15 * x ** 7)[:, None]
    hs, hv = P["emb"][species.long()], torch.zeros((n, 3, V), dtype=F64, device=dev)
    for t in range(2):
        A, B, R = hs @ P[f"WA{t}"], hv @ P[f"WB{t}"], e @ P[f"WR{t}"]
        Aj, Bj = A[j], B[j]
        ms = torch.cat([R[:, :S] * Aj[:, :S],
                        R[:, S:S + V] * torch.einsum("ea,eac->ec", h, Bj[:, :, :V])], 1)
        mv = torch.cat([(R[:, S + V:S + 2 * V] * Aj[:, S:])[:, None, :] * h[:, :, None],
                        R[:, None, S + 2 * V:] * Bj[:, :, V:]], 2)
        ms = torch.zeros((n, S + V), dtype=F64, device=dev).index_add(0, i, ms) / 16
        mv = torch.zeros((n, 3, 2 * V), dtype=F64, device=dev).index_add(0, i, mv) / 16
        U = ms @ P[f"WU{t}"]
        hs = hs + torch.nn.functional.silu(U[:, :S])
        hv = hv + torch.sigmoid(U[:, S:])[:, None, :] * (mv @ P[f"WY{t}"])
    H = torch.nn.functional.silu(hs @ P["Wh"] + P["bh"])
    q = H[:, :S] @ P["wq"] + P["bq"]
    q = torch.cat([t - t.mean() for t in torch.split(q, np.diff(offsets).tolist())])
    site = H[:, S:] @ P["wE"] + P["bE"]
    return q, hv @ P["wmu"], torch.stack([t.sum() for t in torch.split(site, np.diff(offsets).tolist())])


def exact(case, seed):
    frames, x = _inputs(case, seed)
    kind = case["kind"]
    x = {k: v.double() if torch.is_tensor(v) and v.is_floating_point() else v for k, v in x.items()}
    model = _Exact(frames, case["rcut"], x["pos"])
    if kind == "train":
        P = {k: v.double().requires_grad_(True) for k, v in x["params"].items()}
        pos = x["pos"].requires_grad_(True)
        q, mu, short = _network(P, pos, x["species"], model.start, model.boxes)
        e = short + model.energy(pos, q, mu)
        force = -torch.autograd.grad(e.sum(), pos, create_graph=True)[0]
        le = (((e - x["e_ref"]) / case["n"]) ** 2).mean()
        lf = ((force - x["f_ref"]) ** 2).mean()
        grads = torch.autograd.grad(le + lf, list(P.values()))
        return dict(loss=torch.stack([le + lf, le, lf]).detach(), force=force.detach(),
                    grad=torch.cat([t.reshape(-1) for t in grads]))
    leaves = [x[k].requires_grad_(True) for k in ("pos", "q", "mu")]
    if kind == "quad":
        t = x["theta"]
        leaves.append(t[:, [0, 3, 4, 3, 1, 5, 4, 5, 2]].reshape(-1, 3, 3).requires_grad_(True))
    second = kind in ("step", "host", "autograd", "quad") or case.get("backward", False)
    strain = torch.zeros((3, 3), dtype=F64, device=x["pos"].device, requires_grad=True) if case.get("virial") else None
    e = model.energy(*leaves, strain=strain)
    g = torch.autograd.grad(e.sum(), leaves + ([strain] if strain is not None else []), create_graph=second)
    if kind == "autograd":
        force = -g[0]
        grads = torch.autograd.grad(((force - x["f_ref"]) ** 2).mean(), leaves)
        return dict(energy=e.detach().reshape(()), force=force.detach(), grads=grads)
    out = dict(energy=e.detach(), force=-g[0].detach(), phi=g[1].detach(), field=-g[2].detach())
    if strain is not None:
        out["virial"] = -g[3].detach()
    if kind == "quad":
        out["field_grad"] = -_six(g[3].detach())
    if second:
        L = (x["ge"] * e).sum() - (x["gf"] * g[0]).sum() + (x["gphi"] * g[1]).sum() - (x["gfield"] * g[2]).sum()
        grads = list(torch.autograd.grad(L, leaves))
        if kind == "quad":
            grads[3] = _six(grads[3])
        out["grads"] = tuple(grads)
    return out
