"""Workloads of this package that its speed is measured on.

Each case is one call (or the few calls) a user's program makes on the public
binding, on inputs it holds in GPU memory: registering whole series with a
prefix scan, adding one frame to a running series, building a handle from
frames, averaging a registered series, and the learned initialiser's forward
and training passes.  Frames come from a small generator (a drifting, distorted
lattice of Gaussian atom columns over a few large blobs, under Poisson noise)
with the lattices, counts and motions of the repository's workloads.
"""
import math
import random

import numpy as np
import torch

import paper_1712_02533_gb300 as reg

SCHEDULES = {"serial": reg.SERIAL, "sklansky": reg.SKLANSKY, "kogge_stone": reg.KOGGE_STONE,
             "brent_kung": reg.BRENT_KUNG, "blelloch": reg.BLELLOCH}

# Lattice spacing, atom sigma, peak counts, drift per frame and distortion (px)
# of the 64^2, 512^2 and 1024^2 workloads.
FINE = dict(spacing=8.0, sigma=1.5, peak=20.0, drift=0.5, dist=1.0)
MIDDLE = dict(spacing=12.0, sigma=2.0, peak=10.0, drift=0.5, dist=1.0)
COARSE = dict(spacing=16.0, sigma=2.0, peak=5.0, drift=1.0, dist=2.0)


def listed():
    return [
        # The smallest series anyone registers (8 frames of 64^2): latency of the
        # solver's steps, hardly any arithmetic.
        dict(name="scan 8x64", kind="scan", sides="64", frames="8", levels=3, schedule="sklansky", bf16=False,
             smooth=0.0, rigid=False, **FINE),
        # Several series of different sides and lengths in one segmented scan,
        # pyramids stored in BF16.
        dict(name="scan mixed bf16", kind="scan", sides="64,256,128", frames="7,11,5", levels=3,
             schedule="sklansky", bf16=True, smooth=0.0, rigid=False, **MIDDLE),
        # An ordinary series: the 512^2 workload's frames with a work-efficient tree.
        dict(name="scan 21x512", kind="scan", sides="512", frames="21", levels=4, schedule="brent_kung", bf16=False,
             smooth=0.0, rigid=False, **MIDDLE),
        # The bulk of a long series: wide batches of 1024^2 operators on five
        # levels, the benchmark's frames and tree.
        dict(name="scan 33x1024", kind="scan", sides="1024", frames="33", levels=5, schedule="sklansky", bf16=False,
             smooth=0.0, rigid=False, **COARSE),
        # During an acquisition: one new 1024^2 frame is registered to its
        # predecessor and combined with the running deformation, one operator
        # at a time.
        dict(name="arrival 1024", kind="arrival", side=1024, levels=5, bf16=False, **COARSE),
        # The smoothed flow of the method's H1-type smoother.
        dict(name="scan smooth 6x256", kind="scan", sides="256", frames="6", levels=4, schedule="sklansky",
             bf16=False, smooth=2.0, rigid=False, **MIDDLE),
        # Registration with rigid maps.
        dict(name="scan rigid 9x256", kind="scan", sides="256", frames="9", levels=3, schedule="sklansky", bf16=False,
             smooth=0.0, rigid=True, **MIDDLE),
        # Opening a series: frames on the GPU to a handle with its pyramids, and
        # the network inputs of its neighbour pairs read from them.
        dict(name="open 40x1024", kind="open", side=1024, frames=40, levels=5, bf16=False, **COARSE),
        # The average image of a registered series.
        dict(name="average 64x1024", kind="average", side=1024, frames=64, levels=5, bf16=False, **COARSE),
        # Starting displacements predicted for a chunk of neighbour pairs, BF16
        # tensor cores.
        dict(name="cnn forward 64", kind="cnn_forward", side=256, batch=64, tensor_cores=True),
        # One minibatch step of training on the tensor cores.
        dict(name="cnn train 32", kind="cnn_train", side=256, batch=32, tensor_cores=True),
        # The same in FP32, the binding's default.
        dict(name="cnn train fp32 32", kind="cnn_train", side=256, batch=32, tensor_cores=False),
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["scan", "scan", "scan", "multi", "smooth", "rigid", "arrival", "open", "average",
                       "cnn_forward", "cnn_train"])
    look = dict(rng.choice([FINE, MIDDLE, COARSE]))
    look["peak"] = round(look["peak"] * rng.uniform(0.8, 1.5), 2)
    look["spacing"] = round(look["spacing"] * rng.uniform(0.9, 1.1), 2)
    bf16 = rng.random() < 0.25

    def scan(sides, frames, levels, schedule, **kw):
        c = dict(kind="scan", sides=",".join(map(str, sides)), frames=",".join(map(str, frames)), levels=levels,
                 schedule=schedule, bf16=bf16, smooth=0.0, rigid=False, **look)
        c.update(kw)
        return c

    if kind == "scan":
        L = rng.choice([6, 7, 8, 9, 10])
        # from 2 frames to as many as keep the batch below the largest listed one
        n = log_int(2, min(48, 33 << (2 * (10 - L))))
        names = ["sklansky", "brent_kung", "blelloch"] + (["kogge_stone"] if L < 10 else []) + (
            ["serial"] if n <= 9 and L < 10 else [])
        return scan([1 << L], [n], rng.randint(2, min(5, L - 3)), rng.choice(names))
    if kind == "multi":
        m = rng.randint(2, 4)
        sides = [1 << rng.choice([6, 7, 8, 9]) for _ in range(m)]
        return scan(sides, [rng.randint(2, 13) for _ in sides], rng.choice([2, 3]), "sklansky")
    if kind == "smooth":
        L = rng.choice([6, 7, 8])
        return scan([1 << L], [rng.randint(2, 6)], rng.randint(2, L - 4), "sklansky",
                    smooth=round(rng.uniform(1.0, 4.0), 1), bf16=False)
    if kind == "rigid":
        L = rng.choice([6, 7, 8])
        return scan([1 << L], [log_int(2, 16)], rng.randint(2, 3), "sklansky", rigid=True, bf16=False)
    if kind == "arrival":
        L = rng.choice([7, 8, 9, 10])
        return dict(kind="arrival", side=1 << L, levels=rng.randint(2, min(5, L - 3)), bf16=bf16, **look)
    if kind in ("open", "average"):
        L = rng.choice([8, 9, 10])
        most = 64 if kind == "average" else 40
        return dict(kind=kind, side=1 << L, frames=log_int(2, most << min(2, 10 - L)),
                    levels=rng.randint(max(1, L - 7), 5), bf16=bf16, **look)
    return dict(kind=kind, side=256, batch=log_int(1, 64 if kind == "cnn_forward" else 32),
                tensor_cores=rng.random() < 0.6)


# --- inputs ------------------------------------------------------------------------

def _motion(seed, n, case, side):
    """Per frame k the displacement d_k of the specimen, as row and column terms
    (d_k(y) = (x-term of the row, y-term of the column))."""
    rng = random.Random(seed)
    ph = [[rng.uniform(0, 2 * math.pi) for _ in range(3)] for _ in range(2)]
    tx = ty = 0.0
    c = torch.arange(side + 1, device="cuda", dtype=torch.float32)
    out = []
    for k in range(n):
        if k:
            tx += rng.gauss(0, case["drift"])
            ty += rng.gauss(0, case["drift"])
        dx, dy = torch.full_like(c, tx), torch.full_like(c, ty)
        for (period, nu), (p0, p1, p2) in zip(((37.0, 1.0), (91.0, 2.0)), ph):
            a = case["dist"] * math.sin(2 * math.pi * k / period + p2)
            dx = dx + a * torch.sin(2 * math.pi * nu / side * c + p0)
            dy = dy + a * torch.sin(2 * math.pi * nu / side * c + p1)
        out.append((dx, dy))
    return out


def _field(motion, k):
    """phi_{0,k} - id = d_0 - d_k to first order, pixels on the vertex grid."""
    fx = (motion[0][0] - motion[k][0])[:, None].expand(-1, motion[0][0].numel())
    fy = (motion[0][1] - motion[k][1])[None, :].expand(motion[0][1].numel(), -1)
    return torch.stack([fx, fy]).contiguous()


def _frames(seed, n, side, case, motion=None):
    rng = random.Random(seed + 7919)
    g = torch.Generator(device="cuda").manual_seed(seed)
    s, sig = case["spacing"], case["sigma"]
    ox, oy = rng.uniform(0, s), rng.uniform(0, s)
    blobs = [(rng.uniform(0, side), rng.uniform(0, side), side * rng.uniform(1 / 16, 1 / 6), rng.uniform(0.5, 1.0))
             for _ in range(6)]
    c = torch.arange(side, device="cuda", dtype=torch.float32)
    out = torch.empty((n, side, side), device="cuda")
    for k, (dx, dy) in enumerate(motion or _motion(seed, n, case, side)):
        z0, z1 = c[None, :] + dx[:side, None], c[:, None] + dy[None, :side]
        q0 = z0 - ox - s * torch.round((z0 - ox) / s)
        q1 = z1 - oy - s * torch.round((z1 - oy) / s)
        v = torch.exp(-(q0 * q0 + q1 * q1) / (2 * sig * sig)) + 0.15
        for bx, by, br, ba in blobs:
            v = v + 0.6 * ba * torch.exp(-((z0 - bx) ** 2 + (z1 - by) ** 2) / (2 * br * br))
        out[k] = torch.poisson(v * (case["peak"] / 1.75), generator=g)
    return out


def _params(case):
    return reg.default_params(n_levels=case["levels"], storage=reg.STORAGE_BF16 if case["bf16"] else reg.STORAGE_F32,
                              smooth=case.get("smooth", 0.0), flags=reg.FLAG_RIGID if case.get("rigid") else 0)


CNN_SHAPES = [(2, 32), (32, 32), (32, 32), (32, 32), (32, 32), (32, 2)]
CNN_STRIDES = [2, 2, 1, 1, 1, 1]


def _theta(seed):
    """Network parameters: He-normal weights, small biases."""
    rng = np.random.default_rng(seed)
    parts = []
    for c, o in CNN_SHAPES:
        parts += [rng.standard_normal(o * c * 9) * math.sqrt(2.0 / (9 * c)), 0.05 * rng.standard_normal(o)]
    return np.concatenate(parts).astype(np.float32)


def _pairs(seed, batch, side):
    """Normalised neighbour pairs, as the network sees them, and displacements of
    the size the plain method finds between them."""
    fr = _frames(seed, batch + 1, side, MIDDLE)
    fr = (fr - fr.mean(dim=(1, 2), keepdim=True)) / fr.std(dim=(1, 2), keepdim=True)
    x = torch.stack([fr[:-1], fr[1:]], 1).contiguous()
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    t = 0.5 * torch.randn((batch, 2, 1, 1), generator=g, device="cuda") + 0.1 * torch.randn(
        (batch, 2, side // 4, side // 4), generator=g, device="cuda")
    return x, t.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "scan":
        sides, counts = ([int(v) for v in case[k].split(",")] for k in ("sides", "frames"))
        fr = [_frames(seed + 31 * i, n, s, case) for i, (n, s) in enumerate(zip(counts, sides))]
        if len(set(sides)) > 1:
            fr = [f.cpu().numpy() for f in fr]  # series of different sides come from host memory
        s = reg.Series(fr, _params(case))
        out = [torch.empty((n, 2, side, side), device="cuda") for n, side in zip(counts, sides)]
        return dict(kind=kind, s=s, out=out, schedule=SCHEDULES[case["schedule"]])
    if kind == "arrival":
        motion = _motion(seed, 3, case, case["side"])
        s = reg.Series(_frames(seed, 3, case["side"], case, motion), _params(case))
        s.set_slot_device(0, _field(motion, 1), 0, 1)
        return dict(kind=kind, s=s)
    if kind == "open":
        fr = _frames(seed, case["frames"], case["side"], case)
        x = torch.empty((case["frames"] - 1, 2, 256, 256), device="cuda")
        return dict(kind=kind, frames=fr, x=x, params=_params(case))
    if kind == "average":
        motion = _motion(seed, case["frames"], case, case["side"])
        s = reg.Series(_frames(seed, case["frames"], case["side"], case, motion), _params(case))
        for k in range(1, case["frames"]):
            s.set_slot_device(k - 1, _field(motion, k), 0, k)
        return dict(kind=kind, s=s, out=torch.empty((case["side"], case["side"]), device="cuda"))
    x, t = _pairs(seed, case["batch"], case["side"])
    net = reg.Cnn(_theta(seed), side=case["side"], max_batch=case["batch"])
    return dict(kind=kind, net=net, x=x, t=t, tc=case["tensor_cores"])


def run(state):
    kind = state["kind"]
    if kind == "scan":
        s = state["s"]
        s.prefix_scan(state["schedule"])
        return [s.get_deformations(i, out=o) for i, o in enumerate(state["out"])]
    if kind == "arrival":
        # phi_{1,2} into slot 1, then phi_{0,2} = phi_{0,1} (.)_B phi_{1,2} in its place
        s = state["s"]
        s.apply_operator_batch([(0, -1, -1, 1, 1, 2)])
        s.apply_operator_batch([(0, 0, 1, 1, 0, 2)])
        return s.get_slot_device(1)
    if kind == "open":
        with reg.Series(state["frames"], state["params"]) as s:
            return s.cnn_pairs(0, s.counts[0] - 1, state["x"])
    if kind == "average":
        return state["s"].average(iterations=0, out=state["out"])
    if kind == "cnn_forward":
        return state["net"].forward(state["x"], tensor_cores=state["tc"])
    loss, grad = state["net"].loss_grad(state["x"], state["t"], want_grad=True, tensor_cores=state["tc"])
    state["net"].adam_step(1e-4)
    return loss, grad


# --- what a pass cannot do without -----------------------------------------------------

def _nodes(side, levels):
    return sum(((side >> k) + 1) ** 2 for k in range(levels))


def _scan_ops(n, schedule):
    """Operator applications over n neighbour pairs."""
    levels, _ = reg.schedule(SCHEDULES[schedule], n)
    return n + sum(1 for lv in levels for o in lv if o[0] == "op")


# Arithmetic of one gradient iteration per node: the direction (warp, mass and
# stiffness stencils) and the energy of two step sizes.
FLOP_ITER = 200.0


def work(case):
    kind = case["kind"]
    if kind in ("scan", "arrival"):
        if kind == "arrival":
            jobs = [(case["side"], 3, 2)]
        else:
            jobs = [(int(s), int(n), _scan_ops(int(n) - 1, case["schedule"]))
                    for s, n in zip(case["sides"].split(","), case["frames"].split(","))]
        img = 2 if case["bf16"] else 4
        nbytes = sum(n * img * _nodes(s, case["levels"]) + n * 8 * s * s for s, n, _ in jobs)
        flops = sum(o * 50 * FLOP_ITER * _nodes(s, case["levels"]) for s, _, o in jobs)
        return dict(bytes=nbytes, flops=flops)
    if kind == "open":
        # frames read; normalised pyramid and mass-weighted pyramid written; pairs written
        px, nd = case["side"] ** 2, _nodes(case["side"], case["levels"])
        return dict(bytes=case["frames"] * (4 * px + (4 + (2 if case["bf16"] else 4)) * nd) +
                    4 * (case["frames"] - 1) * 2 * 256 * 256, flops=40.0 * case["frames"] * nd)
    if kind == "average":
        px = case["side"] ** 2
        return dict(bytes=case["frames"] * px * (8 + (2 if case["bf16"] else 4)) + 4 * px,
                    flops=12.0 * case["frames"] * px)
    q, fl = case["side"], 0.0
    for (c, o), st in zip(CNN_SHAPES, CNN_STRIDES):
        q //= st
        fl += 2.0 * q * q * c * o * 9
    x, y = 2 * case["side"] ** 2, 2 * q * q
    if kind == "cnn_forward":
        return dict(bytes=4.0 * case["batch"] * (x + y), flops=fl * case["batch"])
    return dict(bytes=4.0 * case["batch"] * (x + y), flops=3 * fl * case["batch"])


# --- the same in 64 bits -----------------------------------------------------------------

def _embed64(frames):
    return torch.nn.functional.pad(frames.double()[:, None], (0, 1, 0, 1), mode="replicate")[:, 0]


def _restrict64(f):
    w = torch.tensor([0.25, 0.5, 0.25], dtype=torch.float64, device=f.device)
    p = torch.nn.functional.pad(f[:, None], (1, 1, 1, 1), mode="reflect")[:, 0]
    p = sum(w[a] * p[:, a:a + f.shape[1]:2, :] for a in range(3))
    return sum(w[b] * p[:, :, b:b + f.shape[2]:2] for b in range(3))


def _normalise64(f):
    """FE mean 0 and FE standard deviation 1 (exact Q1 element integrals)."""
    h2 = 1.0 / (f.shape[1] - 1) ** 2

    def corners(v):
        return v[:, :-1, :-1], v[:, :-1, 1:], v[:, 1:, 1:], v[:, 1:, :-1]

    mean = h2 * 0.25 * sum(v.sum(dim=(1, 2)) for v in corners(f))
    f = f - mean[:, None, None]
    a, b, c, d = corners(f)
    q = 4 * (a * a + b * b + c * c + d * d) + 4 * (a * b + b * c + c * d + d * a) + 2 * (a * c + b * d)
    return f / (h2 * q.sum(dim=(1, 2)) / 36.0).sqrt()[:, None, None]


def _sample64(img, u):
    """Bilinear interpolant of an n x n nodal image at the nodes moved by u, clamped."""
    n = img.shape[0]
    c = torch.arange(n, device=img.device, dtype=torch.float64)
    x, y = (c[None, :] + u[0]).clamp(0, n - 1), (c[:, None] + u[1]).clamp(0, n - 1)
    jx, jy = x.floor().clamp(max=n - 2).long(), y.floor().clamp(max=n - 2).long()
    ax, ay = x - jx, y - jy
    v = img.reshape(-1)
    i = jy * n + jx
    return (1 - ay) * ((1 - ax) * v[i] + ax * v[i + 1]) + ay * ((1 - ax) * v[i + n] + ax * v[i + n + 1])


def _net64(theta, x):
    a, off = x.double(), 0
    for k, ((c, o), st) in enumerate(zip(CNN_SHAPES, CNN_STRIDES)):
        w = theta[off:off + o * c * 9].reshape(o, c, 3, 3)
        b = theta[off + o * c * 9:off + o * c * 9 + o]
        off += o * c * 9 + o
        # the convolution as nine shifted products
        p, q = torch.nn.functional.pad(a, (1, 1, 1, 1)), a.shape[2] // st
        z = b[None, :, None, None].expand(a.shape[0], o, q, q)
        for dy in range(3):
            for dx in range(3):
                z = z + torch.einsum("bchw,oc->bohw", p[:, :, dy:dy + st * (q - 1) + 1:st, dx:dx + st * (q - 1) + 1:st],
                                     w[:, :, dy, dx])
        a = z if k == 5 else torch.relu(z)
    return a


def exact(case, seed):
    kind = case["kind"]
    if kind in ("scan", "arrival"):
        # an iterative flow whose 64-bit form takes minutes
        return None
    if kind == "open":
        fr = _frames(seed, case["frames"], case["side"], case)
        f = torch.empty((case["frames"], 256, 256), dtype=torch.float64, device="cuda")
        for k in range(0, case["frames"], 8):
            v = _embed64(fr[k:k + 8])
            while v.shape[1] > 257:
                v = _restrict64(v)
            f[k:k + 8] = _normalise64(v)[:, :256, :256]
        return torch.stack([f[:-1], f[1:]], 1)
    if kind == "average":
        side, n = case["side"], case["frames"]
        motion = _motion(seed, n, case, side)
        fr = _frames(seed, n, side, case, motion)
        acc = torch.zeros((side + 1, side + 1), dtype=torch.float64, device="cuda")
        for k in range(n):
            img = _embed64(fr[k:k + 1])[0]
            acc += _sample64(img, _field(motion, k).double()) if k else img
        return acc[:side, :side] / n
    x, t = _pairs(seed, case["batch"], case["side"])
    theta = torch.from_numpy(_theta(seed)).cuda().double()
    if kind == "cnn_forward":
        return torch.cat([_net64(theta, x[k:k + 8]) for k in range(0, case["batch"], 8)])
    theta.requires_grad_(True)
    loss, grad = 0.0, torch.zeros_like(theta)
    for k in range(0, case["batch"], 4):
        part = ((_net64(theta, x[k:k + 4]) - t[k:k + 4].double()) ** 2).sum() / t.numel()
        grad += torch.autograd.grad(part, theta)[0]
        loss += float(part)
    return loss, grad.cpu().numpy()
