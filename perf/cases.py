"""The work that users of the denoiser have it do, as cases a program can time.

Every case goes through the public front end (``Denoiser``, ``Params``,
``SoftRemoval``) with the clouds the method is meant for: an object scan, a
dense scan of several objects, spinning-LiDAR frames with snow, single or as a
batch, the calibration step, the cross-leaf variant, one leaf for the whole
cloud, the evaluation metrics and the Sec. 2.2 baseline.  The clouds are
seeded and made on the GPU.

A case is a dict of plain values:
  kind     what is called (see ``run``)
  cloud    "object", "scan", "lidar" (32 beams) or "street" (128 beams)
  n        points (of the whole batch for kind "batch")
  frames   frames of a batch
  k, capacity, rescore, scale   method parameters and the coordinates' unit
"""

from __future__ import annotations

import math
import random

import torch

from paper_2512_10386_gb300 import Denoiser, Params, SoftRemoval, soft_f1_loss

ONE_LEAF = 0xFFFFFFFF  # leaf capacity of the "without octree" configuration


def _case(name, kind, cloud, n, k, capacity=512, frames=1, rescore=0, scale=1.0):
    c = {"kind": kind, "cloud": cloud, "n": n, "frames": frames, "k": k, "capacity": capacity,
         "rescore": rescore, "scale": scale}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a cropped object or a region of interest with the default parameters: latency
        _case("object_1500", "sync", "object", 1500, 12),
        # a whole object scan (the paper's Bunny has about this many points)
        _case("object_36750", "sync", "object", 36750, 16),
        # one 32-beam LiDAR frame with snow, as it arrives from a sensor
        _case("lidar_96413", "stream", "lidar", 96413, 24),
        # the dense scan of the benchmark, device to device
        _case("scan_560000", "stream", "scan", 560000, 32),
        # the same kind of scan from and to a program's pinned host buffers
        _case("scan_host_410027", "host", "scan", 410027, 32),
        # a dense 128-beam street frame of a serving program
        _case("street_1111111", "stream", "street", 1111111, 24),
        # 64 LiDAR frames as one batch (one CUDA graph), offline processing of a drive
        _case("lidar_batch_64", "batch", "lidar", 6080000, 24, capacity=256, frames=64),
        # one calibration step on a labelled frame: soft removal, loss, gradients
        _case("train_560000", "train", "scan", 560000, 32),
        # neighbours searched across leaf borders
        _case("cross_leaf_560000", "cross", "scan", 560000, 32),
        # PSNR and Chamfer distance of a denoised scan against its clean points
        _case("metrics_500000", "metrics", "scan", 500000, 1),
        # the comparison method of Sec. 2.2 on a scan in millimetres
        _case("baseline_560000", "baseline", "scan", 560000, 1, scale=1000.0),
        # "without octree" (Table 8): the whole object is one leaf
        _case("one_leaf_36750", "sync", "object", 36750, 16, capacity=ONE_LEAF),
    ]


def draw(rng: random.Random):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["object", "lidar", "scan", "host", "street", "batch", "train", "cross", "metrics", "baseline",
                       "one_leaf"])
    caps = [64, 100, 128, 256, 512, 512, 1000, 2048]
    if kind == "object":
        return _case(None, rng.choice(["sync", "stream"]), "object", size(300, 60000), rng.choice([8, 12, 16, 24, 64]),
                     rng.choice(caps), rescore=rng.choice([0, 0, 1]))
    if kind == "lidar":
        return _case(None, rng.choice(["sync", "stream"]), "lidar", size(20000, 130000), rng.choice([12, 16, 24, 32]),
                     rng.choice(caps))
    if kind == "scan":
        return _case(None, "stream", "scan", size(60000, 560000), rng.choice([12, 16, 24, 32, 48, 64]),
                     rng.choice(caps), rescore=rng.choice([0, 0, 1]))
    if kind == "host":
        return _case(None, "host", rng.choice(["object", "scan", "lidar"]), size(2000, 560000) if rng.random() < 0.7
                     else size(2000, 60000), rng.choice([12, 24, 32]))
    if kind == "street":
        return _case(None, "stream", "street", size(300000, 1111111), rng.choice([16, 24, 32]), rng.choice([256, 512]))
    if kind == "batch":
        f = size(2, 64)
        return _case(None, "batch", "lidar", f * size(60000, 95000), rng.choice([12, 24]), rng.choice([128, 256, 512]),
                     frames=f)
    if kind == "train":
        return _case(None, "train", rng.choice(["scan", "lidar"]), size(30000, 560000), rng.choice([12, 16, 32]))
    if kind == "cross":
        return _case(None, "cross", "scan", size(20000, 560000), rng.choice([12, 16, 24, 32]), rng.choice([128, 256, 512]))
    if kind == "metrics":
        return _case(None, "metrics", rng.choice(["object", "scan", "lidar"]), size(2000, 500000), 1)
    if kind == "baseline":
        return _case(None, "baseline", rng.choice(["object", "scan"]), size(3000, 560000), 1,
                     scale=rng.choice([1.0, 30.0, 150.0, 1000.0]))
    return _case(None, "sync", "object", size(1000, 36750), rng.choice([8, 12, 16, 32]), ONE_LEAF)


# ---------------------------------------------------------------------------
# clouds
# ---------------------------------------------------------------------------
class _Rand:
    """Seeded uniform and normal draws on the GPU."""

    def __init__(self, seed):
        self.dev = torch.device("cuda")
        self.g = torch.Generator(device=self.dev).manual_seed(int(seed) & 0x7FFFFFFFFFFF)
        self.host = random.Random(int(seed) * 7919 + 1)

    def uniform(self, *shape, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(*shape, generator=self.g, device=self.dev, dtype=torch.float64)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device=self.dev, dtype=torch.float64)

    def box(self, lo, hi, count, scale=1.2):
        c, half = 0.5 * (lo + hi), 0.5 * (hi - lo) * scale
        return c + half * self.uniform(count, 3, lo=-1.0, hi=1.0)


def _finish(r: _Rand, parts):
    """(xyz float32 [n, 3], noise labels float32 [n]) of (points, label) parts, shuffled."""
    xyz = torch.cat([p for p, _ in parts]).float()
    lab = torch.cat([torch.full((len(p),), float(v), device=r.dev) for p, v in parts])
    perm = torch.randperm(len(xyz), generator=r.g, device=r.dev)
    return xyz[perm].contiguous(), lab[perm].contiguous()


def _object(r: _Rand, n):
    """Unit sphere with an attached torus, jitter 0.005, 5 % uniform outliers."""
    n_out = max(1, int(round(n * 0.05 / 1.05)))
    surf = n - n_out
    big, small, zc = 0.6, 0.15, 0.8
    a_sph, a_tor = 4 * math.pi, 4 * math.pi ** 2 * big * small
    n_sph = int(round(surf * a_sph / (a_sph + a_tor)))
    v = r.normal(n_sph, 3)
    sph = v / v.norm(dim=1, keepdim=True)
    m = surf - n_sph
    th = r.uniform(4 * m + 64, hi=2 * math.pi)
    keep = r.uniform(len(th)) < (big + small * torch.cos(th)) / (big + small)
    order = torch.argsort((~keep).to(torch.int8), stable=True)
    th = th[order][:m]
    ph = r.uniform(m, hi=2 * math.pi)
    ring = big + small * torch.cos(th)
    tor = torch.stack([ring * torch.cos(ph), ring * torch.sin(ph), zc + small * torch.sin(th)], 1)
    pts = torch.cat([sph, tor])
    pts = pts + 0.005 * r.normal(len(pts), 3)
    out = r.box(pts.amin(0), pts.amax(0), n_out)
    return _finish(r, [(pts, 0), (out, 1)])


def _scan(r: _Rand, n):
    """Eight random superquadrics, 0.5 % jitter, 10 % outliers, 2 % in 20 Gaussian blobs."""
    n_out, per = int(round(n * 0.10 / 1.12)), int(round(n * 0.02 / 1.12)) // 20
    surf = n - n_out - 20 * per

    def spow(v, e):
        return torch.sign(v) * v.abs() ** e

    def points(eta, om, ax, e1, e2):
        ce, se, co, so = torch.cos(eta), torch.sin(eta), torch.cos(om), torch.sin(om)
        return torch.stack([ax[0] * spow(ce, e1) * spow(co, e2), ax[1] * spow(ce, e1) * spow(so, e2),
                            ax[2] * spow(se, e1)], -1)

    shapes = []
    eta = torch.linspace(-math.pi / 2, math.pi / 2, 129, device=r.dev, dtype=torch.float64)
    om = torch.linspace(-math.pi, math.pi, 257, device=r.dev, dtype=torch.float64)
    grid_e, grid_o = torch.meshgrid(eta, om, indexing="ij")
    for _ in range(8):
        h = r.host
        size, ratios = h.uniform(0.1, 1.0), [h.uniform(0.5, 1.0) for _ in range(3)]
        ax = [0.5 * size * q / max(ratios) for q in ratios]
        e1, e2 = h.uniform(0.3, 1.5), h.uniform(0.3, 1.5)
        rot = torch.linalg.qr(r.normal(3, 3).cpu())[0].to(r.dev)
        centre = r.uniform(3, lo=-1.0, hi=1.0)
        p = points(grid_e, grid_o, ax, e1, e2)
        area = torch.linalg.cross(p[1:, :-1] - p[:-1, :-1], p[:-1, 1:] - p[:-1, :-1]).norm(dim=-1)
        shapes.append((ax, e1, e2, rot, centre, area))
    tot = [float(s[5].sum()) for s in shapes]
    counts = [int(surf * t / sum(tot)) for t in tot]
    counts[0] += surf - sum(counts)
    parts = []
    for (ax, e1, e2, rot, centre, area), cnt in zip(shapes, counts):
        cum = torch.cumsum(area.flatten(), 0)
        cell = torch.searchsorted(cum, r.uniform(cnt) * cum[-1]).clamp_(max=area.numel() - 1)
        i, j = cell // area.shape[1], cell % area.shape[1]
        e = eta[i] + r.uniform(cnt) * (eta[1] - eta[0])
        o = om[j] + r.uniform(cnt) * (om[1] - om[0])
        parts.append(points(e, o, ax, e1, e2) @ rot.T + centre)
    pts = torch.cat(parts)
    lo, hi = pts.amin(0), pts.amax(0)
    pts = pts + 0.005 * float((hi - lo).norm()) * r.normal(len(pts), 3)
    out = r.box(lo, hi, n_out)
    centres = lo + (hi - lo) * r.uniform(20, 3)
    blob = (centres[:, None, :] + 0.01 * r.normal(20, per, 3)).reshape(-1, 3)
    return _finish(r, [(pts, 0), (out, 1), (blob, 1)])


def _lidar(r: _Rand, n, beams):
    """A spinning sensor among boxes and poles on a ground plane; as many sweeps as the
    size needs.  32 beams: 12 % near-range snow; 128 beams: 10 % uniform outliers."""
    h, dev = r.host, r.dev
    sensor, max_range = 1.8, 80.0
    n_noise = int(round(n * (0.12 if beams == 32 else 0.10)))
    need = n - n_noise
    nb, nc = h.randint(10, 30), h.randint(20, 60)
    rb, ab, yaw = r.uniform(nb, lo=5, hi=60), r.uniform(nb, hi=2 * math.pi), r.uniform(nb, hi=math.pi)
    dims = torch.tensor([4.5, 1.8, 1.5], device=dev, dtype=torch.float64) * r.uniform(nb, 3, lo=0.9, hi=1.1)
    bx, by = rb * torch.cos(ab), rb * torch.sin(ab)
    rc, ac = r.uniform(nc, lo=3, hi=70), r.uniform(nc, hi=2 * math.pi)
    px, py = rc * torch.cos(ac), rc * torch.sin(ac)
    prad, ph = r.uniform(nc, lo=0.1, hi=0.3), r.uniform(nc, lo=3, hi=8)
    el = torch.deg2rad(torch.linspace(-25, 15, beams, device=dev, dtype=torch.float64))
    base_az = torch.arange(1800, device=dev, dtype=torch.float64) * 0.2

    def sweep(phase):
        az = torch.deg2rad(base_az + phase)
        e, a = torch.meshgrid(el, az, indexing="ij")
        d = torch.stack([torch.cos(e) * torch.cos(a), torch.cos(e) * torch.sin(a), torch.sin(e)], -1).reshape(-1, 3)
        inf = torch.full_like(d[:, 0], math.inf)
        t = torch.where(d[:, 2] < 0, -sensor / d[:, 2], inf)
        cy, sy = torch.cos(yaw), torch.sin(yaw)
        ox, oy = -(cy * bx + sy * by), sy * bx - cy * by
        dx = d[:, :1] * cy + d[:, 1:2] * sy
        dy = d[:, 1:2] * cy - d[:, :1] * sy
        dz = d[:, 2:3].expand_as(dx)
        t1, t2 = (-dims[:, 0] / 2 - ox) / dx, (dims[:, 0] / 2 - ox) / dx
        u1, u2 = (-dims[:, 1] / 2 - oy) / dy, (dims[:, 1] / 2 - oy) / dy
        v1, v2 = -sensor / dz, (dims[:, 2] - sensor) / dz
        near = torch.maximum(torch.maximum(torch.minimum(t1, t2), torch.minimum(u1, u2)), torch.minimum(v1, v2))
        far = torch.minimum(torch.minimum(torch.maximum(t1, t2), torch.maximum(u1, u2)), torch.maximum(v1, v2))
        t = torch.minimum(t, torch.where((far >= near) & (near > 0), near, math.inf).amin(1))
        aa = d[:, :1] ** 2 + d[:, 1:2] ** 2
        bb = -2 * (d[:, :1] * px + d[:, 1:2] * py)
        disc = bb * bb - 4 * aa * (px ** 2 + py ** 2 - prad ** 2)
        tc = (-bb - disc.clamp(min=0).sqrt()) / (2 * aa)
        zc = sensor + tc * d[:, 2:3]
        ok = (disc > 0) & (tc > 0) & (zc >= 0) & (zc <= ph)
        t = torch.minimum(t, torch.where(ok, tc, math.inf).amin(1))
        hit = t <= max_range
        d, t = d[hit], t[hit]
        p = d * (t + 0.02 * r.normal(len(t)))[:, None]
        p[:, 2] += sensor
        return p

    surf = [sweep(0.0)]
    s = 1
    while sum(len(p) for p in surf) < need:  # further sweeps at phases between the columns
        surf.append(sweep(0.2 * ((s * 0.6180339887) % 1.0)))
        s += 1
    surf = torch.cat(surf)
    surf = surf[torch.randperm(len(surf), generator=r.g, device=dev)[:need]]
    if beams == 32:
        m = 2 * n_noise + 64
        rad = (0.25 + (225 - 0.25) * r.uniform(m)).sqrt()
        az = r.uniform(m, hi=2 * math.pi)
        sel = r.uniform(m, lo=math.sin(math.radians(-25)), hi=math.sin(math.radians(15)))
        cel = (1 - sel ** 2).sqrt()
        p = torch.stack([rad * cel * torch.cos(az), rad * cel * torch.sin(az), (sensor + rad * sel).abs()], 1)
        noise = p[:n_noise]
    else:
        noise = r.box(surf.amin(0), surf.amax(0), n_noise)
    return _finish(r, [(surf, 0), (noise, 1)])


def _cloud(kind, seed, n):
    r = _Rand(seed)
    if kind == "object":
        return _object(r, n)
    if kind == "scan":
        return _scan(r, n)
    return _lidar(r, n, 32 if kind == "lidar" else 128)


def _offsets(case, seed):
    """Frame offsets of a batch: sizes within about a third of their mean."""
    f, n = case["frames"], case["n"]
    rng = random.Random(seed * 31 + 5)
    w = [rng.uniform(0.66, 1.34) for _ in range(f)]
    offs = [0]
    for i in range(f):
        offs.append(n if i == f - 1 else offs[-1] + int(n * w[i] / sum(w)))
    return offs


def _inputs(case, seed):
    """(xyz, noise labels, frame offsets) of a case."""
    if case["kind"] == "batch":
        offs = _offsets(case, seed)
        parts = [_cloud(case["cloud"], seed * 1009 + f, offs[f + 1] - offs[f]) for f in range(case["frames"])]
        return torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts]), offs
    xyz, lab = _cloud(case["cloud"], seed * 1009, case["n"])
    if case["scale"] != 1.0:
        xyz = xyz * case["scale"]
    return xyz, lab, [0, case["n"]]


def _pair(case, seed):
    """A clean cloud and a denoised one: 97 % of its points with the sensor's jitter (0.1 % of
    the extent) and as many left-over noise points as 5 % of it."""
    xyz, _, _ = _inputs(case, seed)
    r = _Rand(seed + 77)
    lo, hi = xyz.amin(0).double(), xyz.amax(0).double()
    kept = xyz[torch.randperm(len(xyz), generator=r.g, device=r.dev)[:int(0.97 * len(xyz))]].double()
    kept = kept + 0.001 * float((hi - lo).norm()) * r.normal(len(kept), 3)
    return xyz, torch.cat([kept, r.box(lo, hi, max(1, len(xyz) // 20))]).float().contiguous()


def _params(case):
    return Params(k=case["k"], leaf_capacity=case["capacity"], rescore_p2=case["rescore"],
                  cross_leaf=int(case["kind"] == "cross"), temperature=0.5 if case["kind"] == "train" else 0.05)


def _theta(case):
    """alpha, sigma, gamma, tau of the calibration step: tau near the lower tenth of the log scores."""
    return 1.0, 1.0, 2.0, round(math.log(case["n"]) - (2.0 if case["cloud"] == "scan" else 5.0), 2)


# ---------------------------------------------------------------------------
# what is timed
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "metrics":
        clean, den = _pair(case, seed)
        return {"case": case, "d": Denoiser(max_points=max(len(clean), len(den))), "clean": clean, "denoised": den}
    xyz, lab, offs = _inputs(case, seed)
    d = Denoiser(max_points=case["n"], max_frames=case["frames"])
    st = {"case": case, "d": d, "params": _params(case), "xyz": xyz}
    if kind == "stream":
        d.set_sync(False)
    elif kind == "host":
        st["xyz"] = xyz.cpu().pin_memory()
        st["out"] = {"mask": torch.empty(case["n"], dtype=torch.uint8, pin_memory=True),
                     "score": torch.empty(case["n"], dtype=torch.float32, pin_memory=True),
                     "stage": torch.empty(case["n"], dtype=torch.uint8, pin_memory=True)}
    elif kind == "batch":
        d.set_sync(False)
        d.set_graphs(True)
        st["offsets"] = offs
        st["out"] = {"mask": torch.empty(case["n"], dtype=torch.uint8, device="cuda"),
                     "score": torch.empty(case["n"], dtype=torch.float32, device="cuda"),
                     "stage": torch.empty(case["n"], dtype=torch.uint8, device="cuda")}
    elif kind == "train":
        d.set_training(True)
        st["noise"] = lab
        st["theta"] = _theta(case)
    elif kind == "cross":
        d.set_cross_leaf(True)
        d.set_sync(False)
    torch.cuda.synchronize()
    return st


def run(state):
    kind, d = state["case"]["kind"], state["d"]
    if kind == "metrics":
        return d.eval_metrics(state["clean"], state["denoised"], per_point=True)
    if kind == "baseline":
        return d.run_baseline(state["xyz"], counts=True)
    if kind == "train":
        theta = torch.tensor(state["theta"], dtype=torch.float64, requires_grad=True)
        removal = SoftRemoval.apply(state["xyz"], theta, d, state["params"])
        loss = soft_f1_loss(removal, state["noise"])
        loss.backward()
        return removal.detach(), loss.detach(), theta.grad
    if kind == "batch":
        r = d.run_batch(state["xyz"], state["offsets"], state["params"], **state["out"])
    else:
        r = d.run(state["xyz"], state["params"], **state.get("out", {}))
    return r.mask, r.score, r.stage


def work(case):
    n, k, kind = case["n"], case["k"], case["kind"]
    if kind == "metrics":  # both clouds in, a nearest distance per point out
        m = n + int(n * 0.97) + max(1, n // 20)
        return {"bytes": 16 * m, "flops": 8 * m}
    if kind == "baseline":  # points in, keep flag and count out
        return {"bytes": 17 * n, "flops": 30 * n}
    per = 20 * k  # a distance (8) and a score term (12) per neighbour
    if kind == "train":  # points and labels in, removal probabilities and their gradient out
        return {"bytes": (12 + 4 + 4 + 4) * n, "flops": n * (per + 40 * k)}
    return {"bytes": (12 + 6) * n, "flops": n * per}


# ---------------------------------------------------------------------------
# the same values in 64 bits (plain torch; the decisions that the method takes on
# FP32 values -- cells, voxels, the order of distances -- are taken on FP32 here too)
# ---------------------------------------------------------------------------
def exact(case, seed):
    if case["kind"] == "metrics":
        return _exact_metrics(*_pair(case, seed))
    xyz, lab, offs = _inputs(case, seed)
    if case["kind"] == "baseline":
        return _exact_baseline(xyz)
    p = _params(case)
    score = torch.zeros(len(xyz), dtype=torch.float64, device=xyz.device)
    terms = []
    for f in range(case["frames"]):
        a, b = offs[f], offs[f + 1]
        frame = _Frame(xyz[a:b], p)
        frame.solve(terms if case["kind"] == "train" else None)
        score[a:b] = frame.score
    if case["kind"] != "train":
        return None, score, None
    return _exact_train(terms, lab, p, _theta(case))


def _exact_metrics(clean, den):
    a, b = clean.double(), den.double()
    nn_a = torch.full((len(a),), math.inf, dtype=torch.float64, device=a.device)
    nn_b = torch.full((len(b),), math.inf, dtype=torch.float64, device=a.device)
    step = max(1, (1 << 28) // len(b))
    bt = b.T.contiguous()
    for s in range(0, len(a), step):
        q = a[s:s + step]
        d2 = (q[:, :1] - bt[0]).square_()
        for c in (1, 2):
            t = q[:, c:c + 1] - bt[c]
            d2.addcmul_(t, t)
        nn_a[s:s + step] = d2.amin(1)
        nn_b = torch.minimum(nn_b, d2.amin(0))
    mse = float(nn_a.mean())
    m2 = float(((a.amax(0) - a.amin(0)) ** 2).sum())
    return {"mse": mse, "chamfer": mse + float(nn_b.mean()), "psnr": 10 * math.log10(m2 / mse) if mse else math.inf,
            "nn_clean": nn_a, "nn_denoised": nn_b}


def _exact_baseline(xyz):
    p = xyz.double()
    h = (p.amax(0) - p.amin(0)).tolist()
    n = len(xyz)
    return {"keep": None, "theta": p.mean(0).tolist(), "R": 6 * (h[0] * h[1] + h[0] * h[2] + h[1] * h[2]) / n,
            "T": 600.0 * 6.67e-11 * sum(h) / n, "n_i": None}


def _exact_train(terms, lab, p, theta0):
    """Soft removal, loss and gradient: autograd over the scored points' neighbour terms."""
    theta = torch.tensor(theta0, dtype=torch.float64, device=lab.device, requires_grad=True)
    alpha, sigma, gamma, tau = theta
    removal = torch.ones(len(lab), dtype=torch.float64, device=lab.device)
    parts, index = [], []
    for idx, valid, d2, lw, r2 in terms:
        dist = d2 ** (gamma / 2) if bool((d2 > 0).all()) else torch.where(
            d2 > 0, d2.clamp(min=1e-300) ** (gamma / 2), torch.zeros_like(d2))
        t = torch.exp(0.5 * alpha * lw - d2 / (2 * sigma ** 2 * r2[:, None])) / (dist + p.eps_k)
        f = torch.where(valid, t, torch.zeros_like(t)).sum(1)
        parts.append(1 - torch.sigmoid((torch.log(f) - tau) / p.temperature))
        index.append(idx)
    removal = removal.index_put((torch.cat(index),), torch.cat(parts))
    y = lab.double()
    loss = 1 - 2 * (removal * y).sum() / (removal.sum() + y.sum())
    loss.backward()
    return removal.detach(), loss.detach().cpu(), theta.grad.cpu()


def _round_d2(dx, dy, dz):
    """FP32 squared distance fma(dz, dz, fma(dy, dy, dx * dx)) of FP32 differences."""
    s = (dx * dx).double()
    dy, dz = dy.double(), dz.double()
    s = (s + dy * dy).float().double()
    return (s + dz * dz).float()


class _Frame:
    """The method on one frame (Sec. 3): octree leaves, voxel gate, kNN, density gate, score."""

    def __init__(self, xyz, p):
        self.p, self.dev, self.n = p, xyz.device, len(xyz)
        self.score = torch.zeros(self.n, dtype=torch.float64, device=self.dev)
        lo = xyz.amin(0)
        side = float((xyz.amax(0) - lo).max())
        side = side if side > 0 else 1.0
        side32 = torch.tensor(side, dtype=torch.float32, device=self.dev)
        self.delta = side32 * torch.tensor(2.0 ** -21, dtype=torch.float32, device=self.dev)
        s = torch.tensor(2097152.0, dtype=torch.float32, device=self.dev) / side32
        q = ((xyz - lo) * s).floor().clamp(max=2097151.0).long()
        key = torch.zeros(self.n, dtype=torch.int64, device=self.dev)
        for b in range(21):
            for c in range(3):
                key |= ((q[:, c] >> b) & 1) << (3 * b + 2 - c)
        self.key, self.order = torch.sort(key, stable=True)
        self.xyz = xyz[self.order]
        self.partition()
        self.voxel_gate()

    def partition(self):
        """leaf[i] of the sorted points; starts, counts, levels of the leaves."""
        n, cap, depth = self.n, self.p.leaf_capacity, self.p.max_depth
        level = torch.full((n,), -1, dtype=torch.int64, device=self.dev)
        for lv in range(depth + 1):
            pre = self.key >> (63 - 3 * lv) if lv else torch.zeros_like(self.key)
            _, inv, cnt = torch.unique_consecutive(pre, return_inverse=True, return_counts=True)
            small = (cnt <= cap) | (lv == depth)
            level = torch.where((level < 0) & small[inv], lv, level)
            if bool((level >= 0).all()):
                break
        pre = (self.key >> (63 - 3 * level).clamp(max=62)) * (level > 0)
        new = torch.ones(n, dtype=torch.bool, device=self.dev)
        new[1:] = (pre[1:] != pre[:-1]) | (level[1:] != level[:-1])
        self.leaf = torch.cumsum(new, 0) - 1
        self.start = torch.nonzero(new).flatten()
        self.count = torch.diff(self.start, append=torch.tensor([n], device=self.dev))
        self.level = level[self.start]

    def voxel_gate(self):
        nl, lf = len(self.start), self.leaf[:, None].expand(-1, 3)
        lo = torch.full((nl, 3), math.inf, device=self.dev).scatter_reduce(0, lf, self.xyz, "amin")
        hi = torch.full((nl, 3), -math.inf, device=self.dev).scatter_reduce(0, lf, self.xyz, "amax")
        ext = torch.maximum(hi - lo, self.delta).double()
        u = ext[:, 0] * ext[:, 1] * ext[:, 2] / self.count.double()
        y = u ** (1.0 / 3.0)
        for _ in range(2):
            y = y - (y * y * y - u) / (3 * y * y)
        h = (float(torch.tensor(self.p.beta, dtype=torch.float32)) * y).float()
        v = ((self.xyz - lo[self.leaf]) / h[self.leaf, None]).floor().clamp(max=2097151.0).long()
        cell = (v[:, 0] << 42) | (v[:, 1] << 21) | v[:, 2]
        order = torch.argsort(cell, stable=True)
        order = order[torch.argsort(self.leaf[order], stable=True)]
        c, lfs = cell[order], self.leaf[order]
        new = torch.ones(self.n, dtype=torch.bool, device=self.dev)
        new[1:] = (c[1:] != c[:-1]) | (lfs[1:] != lfs[:-1])
        run_id = torch.cumsum(new, 0) - 1
        occ = torch.empty(self.n, dtype=torch.int64, device=self.dev)
        occ[order] = torch.bincount(run_id)[run_id]
        self.in1 = occ >= self.p.min_vox_count

    def solve(self, terms):
        """Scores (input order); with `terms` also every scored point's neighbour terms."""
        members = torch.nonzero(self.in1).flatten()  # sorted positions of P_1
        if self.p.cross_leaf:
            nbr, d2, keff = self.cross_knn(members)
        else:
            nbr, d2, keff = self.leaf_knn(members)
        alive = self.gate(members, d2, keff)
        if self.p.rescore_p2:
            members = members[alive]
            nbr, d2, keff = self.leaf_knn(members)
            alive = torch.ones(len(members), dtype=torch.bool, device=self.dev)
        self.weigh(members, nbr, d2, keff, alive, terms)

    def leaf_knn(self, members):
        """Neighbours (indices into `members`), FP32 d^2 and k_eff of every member within its leaf."""
        k, m = self.p.k, len(members)
        nbr = torch.zeros((m, k), dtype=torch.int64, device=self.dev)
        d2 = torch.full((m, k), math.inf, device=self.dev)
        leaf = self.leaf[members]
        uniq, cnt = torch.unique_consecutive(leaf, return_counts=True)
        first = torch.cumsum(cnt, 0) - cnt
        keff = torch.clamp(torch.repeat_interleave(cnt, cnt) - 1, max=k)
        pts, gid = self.xyz[members], self.order[members]
        size = 2
        while bool((cnt > size // 2).any()):
            sel = torch.nonzero((cnt > size // 2) & (cnt <= size)).flatten()
            width = int(cnt[sel].max()) if len(sel) else 0
            rows = max(1, (1 << 25) // max(1, width * width)) if width * width <= (1 << 25) else 1
            for s in range(0, len(sel), rows):
                g = sel[s:s + rows]
                col = torch.arange(width, device=self.dev)
                pos = (first[g][:, None] + col).clamp(max=m - 1)
                ok = col < cnt[g][:, None]
                qstep = width if rows > 1 or width * width <= (1 << 25) else max(1, (1 << 25) // width)
                for q0 in range(0, width, qstep):
                    qp, qok = pos[:, q0:q0 + qstep], ok[:, q0:q0 + qstep]
                    diff = pts[pos][:, None, :, :] - pts[qp][:, :, None, :]
                    dd = _round_d2(diff[..., 0], diff[..., 1], diff[..., 2])
                    key = (dd.view(torch.int32).long() << 32) | gid[pos][:, None, :]
                    bad = ~ok[:, None, :] | (pos[:, None, :] == qp[:, :, None])
                    key = torch.where(bad, torch.iinfo(torch.int64).max, key)
                    kk = min(k, width)
                    val, loc = torch.topk(key, kk, dim=-1, largest=False)
                    found = torch.gather(pos[:, None, :].expand(-1, qp.shape[1], -1), 2, loc)
                    rows_q = qp[qok]
                    nbr[rows_q, :kk] = found[qok]
                    dist = (val >> 32).int().view(torch.float32)
                    d2[rows_q, :kk] = torch.where(val == torch.iinfo(torch.int64).max, math.inf, dist)[qok]
            size *= 2
        return nbr, d2, keff

    def cross_knn(self, members):
        """The same over the 27 same-level cells around each leaf."""
        k, m = self.p.k, len(members)
        nbr = torch.zeros((m, k), dtype=torch.int64, device=self.dev)
        d2 = torch.full((m, k), math.inf, device=self.dev)
        keff = torch.zeros(m, dtype=torch.int64, device=self.dev)
        pts, gid, keys = self.xyz[members], self.order[members], self.key[members]
        leaf = self.leaf[members]
        uniq, cnt = torch.unique_consecutive(leaf, return_counts=True)
        first = torch.cumsum(cnt, 0) - cnt
        # cells of all leaves at once: [leaves, 27] ranges of the members
        lv = self.level[uniq]
        k0 = self.key[self.start[uniq]]
        axes = []
        for c in range(3):
            q = torch.zeros_like(k0)
            for b in range(21):
                q |= ((k0 >> (3 * b + 2 - c)) & 1) << b
            axes.append(q >> (21 - lv))
        off = torch.tensor([(i, j, l) for i in (-1, 0, 1) for j in (-1, 0, 1) for l in (-1, 0, 1)], device=self.dev)
        cell = torch.stack(axes, 1)[:, None, :] + off
        ok = ((cell >= 0) & (cell < (1 << lv)[:, None, None])).all(2)
        pre = torch.zeros(ok.shape, dtype=torch.int64, device=self.dev)
        for b in range(21):
            for c in range(3):
                pre |= ((cell[..., c].clamp(min=0) >> b) & 1) << (3 * b + 2 - c)
        sh = (3 * (21 - lv))[:, None]
        # prefixes of at most 62 bits after the shift (the last cell's end is past every key)
        a = torch.searchsorted(keys, torch.where(lv[:, None] > 0, pre << sh.clamp(max=62), 0))
        end = torch.where(lv[:, None] > 0, (pre << sh.clamp(max=62)) + ((1 << sh.clamp(max=62)) - 1),
                          torch.iinfo(torch.int64).max)
        b = torch.searchsorted(keys, end, right=True)
        a, b = torch.where(ok, a, 0).tolist(), torch.where(ok, b, 0).tolist()
        first, cnt, lvl = first.tolist(), cnt.tolist(), lv.tolist()
        for li in range(len(cnt)):
            rng = [(0, m)] if lvl[li] == 0 else [(x, y) for x, y in zip(a[li], b[li]) if y > x]
            cand = torch.cat([torch.arange(x, y, device=self.dev) for x, y in rng])
            ke = min(k, len(cand) - 1)
            q_all = torch.arange(first[li], first[li] + cnt[li], device=self.dev)
            keff[q_all] = max(0, ke)
            if ke < 1:
                continue
            step = max(1, (1 << 26) // len(cand))
            for q0 in range(0, len(q_all), step):
                q = q_all[q0:q0 + step]
                diff = pts[cand][None] - pts[q][:, None]
                dd = _round_d2(diff[..., 0], diff[..., 1], diff[..., 2])
                key = (dd.view(torch.int32).long() << 32) | gid[cand][None]
                key = torch.where(cand[None] == q[:, None], torch.iinfo(torch.int64).max, key)
                val, loc = torch.topk(key, ke, dim=-1, largest=False)
                nbr[q, :ke] = cand[loc]
                d2[q, :ke] = (val >> 32).int().view(torch.float32)
        return nbr, d2, keff

    def kth(self, d2, keff):
        """The floored FP32 k_eff-th squared distance."""
        last = d2.gather(1, (keff - 1).clamp(min=0)[:, None])[:, 0]
        return torch.maximum(last, self.delta * self.delta)

    def gate(self, members, d2, keff):
        """Eq. 14 per leaf, as a rank cut on the FP32 r_K^2; a point without neighbours fails."""
        r2 = self.kth(d2, keff)
        leaf = self.leaf[members]
        _, inv, cnt = torch.unique_consecutive(leaf, return_inverse=True, return_counts=True)
        order = torch.argsort(r2, stable=True)
        order = order[torch.argsort(inv[order], stable=True)]
        first = torch.cumsum(cnt, 0) - cnt
        q = float(torch.tensor(self.p.rho_percentile, dtype=torch.float32))
        c = torch.ceil(cnt.double() * q / 100.0 + 0.5).long().clamp(min=1)
        c = torch.minimum(c, cnt)
        cut = r2[order[first + cnt - c]]
        return (r2 <= cut[inv]) & (keff > 0)

    def weigh(self, members, nbr, d2f, keff, alive, terms):
        """Eq. 16-21 in FP64 for the members that are alive."""
        p, leaf = self.p, self.leaf[members]
        if not len(members):
            return
        pts = self.xyz[members].double()
        fl = (self.delta * self.delta).double()
        k = min(p.k, nbr.shape[1])
        col = torch.arange(k, device=self.dev)
        valid = col < keff[:, None]
        rows = (1 << 25) // k
        d2 = torch.empty(nbr.shape, dtype=torch.float64, device=self.dev)
        for s in range(0, len(members), rows):
            d2[s:s + rows] = (pts[nbr[s:s + rows]] - pts[s:s + rows, None]).square().sum(2)
        r2 = torch.maximum(torch.where(valid, d2, 0.0).amax(1), fl)
        rho = keff.double() / (4.0 / 3.0 * math.pi * r2 * r2.sqrt())
        # median of each leaf's alive points
        _, inv = torch.unique_consecutive(leaf, return_inverse=True)
        nl = int(inv.max()) + 1
        ai = torch.nonzero(alive).flatten()
        if not len(ai):
            return
        order = ai[torch.argsort(rho[ai], stable=True)]
        order = order[torch.argsort(inv[order], stable=True)]
        cnt = torch.bincount(inv[ai], minlength=nl)
        first = torch.cumsum(cnt, 0) - cnt
        sorted_rho = rho[order]
        has = cnt > 0
        lo_i = (first + (cnt - 1).clamp(min=0) // 2).clamp(max=len(order) - 1)
        hi_i = (first + cnt // 2).clamp(max=len(order) - 1)
        med = torch.where(has, 0.5 * (sorted_rho[lo_i] + sorted_rho[hi_i]), 1.0)
        ref = (med * med + p.eps_rho).sqrt()
        out = torch.zeros(len(members), dtype=torch.float64, device=self.dev)
        for s in range(0, len(ai), rows):
            i = ai[s:s + rows]
            lw = torch.log(rho[nbr[i]] / ref[inv[i]][:, None]) + torch.log(rho[i] / ref[inv[i]])[:, None]
            di, ok = d2[i], valid[i]
            t = torch.exp(0.5 * p.alpha * lw - di / (2 * p.sigma ** 2 * r2[i])[:, None]) / (di ** (p.gamma / 2) + p.eps_k)
            out[i] = torch.where(ok, t, 0.0).sum(1)
            if terms is not None:
                terms.append((self.order[members[i]], ok, torch.where(ok, di, 1.0), torch.where(ok, lw, 0.0), r2[i]))
        self.score[self.order[members]] = out
