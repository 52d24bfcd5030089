"""The workloads whose speed is measured: what users of the library have it do, each through a public call.

Inputs are synthetic and made on the GPU from the seed: depth images of a procedural scene (a ground plane, a
far wall, 20 spheres and boxes, 5 mm of depth noise, dropped pixels; one or several posed frames, with an
intensity channel for the 4D calls) and clouds drawn from random mixtures.  Models that a program holds before
the call (for scoring, registration, refinement, resampling) have the moments of a partition of such a scan.
`exact` computes the same outputs in 64 bits with plain torch and numpy; the k-means decisions, which are
defined in binary32 and exact integers, are taken as they are defined.
"""
import math
import random

import numpy as np
import torch

from paper_2307_00071_gb300 import autograd, gira

DEV = "cuda"
REG = 1e-4      # metres^2 on every covariance diagonal: (1 cm)^2, above the sensor's noise, so that thousands of
                # components on 5 mm surfaces stay well conditioned over the iterations
MODES = 8192    # room in the table of modes (the fits' largest K)
LLOYD = 10      # Lloyd iterations of KInit: the fits' default


def listed():
    return [
        # Twelve uses, from a control loop's single score (tens of microseconds) to a refined map.
        # A tracker scores a small thinned scan against a small local model in a loop that may not allocate.
        {"name": "score_control_loop", "kind": "score_noalloc", "n": 2053, "k": 64},
        # One object's cloud: the whole fit at the smallest size a user would fit.
        {"name": "fit_small_cloud", "kind": "fit_cloud", "n": 20000, "k": 8, "iters": 20, "tol": 0.0},
        # One 640x480 depth frame, the whole fit: the headline workload.
        {"name": "fit_frame", "kind": "fit_frame", "n": 276348, "k": 512, "iters": 30, "tol": 1e-4},
        # The same frame with intensity (4D): the paper's model of a frame.
        {"name": "fit_frame_intensity", "kind": "fit_frame4", "n": 276348, "k": 512, "iters": 12, "tol": 1e-4},
        # Many segments of uneven size fitted in one call.
        {"name": "fit_segments_batched", "kind": "fit_batch", "batch": 48, "n_lo": 2000, "n_hi": 200000,
         "k_lo": 16, "k_hi": 512, "sizes": 7, "iters": 12, "tol": 0.0},
        # A map of 16 frames refined from the model of the previous pass: K above 1024.
        {"name": "refine_large_map", "kind": "refine_map", "n": 4000000, "k": 8192, "iters": 2, "tol": 0.0},
        # Seeding for a map of several frames: more points than the one-launch seeding kernels hold.
        {"name": "kmeans_map", "kind": "kmeans", "n": 1000003, "k": 768},
        # Change detection: every point of a new frame scored against a frame's model (odd K, above 1024 too in draws).
        {"name": "score_frame", "kind": "score", "n": 276347, "k": 1023},
        # One training / registration step through autograd: value, and the gradient of every input.
        {"name": "autograd_scan", "kind": "autograd", "n": 100000, "k": 1024, "offset": 0.3},
        # Many registrations advanced together: value and twist of every scan, each with its own model.
        {"name": "register_batched", "kind": "register", "batch": 16, "n_lo": 20000, "n_hi": 100000, "k": 1024,
         "sizes": 3},
        # A 640x480 cloud resampled from the 4D model and its intensity inferred at the sampled positions.
        {"name": "resample_and_infer", "kind": "resample", "n": 307200, "k": 1163},
        # The number of components from a bandwidth (the step before the 4D fit).
        {"name": "modes_frame", "kind": "gbms", "n": 276348, "h": 0.05},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["score_noalloc", "fit_cloud", "fit_frame", "fit_frame4", "fit_batch", "refine_map", "kmeans",
                       "score", "autograd", "register", "resample", "gbms"])
    c = {"kind": kind}
    if kind == "score_noalloc":
        c.update(n=_log_int(rng, 600, 20000), k=_log_int(rng, 8, 256))
    elif kind == "fit_cloud":
        c.update(n=_log_int(rng, 2000, 200000), k=_log_int(rng, 2, 64), iters=20, tol=0.0)
    elif kind == "fit_frame":
        c.update(n=_log_int(rng, 17000, 300000), k=_log_int(rng, 64, 1024), iters=30, tol=1e-4)
    elif kind == "fit_frame4":
        c.update(n=_log_int(rng, 17000, 300000), k=_log_int(rng, 64, 1024), iters=12, tol=1e-4)
    elif kind == "fit_batch":
        c.update(batch=_log_int(rng, 8, 48), n_lo=2000, n_hi=rng.choice([20000, 200000]), k_lo=16,
                 k_hi=rng.choice([128, 512]), sizes=rng.randrange(1000), iters=12, tol=0.0)
    elif kind == "refine_map":
        c.update(n=_log_int(rng, 500000, 4000000), k=_log_int(rng, 1025, 8192), iters=2, tol=0.0)
    elif kind == "kmeans":
        c.update(n=_log_int(rng, 300000, 2000000), k=_log_int(rng, 128, 768))
    elif kind == "score":
        c.update(n=_log_int(rng, 17000, 300000), k=_log_int(rng, 64, 2048))
    elif kind == "autograd":
        c.update(n=_log_int(rng, 5000, 100000), k=_log_int(rng, 64, 1024), offset=round(rng.uniform(0.0, 1.0), 3))
    elif kind == "register":
        c.update(batch=_log_int(rng, 2, 16), n_lo=5000, n_hi=100000, k=_log_int(rng, 64, 1024),
                 sizes=rng.randrange(1000))
    elif kind == "resample":
        c.update(n=_log_int(rng, 17000, 307200), k=_log_int(rng, 100, 1534))
    else:
        c.update(n=_log_int(rng, 30000, 300000), h=round(rng.uniform(0.05, 0.15), 3))
    return c


def _sizes(case):
    """The points (and components) of each instance of a batch, log-uniform, the same for every seed."""
    r = random.Random(case["sizes"])
    ns = [_log_int(r, case["n_lo"], case["n_hi"]) for _ in range(case["batch"])]
    if "k" in case:
        return ns, [case["k"]] * case["batch"]
    ks = [k for k in (16, 32, 64, 128, 256, 512) if case["k_lo"] <= k <= case["k_hi"]]
    return ns, [r.choice(ks) for _ in ns]


# ------------------------------------------------------------------------------------------------ inputs
def _gen(*seed):
    return torch.Generator(DEV).manual_seed(int(np.random.SeedSequence(seed).generate_state(1)[0]))


def _frame(n, scene, gen):
    """n points of a depth image of the scene, in pixel order (camera frame, metres, float64)."""
    w = math.ceil(math.sqrt(n / 0.9 * 4 / 3))
    h = math.ceil(n / 0.9 / w)
    f = 525.0 * w / 640
    r = np.random.default_rng(scene)
    pitch = np.deg2rad(r.uniform(20.0, 30.0))
    c, s = math.cos(pitch), math.sin(pitch)
    pix = torch.arange(w * h, device=DEV)
    cam = torch.stack([(pix % w - (w - 1) / 2) / f, (pix // w - (h - 1) / 2) / f, torch.ones_like(pix)], 1).double()
    rot = torch.tensor([[1.0, 0, 0], [0, -s, c], [0, -c, -s]], dtype=torch.float64, device=DEV)
    d = cam @ rot.T                                     # world directions: x right, y ahead, z up
    o = np.array([0.0, 0.0, 1.5])
    inf = torch.full((w * h,), math.inf, dtype=torch.float64, device=DEV)
    t = torch.where(d[:, 2] < 0, -o[2] / d[:, 2], inf)
    t = torch.minimum(t, torch.where(d[:, 1] > 0, 8.0 / d[:, 1], inf))
    half = math.atan(319.5 / 525.0)
    for j in range(20):
        dist, size = r.uniform(0.5, 8.0), r.uniform(0.2, 1.5)
        side = r.uniform(-1.0, 1.0) * math.tan(half) * dist
        if j % 2:
            oc = torch.tensor(o - [side, dist, size / 2], device=DEV)
            a, b = (d * d).sum(1), d @ oc
            q = b * b - a * (oc @ oc - size * size / 4)
            hit = torch.where(q >= 0, (-b - q.clamp_min(0).sqrt()) / a, inf)
        else:
            box = 0.5 * r.uniform(0.2, 1.5, size=3)
            yaw = r.uniform(0, math.pi)
            rz = np.array([[math.cos(yaw), -math.sin(yaw), 0], [math.sin(yaw), math.cos(yaw), 0], [0, 0, 1.0]])
            ol = torch.tensor(rz.T @ (o - [side, dist, box[2]]), device=DEV)
            dl = d @ torch.tensor(rz, device=DEV)
            box = torch.tensor(box, device=DEV)
            lo, hi = (-box - ol) / dl, (box - ol) / dl
            near, far = torch.minimum(lo, hi).amax(1), torch.maximum(lo, hi).amin(1)
            hit = torch.where((far >= near) & (near > 0), near, inf)
        t = torch.where((hit > 1e-3) & (hit < t), hit, t)
    t = (t + 0.005 * torch.randn(w * h, generator=gen, dtype=torch.float64, device=DEV)).clamp_min(0.05)
    keep = torch.randperm(w * h, generator=gen, device=DEV)[:n].sort().values
    return cam[keep] * t[keep, None]


def _scan(n, seed, d=3, scan=0):
    """n points (float32) of the scene of `seed`: one frame, or several posed ones for a map; `scan` is the sensor's
    noise and dropout.  d = 4 adds intensity, a texture of the position with noise, in [0, 1]."""
    frames = math.ceil(n / 300000)
    r = np.random.default_rng([seed, 17])
    out = []
    for j in range(frames):
        m = n * (j + 1) // frames - n * j // frames
        p = _frame(m, [seed, j], _gen(seed, j, scan))
        if frames > 1:
            yaw, at = r.uniform(0, 2 * math.pi), r.uniform(-10, 10, size=3)
            rot = torch.tensor([[math.cos(yaw), 0, math.sin(yaw)], [0, 1.0, 0], [-math.sin(yaw), 0, math.cos(yaw)]],
                               dtype=torch.float64, device=DEV)
            p = p @ rot.T + torch.tensor(at, device=DEV)
        out.append(p)
    p = torch.cat(out)
    if d == 4:
        x, y, z = p.unbind(1)
        tex = 0.5 + 0.25 * torch.sin(3 * x) * torch.cos(2 * y) + 0.15 * torch.sin(1.3 * z + 0.5 * x) - 0.02 * z
        tex = tex + 0.01 * torch.randn(n, generator=_gen(seed, 99, scan), dtype=torch.float64, device=DEV)
        p = torch.cat([p, tex.clamp(0, 1)[:, None]], 1)
    return p.float().contiguous()


def _model(points, k, seed):
    """(weights, means, covs) float32: the moments of the points' partition by k of their own as centres (64-bit
    integer sums, so the values do not depend on the order of the sums)."""
    n, d = points.shape
    gen = _gen(seed, 5)
    m = min(n, 64 * k)
    sub = points[torch.randperm(n, generator=gen, device=DEV)[:m]].contiguous()
    c = sub[:k].double()
    label = torch.empty(m, dtype=torch.int64, device=DEV)
    for a in range(0, m, 1 << 16):
        x = sub[a:a + (1 << 16)].double()
        label[a:a + (1 << 16)] = ((c * c).sum(1) - 2 * x @ c.T).argmin(1)
    q = ((sub.double() - c[label]) * 2.0 ** 20).round().long()
    cnt = torch.zeros(k, dtype=torch.int64, device=DEV).index_add_(0, label, torch.ones_like(label)).clamp_min(1)
    s1 = torch.zeros(k, d, dtype=torch.int64, device=DEV).index_add_(0, label, q)
    s2 = torch.zeros(k, d, d, dtype=torch.int64, device=DEV).index_add_(0, label, q[:, :, None] * q[:, None, :])
    mean = s1 / cnt[:, None] * 2.0 ** -20
    cov = s2 / cnt[:, None, None] * 2.0 ** -40 - mean[:, :, None] * mean[:, None, :]
    cov = cov + 1e-5 * torch.eye(d, dtype=torch.float64, device=DEV)
    return (cnt / cnt.sum()).float(), (c + mean).float(), cov.float().contiguous()


def _clouds(ns, ks, seed):
    """One cloud per instance, each drawn from its own random 8-component mixture, stacked (float32)."""
    out = []
    for i, n in enumerate(ns):
        r = np.random.default_rng([seed, i])
        mu = r.uniform(-2, 2, size=(8, 3))
        q = np.linalg.qr(r.standard_normal((8, 3, 3)))[0]
        a = q * np.exp(0.5 * r.uniform(np.log(1e-4), np.log(1e-2), size=(8, 1, 3)))
        comp = torch.tensor(r.choice(8, size=n, p=r.dirichlet(np.ones(8))), device=DEV)
        z = torch.randn(n, 3, generator=_gen(seed, i), dtype=torch.float64, device=DEV)
        a, mu = torch.tensor(a, device=DEV), torch.tensor(mu, device=DEV)
        out.append(mu[comp] + (a[comp] @ z[:, :, None])[:, :, 0])
    return torch.cat(out).float().contiguous()


def _pose(r, offset):
    """A rotation (<= 15 degrees) and a translation (<= 0.5 m per axis), scaled by `offset`."""
    axis = r.normal(size=3)
    axis /= np.linalg.norm(axis)
    g = math.radians(r.uniform(0.0, 15.0)) * offset
    k = np.array([[0, -axis[2], axis[1]], [axis[2], 0, -axis[0]], [-axis[1], axis[0], 0]])
    return np.eye(3) + math.sin(g) * k + (1 - math.cos(g)) * (k @ k), r.uniform(-0.5, 0.5, size=3) * offset


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind == "fit_cloud":
        s["points"] = _clouds([case["n"]], [case["k"]], seed)
    elif kind in ("fit_frame", "kmeans"):
        s["points"] = _scan(case["n"], seed)
    elif kind in ("fit_frame4", "gbms"):
        s["points"] = _scan(case["n"], seed, 4)
    elif kind == "fit_batch":
        ns, s["ks"] = _sizes(case)
        s["points"] = _clouds(ns, s["ks"], seed)
        s["offsets"] = np.concatenate([[0], np.cumsum(ns)]).astype(np.int64)
    elif kind == "refine_map":
        s["points"] = _scan(case["n"], seed)
        s["model"] = _model(s["points"], case["k"], seed)
    elif kind in ("score", "score_noalloc"):    # a second scan of the modelled scene
        s["points"] = _scan(case["n"], seed, scan=1)
        s["model"] = _model(_scan(276348, seed), case["k"], seed)
    elif kind == "autograd":
        w, mu, cov = _model(_scan(276348, seed), case["k"], seed)
        scan = _scan(case["n"], seed, scan=1).double()
        R, t = _pose(np.random.default_rng([seed, 23]), case["offset"])
        leaf = {"points": ((scan - scan.mean(0)) @ torch.tensor(R, device=DEV) + torch.tensor(t, device=DEV)).float(),
                "logits": w.double().log().float(), "means": mu, "chol": torch.linalg.cholesky(cov.double()).float(),
                "R": torch.eye(3, device=DEV), "t": scan.mean(0).float()}
        s["leaf"] = {k: v.contiguous().requires_grad_() for k, v in leaf.items()}
    elif kind == "register":
        ns, s["ks"] = _sizes(case)
        w, mu, cov = _model(_scan(276348, seed), case["k"], seed)
        r = np.random.default_rng([seed, 29])
        scans, poses = [], []
        for i, n in enumerate(ns):
            p = _scan(n, seed, scan=1 + i).double()
            R, t = _pose(r, r.uniform(0.0, 1.0))    # each registration is somewhere on its way
            scans.append(((p - p.mean(0)) @ torch.tensor(R, device=DEV) + torch.tensor(t, device=DEV)).float())
            poses.append(torch.cat([torch.eye(3, device=DEV).reshape(9), p.mean(0).float()]))
        s["points"], s["poses"] = torch.cat(scans).contiguous(), torch.stack(poses).contiguous()
        s["offsets"] = np.concatenate([[0], np.cumsum(ns)]).astype(np.int64)
        s["model"] = [torch.cat([a] * case["batch"]).contiguous()
                      for a in (w.double().log().float(), mu, torch.linalg.cholesky(cov.double()).float())]
    elif kind == "resample":
        s["model"] = _model(_scan(276348, seed, 4), case["k"], seed)
        s["locs"] = _scan(case["n"], seed, scan=1)
        s["seed"] = seed
    return s


# ------------------------------------------------------------------------------------------------ one pass
def _log(v, iters=None):
    """Log-likelihoods as a program logs them (they are sums of binary32 terms): a trace in a row of `iters` entries,
    NaN after the fit stopped, as the batched call gives it."""
    v = np.asarray(v, np.float32)
    return v if iters is None else np.concatenate([v, np.full(iters - len(v), np.nan, np.float32)])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("fit_cloud", "fit_frame", "fit_frame4"):
        fit = gira.gira_gmm_fit4 if kind == "fit_frame4" else gira.gira_gmm_fit
        r = fit(state["points"], case["k"], iters=case["iters"], tol=case["tol"], reg_covar=REG, seed=0,
                lloyd_iters=LLOYD)
        return dict(r, trace=_log(r["trace"], case["iters"]))
    if kind == "refine_map":
        r = gira.gira_gmm_fit(state["points"], case["k"], iters=case["iters"], tol=case["tol"], reg_covar=REG,
                              init=state["model"])
        return dict(r, trace=_log(r["trace"], case["iters"]))
    if kind == "fit_batch":
        r = gira.gira_gmm_fit_batched(state["points"], state["offsets"], state["ks"], iters=case["iters"],
                                      tol=case["tol"], reg_covar=REG, seed=0, lloyd_iters=LLOYD)
        return dict(r, trace=_log(r["trace"]), final_loglik=_log(r["final_loglik"]))
    if kind == "kmeans":
        centers, labels, iters = gira.gira_kmeans_init(state["points"], case["k"], seed=0, lloyd_iters=LLOYD)
        return {"centers": centers, "labels": labels, "iters_done": iters}
    if kind in ("score", "score_noalloc"):
        call = gira.gira_gmm_loglik if kind == "score" else gira.gira_gmm_loglik_noalloc
        mean, per_point = call(state["points"], *state["model"], per_point=True)
        return {"mean": mean, "per_point": per_point}
    if kind == "autograd":
        leaf = state["leaf"]
        for v in leaf.values():
            v.grad = None
        loss = autograd.gmm_loglik(leaf["points"], leaf["logits"], leaf["means"], leaf["chol"], leaf["R"], leaf["t"])
        loss.backward()
        return dict({"grad_" + k: v.grad for k, v in leaf.items()}, loss=loss.detach().float())
    if kind == "register":
        r = gira.gira_gmm_loglik_grad_batched(state["points"], state["offsets"], state["ks"], *state["model"],
                                              state["poses"], want=("twist",))
        # the poses are binary32, and so are their gradients in an optimiser
        return {"loglik": _log(r["loglik"]), "status": r["status"], "twist": r["grad_twist"].float()}
    if kind == "resample":
        points, comp = gira.gira_gmm_sample(case["n"], *state["model"], seed=state["seed"])
        mean, var = gira.gira_gmm_conditional4(state["locs"], *state["model"])
        return {"points": points, "components": comp, "mean": mean, "var": var}
    modes, counts = gira.gira_gbms(state["points"], case["h"])
    room = MODES - len(counts)      # into tables of a fixed size, as the number of modes varies with the scene
    return {"k": len(counts), "modes": torch.nn.functional.pad(modes, (0, 0, 0, room)),
            "counts": torch.nn.functional.pad(counts, (0, room))}


# ------------------------------------------------------------------------------------------------ what a pass needs
def work(case):
    """Inputs read once and outputs written once; operations by the definition of each step over every (point,
    component) pair: 23 an EM unit in 3D and 33 in 4D, 12 a log-density, 32 a gradient, 8 (11) a squared distance."""
    kind = case["kind"]
    if kind == "gbms":
        return {"bytes": 16.0 * case["n"] + 36.0 * case["n"] / 100, "flops": 300.0 * case["n"]}
    if kind in ("fit_batch", "register"):
        ns, ks = _sizes(case)
        nk, n, k = float(sum(a * b for a, b in zip(ns, ks))), float(sum(ns)), float(sum(ks))
    else:
        n, k = float(case["n"]), float(case["k"])
        nk = n * k
    kinit = (2 + LLOYD) * 8 * nk
    if kind in ("fit_cloud", "fit_frame", "fit_batch"):
        return {"bytes": 12 * n + 52 * k, "flops": 23 * nk * case["iters"] + kinit}
    if kind == "fit_frame4":
        return {"bytes": 16 * n + 84 * k, "flops": 33 * nk * case["iters"] + kinit * 11 / 8}
    if kind == "refine_map":
        return {"bytes": 12 * n + 104 * k, "flops": 23 * nk * case["iters"] + 12 * nk}
    if kind == "kmeans":
        return {"bytes": 16 * n + 12 * k, "flops": kinit}
    if kind in ("score", "score_noalloc"):
        return {"bytes": 16 * n + 52 * k, "flops": 12 * nk}
    if kind == "autograd":
        return {"bytes": 24 * n + 104 * k, "flops": 32 * nk}
    if kind == "register":
        return {"bytes": 12 * n + 52 * k, "flops": 32 * nk}
    return {"bytes": 40 * n + 84 * k, "flops": 16 * nk + 60 * n}


# ------------------------------------------------------------------------------------------------ 64-bit results
def _splitmix(seed, i):
    """Draws i (array) of the SplitMix64 counter stream: the top 53 bits of output i + 1."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (np.asarray(i, np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return (z ^ (z >> np.uint64(31))) >> np.uint64(11)


def _dist2(x, c):
    """Binary32 squared distances in the defined order, each operation rounded."""
    s = None
    for j in range(x.shape[-1]):
        e = x[..., j] - c[..., j]
        s = e * e if s is None else s + e * e
    return s


def _kmeans(x, k, seed=0):
    """(centres, labels, updates): k-means++ in exact fixed point, then Lloyd, by their definitions."""
    n = len(x)
    u = [int(v) for v in _splitmix(seed, np.arange(k))]
    at = [u[0] * n >> 53]
    d2 = torch.full((n,), math.inf, device=DEV)
    for j in range(1, k):
        d2 = torch.minimum(d2, _dist2(x, x[at[-1]]))
        fx = (d2.double() * 2.0 ** 48).long()
        hi, lo = (fx >> 24).cumsum(0), (fx & 0xFFFFFF).cumsum(0)
        hi, lo = hi + (lo >> 24), lo & 0xFFFFFF
        last = torch.stack([hi[-1], lo[-1]]).tolist()
        total = (last[0] << 24) + last[1]
        thr = u[j] * total >> 53
        over = (hi > thr >> 24) | ((hi == thr >> 24) & (lo > (thr & 0xFFFFFF)))
        at.append(int(over.to(torch.uint8).argmax()) if total else u[j] * n >> 53)
    c = x[torch.tensor(at, device=DEV)].clone()

    def assign():
        step = max(1, (1 << 28) // k)
        return torch.cat([_dist2(x[a:a + step, None], c[None]).argmin(1) for a in range(0, n, step)])

    label, done = assign(), 0
    while done < LLOYD:
        cnt = torch.bincount(label, minlength=k).double()
        s = torch.zeros(k, x.shape[1], dtype=torch.float64, device=DEV).index_add_(0, label, x.double())
        c = torch.where(cnt[:, None] > 0, (s / cnt[:, None]).float(), c)
        done += 1
        before, label = label, assign()
        if torch.equal(before, label):
            break
    return c, label, done


def _mstep(s0, s1, s2, reg):
    nb = s0 + 10 * np.finfo(np.float64).eps
    mu = s1 / nb[:, None]
    d = mu.shape[1]
    cov = s2.reshape(-1, d, d) / nb[:, None, None] - mu[:, :, None] * mu[:, None, :]
    return nb / nb.sum(), mu, cov + reg * torch.eye(d, dtype=torch.float64, device=DEV)


def _outer(x):
    return (x[:, :, None] * x[:, None, :]).reshape(len(x), -1)


def _logits(x, logw, mu, P):
    """ln pi_b + ln N(x_n | mu_b, (P_b^T P_b)^-1), N x K."""
    d = x.shape[1]
    c = logw + P.diagonal(dim1=1, dim2=2).log().sum(1) - 0.5 * d * math.log(2 * math.pi)
    at = (P @ mu[:, :, None])[:, :, 0]
    q = torch.zeros(len(x), len(mu), dtype=torch.float64, device=DEV)
    for j in range(d):
        y = x[:, :j + 1] @ P[:, j, :j + 1].T
        y -= at[:, j]
        q.addcmul_(y, y, value=-0.5)
    return q.add_(c)


def _precision(cov):
    L = torch.linalg.cholesky(cov)
    return _inverse(L)


def _inverse(L):
    eye = torch.eye(L.shape[1], dtype=torch.float64, device=DEV)
    return torch.linalg.solve_triangular(L, eye.expand_as(L), upper=False)


def _estep(x, w, mu, cov, stats=True):
    """(log-likelihood per point, S0, S1, S2) of 64-bit points."""
    P, k, d = _precision(cov), len(w), x.shape[1]
    s = [torch.zeros(k, m, dtype=torch.float64, device=DEV) for m in (1, d, d * d)]
    lls, step = [], max(1, (1 << 28) // k)
    for a in range(0, len(x), step):
        xa = x[a:a + step]
        g = _logits(xa, w.log(), mu, P)
        lls.append(g.logsumexp(1))
        if stats:
            g = g.sub_(lls[-1][:, None]).exp_().T
            for t, f in zip(s, (torch.ones_like(xa[:, :1]), xa, _outer(xa))):
                t += g @ f
    return torch.cat(lls), s[0][:, 0], s[1], s[2]


def _em(x, model, iters, tol, reg=REG):
    """EM from a model (64 bits), about the points' mean."""
    off = x.mean(0)
    x, (w, mu, cov) = x - off, model
    mu, trace = mu - off, []
    for _ in range(iters):
        ll, s0, s1, s2 = _estep(x, w, mu, cov)
        trace.append(float(ll.mean()))
        w, mu, cov = _mstep(s0, s1, s2, reg)
        if len(trace) > 1 and abs(trace[-1] - trace[-2]) < tol:
            break
    return {"weights": w, "means": mu + off, "covs": cov, "iters_done": len(trace),
            "trace": np.array(trace + [math.nan] * (iters - len(trace))),
            "final_loglik": float(_estep(x, w, mu, cov, False)[0].mean())}


def _fit(x, case, k):
    _, label, _ = _kmeans(x, k)
    x = x.double()
    off = x.mean(0)
    y = x - off
    s = [torch.zeros(k, f.shape[1], dtype=torch.float64, device=DEV).index_add_(0, label, f)
         for f in (torch.ones_like(y[:, :1]), y, _outer(y))]
    w, mu, cov = _mstep(s[0][:, 0], s[1], s[2], REG)
    return _em(x, (w, mu + off, cov), case["iters"], case["tol"])


def _gradient(x, R, t, logits, mu, L):
    """L = sum_n ln p(R x_n + t) and its gradients, all in 64 bits."""
    P = _inverse(L)
    lam, logw = P.mT @ P, logits.log_softmax(0)
    off = mu.mean(0)
    y, m = x @ R.T + t - off, mu - off
    k, step = len(m), max(1, (1 << 27) // len(m))
    lam_m = (lam @ m[:, :, None])[:, :, 0]
    s = [torch.zeros(k, j, dtype=torch.float64, device=DEV) for j in (1, 3, 9)]
    total, gs = 0.0, []
    for a in range(0, len(y), step):
        ya = y[a:a + step]
        g = _logits(ya, logw, m, P)
        ll = g.logsumexp(1)
        total += float(ll.sum())
        g = g.sub_(ll[:, None]).exp_()
        A = (g @ lam.reshape(k, 9)).reshape(-1, 3, 3)
        gs.append(g @ lam_m - (A @ ya[:, :, None])[:, :, 0])
        for u, f in zip(s, (torch.ones_like(ya[:, :1]), ya, _outer(ya))):
            u += g.T @ f
    s0, s1, g, xm = s[0][:, 0], s[1], torch.cat(gs), y + off
    c1 = s1 - s0[:, None] * m
    c2 = s[2].reshape(k, 3, 3) - s1[:, :, None] * m[:, None] - m[:, :, None] * s1[:, None] \
        + s0[:, None, None] * m[:, :, None] * m[:, None]
    chol = P.mT @ (P @ c2 @ P.mT) - s0[:, None, None] * torch.diag_embed(1 / L.diagonal(dim1=1, dim2=2))
    return {"loss": total, "grad_points": g @ R, "grad_logits": s0 - len(y) * logw.exp(),
            "grad_means": (lam @ c1[:, :, None])[:, :, 0], "grad_chol": chol.tril(), "grad_R": g.T @ x,
            "grad_t": g.sum(0), "twist": torch.cat([torch.linalg.cross(xm, g).sum(0), g.sum(0)])}


def _conditional(x, w, mu, cov):
    sxx, sxi, sii = cov[:, :3, :3], cov[:, :3, 3], cov[:, 3, 3]
    b = torch.linalg.solve(sxx, sxi[:, :, None])[:, :, 0]
    v = sii - (sxi * b).sum(1)
    P, off, out = _precision(sxx), mu[:, 3] - (b * mu[:, :3]).sum(1), []
    for a in range(0, len(x), 1 << 16):
        xa = x[a:a + (1 << 16)]
        g = _logits(xa, w.log(), mu[:, :3], P).softmax(1)
        m = xa @ b.T + off
        e = (g * m).sum(1)
        out.append((e, (g * (v + (m - e[:, None]) ** 2)).sum(1)))
    return torch.cat([e for e, _ in out]), torch.cat([q for _, q in out])


def _sample(n, w, mu, cov, seed):
    i = 5 * np.arange(n, dtype=np.uint64)
    u = [_splitmix(seed, i + np.uint64(j)).astype(np.float64) / 2.0 ** 53 for j in range(5)]
    cum = np.cumsum(w.cpu().numpy())
    b = torch.tensor(np.minimum(np.searchsorted(cum, u[0] * cum[-1], side="right"), len(cum) - 1), device=DEV)
    r1, r2 = np.sqrt(-2 * np.log1p(-u[1])), np.sqrt(-2 * np.log1p(-u[3]))
    a1, a2 = 2 * np.pi * u[2], 2 * np.pi * u[4]
    z = torch.tensor(np.stack([r1 * np.cos(a1), r1 * np.sin(a1), r2 * np.cos(a2), r2 * np.sin(a2)], 1), device=DEV)
    L = torch.linalg.cholesky(cov)
    return mu[b] + (L[b] @ z[:, :mu.shape[1], None])[:, :, 0], b


def exact(case, seed):
    kind = case["kind"]
    if kind == "gbms":      # decided in exact integers and binary64: the start's own modes are the definition's
        return None
    s = prepare(case, seed)
    if kind == "kmeans":
        c, label, done = _kmeans(s["points"], case["k"])
        return {"centers": c.double(), "labels": label, "iters_done": done}
    if kind in ("fit_cloud", "fit_frame", "fit_frame4"):
        return _fit(s["points"], case, case["k"])
    if kind == "refine_map":
        return _em(s["points"].double(), [v.double() for v in s["model"]], case["iters"], case["tol"])
    if kind == "fit_batch":
        o = s["offsets"]
        fits = [_fit(s["points"][o[i]:o[i + 1]], case, k) for i, k in enumerate(s["ks"])]
        r = {k: torch.cat([f[k] for f in fits]) for k in ("weights", "means", "covs")}
        return dict(r, trace=np.stack([f["trace"] for f in fits]), iters_done=np.array([f["iters_done"] for f in fits]),
                    final_loglik=np.array([f["final_loglik"] for f in fits]), status=np.zeros(len(fits), np.int32))
    if kind in ("score", "score_noalloc"):
        x, (w, mu, cov) = s["points"].double(), [v.double() for v in s["model"]]
        off = x.mean(0)
        ll = _estep(x - off, w, mu - off, cov, False)[0]
        return {"mean": float(ll.mean()), "per_point": ll}
    if kind == "autograd":
        v = {k: t.detach().double() for k, t in s["leaf"].items()}
        g = _gradient(v["points"], v["R"], v["t"], v["logits"], v["means"], v["chol"])
        return {k: t for k, t in g.items() if k != "twist"}
    if kind == "register":
        o, b = s["offsets"], 0
        ll, tw = [], []
        for i, k in enumerate(s["ks"]):
            p = s["poses"][i].double()
            g = _gradient(s["points"][o[i]:o[i + 1]].double(), p[:9].reshape(3, 3), p[9:],
                          *[v[b:b + k].double() for v in s["model"]])
            ll.append(g["loss"])
            tw.append(g["twist"])
            b += k
        return {"loglik": np.array(ll), "status": np.zeros(len(ll), np.int32), "twist": torch.stack(tw)}
    model = [v.double() for v in s["model"]]
    points, comp = _sample(case["n"], *model, s["seed"])
    mean, var = _conditional(s["locs"].double(), *model)
    return {"points": points, "components": comp, "mean": mean, "var": var}
