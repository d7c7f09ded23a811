"""The workloads whose time is measured, each through the entry points that a
program using this package calls.

Scenes are ray cast on the GPU in 64 bits: rectangles and infinite planes, some
moving, seen by a camera on a random trajectory, with the flow noise of the
Fisk residual model. They come in the package's three kinds: `planes` (a few
tilted patches before a wall), `handheld` (an indoor scene at 0.5 to 8 m with
non-rigid patches) and `driving` (a ground plane, facades and moving cars).
Sizes are those of the package's own configurations and tests: windows from
160x120 with 3 flows and 256 hypotheses per frame to 1242x375 with 8 flows and
8192.
"""
import math
import os

import numpy as np
import torch

from paper_2104_06789_gb300 import voldor, vo

SCENES = {                      # focal length over width, inverse depth range
    "planes": (0.75, (1 / 40.0, 1.0)),
    "handheld": (0.82, (1 / 16.0, 4.0)),
    "driving": (0.578, (1 / 160.0, 1 / 1.5)),
}


def listed():
    w = dict(op="window", init="given", flows="device", criterion="mie", residual="fisk")
    return [
        # one small window: what a low-resolution tracker runs for every new flow
        dict(w, name="window_small", scene="planes", W=160, H=120, T=3, S=256, iters=3, dtype="f32"),
        # an indoor window whose flows arrive in host memory
        dict(w, name="window_handheld", scene="handheld", W=640, H=480, T=5, S=4096, iters=5, dtype="f32",
             flows="host"),
        # the driving window that bench.py times: full size, half-precision flows
        dict(w, name="window_driving", scene="driving", W=1242, H=375, T=8, S=8192, iters=5, dtype="f16"),
        # the learned rigidness prior in place of the plain bootstrap, and the fewer iterations it needs
        dict(w, name="window_learned", scene="handheld", W=1242, H=375, T=8, S=4096, iters=3, dtype="f16",
             init="learned"),
        # the ablation's likelihood criterion and Gaussian residual, as a parameter study runs them
        dict(w, name="window_ablation", scene="handheld", W=320, H=240, T=6, S=2048, iters=5, dtype="f32",
             criterion="mle", residual="gaussian"),
        # odometry over a short sequence: overlapping windows, absolute scale from the ground plane
        dict(op="sequence", name="sequence", W=414, H=125, T=6, n=10, stride=2, S=1024, iters=5, dtype="f16"),
        # several cameras' windows of mixed size in one graph
        dict(op="batch", name="batch", n=6, S=1024, iters=5, dtype="f16"),
        # the first window of a sequence: T_1 from the epipolar geometry of its first flow
        dict(op="epipolar", name="epipolar", scene="driving", W=1242, H=375, M=512, dtype="f16"),
        # one frame's pose alone, on a known depth and rigidness
        dict(op="pose", name="pose_update", scene="handheld", W=640, H=480, T=5, t=3, S=4096, dtype="f32"),
        # depth and rigidness alone, on known poses: a sweep in each of the four directions
        dict(op="refine", name="refine", scene="driving", W=1242, H=375, T=8, dtype="f16"),
        # the proposal network: inference on a batch of windows, and a training step
        dict(op="net_forward", name="net_forward", W=1242, H=375, T=8, B=8, dtype="f16"),
        dict(op="net_train", name="net_train", W=1242, H=375, T=8, B=2, dtype="f16"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["window"] * 5 + ["sequence", "batch", "epipolar", "pose", "refine", "net_forward", "net_train"])
    dtype = rng.choice(["f16", "f32"])
    W = _spread(rng, 160, 1242)
    H = min(_spread(rng, 0.3 * W, 0.8 * W), 465750 // W)
    if op == "sequence":
        T = rng.randint(4, 6)
        return dict(op=op, W=_spread(rng, 300, 500), H=_spread(rng, 90, 200), T=T, n=T + rng.randint(2, 6),
                    stride=rng.randint(1, 3),
                    S=_spread(rng, 256, 2048), iters=rng.randint(3, 5), dtype=dtype)
    if op == "batch":
        return dict(op=op, n=rng.randint(3, 8), S=_spread(rng, 512, 2048), iters=rng.randint(3, 5), dtype=dtype)
    if op == "epipolar":
        return dict(op=op, scene=rng.choice(["handheld", "driving"]), W=W, H=H, M=_spread(rng, 128, 1024), dtype=dtype)
    if op in ("net_forward", "net_train"):
        most = 8 if op == "net_forward" else 2
        return dict(op=op, W=W, H=H, T=rng.randint(3, 8), B=rng.randint(1, most), dtype=dtype)
    scene = rng.choice(sorted(SCENES))
    T = rng.randint(3, 8)
    if op == "refine":
        return dict(op=op, scene=scene, W=W, H=H, T=T, dtype=dtype)
    S = _spread(rng, 256, 8192)
    if op == "pose":
        return dict(op=op, scene=scene, W=W, H=H, T=T, t=rng.randint(1, T), S=S, dtype=dtype)
    init = "learned" if T == 8 and rng.random() < 0.5 else "given"
    plain = rng.random() < 0.7
    return dict(op=op, init=init, flows=rng.choice(["device", "device", "host"]), scene=scene, W=W, H=H, T=T, S=S,
                iters=rng.randint(3, 5), dtype=dtype,
                criterion="mie" if plain else rng.choice(["mie", "mle"]), residual="fisk" if plain else "gaussian")


# ---------------------------------------------------------------------------
# Scenes
# ---------------------------------------------------------------------------
def _rotation(axis, angle):
    axis = np.asarray(axis, float) / np.linalg.norm(axis)
    k = np.array([[0, -axis[2], axis[1]], [axis[2], 0, -axis[0]], [-axis[1], axis[0], 0]])
    return np.eye(3) + np.sin(angle) * k + (1 - np.cos(angle)) * k @ k


def _surfaces(scene, rng, K, W, H):
    """Rectangles: centre, normal, in-plane axis, half sizes along it and across (inf: a plane), velocity per frame."""
    f, _, cx, cy = K
    inf, still = math.inf, (0.0, 0.0, 0.0)
    if scene == "driving":
        out = [((0, 1.65, 0), (0, -1, 0), (1, 0, 0), inf, inf, still), ((0, 0, 80), (0, 0, -1), (1, 0, 0), inf, inf, still)]
        for side in (-1, 1):
            z = 0.0
            while z < 80:
                seg, x, h = rng.uniform(6, 20), side * rng.uniform(5, 15), rng.uniform(4, 20)
                out.append(((x, 1.65 - h / 2, z + seg / 2), (-side, 0, 0), (0, 0, 1), seg / 2, h / 2, still))
                z += seg
        for _ in range(10):         # the backs of cars
            x, z = rng.uniform(-5, 5), rng.uniform(8, 35)
            vel = (rng.uniform(-0.1, 0.1), 0.0, rng.uniform(0.2, 2.0) if z < 20 else rng.uniform(-1.0, 2.0))
            out.append(((x, 0.9, z), (0, 0, -1), (1, 0, 0), 0.9, 0.75, vel))
        return out
    near, far, count = (2.0, 20.0, 4) if scene == "planes" else (0.5, 8.0, 20)
    out = [((0, 0, far), (0, 0, -1), (1, 0, 0), inf, inf, still)]
    for _ in range(count):
        z = rng.uniform(near, far)
        c = ((rng.uniform(0.1, 0.9) * W - cx) / f * z, (rng.uniform(0.1, 0.9) * H - cy) / f * z, z)
        n = _rotation([rng.normal(), rng.normal(), 0.0], rng.uniform(0, math.pi / 3)) @ np.array([0.0, 0.0, -1.0])
        u = np.cross(n, [0.0, 1.0, 0.0])
        out.append((c, n, u / np.linalg.norm(u), z * rng.uniform(0.15, 0.4) * W / f, z * rng.uniform(0.15, 0.4) * H / f,
                    still))
    return out


def _step(scene, rng):
    M = np.eye(4)
    axis, way = rng.normal(size=3), rng.normal(size=3)
    if scene == "driving":
        M[:3, :3], M[:3, 3] = _rotation([0, 1, 0], math.radians(rng.uniform(-1, 1))), (0, 0, -1.0)
    else:
        most, size = (2.0, 0.1) if scene == "planes" else (5.0, rng.uniform(0.01, 0.05))
        M[:3, :3], M[:3, 3] = _rotation(axis, math.radians(rng.uniform(0, most))), size * way / np.linalg.norm(way)
    return M


def _flows(scene, seed, W, H, T, dtype, focal=None):
    """Flows X_1..X_T on the GPU, the intrinsics, the true T_t and the depth of the first image."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator("cuda").manual_seed(seed)
    f64 = dict(dtype=torch.float64, device="cuda")
    fl = focal or SCENES[scene][0] * W
    K = (fl, fl, (W - 1) / 2.0, (H - 1) / 2.0)
    surfaces = _surfaces(scene, rng, K, W, H)
    patches = []
    for _ in range({"planes": 1, "handheld": 3, "driving": 0}[scene]):
        side = math.sqrt({"planes": 0.10, "handheld": 0.067}[scene])
        pw, ph = max(1, round(side * W)), max(1, round(side * H))
        patches.append((int(rng.integers(0, W - pw + 1)), int(rng.integers(0, H - ph + 1)), pw, ph))
    ys, xs = torch.meshgrid(torch.arange(H, **f64), torch.arange(W, **f64), indexing="ij")
    rays = torch.stack([(xs - K[2]) / fl, (ys - K[3]) / fl, torch.ones_like(xs)], -1)
    steps = [_step(scene, rng) for _ in range(T)]
    M, out, depth0 = np.eye(4), [], None
    for t, rel in enumerate(steps):
        o, R = -M[:3, :3].T @ M[:3, 3], torch.tensor(M[:3, :3], **f64)
        d = rays @ R
        best = torch.full((H, W), math.inf, **f64)
        move = torch.zeros(H, W, 3, **f64)
        for c, n, u, hu, hv, vel in surfaces:
            c, n, u, vel = (np.asarray(v, float) for v in (c, n, u, vel))
            at, v = c + vel * t, np.cross(n, u)
            dist = float((at - o) @ n) / (d @ torch.tensor(n, **f64))
            hit = dist > 1e-6
            if math.isfinite(hu):
                for axis, half in ((u, hu), (v, hv)):
                    hit &= (float((o - at) @ axis) + dist * (d @ torch.tensor(axis, **f64))).abs() <= half
            hit &= dist < best
            best = torch.where(hit, dist, best)
            move = torch.where(hit[..., None], torch.tensor(vel, **f64), move)
        depth0 = best if depth0 is None else depth0
        M = rel @ M
        P = (torch.tensor(o, **f64) + best[..., None] * d + move) @ torch.tensor(M[:3, :3].T.copy(), **f64)
        P = P + torch.tensor(M[:3, 3], **f64)
        x = torch.stack([fl * P[..., 0] / P[..., 2] + K[2] - xs, fl * P[..., 1] / P[..., 2] + K[3] - ys], -1)
        lost = ~torch.isfinite(x).all(-1) | (P[..., 2] <= 0.5 * (scene == "driving")) | (x.abs().amax(-1) > max(W, H))
        x = torch.where(lost[..., None], torch.rand(H, W, 2, generator=gen, **f64) * 40 - 20, x)
        for x0, y0, pw, ph in patches:
            x[y0:y0 + ph, x0:x0 + pw] += torch.tensor(rng.uniform(-8, 8, size=2), **f64)
        n = x.norm(dim=-1).clamp(max=40.0)
        p = torch.rand(H, W, generator=gen, **f64).clamp(1e-12, 1 - 1e-12)
        epe = (0.01 * torch.exp(0.09 * n) * (p / (1 - p)) ** (1 / (1 - 0.0022 * n))).sqrt().clamp(max=1e4)
        way = 2 * math.pi * torch.rand(H, W, generator=gen, **f64)
        out.append(x + torch.stack([epe * way.cos(), epe * way.sin()], -1))
    flows = torch.stack(out).to(torch.float16 if dtype == "f16" else torch.float32)
    return flows, K, np.array(steps), depth0.clamp(0.1, 1e3)


def _params(case, scene, seed):
    lo, hi = SCENES[scene][1]
    return voldor.default_params(
        hyps_per_frame=case.get("S", 256), inv_depth_min=lo, inv_depth_max=hi, seed=seed & 0xffff,
        criterion=voldor.CRITERION_MLE if case.get("criterion") == "mle" else voldor.CRITERION_MIE,
        residual=voldor.RESIDUAL_GAUSSIAN if case.get("residual") == "gaussian" else voldor.RESIDUAL_FISK)


def _known_state(case, poses, depth0, seed):
    """Poses, depth and rigidness as a previous estimate leaves them: near the truth, most pixels rigid."""
    gen = torch.Generator("cuda").manual_seed(seed + 1)
    shape = (case["H"], case["W"])
    depth = depth0 * (1 + 0.05 * torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)).clamp(0.5, 2)
    rigid = torch.rand((case["T"],) + shape, generator=gen, device="cuda") ** 0.25
    return poses, depth.float().cpu().numpy(), rigid.cpu().numpy()


def _weights(T, seed):
    """Weights of the proposal network: the trained ones the package ships for T = 8, else a fresh initialisation."""
    here = os.path.join(os.path.dirname(voldor.__file__), "weights", "proposal_handheld_1242x375_T8.npy")
    if T == 8:
        return np.load(here)
    rng = np.random.default_rng(seed)
    out = []
    for cin, cout in [(2 * T, 32)] + [(32, 32)] * 4 + [(32, 2)]:
        out += [rng.normal(size=cout * 9 * cin) * math.sqrt(2.0 / (9 * cin)), np.zeros(cout)]
    return np.concatenate(out).astype(np.float32)


def _batch_sizes(case):
    """Width, height and flows of a batch's windows: three resolutions in turn, 3 to 8 flows."""
    return [((320, 240), (640, 480), (1242, 375))[i % 3] + (3 + 5 * i % 6,) for i in range(case["n"])]


def _net_inputs(case, seed):
    made = [_flows("handheld", 131 * seed + b, case["W"], case["H"], case["T"], case["dtype"]) for b in range(case["B"])]
    depth = torch.stack([m[3] for m in made]).log()
    gen = torch.Generator("cuda").manual_seed(seed + 1)
    rigid = torch.rand(depth.shape, generator=gen, device="cuda", dtype=torch.float64) ** 0.25
    target = torch.stack([depth - depth.flatten(1).median(dim=1).values[:, None, None], rigid], -1).float()
    return torch.stack([m[0] for m in made]), target


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def prepare(case, seed):
    op = case["op"]
    s = {"case": case}
    if op in ("net_forward", "net_train"):
        s["flows"], s["target"] = _net_inputs(case, seed)
        s["net"] = voldor.Net(case["T"], _weights(case["T"], seed))
        return s
    if op == "sequence":
        s["flows"], K, poses, _ = _flows("driving", seed, case["W"], case["H"], case["n"], case["dtype"])
        s["T1"] = poses[0]
        s["vo"] = vo.SlidingWindowVO(K, case["T"], case["stride"], case["iters"], _params(case, "driving", seed))
        return s
    if op == "batch":
        s["windows"], s["T1"] = [], []
        for i, (W, H, T) in enumerate(_batch_sizes(case)):
            scene = "driving" if W == 1242 else "handheld"
            flows, K, poses, _ = _flows(scene, 131 * seed + i, W, H, T, case["dtype"])
            s["windows"].append(voldor.Window(flows, K, _params(case, scene, seed + i)))
            s["T1"].append(poses[0])
        for w, T1 in zip(s["windows"], s["T1"]):
            w.bootstrap(T1)
        s["batch"] = voldor.Batch(s["windows"], case["iters"])
        return s
    scene = case["scene"]
    flows, K, poses, depth0 = _flows(scene, seed, case["W"], case["H"], case.get("T", 1), case["dtype"])
    s["flows"] = flows.cpu().numpy() if case.get("flows") == "host" else flows
    s["T1"] = poses[0]
    s["window"] = voldor.Window(s["flows"], K, _params(case, scene, seed))
    if case.get("init") == "learned":
        s["net"] = voldor.Net(case["T"], _weights(case["T"], seed))
    if op in ("pose", "refine"):
        s["window"].set_state(*_known_state(case, poses, depth0, seed))
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "window":
        w = s["window"]
        w.set_flows(s["flows"])
        if case["init"] == "learned":
            s["net"].bootstrap(w, s["T1"], depth=False)
        else:
            w.bootstrap(s["T1"])
        w.em_step(case["iters"])
        return w.get_pose_depth_rigidness()
    if op == "sequence":
        r = s["vo"].run(s["flows"], T1=s["T1"], camera_height=1.65)
        return r["relative"], r["trajectory"]
    if op == "batch":
        for w, T1 in zip(s["windows"], s["T1"]):
            w.bootstrap(T1)
        s["batch"].run(latency=False)
        return [w.get_pose_depth_rigidness() for w in s["windows"]]
    if op == "epipolar":
        return s["window"].bootstrap_epipolar(case["M"], 1.0)
    if op == "pose":
        s["window"].pose_update(0, case["t"])
        return s["window"].get_pose_depth_rigidness(depth=False, rigidness=False)[0]
    if op == "refine":
        for k in range(4):
            s["window"].rigidness_smooth(k)
            s["window"].depth_update(k)
            s["window"].rigidness_update()
        return s["window"].get_pose_depth_rigidness(poses=False)[1:]
    if op == "net_forward":
        return s["net"].forward(s["flows"])
    loss = s["net"].train_step(s["flows"], s["target"], 1e-3)
    return {"loss": loss, "grads": s["net"].get_grads()}


def work(case):
    """A pass's inputs and outputs, and its arithmetic: about 60 operations for a (hypothesis, pixel) pair of the dense
    scoring (three in five pixels of a frame keep their correspondence), 200 for a pixel of a frame in each per-pixel
    pass, 50 for a (sample, pixel) pair of the epipolar estimate, two for a multiply-add of the network."""
    op = case["op"]
    per = 4 if case["dtype"] == "f16" else 8
    if op == "batch":
        w = [(W * H, T) for W, H, T in _batch_sizes(case)]
        return {"bytes": sum(n * (T * (per + 4) + 4) for n, T in w),
                "flops": sum(n * T * case["iters"] * (0.6 * 60 * case["S"] + 600) for n, T in w)}
    N = case["W"] * case["H"]
    if op == "sequence":
        windows = len(vo.window_starts(case["n"], case["T"], min(case["stride"], case["T"] - 1)))
        return {"bytes": N * case["n"] * per,
                "flops": windows * N * case["T"] * case["iters"] * (0.6 * 60 * case["S"] + 600)}
    if op == "epipolar":
        return {"bytes": N * per, "flops": 50 * N * case["M"]}
    T = case["T"]
    if op in ("net_forward", "net_train"):
        n = case["B"] * N
        forward = 2 * 9 * (2 * T * 32 + 4 * 32 * 32 + 32 * 2) * n
        if op == "net_forward":
            return {"bytes": n * (T * per + 32), "flops": forward}
        return {"bytes": n * (T * per + 8), "flops": 3 * forward}
    if op == "pose":
        return {"bytes": N * (per + 4 + 4), "flops": N * 0.6 * 60 * case["S"]}
    if op == "refine":
        return {"bytes": N * (T * (per + 4 + 4) + 8), "flops": 4 * 600 * N * T}
    return {"bytes": N * (T * (per + 4) + 4), "flops": N * T * case["iters"] * (0.6 * 60 * case["S"] + 600)}


def exact(case, seed):
    """The network's prediction, and the gradient of its loss, in 64 bits. The other paths choose among candidates
    (a hypothesis, a depth, a sample): their results follow the choice and have no value of their own."""
    if case["op"] not in ("net_forward", "net_train"):
        return None
    T, B, H, W = case["T"], case["B"], case["H"], case["W"]
    flows, target = _net_inputs(case, seed)
    weights = torch.from_numpy(_weights(T, seed)).double().cuda()
    mean = flows.double().norm(dim=-1).mean(dim=(2, 3))
    x = flows.double() / mean[..., None, None, None]
    x = x.permute(0, 1, 4, 2, 3).reshape(B, 2 * T, H, W)
    at, layers = 0, []
    for cin, cout in [(2 * T, 32)] + [(32, 32)] * 4 + [(32, 2)]:
        n = cout * 9 * cin
        layers.append((weights[at:at + n].clone().requires_grad_(), weights[at + n:at + n + cout].clone().requires_grad_()))
        at += n + cout

    def predict(x):
        for i, (w, b) in enumerate(layers):
            w = w.reshape(b.numel(), 3, 3, -1)
            pad = torch.nn.functional.pad(x, (1, 1, 1, 1))
            y = b[:, None, None]
            for ky in range(3):
                for kx in range(3):
                    y = y + torch.einsum("oc,bchw->bohw", w[:, ky, kx], pad[:, :, ky:ky + H, kx:kx + W])
            x = y.relu() if i < 5 else y
        return x

    if case["op"] == "net_forward":
        out = torch.zeros(B, H, W, 8, dtype=torch.float64, device="cuda")
        with torch.no_grad():
            for b in range(B):
                out[b, :, :, :2] = predict(x[b:b + 1])[0].permute(1, 2, 0)
        return out
    total = 0.0
    for b in range(B):
        z = predict(x[b:b + 1])[0]
        d, logit = z[0] - target[b, :, :, 0].double(), z[1]
        huber = torch.where(d.abs() < 0.1, 5 * d * d, d.abs() - 0.05)
        loss = (huber + torch.nn.functional.softplus(logit) - target[b, :, :, 1].double() * logit).sum() / (B * H * W)
        loss.backward()
        total += float(loss)
    return {"loss": total, "grads": torch.cat([p.grad.reshape(-1) for layer in layers for p in layer])}
