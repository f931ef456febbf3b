"""The work this framework is used for, as timed cases: single seam searches, energies, whole carves,
forward energy, seam insertion, a batch and a serving burst, each through the Python binding as a
program calls it. Images are a colour gradient with solid rectangles and Gaussian noise, as the
benchmark's; maps are the e1 energies of such images. Sizes are the benchmark's configurations, the
thumbnail of the tests and one odd size; ``draw`` gives others of the same ranges."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_21207_gb300 import binding as sc


def listed():
    return [
        # the smallest call: one seam of a thumbnail's energy map (latency and launches)
        {"name": "seam_64x48", "kind": "seam", "W": 64, "H": 48, "C": 3},
        # one seam of a full-HD map: what an interactive tool asks per step
        {"name": "seam_1920x1080", "kind": "seam", "W": 1920, "H": 1080, "C": 3},
        # the seams of many UHD frames in one call (a video's frames, one GPU full of maps)
        {"name": "seams_58x3840x2160", "kind": "seams", "n": 58, "W": 3840, "H": 2160, "C": 3},
        # the e1 energy of a full-HD photograph alone (importance map for display or masking)
        {"name": "energy_1920x1080", "kind": "energy", "W": 1920, "H": 1080, "C": 3},
        # a thumbnail of uniform bytes narrowed by 16 seams: every launch counts
        {"name": "carve_64x48", "kind": "carve", "W": 64, "H": 48, "C": 3, "tw": 48, "th": 48, "uniform": True},
        # odd sizes, four channels, both directions: an RGBA picture fitted to a layout
        {"name": "carve_1279x853_rgba", "kind": "carve", "W": 1279, "H": 853, "C": 4, "tw": 1021, "th": 701},
        # the headline: full HD narrowed to three quarters
        {"name": "carve_1920x1080", "kind": "carve", "W": 1920, "H": 1080, "C": 3, "tw": 1440, "th": 1080},
        # the largest: UHD reduced to three quarters in both directions
        {"name": "carve_3840x2160", "kind": "carve", "W": 3840, "H": 2160, "C": 3, "tw": 2880, "th": 1620},
        # full HD narrowed with forward energy
        {"name": "forward_1920x1080", "kind": "forward", "W": 1920, "H": 1080, "C": 3, "tw": 1440, "th": 1080},
        # full HD widened by a quarter through seam insertion
        {"name": "enlarge_1920x1080", "kind": "enlarge", "W": 1920, "H": 1080, "C": 3, "tw": 2400, "th": 1080},
        # a set of 256 pictures of mixed sizes narrowed by one replayed plan
        {"name": "batch_256", "kind": "batch", "n": 256, "C": 3, "sizes": 4},
        # a burst of requests of mixed sizes to the server, host pictures in and out
        {"name": "serve_64", "kind": "serve", "n": 64, "C": 3, "sizes": 5},
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    """One more case: any kind, sizes spread over the logarithm of the listed cases' range."""
    kind = rng.choice(["seam", "seams", "energy", "carve", "carve", "carve", "forward", "enlarge", "batch", "serve"])
    C = rng.choice([1, 3, 3, 4])
    if kind in ("batch", "serve"):
        n = _log_int(rng, 8, 256) if kind == "batch" else _log_int(rng, 4, 48)
        while True:   # no single request heavier than the largest listed carve
            case = {"kind": kind, "n": n, "C": C, "sizes": rng.randrange(1, 1 << 20)}
            if max(H * (W - tw) + tw * (H - th) for W, H, tw, th in _jobs(case)) < 2_500_000:
                return case
    small = kind in ("forward", "enlarge")
    W = _log_int(rng, 64, 1920 if small else 3840)
    H = _log_int(rng, 48, 1080 if small else 2160)
    case = {"kind": kind, "W": W, "H": H, "C": C}
    if kind == "seams":
        case["n"] = _log_int(rng, 2, 58)
    if kind in ("carve", "forward"):
        case["tw"] = max(1, int(W * rng.uniform(0.75, 0.97)))
        case["th"] = H if rng.random() < 0.5 else max(1, int(H * rng.uniform(0.75, 0.97)))
        if kind == "forward":
            case["th"] = H
    if kind == "enlarge":
        case["tw"], case["th"] = W + max(1, int(W * rng.uniform(0.03, 0.25))), H
    return case


# ---- inputs ----
def _image(W, H, C, seed, uniform=False):
    """uint8 H x W x C on the GPU: gradient, solid rectangles, noise of standard deviation 8."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if uniform:
        return torch.randint(0, 256, (H, W, C), generator=g, device="cuda", dtype=torch.uint8)
    r = np.random.default_rng(seed)
    a, b = r.integers(0, 256, C), r.integers(0, 256, C)
    th = r.uniform(0.0, 2.0 * math.pi)
    xs = torch.arange(W, device="cuda", dtype=torch.float32)[None, :] * math.cos(th)
    ys = torch.arange(H, device="cuda", dtype=torch.float32)[:, None] * math.sin(th)
    t = xs + ys
    t = (t - t.min()) / max(float(t.max() - t.min()), 1e-6)
    a32 = torch.tensor(a, device="cuda", dtype=torch.float32)
    b32 = torch.tensor(b, device="cuda", dtype=torch.float32)
    img = a32 + (b32 - a32) * t[:, :, None]
    side = max(20, min(300, W, H))
    for _ in range(max(1, round(40.0 * W * H / (1920.0 * 1080.0)))):
        w, h = r.integers(20, side + 1, 2)
        x0, y0 = int(r.integers(0, W)), int(r.integers(0, H))
        img[y0:y0 + h, x0:x0 + w] = torch.tensor(r.integers(0, 256, C), device="cuda", dtype=torch.float32)
    img += 8.0 * torch.randn(img.shape, generator=g, device="cuda")
    return img.round_().clamp_(0, 255).to(torch.uint8).contiguous()


def _energy_map(img):
    """The e1 energy of an image as a caller with its own code would make it: uint16 H x W."""
    x = img.to(torch.int32)
    H, W = x.shape[:2]
    j, i = torch.arange(W, device=x.device), torch.arange(H, device=x.device)
    dx = (x[:, (j + 1).clamp(max=W - 1)] - x[:, (j - 1).clamp(min=0)]).abs()
    dy = (x[(i + 1).clamp(max=H - 1)] - x[(i - 1).clamp(min=0)]).abs()
    return (dx + dy).sum(2).to(torch.int16).view(torch.uint16).contiguous()   # at most 2040


def _maps(case, seed):
    base = [_energy_map(_image(case["W"], case["H"], case["C"], seed * 16 + k)) for k in range(min(4, case["n"]))]
    return [torch.roll(base[k % len(base)].view(torch.int16), 13 * (k // len(base)), 1).view(torch.uint16).contiguous()
            for k in range(case["n"])]


def _jobs(case):
    """(W, H, tw, th) of a batch's pictures or a burst's requests: the benchmark's distributions."""
    r = np.random.default_rng(case["sizes"])
    jobs = []
    for _ in range(case["n"]):
        if case["kind"] == "batch":
            W, H = int(r.integers(240, 1281)), int(r.integers(180, 961))
            jobs.append((W, H, W - int(r.uniform(0.10, 0.40) * W), H))
        else:
            W = int(round(math.exp(r.uniform(math.log(128), math.log(4096)))))
            H = int(round(math.exp(r.uniform(math.log(128), math.log(2160)))))
            jobs.append((W, H, max(1, int(r.uniform(0.5, 0.9) * W)), max(1, int(r.uniform(0.8, 1.0) * H))))
    return jobs


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "seams":
        st["maps"] = _maps(case, seed)
    elif kind in ("batch", "serve"):
        jobs = _jobs(case)
        imgs = [_image(W, H, case["C"], seed * 1000 + k) for k, (W, H, _, _) in enumerate(jobs)]
        st["targets"] = [(tw, th) for _, _, tw, th in jobs]
        if kind == "batch":
            # the plan a program builds once and replays; balanced by the library's own model
            st["plan"] = sc.BatchPlan(imgs, st["targets"], autotune=2)
        else:
            st["imgs"] = [i.cpu().numpy() for i in imgs]
            st["server"] = sc.Server(budget_bytes=8 << 30)
    else:
        img = _image(case["W"], case["H"], case["C"], seed, case.get("uniform", False))
        st["in"] = _energy_map(img) if kind == "seam" else img
    torch.cuda.synchronize()
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "seam":
        return sc.find_seam(state["in"])
    if kind == "seams":
        return sc.find_seam_multi(state["maps"])
    if kind == "energy":
        return sc.energy(state["in"])
    if kind == "carve":
        return sc.carve(state["in"], case["tw"], case["th"], with_log=True)
    if kind == "forward":
        return sc.carve_forward(state["in"], case["tw"], case["th"], with_log=True)
    if kind == "enlarge":
        return sc.enlarge(state["in"], case["tw"], with_cols=True)
    if kind == "batch":   # the set handed on as one buffer
        return torch.cat([o.view(-1) for o in state["plan"].run()])
    server = state["server"]
    tickets = [server.submit(i, tw, th) for i, (tw, th) in zip(state["imgs"], state["targets"])]
    server.drain()
    outs = np.concatenate([server.result(t).reshape(-1) for t in tickets])
    for t in tickets:
        server.release(t)
    return outs


# ---- what a pass cannot do without ----
def _pixel_seams(W, H, tw, th):
    nv, nh = W - tw, H - th
    return H * (nv * W - nv * (nv - 1) // 2) + tw * (nh * H - nh * (nh - 1) // 2)


def work(case):
    """Inputs read once, outputs written once; per searched pixel two minima and an addition, per
    image pixel the energy's differences and sums (4 per channel)."""
    kind, C = case["kind"], case["C"]
    if kind in ("batch", "serve"):
        jobs = _jobs(case)
        return {"bytes": sum((W * H + tw * th) * C for W, H, tw, th in jobs),
                "flops": sum(3 * _pixel_seams(*j) + 4 * C * j[0] * j[1] for j in jobs)}
    W, H = case["W"], case["H"]
    if kind == "seam":
        return {"bytes": 2 * W * H + 4 * H + 8, "flops": 3 * W * H}
    if kind == "seams":
        return {"bytes": case["n"] * (2 * W * H + 4 * H + 8), "flops": 3 * W * H * case["n"]}
    if kind == "energy":
        return {"bytes": (C + 2) * W * H, "flops": 4 * C * W * H}
    tw, th = case["tw"], case["th"]
    if kind == "enlarge":
        k = tw - W
        return {"bytes": (W + tw) * H * C + 4 * k * H, "flops": 3 * _pixel_seams(W, H, W - k, H) + 4 * C * W * H}
    seams, log = W - tw + H - th, (W - tw) * H + (H - th) * tw
    return {"bytes": (W * H + tw * th) * C + 4 * log + 8 * seams,
            "flops": 3 * _pixel_seams(W, H, tw, th) + 4 * C * W * H}


# ---- the same results in 64-bit numpy ----
def _seam64(cu, dl=None, dr=None):
    """Algorithm 3 (leftmost ties) of int64 maps [n, H, W]: seams [n, H] and costs [n]."""
    n, H, W = cu.shape
    big = np.int64(1) << 60
    pad = np.full((H, n, W + 2), big, dtype=np.int64)
    pad[0, :, 1:-1] = cu[:, 0]
    for i in range(1, H):
        p = pad[i - 1]
        a, b, c = p[:, :-2], p[:, 1:-1], p[:, 2:]
        if dl is not None:
            a, c = a + dl[:, i], c + dr[:, i]
        pad[i, :, 1:-1] = cu[:, i] + np.minimum(np.minimum(a, b), c)
    seams = np.empty((n, H), dtype=np.int32)
    costs = np.empty(n, dtype=np.int64)
    for k in range(n):
        j = int(np.argmin(pad[H - 1, k]))
        costs[k] = pad[H - 1, k, j]
        for i in range(H - 1, -1, -1):
            seams[k, i] = j - 1
            if i:
                three = pad[i - 1, k, j - 1:j + 2]
                if dl is not None:
                    three = three + np.array([dl[k, i, j - 1], 0, dr[k, i, j - 1]])
                j += int(np.argmin(three)) - 1
    return seams, costs


def _energy64(x):
    xp = np.concatenate([x[:, :1], x, x[:, -1:]], 1)
    yp = np.concatenate([x[:1], x, x[-1:]], 0)
    return (np.abs(xp[:, 2:] - xp[:, :-2]) + np.abs(yp[2:] - yp[:-2])).sum(2, dtype=np.int64)


def _forward64(x):
    H, W, _ = x.shape
    cu, dl, dr = (np.zeros((H, W), dtype=np.int64) for _ in range(3))
    cu[:, 1:-1] = np.abs(x[:, 2:] - x[:, :-2]).sum(2)
    dl[1:, 1:] = np.abs(x[:-1, 1:] - x[1:, :-1]).sum(2)
    dr[1:, :-1] = np.abs(x[:-1, :-1] - x[1:, 1:]).sum(2)
    return cu, dl, dr


def _pass64(x, count, forward):
    logs, costs = [], []
    for _ in range(count):
        planes = _forward64(x) if forward else (_energy64(x),)
        s, c = _seam64(*[p[None] for p in planes])
        logs.append(s[0])
        costs.append(int(c[0]))
        keep = np.ones(x.shape[:2], dtype=bool)
        keep[np.arange(x.shape[0]), s[0]] = False
        x = x[keep].reshape(x.shape[0], x.shape[1] - 1, x.shape[2])
    return x, logs, costs


def _carve64(img, tw, th, forward=False):
    x = img.astype(np.int64)
    H, W, _ = x.shape
    x, l0, c0 = _pass64(x, W - tw, forward)
    x, l1, c1 = _pass64(x.transpose(1, 0, 2), H - th, forward)
    log = np.concatenate(l0 + l1) if l0 or l1 else np.empty(0, dtype=np.int32)
    out = np.ascontiguousarray(x.transpose(1, 0, 2)).astype(np.uint8)
    return out, log.astype(np.int32), np.array(c0 + c1, dtype=np.int64), l0


def exact(case, seed):
    kind, C = case["kind"], case["C"]
    if kind == "seams":
        if case["n"] * case["W"] * case["H"] > 1 << 29:
            return None   # 64-bit tables of all maps at once
        m = np.stack([e.cpu().view(torch.int16).numpy().view(np.uint16) for e in _maps(case, seed)]).astype(np.int64)
        return _seam64(m)
    if kind in ("batch", "serve"):
        jobs = _jobs(case)
        if sum(_pixel_seams(*j) for j in jobs) > 2e8:
            return None   # minutes in numpy
        return np.concatenate([_carve64(_image(W, H, C, seed * 1000 + k).cpu().numpy(), tw, th)[0].reshape(-1)
                               for k, (W, H, tw, th) in enumerate(jobs)])
    img = _image(case["W"], case["H"], C, seed, case.get("uniform", False)).cpu().numpy()
    if kind in ("seam", "energy"):
        e = _energy64(img.astype(np.int64))
        if kind == "energy":
            return e
        s, c = _seam64(e[None])
        return s[0], c
    k = case["tw"] - case["W"]
    tw = case["W"] - k if kind == "enlarge" else case["tw"]
    if _pixel_seams(case["W"], case["H"], tw, case["th"]) > (1e8 if kind == "forward" else 2e8):
        return None       # minutes in numpy
    out, log, costs, seams = _carve64(img, tw, case["th"], kind == "forward")
    if kind != "enlarge":
        return out, log, costs
    # each seam's column in the input, and the rounded-up mean after every such pixel
    H, W = case["H"], case["W"]
    cols = np.empty((k, H), dtype=np.int32)
    wide = np.empty((H, case["tw"], C), dtype=np.uint8)
    for i in range(H):
        left = list(range(W))
        for t in range(k):
            cols[t, i] = left.pop(int(seams[t][i]))
        row = img[i].astype(np.int64)
        mean = (row + np.concatenate([row[1:], row[-1:]], 0) + 1) >> 1
        at = np.sort(cols[:, i])
        wide[i] = np.insert(row, at + 1, mean[at], axis=0).astype(np.uint8)
    return wide, cols
