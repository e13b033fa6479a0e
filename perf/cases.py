"""Workloads of the light-field renderer as a program drives it through
``Renderer``: light-field frames in every mode, batches of small frames in one
launch, and the set-up of a panel's tables.

A case names its kind ("frame", "batch" or "display"), the panel and, where one
is rendered, the scene and the mode.  ``prepare`` loads the scene and sets the
display up, ``run`` is the call that the program repeats, ``exact`` is the same
result in 64 bits in plain torch."""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as W
from paper_2407_14053_gb300 import Renderer
from paper_2407_14053_gb300 import _binding as B

_TORCH_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


# ------------------------------------------------------------------ cases ---
def _panel(d) -> dict:
    return {"width": d.width, "height": d.height, "views": d.num_views, "pitch": d.pitch_lx,
            "tan": d.tan_slant, "offset": d.offset_k, "span": d.view_span_deg, "fov": d.fov_x_deg,
            "p_w": d.p_w, "rig": d.rig}


def _frame(name: str, display, n: int, sh: int, dtype: str, mode: str, **more) -> dict:
    return {"name": name, "kind": "frame", **_panel(display), "n": n, "sh": sh, "dtype": dtype,
            "mode": mode, **more}


def listed() -> list:
    tiny, p1080, p4k, p8k = (W.WORKLOADS[k] for k in ("tiny", "1080p", "4k", "8k"))
    return [
        # the smallest frame anyone renders: a thumbnail panel, launch-bound
        _frame("directl-tiny", tiny.display, tiny.scene.n, 0, "f32", "directl"),
        # an odd-sized panel on the off-axis rig, a small half-precision scene
        # without the highest SH band: previews while a scene is edited
        _frame("directl-ragged", W.Display(955, 541, 37, 6.7, -0.21, 1.5, rig=1), 41_003, 2, "f16",
               "directl"),
        # the desktop panel at full precision
        _frame("directl-1080p", p1080.display, p1080.scene.n, 3, "f32", "directl"),
        # the calibrated 7.9-inch portrait panel of the paper's Table 1, a
        # scene whose size is no multiple of anything
        _frame("directl-7.9in", W.PAPER_PANELS["7.9in"], 500_009, 3, "f16", "directl"),
        # the headline: a 4K panel, one million Gaussians
        _frame("directl-4k", p4k.display, p4k.scene.n, 3, "bf16", "directl"),
        # the largest: an 8K panel, 100 views, three million Gaussians
        _frame("directl-8k", p8k.display, p8k.scene.n, 3, "bf16", "directl"),
        # the standard paradigm (every view, then the interweave), which a
        # program runs for comparison and for panels without repurposing
        _frame("standard-1080p", p1080.display, p1080.scene.n, 3, "f32", "standard"),
        _frame("standard-4k", p4k.display, p4k.scene.n, 3, "bf16", "standard"),
        # its low-resolution variant: views at 800x450, upsampled
        _frame("standard-4k-lr", p4k.display, p4k.scene.n, 3, "bf16", "standard", view_w=800,
               view_h=450),
        # ray-order rendering (the paper's Alg. 3) of the desktop panel
        _frame("raycast-1080p", p1080.display, p1080.scene.n, 3, "f32", "raycast", heap=128),
        # sixteen small frames in one captured launch: a server's thumbnails
        {"name": "batch-16", "kind": "batch", "slots": 16, "sh": 3, "dtype": "f16", "n_min": 5000,
         "n_max": 40_000},
        # a panel's tables (view map, repurposing, ray table): what a program
        # pays when a panel is attached or calibrated again
        {"name": "display-4k", "kind": "display", **_panel(p4k.display)},
    ]


def _log_uniform(rng, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_panel(rng, max_w: int) -> W.Display:
    w = int(round(_log_uniform(rng, 160, max_w)))
    h = max(90, int(round(w * rng.choice([9 / 16, 9 / 16, 3 / 4, 4 / 3, 5 / 8]))))
    if w * h > max_w * max_w * 9 // 16:
        h = max_w * max_w * 9 // 16 // w
    tan = rng.choice([1, 1, 1, -1]) * rng.uniform(0.05, 0.3)
    return W.Display(w, h, rng.randint(8, 64), round(rng.uniform(4.0, 12.0), 4), round(tan, 5),
                     round(rng.uniform(0.0, 20.0), 4), round(rng.uniform(20.0, 60.0), 1),
                     round(rng.uniform(25.0, 60.0), 1), rng.choice([1, 2, 2, 3]), 1, 0,
                     rng.choice([0, 0, 1]))


def _draw_n(rng, d, most: int) -> int:
    return int(min(most, max(500, d.width * d.height * _log_uniform(rng, 0.02, 0.4))))


def draw(rng) -> dict:
    kind = rng.choices(["directl", "required_only", "standard", "standard_lr", "standard_sr",
                        "raycast", "batch", "display"], [8, 2, 2, 1, 1, 2, 2, 2])[0]
    if kind == "batch":
        lo = int(_log_uniform(rng, 1000, 10_000))
        return {"kind": "batch", "slots": rng.randint(2, 24), "sh": rng.randint(0, 3),
                "dtype": rng.choice(["f32", "bf16", "f16"]), "n_min": lo,
                "n_max": int(lo * rng.uniform(1.0, 8.0))}
    if kind == "display":
        return {"kind": "display", **_panel(_draw_panel(rng, 3840))}
    d = _draw_panel(rng, {"raycast": 1600}.get(kind, 3840))
    n = _draw_n(rng, d, 1_000_000 if kind in ("directl", "required_only") else 400_000)
    if kind.startswith("standard"):
        d = d.replace(num_views=min(d.num_views, 45))
    c = _frame("", d, n, rng.randint(0, 3), rng.choice(["f32", "bf16", "f16"]),
               "standard" if kind == "standard_lr" else kind)
    del c["name"]
    if kind == "standard_lr":
        f = rng.uniform(0.15, 0.6)
        c["view_w"], c["view_h"] = max(16, int(d.width * f)), max(16, int(d.height * f))
    if kind == "raycast":
        c["heap"] = rng.choice([32, 128, 256])
    return c


# ----------------------------------------------------------------- inputs ---
def _display(case: dict, seed: int) -> W.Display:
    d = W.Display(case["width"], case["height"], case["views"], case["pitch"], case["tan"],
                  case["offset"], case["span"], case["fov"], case["p_w"], 1, 0, case["rig"])
    if case["kind"] == "display":  # every unit of a panel has a calibration of its own
        rng = np.random.default_rng(seed)
        d = d.replace(pitch_lx=d.pitch_lx * (1.0 + 0.002 * rng.uniform(-1, 1)),
                      tan_slant=d.tan_slant * (1.0 + 0.01 * rng.uniform(-1, 1)),
                      offset_k=d.offset_k + rng.uniform(0, 1))
    return d


def _scene(n: int, sh: int, seed: int) -> dict:
    """The distributions of ``workloads.make_scene`` (the clustered layout,
    and the uniform one for the smallest scenes), drawn on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device="cuda")

    if n <= 4000:
        mean = 2.0 * uniform(n, 3) - 1.0
    else:
        core = 0.5 * normal(n, 3)
        back = 6.0 * uniform(n, 3) - 3.0
        mean = torch.where(uniform(n, 1) < 0.2, back, core)
    q = normal(n, 4)
    coef = torch.empty(n, (sh + 1) ** 2, 3, device="cuda")
    coef[:, 0] = (uniform(n, 3) - 0.5) / (0.5 / math.sqrt(math.pi))
    coef[:, 1:] = 0.1 * normal(n, (sh + 1) ** 2 - 1, 3)
    return {"mean": mean, "log_scale": (-3.0 - 0.5 * math.log(n / 2000.0)) + 0.5 * normal(n, 3),
            "rot_wxyz": q / q.norm(dim=1, keepdim=True), "opacity_logit": normal(n), "sh": coef,
            "sh_degree": sh}


def _pose(seed: int) -> np.ndarray:
    return W.light_field_centre(4.0, float(np.random.default_rng(seed).uniform(-5.0, 5.0)))


def _load(r: Renderer, scene: dict, dtype: str) -> int:
    host = {k: (v.cpu().numpy() if torch.is_tensor(v) else v) for k, v in scene.items()}
    return r.load_gaussians(host, dtype)


def _batch_frames(case: dict, seed: int) -> list:
    """(display, Gaussians, scene seed, pose) of every slot."""
    small = W.WORKLOADS["tiny"].display
    displays = [small, small.replace(width=480, height=270)]
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["slots"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"] + 1)))))
        out.append((displays[i % 2], n, seed * 64 + i, _pose(seed * 64 + i)))
    return out


def prepare(case: dict, seed: int) -> dict:
    r = Renderer(0)
    if case["kind"] == "display":
        d = _display(case, seed)
        # (view, row, col) of up to 3 w h rays; the rows past the panel's rays stay -1
        rays = torch.full((3 * d.width * d.height, 3), -1, dtype=torch.int32, device="cuda")
        return {"kind": "display", "r": r, "display": d, "rays": rays}
    if case["kind"] == "batch":
        frames = _batch_frames(case, seed)
        dids = {}
        plans, outs, poses = [], [], []
        for d, n, sseed, pose in frames:
            if d not in dids:
                dids[d] = r.set_display(d)
            sid = _load(r, _scene(n, case["sh"], sseed), case["dtype"])
            plans.append((sid, dids[d], None, pose))
            outs.append(torch.empty(d.height, d.width, 3, device="cuda"))
            poses.append(pose)
        batch = r.batch(plans)
        for i, (sid, did, _, pose) in enumerate(plans):
            batch.assign(i, sid, did, outs[i])
            batch.set_pose(i, pose)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            batch.capture()
        return {"kind": "batch", "r": r, "batch": batch, "outs": outs, "poses": poses}
    did = r.set_display(_display(case, seed))
    sid = _load(r, _scene(case["n"], case["sh"], seed), case["dtype"])
    if "view_w" in case:
        r.set_standard_view_size(case["view_w"], case["view_h"])
    if "heap" in case:
        r.set_heap_capacity(case["heap"])
    out = torch.empty(case["height"], case["width"], 3, device="cuda")
    return {"kind": "frame", "r": r, "sid": sid, "did": did, "pose": _pose(seed),
            "mode": case["mode"], "out": out}


def run(state: dict):
    r = state["r"]
    if state["kind"] == "frame":
        return r.render(state["sid"], state["did"], state["pose"], state["mode"], state["out"])
    if state["kind"] == "batch":
        for i, pose in enumerate(state["poses"]):
            state["batch"].set_pose(i, pose)
        state["batch"].launch()
        return state["outs"]
    d = state["display"]
    did = r.set_display(d)
    rays = state["rays"]
    stream = torch.cuda.current_stream().cuda_stream
    # unsigned 16- and 32-bit tables, held in signed tensors of the same width
    view_map = torch.empty(d.height, 3 * d.width, dtype=torch.int16, device="cuda")
    source = torch.empty(d.height, d.width, 3, dtype=torch.int32, device="cuda")
    ray_of = torch.empty(d.height, d.width, 3, dtype=torch.int32, device="cuda")
    B.dl_get_view_map(r.ctx, did, view_map.data_ptr(), 1, stream)
    B.dl_get_subpixel_map(r.ctx, did, source.data_ptr(), 1, stream)
    B.dl_get_ray_table(r.ctx, did, ray_of.data_ptr(), rays.data_ptr(), 1, stream)
    r.free_display(did)
    return {"view_map": view_map, "source": source, "ray_of": ray_of, "rays": rays}


# ------------------------------------------------------------------- work ---
def _scene_bytes(n: int, sh: int, dtype: str) -> float:
    return n * (12.0 + (8 + 3 * (sh + 1) ** 2) * (4 if dtype == "f32" else 2))


def _frame_work(w, h, views, n, sh, dtype, mode, view_w=0, view_h=0) -> tuple:
    """Bytes: the scene in, the image and the panel's per-subpixel table.
    Operations: about 150 (and 6 an SH coefficient) per Gaussian and view,
    and per ray about 30 contributors of 22 operations (the scenes keep that
    number over n and resolution); DirectL composites about 1.5 rays a pixel,
    the standard paradigm every pixel of every view."""
    rays = {"directl": 1.5, "raycast": 1.5, "required_only": 3.0}.get(mode, 0) * w * h
    if not rays:
        rays = views * (view_w or w) * (view_h or h)
    return (_scene_bytes(n, sh, dtype) + 24.0 * w * h,
            views * n * (150.0 + 6.0 * (sh + 1) ** 2) + rays * 30 * 22.0)


def work(case: dict) -> dict:
    if case["kind"] == "display":  # tables out: 2 + 4 + 4 bytes a subpixel, 12 a ray
        px = case["width"] * case["height"]
        return {"bytes": 30.0 * px + 18.0 * px, "flops": 0.0}
    if case["kind"] == "batch":
        b = f = 0.0
        for d, n, _, _ in _batch_frames(case, 1):
            x, y = _frame_work(d.width, d.height, d.num_views, n, case["sh"], case["dtype"],
                               "directl")
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    b, f = _frame_work(case["width"], case["height"], case["views"], case["n"], case["sh"],
                       case["dtype"], case["mode"], case.get("view_w", 0), case.get("view_h", 0))
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------ 64-bit result ---
_Q32 = 1 << 32
_EMPTY = -1


def _quantise(d) -> tuple:
    def q(x):
        return int(np.rint(x * float(_Q32)))
    return q(3.0 * d.tan_slant), q(d.pitch_lx), q(d.offset_k)


def _d_offset(d) -> torch.Tensor:
    """d_offset (Eq. (1)) of every subpixel, Q32, as (h, 3w)."""
    t3, _, k = _quantise(d)
    x = torch.arange(d.height, device="cuda").unsqueeze(1)
    s = torch.arange(3 * d.width, device="cuda").unsqueeze(0)
    return s * _Q32 + x * t3 - k


def _view_map(d) -> torch.Tensor:
    _, lq, _ = _quantise(d)
    return torch.div(torch.remainder(_d_offset(d), lq) * d.num_views, lq, rounding_mode="floor")


def _repurpose_steps(d) -> float:
    return d.height * d.p_w * d.pitch_lx


def _repurpose(d, V: torch.Tensor) -> torch.Tensor:
    """Alg. 2: source pixel (row * w + column) of every subpixel.  Areas are
    independent; all of them advance together, one filled subpixel a step."""
    _, lq, _ = _quantise(d)
    w, h, S = d.width, d.height, 3 * d.width
    area = torch.div(torch.div(_d_offset(d), lq, rounding_mode="floor"), d.p_w,
                     rounding_mode="floor").reshape(-1)
    area = area - area.min()
    order = torch.sort(area, stable=True).indices
    ends = torch.cumsum(torch.bincount(area), 0)
    V = V.reshape(-1)
    src = torch.full_like(V, _EMPTY)
    ptr = torch.cat([ends.new_zeros(1), ends[:-1]])
    lanes = torch.arange(ends.numel(), device=V.device)
    dx = (5 * d.num_views * (1 << 31)) // lq
    dy = (d.num_views * _Q32 + 3 * lq - 1) // (3 * lq)
    step = 1 if d.tan_slant < 0 else -1
    j = torch.arange(max(dx - 1, 0) * (dy + 1) * 3, device=V.device)
    j_row, j_col, j_ch = j // (3 * (dy + 1)), (j // 3) % (dy + 1), j % 3
    look = torch.arange(16, device=V.device)
    cur = torch.full_like(lanes, _EMPTY)  # subpixel the area's chain stands at
    buf = torch.full((lanes.numel(), 3), _EMPTY, device=V.device, dtype=torch.int64)
    last = order.numel() - 1
    count = 0
    while True:
        if count % 64 == 0 and not bool(((ptr < ends) | (cur != _EMPTY)).any()):
            return src
        count += 1
        # areas without a chain look for their next empty subpixel
        idle = cur == _EMPTY
        at = ptr.unsqueeze(1) + look
        free = (src[order[at.clamp(max=last)]] == _EMPTY) & (at < ends.unsqueeze(1))
        skip = torch.where(free, look, 16).amin(1)
        ptr = torch.where(idle, torch.minimum(ptr + skip, ends), ptr)
        cur = torch.where(idle & (skip < 16), order[ptr.clamp(max=last)], cur)
        live = cur != _EMPTY
        i = cur.clamp(min=0)
        x, y, k = i // S, (i % S) // 3, i % 3
        own = x * w + y
        bk = buf.gather(1, k.unsqueeze(1)).squeeze(1)
        used = bk != _EMPTY
        src[i[live]] = torch.where(used, bk, own)[live]
        is_k = look[:3].unsqueeze(0) == k.unsqueeze(1)
        buf = torch.where(used.unsqueeze(1), torch.where(is_k, _EMPTY, buf),
                          torch.where(is_k, buf, own.unsqueeze(1)))
        r = torch.minimum(x + 2, torch.full_like(x, h - 1)).unsqueeze(1) + j_row
        c = y.unsqueeze(1) + step * j_col
        ok = (r <= torch.minimum(x + dx, torch.full_like(x, h - 1)).unsqueeze(1)) & (c >= 0) & (c < w)
        cand = (r * S + 3 * c + j_ch).clamp(0, S * h - 1)
        hit = ok & (V[cand] == V[i].unsqueeze(1)) & (buf[:, j_ch] != _EMPTY)
        first = torch.where(hit, j, j.numel()).amin(1) if j.numel() else torch.zeros_like(lanes)
        found = first < j.numel()
        nxt = cand.gather(1, first.clamp(max=max(j.numel() - 1, 0)).unsqueeze(1)).squeeze(1) \
            if j.numel() else i
        go = live & found & (area[nxt] == lanes) & (src[nxt] == _EMPTY)
        cur = torch.where(go, nxt, torch.full_like(cur, _EMPTY))
        buf = torch.where(go.unsqueeze(1), buf, torch.full_like(buf, _EMPTY))


def _cameras(d, w: int, pose: np.ndarray) -> list:
    """(world-to-camera rotation, translation, centre, principal shift)."""
    focal = 0.5 * w / math.tan(0.5 * math.radians(d.fov_x_deg))
    depth = -float(pose[:3, 2] @ pose[:3, 3])
    out = []
    for v in range(d.num_views):
        th = 0.0
        if d.num_views > 1:
            th = math.radians(-0.5 * d.view_span_deg + v * d.view_span_deg / (d.num_views - 1))
        T, shift = pose.copy(), 0.0
        if d.rig == 1:
            xv = depth * math.tan(th)
            T[:3, 3] += xv * pose[:3, 0]
            shift = focal * xv / depth
        else:
            c, s = math.cos(-th), math.sin(-th)
            T[:3] = np.array([[c, 0, s], [0, 1, 0], [-s, 0, c]]) @ pose[:3]
        R = T[:3, :3].T
        out.append((torch.tensor(R.copy(), device="cuda"), torch.tensor(-R @ T[:3, 3], device="cuda"),
                    torch.tensor(T[:3, 3].copy(), device="cuda"), shift))
    return out


def _sh(deg: int, dirs: torch.Tensor) -> torch.Tensor:
    """Real spherical harmonics of degree 0 to deg, (m, (deg + 1)^2)."""
    x, y, z = dirs.unbind(-1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if deg >= 1:
        a = math.sqrt(3 / (4 * pi))
        Y += [-a * y, a * z, -a * x]
    if deg >= 2:
        a, b, c = math.sqrt(15 / pi) / 2, math.sqrt(5 / pi) / 4, math.sqrt(15 / pi) / 4
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z, c * (x * x - y * y)]
    if deg >= 3:
        a, b = math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi) / 2
        c, e, f = math.sqrt(21 / (2 * pi)) / 4, math.sqrt(7 / pi) / 4, math.sqrt(105 / pi) / 4
        q = 4 * z * z - x * x - y * y
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * q,
              e * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * q, f * z * (x * x - y * y),
              -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


_TILE = 16
_PAIRS = 1 << 25  # (ray, Gaussian) pairs evaluated together


def _render_rays(scene: dict, dtype: str, d, pose, w: int, h: int, view, row, col, chan,
                 heap: int = 0) -> torch.Tensor:
    """Channel ``chan`` of the rays (view, row, col) of w x h views: the
    projected splats in depth order (heap == 0), or the ``heap`` nearest
    intersections along the ray (Alg. 3)."""
    dt = _TORCH_DTYPE[dtype]
    mean, ls, q, op, sh = (scene[k].to(torch.float32 if k == "mean" else dt).double()
                           for k in ("mean", "log_scale", "rot_wxyz", "opacity_logit", "sh"))
    deg = scene["sh_degree"]
    q = q / q.norm(dim=1, keepdim=True)
    a, b, c, e = q.unbind(1)
    R = torch.stack([1 - 2 * (c * c + e * e), 2 * (b * c - a * e), 2 * (b * e + a * c),
                     2 * (b * c + a * e), 1 - 2 * (b * b + e * e), 2 * (c * e - a * b),
                     2 * (b * e - a * c), 2 * (c * e + a * b), 1 - 2 * (b * b + c * c)],
                    1).reshape(-1, 3, 3)
    cov = (R * torch.exp(2 * ls).unsqueeze(1)) @ R.transpose(1, 2)
    inv = (R * torch.exp(-2 * ls).unsqueeze(1)) @ R.transpose(1, 2) if heap else None
    opac = torch.sigmoid(op)
    vis = opac > 1 / 255
    K = 2 * torch.log((255 * opac).clamp(min=1.0))
    focal = 0.5 * w / math.tan(0.5 * math.radians(d.fov_x_deg))
    lim_x, lim_y = 1.3 * 0.5 * w / focal, 1.3 * 0.5 * h / focal
    ntx = (w + _TILE - 1) // _TILE
    nty = (h + _TILE - 1) // _TILE
    out = torch.zeros(view.numel(), device="cuda", dtype=torch.float64)
    tile = (row // _TILE) * ntx + col // _TILE
    perm = torch.argsort(view * (ntx * nty) + tile)
    bounds = torch.searchsorted(view[perm], torch.arange(d.num_views + 1, device="cuda")).tolist()
    for v, (Rw, t, centre, shift) in enumerate(_cameras(d, w, pose)):
        mine = perm[bounds[v]:bounds[v + 1]]
        if not mine.numel():
            continue
        X = mean @ Rw.T + t
        z = X[:, 2]
        cc = Rw @ cov @ Rw.T  # covariance in the camera's axes
        if heap:
            hx = torch.sqrt((K.unsqueeze(1) * torch.diagonal(cc, dim1=1, dim2=2)).clamp(min=0)) * 1.001
            keep = vis & (z + hx[:, 2] > 0.1)
            near, far = z - hx[:, 2], z + hx[:, 2]
            whole = near < 0.05
            near = torch.where(whole, 0.05, near)
            lo, hi = X - hx, X + hx
            box = []
            for ax, half, size, sf in ((0, 0.5 * w, w, shift), (1, 0.5 * h, h, 0.0)):
                m0 = focal * torch.minimum(lo[:, ax] / near, lo[:, ax] / far) + half + sf
                m1 = focal * torch.maximum(hi[:, ax] / near, hi[:, ax] / far) + half + sf
                box += [torch.where(whole, -1.0, m0 - 0.01), torch.where(whole, float(size), m1 + 0.01)]
            c0, c1, r0, r1 = box
        else:
            zs = torch.where(z > 0.2, z, 1.0)
            sz = shift / focal
            xz = (X[:, 0] / zs).clamp(-lim_x - sz, lim_x - sz)
            yz = (X[:, 1] / zs).clamp(-lim_y, lim_y)
            J = torch.zeros(z.numel(), 2, 3, device="cuda", dtype=torch.float64)
            J[:, 0, 0] = J[:, 1, 1] = focal / zs
            J[:, 0, 2], J[:, 1, 2] = -focal / zs * xz, -focal / zs * yz
            s2 = J @ cc @ J.transpose(1, 2)
            sxx, sxy, syy = s2[:, 0, 0] + 0.3, s2[:, 0, 1], s2[:, 1, 1] + 0.3
            det = sxx * syy - sxy * sxy
            keep = vis & (z > 0.2) & (det > 0)
            det = torch.where(keep, det, 1.0)
            u = focal * X[:, 0] / zs + 0.5 * w + shift
            vv = focal * X[:, 1] / zs + 0.5 * h
            rx, ry = torch.sqrt(K * sxx) + 0.01, torch.sqrt(K * syy) + 0.01
            c0, c1, r0, r1 = u - rx, u + rx, vv - ry, vv + ry
        keep = keep & (c1 >= 0) & (r1 >= 0) & (c0 <= w - 1) & (r0 <= h - 1)
        g = keep.nonzero().squeeze(1)
        if not g.numel():
            continue
        g = g[torch.argsort(z[g], stable=True)]
        tx0 = (c0[g].clamp(min=0) / _TILE).long()
        tx1 = (c1[g].clamp(max=w - 1) / _TILE).long()
        ty0 = (r0[g].clamp(min=0) / _TILE).long()
        ty1 = (r1[g].clamp(max=h - 1) / _TILE).long()
        nt = (tx1 - tx0 + 1) * (ty1 - ty0 + 1)
        o = torch.repeat_interleave(torch.arange(g.numel(), device="cuda"), nt)
        k = torch.arange(o.numel(), device="cuda") - (torch.cumsum(nt, 0) - nt)[o]
        span = (tx1 - tx0 + 1)[o]
        kt = (ty0[o] + k // span) * ntx + tx0[o] + k % span
        kt, by = torch.sort(kt, stable=True)  # by tile, then depth
        lists = o[by]
        start = torch.searchsorted(kt, torch.arange(ntx * nty + 1, device="cuda"))
        if not heap:
            dirs = mean[g] - centre
            Y = _sh(deg, dirs / dirs.norm(dim=1, keepdim=True))
            colour = (torch.einsum("gc,gcx->gx", Y, sh[g]) + 0.5).clamp(min=0)
        tl = tile[mine]
        nr = start[tl + 1] - start[tl]
        cum = torch.cumsum(nr, 0)
        first = 0
        while first < mine.numel():
            base = int(cum[first - 1]) if first else 0
            end = max(first + 1, int(torch.searchsorted(cum, base + _PAIRS, right=True)))
            ray = torch.repeat_interleave(torch.arange(first, end, device="cuda"), nr[first:end])
            pos = torch.arange(ray.numel(), device="cuda") + base - (cum - nr)[ray]
            gi = lists[start[tl[ray]] + pos]
            ids = mine[ray]
            px, py = col[ids].double(), row[ids].double()
            if heap:
                gg = g[gi]
                dc = torch.stack([(px - 0.5 * w - shift) / focal, (py - 0.5 * h) / focal,
                                  torch.ones_like(px)], 1) @ Rw
                dc = dc / dc.norm(dim=1, keepdim=True)
                S = inv[gg]
                m = mean[gg] - centre
                Sd = (S @ dc.unsqueeze(2)).squeeze(2)
                tt = (m * Sd).sum(1) / (dc * Sd).sum(1)
                p = tt.unsqueeze(1) * dc - m
                alpha = (opac[gg] * torch.exp(-0.5 * (p * (S @ p.unsqueeze(2)).squeeze(2)).sum(1)))
                alpha = alpha.clamp(max=0.99)
                ok = ((alpha >= 1 / 255) & (tt > 0.2)).nonzero().squeeze(1)
                ok = ok[torch.argsort(tt[ok], stable=True)]
                ok = ok[torch.sort(ray[ok], stable=True).indices]
                rr = ray[ok]
                rank = torch.arange(ok.numel(), device="cuda") - torch.searchsorted(rr, rr)
                ok = ok[rank < heap]
                Y = _sh(deg, dc[ok])
                s = sh[gg[ok]].gather(2, chan[ids[ok]].reshape(-1, 1, 1).expand(-1, Y.shape[1], 1))
                value = ((Y * s.squeeze(2)).sum(1) + 0.5).clamp(min=0)
            else:
                gg = g[gi]
                dxp, dyp = px - u[gg], py - vv[gg]
                power = (syy[gg] * dxp * dxp - 2 * sxy[gg] * dxp * dyp + sxx[gg] * dyp * dyp) / det[gg]
                alpha = (opac[gg] * torch.exp(-0.5 * power)).clamp(max=0.99)
                ok = (alpha >= 1 / 255).nonzero().squeeze(1)
                value = colour[gi[ok], chan[ids[ok]]]
            al, rr = alpha[ok], ray[ok] - first
            lg = torch.cumsum(torch.log1p(-al), 0)
            before = lg - torch.log1p(-al)
            head = torch.searchsorted(rr, rr)  # first contributor of the pair's ray
            T = torch.exp(before - before[head])
            add = torch.where(T * (1 - al) >= 1e-4, al * T * value, 0.0)
            out[mine[first:end]] = out.new_zeros(end - first).index_add_(0, rr, add)
            first = end
    return out


def _exact_frame(scene, dtype, d, pose, mode, view_w=0, view_h=0, heap=0):
    w, h = d.width, d.height
    V = _view_map(d).reshape(-1)
    i = torch.arange(3 * w * h, device="cuda")
    chan = i % 3
    if view_w and mode == "standard":
        row, col = i // (3 * w), (i // 3) % w
        ny, nx = row * view_h, col * view_w
        y0, x0 = ny // h, nx // w
        fy, fx = (ny - y0 * h).double() / h, (nx - x0 * w).double() / w
        y1, x1 = (y0 + 1).clamp(max=view_h - 1), (x0 + 1).clamp(max=view_w - 1)
        out = 0.0
        for yy, xx, wt in ((y0, x0, (1 - fy) * (1 - fx)), (y0, x1, (1 - fy) * fx),
                           (y1, x0, fy * (1 - fx)), (y1, x1, fy * fx)):
            out = out + wt * _render_rays(scene, dtype, d, pose, view_w, view_h, V, yy, xx, chan)
        return out.reshape(h, w, 3)
    src = i // 3 if mode in ("standard", "required_only") else _repurpose(d, V)
    return _render_rays(scene, dtype, d, pose, w, h, V, src // w, src % w, chan,
                        heap if mode == "raycast" else 0).reshape(h, w, 3)


def exact(case: dict, seed: int):
    if case["kind"] == "display":
        return None  # whole numbers throughout
    if case["kind"] == "batch":
        # Alg. 2 of the two panels takes seconds, so do sixteen frames
        return [_exact_frame(_scene(n, case["sh"], s), case["dtype"], d, pose, "directl")
                if i < 4 else None for i, (d, n, s, pose) in enumerate(_batch_frames(case, seed))]
    d = _display(case, seed)
    mode = case["mode"]
    if mode in ("directl", "standard_sr", "raycast") and _repurpose_steps(d) > 26_000:
        return None  # Alg. 2 is a serial walk down every area: over 20 s from here
    if mode == "raycast" and d.width * d.height > 400_000:
        return None  # the pairs' 3 x 3 matrices in 64 bits: over 20 s
    return _exact_frame(_scene(case["n"], case["sh"], seed), case["dtype"], d, _pose(seed), mode,
                        case.get("view_w", 0), case.get("view_h", 0), case.get("heap", 0))
