"""What the raycaster's performance is measured on: listed cases, cases drawn from the same
ranges, their inputs, one pass through the public entry points, the work a pass cannot do
without, and the outputs in 64 bits from plain torch.

Kinds of case
  frame    one amr_render of one view (the framework's main path)
  batch    one amr_render_batch of many views of uneven sizes
  learned  one amr_render with the learned segment proposal installed
  log      log_segments over a few poses (what the proposal is trained on)
  train    one minibatch of the proposal's training: loss, gradient, Adam
  predict  the proposal's forward pass over logged segments

Datasets (seeded; the field, the boxes, the camera and the transfer function all follow the
seed): "tiny" 2 levels, 12 patches, sum of Gaussians; "mid" a 64^3 root and 4 levels;
"large" a 128^3 root and 5 levels (about 1.3e8 cells, the size most figures are quoted at);
"deep" a 128^3 root and 8 levels, each refined level capped.  The last three are lognormal
fields refined on their density peaks, fine patches straddling coarse ones.
"""
import math
import types

import numpy as np
import torch

import paper_1212_3333_gb300 as amr
from paper_1212_3333_gb300 import proposal

DEV = "cuda"

# per dataset: root cells per axis, level-0 patch, levels, growth of the refinement
# threshold per level, cap of cells per refined level, and for work(): cells in all, leaves a
# ray crosses and samples it takes (means over orbit views)
DATA = {
    "tiny": dict(n0=32, levels=2, cells=6.4e4, leaves=3.2, samples=39.0),
    "mid": dict(n0=64, patch0=16, levels=4, growth=2.25, cap=None,
                cells=1.55e7, leaves=11.0, samples=230.0),
    "large": dict(n0=128, patch0=32, levels=5, growth=2.25, cap=None,
                  cells=1.33e8, leaves=22.0, samples=480.0),
    "deep": dict(n0=128, patch0=32, levels=8, growth=1.0, cap=6_000_000,
                 cells=3.7e7, leaves=15.0, samples=190.0),
}
CELL_BYTES = {"f32": 4, "f16": 2, "bf16": 2}
MLP = [(64, 12), (64,), (64, 64), (64,), (64, 64), (64,), (1, 64), (1,)]
MLP_PARAMS = sum(math.prod(s) for s in MLP)
MLP_MACS = 12 * 64 + 2 * 64 * 64 + 64
EXACT_SAMPLES = 1.6e8  # largest plain frame whose 64-bit image is computed (about 20 s)


def _frame(name, data, width, height, **options):
    case = dict(kind="frame", data=data, width=width, height=height, cells="f32", storage="ptr",
                gradient=False, halo=1, maxbrick=False, shade=1, skip=0, lod=0.0, shadow=0)
    case.update(options)
    return dict(case, name=name) if name else case


FULL = dict(gradient=True, halo=2, maxbrick=True)  # every brick the library can keep


def listed():
    return [
        # the smallest call: a two-level hierarchy, plain compositing, default build
        _frame("frame_256_tiny_plain", "tiny", 256, 256, shade=0),
        # an interactive window on a medium hierarchy in the packed atlas
        _frame("frame_512_mid_atlas", "mid", 512, 512, storage="atlas_linear", gradient=True),
        # shaded with a point light inside the data: secondary rays
        _frame("frame_393x371_mid_shadow", "mid", 393, 371, gradient=True, shadow=1),
        # the usual picture of the large hierarchy, shaded, at three sizes
        _frame("frame_640x479_large", "large", 640, 479, **FULL),
        _frame("frame_1024_large", "large", 1024, 1024, **FULL),
        _frame("frame_2048_large", "large", 2048, 2048, **FULL),
        # 16-bit cells: a plain overview frame, and the deep hierarchy shaded
        _frame("frame_1917x1083_large_f16", "large", 1917, 1083, cells="f16", shade=0, halo=2,
               maxbrick=True),
        _frame("frame_1500x1100_deep_bf16", "deep", 1500, 1100, cells="bf16", **FULL),
        # a contact sheet of views of uneven sizes with four transfer functions
        dict(name="batch_32_large", kind="batch", data="large", views=32, lo=64, hi=512, **FULL),
        # the learned proposal: logging what it is trained on, a training step at the
        # minibatch the trainer uses, and a frame that it thins out
        dict(name="log_8x96_large", kind="log", data="large", poses=8, size=96, keep=0.3, **FULL),
        dict(name="train_16384", kind="train", rows=1 << 20, batch=16384),
        dict(name="learned_1024_large", kind="learned", data="large", width=1024, height=1024,
             shade=1, mode=2, factor=32, tau=1e-2, **FULL),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["frame", "batch", "learned", "log", "train", "predict"],
                       weights=[10, 2, 1, 1, 2, 1])[0]
    data = rng.choice(["tiny", "mid", "mid", "large", "deep"])
    if kind == "frame":
        width, height = _log_uniform(rng, 150, 2048), _log_uniform(rng, 150, 2048)
        storage = rng.choice(["ptr", "ptr", "ptr", "atlas_linear"])
        shade = rng.choice([0, 1, 1])
        shadow = 1 if shade and data in ("tiny", "mid") and rng.random() < 0.15 else 0
        if shadow:
            width, height = min(width, 400), min(height, 400)
        cells = "f32" if shadow else rng.choice(["f32", "f32", "f16", "bf16"])
        return _frame(None, data, width, height, cells=cells, storage=storage,
                      gradient=bool(shade and rng.random() < 0.7), halo=rng.choice([1, 2]),
                      maxbrick=storage == "ptr" and rng.random() < 0.6, shade=shade,
                      skip=rng.choice([0, 0, 1]), shadow=shadow,
                      lod=rng.choice([0.0, 0.0, 0.0, 2.0]))
    if kind == "batch":
        lo = _log_uniform(rng, 32, 200)
        return dict(kind=kind, data=data, views=rng.randint(2, 48), lo=lo,
                    hi=lo + rng.randint(0, 400), gradient=rng.random() < 0.7,
                    halo=rng.choice([1, 2]), maxbrick=rng.random() < 0.7)
    if kind == "learned":
        return dict(kind=kind, data=data, width=_log_uniform(rng, 200, 1400),
                    height=_log_uniform(rng, 200, 1400), shade=rng.choice([0, 1, 1]),
                    mode=rng.choice([1, 2, 2]), factor=rng.choice([16, 32, 64]),
                    tau=10.0 ** rng.uniform(-4, -2), **FULL)
    if kind == "log":
        return dict(kind=kind, data=data, poses=rng.randint(1, 16), size=_log_uniform(rng, 48, 160),
                    keep=round(rng.uniform(0.05, 1.0), 3), gradient=False, halo=rng.choice([1, 2]),
                    maxbrick=False)
    if kind == "train":
        return dict(kind=kind, rows=_log_uniform(rng, 1 << 17, 1 << 21),
                    batch=_log_uniform(rng, 300, 1 << 17))
    return dict(kind=kind, rows=_log_uniform(rng, 1000, 1 << 23))


# ----------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------


def _fill_lognormal(rng, d, modes=512):
    """Boxes level by level and exp(Gaussian random field) at their cell centres: `modes`
    plane waves, |k| uniform up to half the root's cells per axis, in separable FP32 products."""
    kmag = rng.uniform(2 * math.pi, math.pi * d["n0"], size=modes)
    cost = rng.uniform(-1.0, 1.0, size=modes)
    phi = rng.uniform(0.0, 2 * math.pi, size=modes)
    sint = np.sqrt(1.0 - cost ** 2)
    k = np.stack([kmag * sint * np.cos(phi), kmag * sint * np.sin(phi), kmag * cost])
    phase = np.stack([np.zeros(modes), np.zeros(modes), rng.uniform(0, 2 * math.pi, size=modes)])
    k, phase = (torch.as_tensor(v, device=DEV) for v in (k, phase))
    n0, p0 = d["n0"], d["patch0"]
    g = np.arange(0, n0, p0)
    lo = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)[:, ::-1]
    boxes = np.concatenate([lo, lo + p0], 1)
    level_boxes, level_cells = [], []
    for level in range(d["levels"]):
        n_l = n0 << level
        x = (torch.arange(n_l, dtype=torch.float64, device=DEV) + 0.5) / n_l
        wave = []
        for a in range(3):
            arg = k[a][:, None] * x[None] + phase[a][:, None]
            wave.append((torch.cos(arg).float(), torch.sin(arg).float()))
        size = (boxes[:, 3:] - boxes[:, :3]).prod(1)
        start = np.concatenate([[0], np.cumsum(size)])
        cells = torch.empty(int(start[-1]), device=DEV)
        for b, s in zip(boxes.tolist(), start.tolist()):
            (xr, xi), (yr, yi), (zr, zi) = [(w[0][:, b[a]:b[3 + a]], w[1][:, b[a]:b[3 + a]])
                                            for a, w in enumerate(wave)]
            re = yr[:, :, None] * xr[:, None] - yi[:, :, None] * xi[:, None]
            im = yr[:, :, None] * xi[:, None] + yi[:, :, None] * xr[:, None]
            v = zr.T @ re.reshape(modes, -1) - zi.T @ im.reshape(modes, -1)
            cells[s:s + v.numel()] = v.reshape(-1)
        cells.mul_(math.sqrt(2.0 / modes)).exp_()
        level_boxes.append(boxes)
        level_cells.append(cells)
        if level + 1 == d["levels"]:
            break
        threshold = 4.0 * math.exp(0.5) * d["growth"] ** level
        coarse = _cluster(cells, boxes, start, n_l, threshold)
        while d["cap"] and len(coarse) and 8 * (coarse[:, 3:] - coarse[:, :3]).prod(1).sum() > d["cap"]:
            threshold *= 1.12
            coarse = _cluster(cells, boxes, start, n_l, threshold)
        if not len(coarse):
            break
        boxes = 2 * coarse
    return level_boxes, level_cells


def _cluster(cells, boxes, start, n_l, threshold, tile=32, least=4):
    """The cells above the threshold, one box per tile of a grid shifted by half a tile: the
    bounding box of the tile's cells grown by one, at least `least` wide inside its tile."""
    at = torch.nonzero(cells > threshold)[:, 0]
    if not len(at):
        return np.zeros((0, 6), dtype=np.int64)
    first, bx = (torch.as_tensor(np.ascontiguousarray(v), device=DEV) for v in (start, boxes))
    p = torch.searchsorted(first, at, right=True) - 1
    r, nx, ny = at - first[p], bx[p, 3] - bx[p, 0], bx[p, 4] - bx[p, 1]
    ijk = torch.stack([r % nx, r // nx % ny, r // (nx * ny)], 1) + bx[p, :3]
    t = (ijk + tile // 2) // tile
    m = n_l // tile + 2
    key, which = torch.unique(t[:, 0] + m * (t[:, 1] + m * t[:, 2]), return_inverse=True)
    at3 = which[:, None].expand(-1, 3)
    lo = torch.full((len(key), 3), n_l, device=DEV, dtype=torch.int64).scatter_reduce(0, at3, ijk, "amin")
    hi = torch.full((len(key), 3), -1, device=DEV, dtype=torch.int64).scatter_reduce(0, at3, ijk, "amax")
    tt = torch.stack([key % m, key // m % m, key // (m * m)], 1).cpu().numpy()
    tlo, thi = np.maximum(tt * tile - tile // 2, 0), np.minimum(tt * tile + tile // 2, n_l)
    lo = np.maximum(lo.cpu().numpy() - 1, tlo)
    hi = np.minimum(hi.cpu().numpy() + 2, thi)
    for _ in range(least):
        short = hi - lo < least
        up = short & (hi < thi)
        hi = hi + up
        lo = lo - (short & ~up & (lo > tlo))
    return np.concatenate([lo, hi], 1)


def _tiny_boxes(rng):
    """Eight 16^3 patches and four level-1 patches of 16-24 cells, one astride two parents."""
    g = np.array([[i, j, k] for k in (0, 16) for j in (0, 16) for i in (0, 16)])
    fine = []
    while len(fine) < 4:
        size = rng.integers(16, 25, size=3)
        lo = np.array([int(rng.integers(0, 64 - s + 1)) for s in size])
        if not fine:
            lo[0] = int(rng.integers(32 - size[0] + 1, 32))
        b = np.concatenate([lo, lo + size])
        if all(any(b[3 + a] <= f[a] or f[3 + a] <= b[a] for a in range(3)) for f in fine):
            fine.append(b)
    return [np.concatenate([g, g + 16], 1), np.array(fine)]


def _fill_tiny(rng, d):
    boxes = _tiny_boxes(rng)
    c, s, a = rng.uniform(size=(8, 3)), rng.uniform(0.05, 0.15, size=8), rng.uniform(0.2, 1.0, size=8)
    cells = []
    for level, bs in enumerate(boxes):
        got = []
        for b in bs:
            xs = [(torch.arange(int(b[q]), int(b[3 + q]), dtype=torch.float64, device=DEV) + 0.5) /
                  (d["n0"] << level) for q in range(3)]
            v = 0.0
            for m in range(8):
                e = [torch.exp(-(xs[q] - c[m, q]) ** 2 / (2 * s[m] ** 2)) for q in range(3)]
                v = v + a[m] * e[2][:, None, None] * e[1][None, :, None] * e[0][None, None]
            got.append(v.float().reshape(-1))
        cells.append(torch.cat(got))
    return boxes, cells


def _hierarchy(name, seed):
    """The hierarchy a program has loaded (host arrays), and its cells on the device."""
    d = DATA[name]
    rng = np.random.default_rng([seed, 11])
    boxes, cells = _fill_tiny(rng, d) if name == "tiny" else _fill_lognormal(rng, d)
    level = np.concatenate([np.full(len(b), i, dtype=np.int32) for i, b in enumerate(boxes)])
    box = np.concatenate(boxes).astype(np.int64)
    flat = torch.cat(cells)
    size = (box[:, 3:] - box[:, :3]).prod(1)
    start = np.concatenate([[0], np.cumsum(size)])
    # transfer functions span the smallest cell to the 99.9th percentile (deep: of level 0,
    # so that its dense regions are opaque)
    part = cells[0] if name == "deep" else flat[:: max(1, len(flat) // 1_000_000)]
    high = torch.sort(part)[0][min(len(part) - 1, int(0.999 * len(part)))]
    return types.SimpleNamespace(num_levels=len(boxes), ratio=2, domain_lo=np.zeros(3),
                                 h0=np.full(3, 1.0 / d["n0"]), patch_level=level, patch_box=box,
                                 flat=flat, start=start, vmin=float(flat.min()), vmax=float(high),
                                 n0=d["n0"])


def _context(case, hier):
    host = hier.flat.cpu().numpy()
    n = hier.patch_box[:, 3:] - hier.patch_box[:, :3]
    hier.data = [host[s:e].reshape(k[2], k[1], k[0])
                 for s, e, k in zip(hier.start[:-1], hier.start[1:], n)]
    ctx = amr.from_hierarchy(hier, case.get("cells", "f32"))
    ctx.amr_build_kdtree(case.get("storage", "ptr"), gradient=case["gradient"], halo=case["halo"],
                         maxbrick=case["maxbrick"])
    hier.data = None
    return ctx


def _camera(rng, width, height):
    """A view of the whole domain from distance 2, any azimuth, elevation up to 60 degrees."""
    az, el = rng.uniform(0, 2 * math.pi), math.radians(rng.uniform(-60, 60))
    out = np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
    right = np.cross(-out, [0.0, 0.0, 1.0])
    right /= np.linalg.norm(right)
    return types.SimpleNamespace(eye=0.5 + 2.0 * out, fwd=-out, right=right,
                                 up=np.cross(right, -out),
                                 tan_half_fov_y=math.tan(math.radians(20.0)), width=width,
                                 height=height)


def _transfer(rng, n=256):
    """A colour ramp whose opacity starts at 8-15 % of the range."""
    t = np.linspace(0.0, 1.0, n)[:, None]
    c0, c1, a = rng.uniform(0, 0.6, 3), rng.uniform(0.3, 1.0, 3), rng.uniform(0.08, 0.15)
    return np.concatenate([(1 - t) * c0 + t * c1, np.clip((t - a) / (1 - a), 0, 1)], 1).astype(np.float32)


def _options(case, hier):
    p = dict(vmin=hier.vmin, vmax=hier.vmax, shade=case.get("shade", 1), skip=case.get("skip", 0),
             lod_pixels=case.get("lod", 0.0))
    if case.get("shadow"):
        p.update(shadow=1, light_step=0.5 / hier.n0)
    return p


def _views(case, rng):
    """Cameras of uneven square sizes (the sizes belong to the case, the poses to the seed)."""
    sides = np.random.default_rng(case["views"]).integers(case["lo"], case["hi"] + 1, size=case["views"])
    return [_camera(rng, int(s), int(s)) for s in sides], [v % 4 for v in range(case["views"])]


_network = {}


def _proposal_weights():
    """A network that has learned how much a segment contributes from its length, its leaf's
    largest value and the opacity before it (plain torch, a fixed seed: the same weights
    whatever the library's own training gives)."""
    if "w" not in _network:
        gen = torch.Generator().manual_seed(3)
        net = [(torch.randn(s, generator=gen) * math.sqrt(2.0 / s[1]) if len(s) == 2
                else torch.zeros(s)).to(DEV).requires_grad_() for s in MLP]
        x = torch.rand((16384, 12), generator=gen).to(DEV)
        x[:, 3:6] = x[:, :3] + 0.04 * (x[:, 3:6] - 0.5)
        x[:, 10:] = 2 * x[:, 10:] - 1
        length = (x[:, 3:6] - x[:, :3]).norm(dim=1)
        y = (1 - x[:, 9]) * (1 - torch.exp(-12.0 * length * x[:, 8] ** 4))
        opt = torch.optim.Adam(net, lr=3e-3)
        for _ in range(250):
            h = x
            for w, b in zip(net[0:6:2], net[1:6:2]):
                h = torch.relu(h @ w.T + b)
            loss = torch.nn.functional.binary_cross_entropy_with_logits((h @ net[6].T + net[7])[:, 0], y)
            opt.zero_grad()
            loss.backward()
            opt.step()
        _network["w"] = torch.cat([w.detach().reshape(-1) for w in net]).cpu().numpy()
    return _network["w"]


def _segments(seed, rows):
    """Features and targets as logging gives them, and a network in training."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.rand((rows, 12), generator=gen, device=DEV)
    x[:, 3:6] = x[:, :3] + 0.05 * (x[:, 3:6] - 0.5)
    x[:, 6] = torch.floor(5 * x[:, 6]) / 4
    x[:, 9] *= x[:, 9]
    x[:, 10:] = 2 * x[:, 10:] - 1
    y = (1 - x[:, 9]) * (1 - torch.exp(-20 * (x[:, 3:6] - x[:, :3]).norm(dim=1) * x[:, 8] ** 3))
    rng = np.random.default_rng([seed, 5])
    w = np.concatenate([(rng.normal(0, math.sqrt(2.0 / s[1]), s) if len(s) == 2 else
                         rng.normal(0, 0.05, s)).ravel() for s in MLP]).astype(np.float32)
    return x, y, w


def prepare(case, seed):
    kind, s = case["kind"], types.SimpleNamespace(case=case)
    rng = np.random.default_rng([seed, 7])
    if kind in ("train", "predict"):
        s.x, s.y, w = _segments(seed, case["rows"])
        s.prop = proposal.Proposal(w)
        if kind == "train":
            s.steps = (case["rows"] + case["batch"] - 1) // case["batch"]
            s.mult = 2 * int(rng.integers(1, case["rows"] // 2)) + 1
            while math.gcd(s.mult, case["rows"]) != 1:
                s.mult += 2
            s.add = int(rng.integers(0, case["rows"]))
        return s
    hier = _hierarchy(case["data"], seed)
    s.ctx = _context(case, hier)
    if kind == "batch":
        cams, which = _views(case, rng)
        s.tf = torch.as_tensor(np.stack([_transfer(rng) for _ in range(4)]), device=DEV)
        s.views, _, total = amr.make_views(cams, which)
        s.out = torch.empty(total, device=DEV)
        s.params = amr.amr_default_params(**_options(case, hier))
        return s
    s.tf = torch.as_tensor(_transfer(rng), device=DEV)
    if kind == "log":
        s.cams = [_camera(rng, case["size"], case["size"]) for _ in range(case["poses"])]
        s.params = amr.amr_default_params(**dict(_options(case, hier), shade=0))
        return s
    s.cam = _camera(rng, case["width"], case["height"])
    s.params = amr.amr_default_params(**_options(case, hier))
    if case.get("shadow"):
        for a, v in enumerate(rng.uniform(0.35, 0.65, 3)):
            s.params.light[a] = v
    if kind == "learned":
        proposal.Proposal(_proposal_weights()).install(s.ctx)
        s.params.learned, s.params.tau = case["mode"], case["tau"]
        s.params.coarse_factor, s.params.skip = case["factor"], 1
    s.out = torch.empty((case["height"], case["width"], 4), device=DEV)
    return s


def run(state):
    s, case = state, state.case
    kind = case["kind"]
    if kind in ("frame", "learned"):
        s.ctx.amr_render(s.cam, s.tf, s.params, s.out)
        return s.out
    if kind == "batch":
        s.ctx.amr_render_batch(s.views, s.tf, s.params, s.out)
        return s.out
    if kind == "log":
        x, y, seen = proposal.log_segments(s.ctx, s.cams, s.tf, s.params, _log_capacity(case),
                                           case["keep"], seed=1)
        return {"features": x, "targets": y, "seen": seen}
    if kind == "train":
        first = (s.prop.step % s.steps) * case["batch"]
        s.prop.loss_grad(s.x, s.y, first, min(case["batch"], case["rows"] - first), s.mult, s.add)
        s.prop.adam(1e-3)
        p = s.prop
        return {"loss": p.loss, "grad": p.grad, "params": p.params, "m": p.m, "v": p.v}
    return s.prop.predict(s.x)


def _log_capacity(case):
    """Records asked for: about half of what the views hold, so the buffer fills up."""
    return int(case["poses"] * case["size"] ** 2 * case["keep"] * DATA[case["data"]]["leaves"] / 2)


# ----------------------------------------------------------------------------------------
# work and tolerance
# ----------------------------------------------------------------------------------------


def _pixels(case):
    if case["kind"] == "batch":
        lo, hi = case["lo"], case["hi"]
        return case["views"] * (lo * lo + lo * hi + hi * hi) / 3.0
    if case["kind"] == "log":
        return case["poses"] * case["size"] ** 2
    return case["width"] * case["height"]


def _samples(case):
    return _pixels(case) * DATA[case["data"]]["samples"]


def work(case):
    kind = case["kind"]
    if kind == "train":
        # forward, and for every layer but the first both gradients
        n = case["batch"]
        return {"bytes": n * 13 * 4 + 8 * 4 * MLP_PARAMS, "flops": n * 2 * (3 * MLP_MACS - 12 * 64)}
    if kind == "predict":
        return {"bytes": case["rows"] * 13 * 4 + 4 * MLP_PARAMS, "flops": case["rows"] * 2 * MLP_MACS}
    # every sample's position, trilinear value and opacity (30 operations), and the shading of
    # the twentieth of them that is opaque (seven more values, 120 operations); each cell that
    # samples can reach once, and the image
    samples = _samples(case)
    flops = samples * 30.0
    if case.get("shade", 1) and kind != "log":
        flops += samples / 20 * (7 * 20 + 120)
    if case.get("shadow"):
        flops += samples / 20 * 30.0 * DATA[case["data"]]["n0"] * 0.7
    if kind == "learned":
        flops = flops / 10 + _pixels(case) * 20 * 2 * MLP_MACS
    cells = min(DATA[case["data"]]["cells"], samples) * CELL_BYTES[case.get("cells", "f32")]
    out = _pixels(case) * 16 if kind != "log" else _log_capacity(case) * 52
    return {"bytes": cells + out, "flops": flops}


def tolerance(case):
    """Four times what the path shows against `exact`, by what rounds it: FP32 positions, values
    and sums; cells stored in 16 bits; the network's 16-bit operands."""
    kind = case["kind"]
    if kind == "train":
        return {"rel": 1e-2, "max": 0.3}
    if kind == "predict":
        return {"rel": 1e-2, "max": 0.1}
    if kind == "learned":
        return {"rel": 5e-3, "max": 0.3}  # a segment at the threshold falls on either side
    if kind == "log":
        return {"rel": 1e-5, "max": 1e-3}
    cells = case.get("cells", "f32")
    if cells != "f32":
        return {"rel": 4e-4, "max": 0.05} if cells == "f16" else {"rel": 2.5e-3, "max": 0.2}
    return {"rel": 1e-4, "max": 0.05}  # a ray that ends within rounding of its last sample


# ----------------------------------------------------------------------------------------
# the same outputs in 64 bits
# ----------------------------------------------------------------------------------------


class _Tree:
    """The kD-tree of a hierarchy in finest cells: per level, leaves are split at the plane that
    crosses the fewest pieces (ties: the most even volumes, the smaller axis, the smaller
    plane) until each is one piece or free of them."""

    def __init__(self, h):
        self.h, L = h, h.num_levels
        sc = 1 << (L - 1 - h.patch_level.astype(np.int64))
        self.fbox = h.patch_box * sc[:, None]
        self.nodes = [[-1, 0, -1, -1, -1]]  # axis, split, first child, patch, level
        n = h.n0 << (L - 1)
        self.box = [np.array([0, 0, 0, n, n, n], dtype=np.int64)]
        for level in range(L):
            ids = np.nonzero(h.patch_level == level)[0]
            leaves = [i for i, nd in enumerate(self.nodes) if nd[0] < 0]
            for i in leaves:
                self._refine(i, self.fbox[ids], ids, 1 << (L - 1 - level), level)
        nd = np.array(self.nodes, dtype=np.int64)
        self.axis, self.split, self.child, self.patch, self.level = (
            torch.as_tensor(np.ascontiguousarray(nd[:, k]), device=DEV) for k in range(5))
        depth = np.zeros(len(nd), dtype=np.int64)
        for i in range(len(nd)):
            if nd[i, 0] >= 0:
                depth[nd[i, 2]:nd[i, 2] + 2] = depth[i] + 1
        self.depth = int(depth.max())

    def _refine(self, i, pieces, ids, step, level):
        todo = [(i, pieces, ids)]
        while todo:
            i, pieces, ids = todo.pop()
            box = self.box[i]
            lo, hi = np.maximum(pieces[:, :3], box[:3]), np.minimum(pieces[:, 3:], box[3:])
            keep = (lo < hi).all(1)
            if not keep.any():
                continue
            lo, hi, ids = lo[keep], hi[keep], ids[keep]
            pieces = np.concatenate([lo, hi], 1)
            if len(ids) == 1 and (pieces[0] == box).all():
                self.nodes[i][3], self.nodes[i][4] = int(ids[0]), level
                continue
            a, s = self._choose(box, lo, hi, step)
            c = len(self.nodes)
            for side in (0, 1):
                b = box.copy()
                b[3 + a if side == 0 else a] = s
                self.box.append(b)
                self.nodes.append([-1, 0, -1, self.nodes[i][3], self.nodes[i][4]])
                todo.append((c + side, pieces, ids))
            self.nodes[i][:3] = [a, s, c]

    @staticmethod
    def _choose(box, lo, hi, step):
        best = None
        for a in range(3):
            l, u = np.sort(lo[:, a]), np.sort(hi[:, a])
            b0, b1 = int(box[a]), int(box[3 + a])
            area = int(np.prod(np.delete(box[3:] - box[:3], a)))
            pos = np.unique(np.concatenate([l, u, [b0, b1]]))
            # the faces, and in each gap between faces the grid plane nearest the centre
            face = pos[(pos > b0) & (pos < b1)]
            cost = np.searchsorted(l, face) - np.searchsorted(u, face, side="right")
            g = b0 + (b1 - b0) // (2 * step) * step
            first, last = pos[:-1] + step, pos[1:] - step
            ok = first <= last
            first, last, left = first[ok], last[ok], pos[:-1][ok]
            g1, g2 = np.clip(g, first, last), np.clip(g + step, first, last)
            e1, e2 = np.abs(2 * g1 - b0 - b1), np.abs(2 * g2 - b0 - b1)
            gap = np.where((e2 < e1) | ((e2 == e1) & (g2 < g1)), g2, g1)
            gcost = np.searchsorted(l, left, side="right") - np.searchsorted(u, left, side="right")
            plane, cost = np.concatenate([face, gap]), np.concatenate([cost, gcost])
            if not len(plane):
                continue
            bal = np.abs(2 * plane - b0 - b1) * area
            k = np.lexsort((plane, bal, cost))[0]
            if best is None or (cost[k], bal[k]) < best[:2]:
                best = (cost[k], bal[k], a, int(plane[k]))
        return best[2], best[3]


class _Field:
    """The cell-centred AMR field in 64 bits: V_l (a level's own cell, else the trilinear value
    of the finest coarser level there), S_l (trilinear in V_l), F (S of the finest level)."""

    def __init__(self, h):
        self.h, self.tree = h, _Tree(h)
        t = lambda v: torch.as_tensor(np.ascontiguousarray(v), device=DEV)  # noqa: E731
        self.lo, self.hi = t(h.patch_box[:, :3]), t(h.patch_box[:, 3:])
        self.start, self.plevel = t(h.start[:-1]), t(h.patch_level.astype(np.int64))
        self.cells = h.flat.double()
        # patches by buckets of each level's index space
        self.side, self.near = [], []
        for level in range(h.num_levels):
            ids = np.nonzero(h.patch_level == level)[0]
            n = h.n0 << level
            side = max(8, n // 64)
            m = -(-n // side)
            lists = {}
            for p in ids:
                b = h.patch_box[p]
                for kk in range(b[2] // side, (b[5] - 1) // side + 1):
                    for jj in range(b[1] // side, (b[4] - 1) // side + 1):
                        for ii in range(b[0] // side, (b[3] - 1) // side + 1):
                            lists.setdefault(ii + m * (jj + m * kk), []).append(p)
            width = max(len(v) for v in lists.values())
            table = np.full((m ** 3, width), -1, dtype=np.int32)
            for key, v in lists.items():
                table[key, :len(v)] = v
            self.side.append((side, m))
            self.near.append(torch.as_tensor(table, device=DEV))

    def patch_at(self, level, c):
        """Patch of one level that holds cells c [N, 3], or -1."""
        side, m = self.side[level]
        b = c // side
        near = self.near[level][b[:, 0] + m * (b[:, 1] + m * b[:, 2])]
        got = torch.full((len(c),), -1, dtype=torch.int64, device=DEV)
        for k in range(near.shape[1]):
            p = near[:, k].long()
            q = p.clamp(min=0)
            inside = (p >= 0) & ((c >= self.lo[q]) & (c < self.hi[q])).all(1)
            got = torch.where(inside, p, got)
        return got

    def cell(self, p, c):
        r, n = c - self.lo[p], self.hi[p] - self.lo[p]
        return self.cells[self.start[p] + r[:, 0] + n[:, 0] * (r[:, 1] + n[:, 1] * r[:, 2])]

    def V(self, level, c, hint):
        """level, hint: per cell (hint: a patch of that level to try first)."""
        n = self.h.n0 << level
        c = torch.minimum(c.clamp(min=0), n[:, None] - 1)
        own = ((c >= self.lo[hint]) & (c < self.hi[hint])).all(1) & (self.plevel[hint] == level)
        v = self.cell(hint, torch.where(own[:, None], c, self.lo[hint]))
        for l in range(self.h.num_levels):
            at = torch.nonzero(~own & (level == l))[:, 0]
            if len(at):
                v[at] = self._coarser(l, c[at])
        return v

    def _coarser(self, level, c):
        v = torch.zeros(len(c), dtype=torch.float64, device=DEV)
        left = torch.arange(len(c), device=DEV)
        for l in range(level, -1, -1):
            p = self.patch_at(l, c[left] >> (level - l))
            found = p >= 0
            at, q = left[found], p[found]
            if len(at):
                if l == level:
                    v[at] = self.cell(q, c[at])
                else:
                    x = (c[at].double() + 0.5) / (self.h.n0 << level)
                    v[at] = self.S(torch.full_like(q, l), x, q)
            left = left[~found]
            if not len(left):
                break
        return v

    def S(self, level, x, patch):
        xi = x * (self.h.n0 << level)[:, None].double() - 0.5
        i0 = torch.floor(xi)
        w = xi - i0
        i0 = i0.long()
        out = 0.0
        for k in range(8):
            d = torch.tensor([k & 1, k >> 1 & 1, k >> 2], device=DEV)
            f = torch.where(d.bool()[None], w, 1.0 - w).prod(1)
            out = out + f * self.V(level, i0 + d, patch)
        return out

    def F(self, x):
        L = self.h.num_levels
        n = self.h.n0 << (L - 1)
        f = torch.floor(x * n).long().clamp(0, n - 1)
        node = self._descend(lambda node, a: f.gather(1, a[:, None])[:, 0] >= self.tree.split[node], len(x))
        return self.S(self.tree.level[node], x, self.tree.patch[node])

    def _descend(self, right, count):
        t = self.tree
        node = torch.zeros(count, dtype=torch.int64, device=DEV)
        for _ in range(t.depth):
            a = t.axis[node]
            go = right(node, a.clamp(min=0)).long()
            node = torch.where(a >= 0, t.child[node] + go, node)
        return node


def _rays(cam):
    W, H = cam.width, cam.height
    t = lambda v: torch.as_tensor(np.asarray(v, dtype=np.float64), device=DEV)  # noqa: E731
    i, j = torch.arange(W, device=DEV).double(), torch.arange(H, device=DEV).double()
    u = (2 * (i + 0.5) / W - 1) * cam.tan_half_fov_y * (W / H)
    v = (1 - 2 * (j + 0.5) / H) * cam.tan_half_fov_y
    d = t(cam.fwd) + u[None, :, None] * t(cam.right) + v[:, None, None] * t(cam.up)
    return t(cam.eye), d.reshape(-1, 3)


def _walk(fld, o, d):
    """Segments of rays o + t d in order: ray, number along the ray, leaf node, t0, t1."""
    tree, n = fld.tree, fld.h.n0 << (fld.h.num_levels - 1)
    inv = 1.0 / d
    ta, tb = (0.0 - o) * inv, (1.0 - o) * inv
    t0 = torch.minimum(ta, tb).max(1)[0].clamp(min=0.0)
    t_out = torch.maximum(ta, tb).min(1)[0]
    ray = torch.nonzero(t0 < t_out)[:, 0]
    t0, t_out, inv = t0[ray], t_out[ray], inv[ray]
    got, k = [], 0
    while len(ray):
        t1 = t_out.clone()

        def right(node, a):
            nonlocal t1
            iv = inv.gather(1, a[:, None])[:, 0]
            ts = (tree.split[node].double() / n - o[a]) * iv
            far = ~(ts >= t1) & (ts <= t0)
            cut = (tree.axis[node] >= 0) & ~far & (ts < t1)
            t1 = torch.where(cut, ts, t1)
            return far == (iv > 0)

        node = fld._descend(right, len(ray))
        got.append((ray, torch.full_like(ray, k), node, t0, t1))
        on = t1 < t_out
        ray, t0, t_out, inv = ray[on], t1[on], t_out[on], inv[on]
        k += 1
    if not got:
        none = torch.zeros(0, dtype=torch.int64, device=DEV)
        return [none] * 3 + [none.double()] * 2
    cols = [torch.cat(c) for c in zip(*got)]
    order = torch.argsort(cols[0] * (k + 1) + cols[1])
    return [c[order] for c in cols]


def _lookup(tf, p, v):
    u = ((v - p["vmin"]) / (p["vmax"] - p["vmin"])).clamp(0, 1) * (len(tf) - 1)
    i = u.long().clamp(max=len(tf) - 2)
    w = (u - i)[:, None]
    return (1 - w) * tf[i] + w * tf[i + 1]


def _light(fld, tf, p, light, x, kappa):
    """Transmittance from points x to the light."""
    D = light - x
    s_out = torch.where(D != 0, ((D > 0).double() - x) / D, torch.inf).min(1)[0].clamp(0, 1)
    length = s_out * D.norm(dim=1)
    n = torch.ceil(length / p["light_step"]).clamp(min=1)
    depth = torch.zeros(len(x), dtype=torch.float64, device=DEV)
    for k in range(int(n.max()) if len(n) else 0):
        at = torch.nonzero(k < n)[:, 0]
        q = x[at] + ((k + 0.5) / n[at] * s_out[at])[:, None] * D[at]
        depth[at] += kappa * _lookup(tf, p, fld.F(q))[:, 3] * length[at] / n[at]
    T = torch.exp(-depth)
    return torch.where(T <= 1e-4, 0.0, T)


def _composite(fld, o, d, tf, p, light=None, ert=1e-4, kappa=8.0):
    """Image [N, 4] of rays o + t d, and their segments with the opacity before and after."""
    ray, num, node, t0, t1 = _walk(fld, o, d)
    h, dn = fld.h, d.norm(dim=1)
    out = torch.zeros((len(d), 4), dtype=torch.float64, device=DEV)
    level, patch = fld.tree.level[node], fld.tree.patch[node]
    length = (t1 - t0) * dn[ray]
    n = torch.ceil(length / (0.5 / (h.n0 << level).double())).clamp(min=1).long()
    seg = torch.repeat_interleave(torch.arange(len(n), device=DEV), n)
    k = torch.arange(len(seg), device=DEV) - (torch.cumsum(n, 0) - n)[seg]
    t = t0[seg] + (k.double() + 0.5) * ((t1 - t0) / n)[seg]
    x = o + t[:, None] * d[ray[seg]]
    rgba = _lookup(tf, p, fld.S(level[seg], x, patch[seg]))
    some = torch.nonzero(rgba[:, 3] > 0)[:, 0]
    seg, x, rgba = seg[some], x[some], rgba[some]
    tau = kappa * rgba[:, 3] * (length / n)[seg]
    per_seg = torch.zeros(len(n), dtype=torch.float64, device=DEV).index_add_(0, seg, tau)
    per_ray = torch.zeros(len(d), dtype=torch.float64, device=DEV).index_add_(0, ray, per_seg)
    base = torch.cumsum(per_ray, 0) - per_ray
    before_seg = torch.cumsum(per_seg, 0) - per_seg - base[ray]
    before = torch.cumsum(tau, 0) - tau - base[ray[seg]]
    a_in, a_out = 1 - torch.exp(-before_seg), 1 - torch.exp(-before_seg - per_seg)
    if ert > 0:
        on = torch.exp(-before) > ert
        seg, x, rgba, tau, before = (v[on] for v in (seg, x, rgba, tau, before))
    r, rgb = ray[seg], rgba[:, :3]
    if p["shade"]:
        hl = 1.0 / (h.n0 << level[seg]).double()
        g = []
        for a in range(3):
            e = torch.zeros((1, 3), dtype=torch.float64, device=DEV)
            e[0, a] = 1.0
            g.append((fld.F(x + hl[:, None] * e) - fld.F(x - hl[:, None] * e)) / (2 * hl))
        g = torch.stack(g, 1)
        den = torch.maximum(g.norm(dim=1), 1e-3 * (p["vmax"] - p["vmin"]) / hl)
        ndl = ((g * d[r]).sum(1) / (den * dn[r])).abs()
        rgb = (rgb * (0.3 + 0.6 * ndl)[:, None] + (0.3 * ndl ** 32)[:, None]).clamp(0, 1)
    if light is not None:
        rgb = rgb * (0.2 + 0.8 * _light(fld, tf, p, light, x, kappa))[:, None]
    w = torch.exp(-before) * (1 - torch.exp(-tau))
    out[:, :3].index_add_(0, r, rgb * w[:, None])
    out[:, 3].index_add_(0, r, w)
    return out, (ray, num, node, t0, t1, a_in, a_out)


def _image(fld, cam, tf, p, light=None):
    o, d = _rays(cam)
    rays = max(1024, int(2.0e7 / DATA[fld.h.name]["samples"]) // (3 if light is not None else 1))
    return torch.cat([_composite(fld, o, d[c:c + rays], tf, p, light)[0]
                      for c in range(0, len(d), rays)])


def _mix(x):
    m = 0xFFFFFFFF
    x = x ^ (x >> 16)
    x = _mul(x, 0x7FEB352D)
    x = x ^ (x >> 15)
    x = _mul(x, 0x846CA68B)
    return (x ^ (x >> 16)) & m


def _mul(x, c):
    """Low 32 bits of x c, for x below 2^32 (in two halves: 64-bit products stay exact)."""
    return ((x & 0xFFFF) * c + (((x >> 16) * c & 0xFFFF) << 16)) & 0xFFFFFFFF


def _logged(fld, cams, tf, p, keep, seed):
    """Features and targets of the segments that the seeded hash keeps, in pixel order."""
    xs, ys = [], []
    tree, h = fld.tree, fld.h
    vmin, vmax = _leaf_range(fld)
    for v, cam in enumerate(cams):
        o, d = _rays(cam)
        _, (ray, num, node, t0, t1, a_in, a_out) = _composite(fld, o, d, tf, dict(p, shade=0), ert=0)
        s = (seed * 1000003 + v) & 0xFFFFFFFF
        i, j = ray % cam.width, ray // cam.width
        inner = _mix((j + (s * 0x85EBCA77 & 0xFFFFFFFF)) & 0xFFFFFFFF)
        hsh = _mix(_mul(i, 0x9E3779B1) ^ inner ^ _mul(num, 0xC2B2AE3D))
        on = (hsh >> 8).double() / 16777216.0 < float(np.float32(keep))
        ray, node, t0, t1, a_in, a_out = (q[on] for q in (ray, node, t0, t1, a_in, a_out))
        u = lambda q: ((q[node] - p["vmin"]) / (p["vmax"] - p["vmin"])).clamp(0, 1)  # noqa: E731
        e = d[ray] / d[ray].abs().sum(1, keepdim=True)
        sgn = torch.where(e >= 0, 1.0, -1.0)
        fold = (1 - e.abs()[:, [1, 0]]) * sgn[:, :2]
        octa = torch.where(e[:, 2:] < 0, fold, e[:, :2])
        xs.append(torch.cat([o + t0[:, None] * d[ray], o + t1[:, None] * d[ray],
                             tree.level[node].double()[:, None] / max(1, h.num_levels - 1),
                             u(vmin)[:, None], u(vmax)[:, None], a_in[:, None], octa], 1))
        ys.append(a_out - a_in)
    return torch.cat(xs), torch.cat(ys)


def _leaf_range(fld):
    """Per node: smallest and largest value that a sample of its leaf can interpolate."""
    tree, h = fld.tree, fld.h
    low = torch.full((len(tree.axis),), math.inf, dtype=torch.float64, device=DEV)
    high = -low
    box = torch.as_tensor(np.array(tree.box), device=DEV)
    leaves = torch.nonzero(tree.axis < 0)[:, 0]
    for part in leaves.split(256):
        level, patch = tree.level[part], tree.patch[part]
        # the cells under the stencils of all points of the box (its faces need not lie on
        # the level's own grid)
        sc = 1 << (h.num_levels - 1 - level)
        b = torch.floor(box[part].double() / sc[:, None] - 0.5).long()
        n = b[:, 3:] - b[:, :3] + 2
        count = n.prod(1)
        at = torch.repeat_interleave(torch.arange(len(part), device=DEV), count)
        r = torch.arange(len(at), device=DEV) - (torch.cumsum(count, 0) - count)[at]
        c = torch.stack([r % n[at, 0], r // n[at, 0] % n[at, 1], r // (n[at, 0] * n[at, 1])], 1)
        v = fld.V(level[at], c + b[at, :3], patch[at])
        low.scatter_reduce_(0, part[at], v, "amin")
        high.scatter_reduce_(0, part[at], v, "amax")
    return low, high


def _network64(w, x):
    out, k = [], 0
    for s in MLP:
        out.append(w[k:k + math.prod(s)].reshape(s))
        k += math.prod(s)
    h = x
    for a, b in zip(out[0:6:2], out[1:6:2]):
        h = torch.relu(h @ a.T + b)
    return (h @ out[6].T + out[7])[:, 0]


def exact(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng([seed, 7])
    if kind in ("train", "predict"):
        x, y, w = _segments(seed, case["rows"])
        w = torch.as_tensor(w, device=DEV).double()
        if kind == "predict":
            return torch.cat([torch.sigmoid(_network64(w, c.double())) for c in x.split(1 << 18)])
        mult = 2 * int(rng.integers(1, case["rows"] // 2)) + 1
        while math.gcd(mult, case["rows"]) != 1:
            mult += 2
        add = int(rng.integers(0, case["rows"]))
        n = min(case["batch"], case["rows"])
        at = (torch.arange(n, device=DEV) * mult + add) % case["rows"]
        w.requires_grad_()
        loss = torch.nn.functional.binary_cross_entropy_with_logits(
            _network64(w, x[at].double()), y[at].double())
        (g,) = torch.autograd.grad(loss, w)
        m, v = 0.1 * g, 0.001 * g * g
        params = w.detach() - 1e-3 * (m / (1 - 0.9)) / (torch.sqrt(v / (1 - 0.999)) + 1e-8)
        return {"loss": loss.detach().reshape(1), "grad": g, "params": params, "m": m, "v": v}
    shaded = case.get("shade", 1) and kind != "log"
    if kind == "learned" or case.get("lod") or case["data"] == "deep" or (
            kind != "frame" and case["data"] == "large") or (
            case.get("shadow") and case["data"] != "tiny") or (
            _samples(case) > EXACT_SAMPLES / (2.5 if shaded else 1)):
        return None
    h = _hierarchy(case["data"], seed)
    h.name = case["data"]
    fld, p = _Field(h), _options(case, h)
    if kind == "batch":
        cams, which = _views(case, rng)
        tfs = [torch.as_tensor(_transfer(rng), device=DEV).double() for _ in range(4)]
        return torch.cat([_image(fld, c, tfs[t], p).reshape(-1) for c, t in zip(cams, which)])
    tf = torch.as_tensor(_transfer(rng), device=DEV).double()
    if kind == "log":
        cams = [_camera(rng, case["size"], case["size"]) for _ in range(case["poses"])]
        x, y = _logged(fld, cams, tf, p, case["keep"], 1)
        n = _log_capacity(case)
        return {"features": x[:n], "targets": y[:n], "seen": None}
    cam = _camera(rng, case["width"], case["height"])
    light = torch.as_tensor(rng.uniform(0.35, 0.65, 3), device=DEV) if case.get("shadow") else None
    return _image(fld, cam, tf, p, light).reshape(case["height"], case["width"], 4)
