"""What a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values.  Its "kind" names the call sequence:

  view       one training view, ViewTrainer.view_step: project, bin/sort, composite, L1 loss, backward, sparse Adam,
             conflict counts against the four views before it; with "active" also the realized active set of the view
  render     forward only (evaluation of a held-out camera): project, bin/sort, composite
  unit       a task unit of two views with one update, ViewTrainer.unit_step
  host       a run of views whose targets live in pinned host memory, ViewTrainer.train_from_host
  admission  scope arithmetic before a task unit is admitted: unions of its views' scopes and their list, hazard counts
             against the units in flight, the delayed-read gate
  graph      the relative locality graph from the measured scopes: pairwise intersections of all views, edge weights,
             retention of the strongest neighbours, scores of the candidate views

Scenes follow the shapes of workloads.py (box, Gaussian blob, unbounded 360-degree capture, city blocks seen from the air
or from the street), drawn on the GPU from the seed.  A training state is one in the middle of a run: a share "seen" of
the primitives has optimizer history, the learning rates are those of the end of a schedule (a pass that is repeated
leaves the scene what it is).
"""
import math

import numpy as np
import torch

from paper_2607_19893_b200 import binding as B
from paper_2607_19893_b200 import workloads as wl
from paper_2607_19893_b200.engine import ViewTrainer

LR = [1e-5] * 6
BETA1, BETA2, EPS = 0.9, 0.999, 1e-15
WINDOW = 4  # a training view is compared with the views before it, as many as this
KEEP = 8    # neighbours an item of the locality graph retains
TAU = 0.05  # admission threshold of the delayed-read gate


def listed():
    return [
        # the smallest call: a toy scene, where launches and the host's own work are all there is
        {"name": "view_1k_sh0_64x64", "kind": "view", "scene": "box", "n": 1024, "sh": 0, "width": 64, "height": 64,
         "log_scale": -3.0, "binning": 0, "seen": 1.0, "active": False},
        # an object-sized capture at preview resolution
        {"name": "view_100k_sh3_256x256", "kind": "view", "scene": "blob", "n": 100_000, "sh": 3, "width": 256,
         "height": 256, "log_scale": -3.0, "binning": 0, "seen": 0.6, "active": False},
        # an unbounded 360-degree capture at full photo resolution: the headline workload of the benchmark
        {"name": "view_1m_sh3_1600x1066", "kind": "view", "scene": "unbounded", "n": 1_000_000, "sh": 3, "width": 1600,
         "height": 1066, "log_scale": -5.0, "binning": 0, "seen": 0.3, "active": False},
        # the same shape with more and larger splats: hundreds of tiles per splat, most of them occluded
        {"name": "view_5m_sh3_1920x1080", "kind": "view", "scene": "unbounded", "n": 5_000_000, "sh": 3, "width": 1920,
         "height": 1080, "log_scale": -4.0, "binning": 0, "seen": 0.3, "active": False},
        # a whole city from the air: the largest pool, two per cent of it visible, nearly all of that blends
        {"name": "view_20m_city_air_1920x1080", "kind": "view", "scene": "air", "n": 20_000_000, "sh": 3, "width": 1920,
         "height": 1080, "log_scale": math.log(0.3), "binning": 0, "seen": 1.0, "active": False},
        # a district from street level: long lists near the horizon
        {"name": "view_2m8_city_street_1920x1080", "kind": "view", "scene": "street", "n": 2_812_500, "sh": 3,
         "width": 1920, "height": 1080, "log_scale": math.log(0.3), "binning": 0, "seen": 1.0, "active": False},
        # odd sizes everywhere, the tight-extent rectangles, degree 2, and the realized active set of the view
        {"name": "view_273k_sh2_1237x823_tight", "kind": "view", "scene": "unbounded", "n": 273_211, "sh": 2,
         "width": 1237, "height": 823, "log_scale": -4.5, "binning": 1, "seen": 0.5, "active": True},
        # a held-out camera is rendered for evaluation, nothing is trained
        {"name": "render_1m_sh3_1600x1066", "kind": "render", "scene": "unbounded", "n": 1_000_000, "sh": 3,
         "width": 1600, "height": 1066, "log_scale": -5.0, "binning": 0},
        # two views per task unit
        {"name": "unit_400k_sh1_800x600", "kind": "unit", "scene": "unbounded", "n": 400_000, "sh": 1, "width": 800,
         "height": 600, "log_scale": -4.5, "binning": 0, "seen": 0.4},
        # the training loop a user runs: target images from the host, loss and counts back after every view
        {"name": "host_4x500k_sh3_1280x720", "kind": "host", "scene": "unbounded", "n": 500_000, "sh": 3, "width": 1280,
         "height": 720, "log_scale": -4.8, "binning": 0, "seen": 0.4, "views": 4},
        # a unit of two views against eight units in flight, on the pool of the larger unbounded capture
        {"name": "admission_5m_8_units", "kind": "admission", "n": 5_000_000, "units": 8},
        # the graph over all 128 views of the city
        {"name": "graph_20m_128_views", "kind": "graph", "n": 20_000_000, "views": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: pools of a thousand to millions of primitives, images from one tile row to
    full HD, every degree, both rules for the rectangles, two to two hundred views in the graph."""
    kind = rng.choice(["view", "view", "view", "view", "render", "unit", "host", "admission", "graph"])
    if kind == "admission":
        return {"kind": kind, "n": _log_int(rng, 20_000, 20_000_000), "units": rng.randint(1, 16)}
    if kind == "graph":
        views = _log_int(rng, 8, 200)
        return {"kind": kind, "n": _log_int(rng, 20_000, min(20_000_000, int(128 * 128 * 2e7 / views ** 2))), "views": views}
    scene = rng.choice(["box", "blob", "unbounded", "unbounded", "air", "street"])
    width = _log_int(rng, 48, 1920)
    height = max(16, int(round(width * rng.uniform(0.5, 0.75))))
    if scene == "box":
        n, log_scale, sh = _log_int(rng, 1_000, 20_000), rng.uniform(-3.5, -2.5), rng.choice([0, 0, 1])
        width, height = min(width, 512), min(height, 384)
    elif scene == "blob":
        n, log_scale, sh = _log_int(rng, 10_000, 400_000), rng.uniform(-3.5, -3.0), rng.choice([1, 2, 3, 3])
        width, height = min(width, 1024), min(height, 768)
    elif scene == "unbounded":
        n, log_scale, sh = _log_int(rng, 50_000, 3_000_000), rng.uniform(-5.2, -4.2), rng.choice([1, 2, 3, 3])
    else:
        grid = rng.randint(8, 40)
        n, log_scale, sh = int(20_000_000 * (grid / 64.0) ** 2) + rng.randint(0, 999), math.log(0.3), rng.choice([2, 3, 3])
        width = max(width, 320)
        height = max(180, int(round(width * rng.uniform(0.5, 0.6))))
    case = {"kind": kind, "scene": scene, "n": n, "sh": sh, "width": width, "height": height,
            "log_scale": round(log_scale, 3), "binning": rng.choice([0, 0, 1])}
    if kind != "render":
        case["seen"] = rng.choice([0.3, 0.6, 1.0])
    if kind == "view":
        case["active"] = rng.random() < 0.2
    if kind == "host":
        case["views"] = rng.randint(2, 6)
    return case


# ------------------------------------------------------------------------------------------------ scenes and cameras
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _scene_tensors(case, g):
    """The five attribute tensors on the GPU, distributed as in workloads.py."""
    n, deg = case["n"], case["sh"]
    k = (deg + 1) ** 2
    rand = lambda *s: torch.rand(s, generator=g, device="cuda")    # noqa: E731
    norm = lambda *s: torch.randn(s, generator=g, device="cuda")   # noqa: E731
    kind = case["scene"]
    if kind == "box":
        means = torch.stack([2 * rand(n) - 1, 2 * rand(n) - 1, 2 + 4 * rand(n)], 1)
    elif kind == "blob":
        means = 2.0 * norm(n, 3)
    elif kind == "unbounded":
        unit = torch.nn.functional.normalize(norm(n, 3), dim=1)
        core = rand(n) < 0.7
        radius = torch.where(core, rand(n) ** (1.0 / 3.0), 3 + 17 * rand(n))
        means = unit * radius[:, None]
    else:  # city blocks of 30 m, stored block by block
        grid = _city_grid(n)
        block = torch.sort(torch.randint(0, grid * grid, (n,), generator=g, device="cuda")).values
        extent = 30.0 * grid
        cap = (40.0 * rand(grid * grid))[block]
        x = ((block % grid).float() + 0.5) * 30.0 - extent / 2 + 24 * rand(n) - 12
        y = (torch.div(block, grid, rounding_mode="floor").float() + 0.5) * 30.0 - extent / 2 + 24 * rand(n) - 12
        means = torch.stack([x, y, cap * rand(n)], 1)
    sigma = 0.3 if kind in ("box", "blob") else 0.5
    log_scales = case["log_scale"] + sigma * norm(n, 3)
    quats = torch.nn.functional.normalize(norm(n, 4), dim=1)
    sh = 0.1 * norm(n, k, 3)
    sh[:, 0] = (rand(n, 3) - 0.5) / wl.SH_DC
    return means.contiguous(), log_scales, quats, norm(n), sh


def _city_grid(n):
    return max(1, int(round(64 * math.sqrt(n / 20_000_000.0))))


def _cameras(case, seed, count):
    """`count` cameras of the scene's kind; neighbours of a ring, or poses over the city."""
    rng = np.random.default_rng(seed)
    w, h, kind = case["width"], case["height"], case["scene"]
    out = []
    for i in range(count):
        zfar = 1.0e9
        if kind == "box":
            f, w2c = w, wl.look_at((0.3 * rng.uniform(-1, 1), 0.3 * rng.uniform(-1, 1), 0.0), (0.0, 0.0, 4.0), up=(0, -1, 0))
        elif kind in ("blob", "unbounded"):
            a = rng.uniform(0, 2 * np.pi) if i == 0 else a + 2 * np.pi / 32
            r, z = (6.0, 0.0) if kind == "blob" else (1.0, 0.2) if case["n"] < 4_000_000 else (0.45, 0.09)
            f = w if kind == "blob" else 0.85 * w
            w2c = wl.look_at((r * np.cos(a), r * np.sin(a), z), (0.0, 0.0, 0.0))
        else:
            grid = _city_grid(case["n"])
            extent, f = 30.0 * grid, w / 1.92
            if kind == "air":
                eye = (rng.uniform(-0.4, 0.4) * extent, rng.uniform(-0.4, 0.4) * extent, 150.0)
                w2c, zfar = wl.pose_from_yaw_pitch(eye, rng.uniform(0, 2 * np.pi), np.deg2rad(-60.0)), 2000.0
            else:
                street = rng.integers(1, max(2, grid)) * 30.0 - extent / 2
                eye = (street, rng.uniform(-0.3, 0.3) * extent, 1.7)
                w2c, zfar = wl.pose_from_yaw_pitch(eye, rng.choice([0.5 * np.pi, 1.5 * np.pi]), 0.0), 400.0
        cam = wl.Camera(w, h, float(f), float(f), w / 2.0, h / 2.0, 0.2, zfar, np.asarray(w2c), np.zeros(3))
        out.append(B.make_camera(cam))
    return out


def _capacities(case):
    """Rows and instances a program leaves room for, whatever the camera."""
    n, p = case["n"], case["width"] * case["height"]
    tiles = ((case["width"] + 15) // 16) * ((case["height"] + 15) // 16)
    base, per_row = {"box": (-3.0, 90.0), "blob": (-3.0, 90.0), "unbounded": (-5.0, 55.0)}.get(case["scene"], (math.log(0.3), 16.0))
    rows = min(n, 1_600_000) if case["scene"] in ("air", "street") else n if case["scene"] != "unbounded" else int((0.5 if n < 4_000_000 else 0.25) * n)
    inst = rows * min(tiles, 4 + per_row * p / 2.07e6 * math.exp(2 * (case["log_scale"] - base)))
    return rows, int(inst) + (1 << 16)


def _trainer(case, seed, n_cams, n_masks):
    """A ViewTrainer on the scene, and its cameras."""
    g = _gen(seed)
    tensors = _scene_tensors(case, g)
    cams = _cameras(case, seed, n_cams)
    n, k = case["n"], (case["sh"] + 1) ** 2
    row_cap, inst_cap = _capacities(case)
    z = lambda *s: np.zeros(s, dtype=np.float32)  # noqa: E731
    tr = ViewTrainer(wl.Scene(case["sh"], z(n, 3), z(n, 3), z(n, 4), z(n), z(n, k, 3)), case["width"], case["height"],
                     row_cap, inst_cap, mask_slots=n_masks, cfg=B.default_config(binning=case["binning"]),
                     extra_render_records=min(inst_cap // 256, 16384))
    for dst, src in zip(tr.params.tensors(), tensors):
        dst.copy_(src)
    seen = case.get("seen", 0.0)
    if seen > 0:  # optimizer history of a run that has lasted a while: gradients of an L1 loss are this small
        size = 0.1 / (3.0 * case["width"] * case["height"])
        has = (torch.rand(n, generator=g, device="cuda") < seen).float() * size
        for m, v in zip(tr.m.tensors(), tr.v.tensors()):
            f = has.view(-1, *([1] * (m.dim() - 1)))
            m.copy_(f * 0.3 * torch.randn(m.shape, generator=g, device="cuda"))
            v.copy_(f * f * (0.05 + torch.rand(m.shape, generator=g, device="cuda")))
        tr.moments_changed()
    # one warm-up projection, then the faster of the two instance orders is kept, as the benchmark does
    tr.project(cams[0])
    tr.choose_instance_sort(cams[0])
    return tr, cams, g


def _targets(case, g, count):
    return [torch.rand((3, case["height"], case["width"]), generator=g, device="cuda") for _ in range(count)]


def _scopes(n, views, g):
    """Touched bitmasks of `views` cameras over a pool stored block by block: a camera sees the blocks around it, and
    most of what they hold.  [views][stride] words."""
    words = (n + 31) // 32
    stride = (words + 3) // 4 * 4
    out = torch.zeros((views, stride), dtype=torch.int32, device="cuda")
    side = 64
    block = torch.arange(n, device="cuda") * (side * side) // n
    bx, by = (block % side).float(), torch.div(block, side, rounding_mode="floor").float()
    weight = (1 << torch.arange(32, device="cuda", dtype=torch.int64))
    for v in range(views):
        c = side * torch.rand(2, generator=g, device="cuda")
        r = 4 + 10 * torch.rand(1, generator=g, device="cuda")
        inside = ((bx - c[0]) ** 2 + (by - c[1]) ** 2 < r * r) & (torch.rand(n, generator=g, device="cuda") < 0.7)
        bits = torch.zeros(words * 32, dtype=torch.bool, device="cuda")
        bits[:n] = inside
        out[v, :words] = (bits.view(words, 32) * weight).sum(1).to(torch.int32)
    return out


# ------------------------------------------------------------------------------------------------ states
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "admission":
        g = _gen(seed)
        n, units = case["n"], case["units"]
        reads = _scopes(n, units + 2, g)  # the units in flight, then the two views of the unit to be admitted
        writes = reads & _scopes(n, units + 2, g).bitwise_or_(_scopes(n, units + 2, g))  # W+ lies inside R+
        s["ctx"] = B.odin_create(0)
        stride = reads.shape[1]
        # the unit's own scopes are built behind the others, in the slot the pairs name
        s["reads"] = torch.cat([reads, torch.zeros((1, stride), dtype=torch.int32, device="cuda")])
        s["writes"] = torch.cat([writes, torch.zeros((1, stride), dtype=torch.int32, device="cuda")])
        s["members"] = torch.tensor([units, units + 1], dtype=torch.int32, device="cuda")
        s["pairs"] = torch.tensor([(a, units + 2) for a in range(units)], dtype=torch.int32, device="cuda")
        s["counts"] = torch.zeros((units, 4), dtype=torch.int64, device="cuda")
        s["idx"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["count"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        s["ws"] = torch.zeros(B.odin_workspace_bytes(s["ctx"], n, 0), dtype=torch.uint8, device="cuda")
        # the realized active set of the producer: part of its write scope, with evidence over several decades
        bits = (writes[0, : (n + 31) // 32, None] >> torch.arange(32, device="cuda")) & 1
        ids = bits.view(-1)[:n].nonzero().view(-1)
        ids = ids[torch.rand(ids.numel(), generator=g, device="cuda") < 0.9]
        s["active"] = ids.to(torch.int32) if ids.numel() else torch.zeros(1, dtype=torch.int32, device="cuda")
        s["evidence"] = torch.exp(2 * torch.randn(s["active"].numel(), generator=g, device="cuda"))
        s["active_count"] = torch.tensor([ids.numel()], dtype=torch.int32, device="cuda")
        s["evidence_sum"] = s["evidence"].double().sum().view(1)
        s["gate"] = torch.zeros(4, dtype=torch.int64, device="cuda")
        return s
    if kind == "graph":
        g = _gen(seed)
        n, views = case["n"], case["views"]
        s["ctx"] = B.odin_create(0)
        s["masks"] = _scopes(n, views, g)
        i, j = torch.triu_indices(views, views, 1, device="cuda")
        s["pairs"] = torch.stack([i, j], 1).to(torch.int32).contiguous()
        s["upper"], s["lower"] = i * views + j, j * views + i
        s["counts"] = torch.zeros(i.numel(), dtype=torch.int64, device="cuda")
        lut = torch.tensor([bin(b).count("1") for b in range(256)], dtype=torch.uint8, device="cuda")
        s["sizes"] = torch.stack([lut[m.view(torch.uint8).long()].sum(dtype=torch.int64) for m in s["masks"]]).to(torch.int32)
        s["edge"] = torch.zeros(i.numel(), device="cuda")
        s["weights"] = torch.zeros((views, views), device="cuda")
        s["graph"] = torch.zeros((views, views), device="cuda")
        s["ws"] = torch.zeros(views * views, dtype=torch.uint8, device="cuda")
        order = torch.randperm(views, generator=g, device="cuda").to(torch.int32)
        s["prev"], s["cand"] = order[:2].contiguous(), order[2:].contiguous()
        s["scores"] = torch.zeros(views - 2, device="cuda")
        return s
    if kind == "render":
        s["tr"], s["cams"], _ = _trainer(case, seed, 1, 1)
        return s
    if kind == "unit":
        tr, s["cams"], g = _trainer(case, seed, 2, 2)
        s["targets"] = _targets(case, g, 2)
        tr.prepare_unit()
    elif kind == "host":
        tr, s["cams"], g = _trainer(case, seed, case["views"], WINDOW + 1)
        s["targets"] = [t.cpu().pin_memory() for t in _targets(case, g, case["views"])]
        tr.prepare_host_io(WINDOW)
    else:
        tr, s["cams"], g = _trainer(case, seed, WINDOW + 1, WINDOW + 1)
        s["target"] = _targets(case, g, 1)[0]
        tr.track_active = bool(case["active"])
    if kind != "unit":
        # the views before this one have left their touched masks
        for k in range(1, WINDOW + 1):
            tr.proj.struct.touched_mask = tr.masks[k].data_ptr()
            tr.project(s["cams"][min(k, len(s["cams"]) - 1)])
        s["pairs"] = torch.tensor([(0, k) for k in range(1, WINDOW + 1)], dtype=torch.int32, device="cuda")
        s["counts"] = torch.zeros(WINDOW, dtype=torch.int64, device="cuda")
    s["tr"], s["step"] = tr, 1000
    return s


def _state_of(tr):
    return {"params": tr.params.tensors(), "m": tr.m.tensors(), "v": tr.v.tensors()}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "view":
        tr, cam = s["tr"], s["cams"][0]
        s["step"] += 1
        tr.target = s["target"]
        tr.view_step(cam, s["step"], LR, BETA1, BETA2, EPS, slot=0, d_pairs=s["pairs"], n_pairs=WINDOW, d_counts=s["counts"])
        out = {"image": tr.out, "final_T": tr.final_T, "n_contrib": tr.n_contrib, "loss": tr.loss, "grad2d": tr.grad2d,
               "rows": tr.count, "mask": tr.masks[0], "conflicts": s["counts"], **_state_of(tr)}
        if case["active"]:
            tr.active_set(0)
            out.update(active_mask=tr.active_masks[0], active_count=tr.active_count, evidence_sum=tr.evidence_sum)
        return out
    if kind == "render":
        tr, cam = s["tr"], s["cams"][0]
        tr.project(cam)
        tr.bin_sort(want_keys=False)
        tr.render_fwd(cam)
        p = tr.proj
        return {"image": tr.out, "final_T": tr.final_T, "n_contrib": tr.n_contrib, "vals": tr.vals, "ranges": tr.ranges,
                "prim_id": p.prim_id, "xy": p.xy, "depth": p.depth, "conic_opacity": p.conic_opacity, "rgb": p.rgb,
                "rect": p.rect, "tiles": p.tiles_touched, "rows": p.num_rows, "instances": p.num_instances}
    if kind == "unit":
        tr = s["tr"]
        s["step"] += 1
        tr.unit_step(s["cams"], s["targets"], s["step"], LR, BETA1, BETA2, EPS, slots=(0, 1))
        u = tr.prepare_unit()
        return {"loss": u["loss"], "union": u["mask"], "count": u["count_u"], "masks": tr.masks, **_state_of(tr)}
    if kind == "host":
        tr, views, got = s["tr"], case["views"], []
        first = s["step"]
        s["step"] += views
        tr.train_from_host(range(first, first + views), cam_of=lambda t: s["cams"][t - first],
                           host_target_of=lambda t: s["targets"][t - first], lr=LR, beta1=BETA1, beta2=BETA2, eps=EPS,
                           pairs_of=lambda t: (s["pairs"], WINDOW), d_counts=s["counts"],
                           on_result=lambda t, loss, touched, counts: got.append((loss, touched, counts)))
        return {"loss": [r[0] for r in got], "touched": [r[1] for r in got], "counts": [r[2] for r in got],
                "image": tr.out, **_state_of(tr)}
    ctx, n = s["ctx"], case["n"]
    if kind == "admission":
        reads, writes, u = s["reads"], s["writes"], case["units"]
        stride, masks = reads.shape[1], reads.shape[0]
        B.odin_mask_union(ctx, reads, masks, stride, n, s["members"], 2, reads[u + 2])
        B.odin_mask_union(ctx, writes, masks, stride, n, s["members"], 2, writes[u + 2])
        B.odin_mask_to_list(ctx, writes[u + 2], n, s["idx"], n, s["count"], s["ws"])
        B.odin_hazard_count(ctx, reads, writes, masks, stride, n, s["pairs"], u, s["counts"])
        B.odin_delayed_read_gate(ctx, reads[u + 2], writes[u + 2], writes[0], n, s["active"], s["evidence"],
                                 s["active_count"], s["evidence_sum"], s["active"].numel(), TAU, s["gate"])
        return {"read": reads[u + 2], "write": writes[u + 2], "idx": s["idx"], "count": s["count"], "hazards": s["counts"],
                "gate": s["gate"]}
    views = case["views"]
    B.odin_conflict_count(ctx, s["masks"], views, s["masks"].shape[1], n, s["pairs"], s["pairs"].shape[0], s["counts"])
    B.odin_rlg_weights(ctx, s["counts"], s["sizes"], s["pairs"], s["pairs"].shape[0], views, s["edge"])
    flat = s["weights"].view(-1)
    flat[s["upper"]] = s["edge"]
    flat[s["lower"]] = s["edge"]
    B.odin_rlg_topk(ctx, s["weights"], views, KEEP, s["graph"], s["ws"])
    B.odin_sds_scores(ctx, s["graph"], views, s["prev"], 2, s["cand"], views - 2, s["scores"])
    return {"counts": s["counts"], "edge": s["edge"], "graph": s["graph"], "scores": s["scores"]}


# ------------------------------------------------------------------------------------------------ work and tolerance
# share of the pool that is visible, tiles per visible primitive at full HD, share of the visible primitives that blend,
# and blended pairs per pixel: what the scenes above show
_SHOWN = {"box": (0.9, 40.0, 1.0, 20.0), "blob": (0.75, 30.0, 0.9, 60.0), "unbounded": (0.3, 35.0, 0.03, 70.0),
          "air": (0.02, 4.5, 0.97, 30.0), "street": (0.04, 4.7, 0.6, 34.0)}


def work(case):
    kind = case["kind"]
    if kind == "admission":
        words = case["n"] / 8.0
        u = case["units"]
        # every scope once, the unit's own written, its list (a tenth of the pool), the evidence of the producer
        return {"bytes": words * (2 * (u + 2) + 2) + 4.0 * 0.1 * case["n"] + 8.0 * 0.1 * case["n"], "flops": words / 4 * 8 * u}
    if kind == "graph":
        v = case["views"]
        return {"bytes": v * case["n"] / 8.0 + 3 * 4.0 * v * v, "flops": v * (v - 1) / 2.0 * case["n"] / 32.0 * 3}
    n, f, p = case["n"], 11 + 3 * (case["sh"] + 1) ** 2, case["width"] * case["height"]
    vis, tiles, blends, pairs = _SHOWN[case["scene"]]
    if case["scene"] in ("air", "street"):  # a camera sees the same number of blocks whatever the size of the city
        vis = min(0.5, vis * 20_000_000 / n)
    rows = vis * n
    inst = rows * max(1.0, tiles * p / 2.07e6 * math.exp(2 * (case["log_scale"] - {"box": -3, "blob": -3, "unbounded": -5}.get(
        case["scene"], math.log(0.3)))))
    inst = min(inst, rows * math.ceil(p / 256.0))
    forward = 12.0 * n + (4 * f - 12) * rows + 4 * n + 61 * rows + 4 * inst + 36 * blends * rows + 20 * p
    flops = 25.0 * pairs * p + 300 * rows
    if kind != "render":
        active = rows * max(blends, case["seen"])
        step = forward + 24 * p + 36 * rows + 12 * rows * blends + 8 * f * blends * rows + 28 * f * active + n / 4.0
        forward, flops = step, 100.0 * pairs * p + 1000 * rows
    times = {"unit": 2, "host": case.get("views", 1)}.get(kind, 1)
    return {"bytes": forward * times, "flops": flops * times}


def tolerance(case):
    if case["kind"] == "admission":
        return "exact"
    if case["kind"] == "graph":  # sums of two weights
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
    if case["kind"] == "render":
        # 32-bit sums; a pixel whose opacity or transmittance sits on a threshold may take one row more or fewer
        return {"rel": 1e-5, "max": 2e-2, "differ": 1e-4}
    # The gradient of an L1 loss is the sign of the residual: a pixel whose residual is within rounding of zero (a few in
    # an image) turns the gradient of the splats that cover it, some of which cover little else.
    return {"rel": 3e-3, "max": 0.5, "differ": 1e-3}
