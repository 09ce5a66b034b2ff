"""The work that users of the edge-alignment library have it do, as measurable cases.

Every case goes through the public entry points (``Scene``, ``EdgeLoss``, ``distance_field``,
``round_bf16``, ``build_viewgraph`` and the C names in ``_binding``).  Inputs are synthetic scenes
of the shapes that the repository's workloads have: 128x96 to 518x518 views (and odd sizes between),
8 to 120 views per scene, each view paired with its nearest ones, edge pixels on 2 to 10 % of the
image, 3 % depth noise, initial poses 2 degrees and 5 % of the scene scale off.

  kind          one pass is
  host_step     ``epo_step_host``: poses in, one optimisation step, poses and loss out
  optimise      poses set, optimiser state cleared, ``steps`` steps, poses and loss read back
  scheduled     the same with a pair budget (Algorithm 3) and the dual-phase schedule
  loss_grad     ``Scene.loss_and_grad``
  autograd      ``EdgeLoss`` forward and backward at non-zero twists
  refine        optimisation steps with the focal and depth modules on (Eqs. 4-5)
  mlp           optimisation steps under the pose MLP (Eq. 3)
  maps          the distance fields of a scene's views (rounded to BF16 where the scene stores it)
  viewgraph     ``build_viewgraph`` (Eq. 2) over all ordered view pairs
  noalloc       ``epo_loss_and_grad_noalloc`` on caller-owned buffers
"""
import math

import numpy as np
import torch

import paper_2607_00579_gb300 as epo

B = epo._binding
CASE = dict(scenes=1, views=32, width=518, height=392, k=8, density=0.1, mixed=False, norm_all=False,
            schedule="default", steps=1, budget=0, stride=4, off_centre=False)


def listed():
    return [
        # a host program stepping a small object capture: all ordered pairs of 8 small views (the
        # repository's smallest scene); launches and latency are everything
        dict(CASE, name="host_step_8v_128x96", kind="host_step", views=8, width=128, height=96, k=0, density=0.14),
        # the ordinary optimisation of one scene in the library's default options (the 32-view ring)
        dict(CASE, name="optimise_32v_518x392", kind="optimise", steps=10),
        # the benchmark's throughput workload: uneven scenes (8 to 120 views, three sizes, 2-8 %
        # edges) in one handle with the schedule that its autotuner picks
        dict(CASE, name="host_step_batch24_uneven", kind="host_step", scenes=24, views=0, width=0, height=0,
             density=0.0, schedule="tex/128/4"),
        # a large collection in the reduced-precision storage (BF16 maps, FP16 depth), 12 neighbours
        dict(CASE, name="optimise_96v_518x518_mixed", kind="optimise", views=96, height=518, k=12, density=0.09,
             mixed=True, schedule="tex/128/4", steps=4),
        # a long walk with Algorithm 3's pair budget and the convergence schedule, checked every 5 steps
        dict(CASE, name="scheduled_120v_518x392", kind="scheduled", views=120, k=10, density=0.05, budget=500, steps=5),
        # one evaluation for an outside optimiser: odd image size, off-centre principal point, Eq. 7's
        # normaliser, every ordered pair
        dict(CASE, name="loss_grad_14v_319x241", kind="loss_grad", views=14, width=319, height=241, k=0,
             density=0.06, norm_all=True, off_centre=True),
        # the objective inside a torch program
        dict(CASE, name="autograd_48v_518x392", kind="autograd", views=48, k=10, density=0.08),
        # focal and per-pixel depth refinement beside the poses
        dict(CASE, name="refine_32v_518x392", kind="refine", density=0.08, steps=2),
        # the paper's own pose parameterisation
        dict(CASE, name="mlp_32v_518x392", kind="mlp", density=0.04, steps=1),
        # building the maps of a scene from its edge masks (Algorithm 1)
        dict(CASE, name="maps_16v_518x392", kind="maps", views=16, density=0.08),
        # choosing the view pairs from predicted depths
        dict(CASE, name="viewgraph_24v_518x392", kind="viewgraph", views=24),
        # a caller that owns all device memory
        dict(CASE, name="noalloc_24v_256x192", kind="noalloc", views=24, width=256, height=192, density=0.06),
    ]


def draw(rng):
    """A case of the same ranges: every kind, sizes spread over their logarithm, odd ones among them."""
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    kind = rng.choice(["host_step", "optimise", "optimise", "scheduled", "loss_grad", "autograd", "refine", "mlp",
                       "maps", "viewgraph", "noalloc"])
    c = dict(CASE, kind=kind, views=log(6, 120), width=log(96, 640), density=rng.uniform(0.02, 0.1))
    c["height"] = max(64, int(c["width"] * rng.uniform(0.6, 1.05)))
    c["k"] = rng.choice([4, 6, 8, 10, 12])
    if c["views"] <= 16 and rng.random() < 0.4:
        c["k"] = 0
    c["off_centre"] = rng.random() < 0.3
    if kind in ("host_step", "optimise", "loss_grad", "autograd"):
        c["mixed"] = rng.random() < 0.25
        c["norm_all"] = rng.random() < 0.25
        c["schedule"] = rng.choice(["default", "default", "tex/128/4"])
    if kind in ("optimise", "scheduled"):
        c["steps"] = rng.choice([1, 5, 10])
    if kind == "scheduled":
        c["budget"] = log(20, 500)
    if kind == "maps":
        c["views"] = log(2, 24)
        c["mixed"] = rng.random() < 0.4
    if kind == "viewgraph":
        c["views"] = log(6, 32)
        c["stride"] = rng.choice([3, 4, 6, 8])
    if kind == "noalloc":
        c["views"] = log(6, 60)
        c["width"], c["height"] = min(c["width"], 400), min(c["height"], 400)
    if kind in ("refine", "mlp"):
        c["views"] = log(6, 64)
    while work(c)["flops"] > 4e9 and c["views"] > 6:  # well below the largest listed cases
        c["views"] -= 1
    return c


# ------------------------------------------------------------------------------------------
# synthetic scenes
# ------------------------------------------------------------------------------------------
def _scene_shapes(case):
    """(views, width, height, density) of every scene of the case: the batch is uneven by its own fixed draw."""
    if case["scenes"] == 1:
        return [(case["views"], case["width"], case["height"], case["density"])]
    r = np.random.default_rng(20260004)
    sizes = [(256, 192), (518, 392), (518, 518)]
    out = []
    for _ in range(case["scenes"]):
        n = int(r.integers(8, 121))
        w, h = sizes[int(r.integers(0, 3))]
        out.append((n, w, h, float(r.uniform(0.02, 0.08))))
    return out


def _hat(w):
    return np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])


def _rotation(w):
    t = float(np.linalg.norm(w))
    if t == 0.0:
        return np.eye(3)
    K = _hat(w / t)
    return np.eye(3) + math.sin(t) * K + (1 - math.cos(t)) * (K @ K)


def _cameras(r, n):
    """n world-to-camera poses on a ring of radius 15 looking at the centre, and their perturbation."""
    gt, init = np.zeros((n, 12)), np.zeros((n, 12))
    for v in range(n):
        th = 2 * math.pi * v / n + r.normal(0, 0.02)
        c = np.array([15 * math.cos(th), 15 * math.sin(th), r.uniform(-1, 1)])
        f = r.normal(0, 0.2, 3) - c
        f /= np.linalg.norm(f)
        x = np.cross(f, [0.0, 0.0, 1.0])
        x /= np.linalg.norm(x)
        R = np.stack([x, np.cross(f, x), f])
        gt[v] = np.concatenate([R, -(R @ c)[:, None]], 1).ravel()
        if v:
            R = _rotation(r.normal(0, math.radians(2.0), 3)) @ R
            c = c + r.normal(0, 0.05 * 15, 3)
        init[v] = np.concatenate([R, -(R @ c)[:, None]], 1).ravel()
    return gt, init


def _pairs(gt, k):
    n = len(gt)
    M = gt.reshape(n, 3, 4)
    C = -np.einsum("nji,nj->ni", M[:, :, :3], M[:, :, 3])
    D = np.linalg.norm(C[:, None] - C[None], axis=2)
    k = n - 1 if k == 0 else min(k, n - 1)
    out = []
    for i in range(n):
        out += [(i, int(j)) for j in np.argsort(D[i], kind="stable") if j != i][:k]
    return np.array(out, dtype=np.int32)


def _intrinsics(case, r, n, w, h):
    K = np.zeros((n, 4))
    K[:, 0] = K[:, 1] = 1.1 * w
    K[:, 2], K[:, 3] = (w - 1) / 2, (h - 1) / 2
    if case["off_centre"]:
        K[:, 2:] += r.uniform(-0.04, 0.04, (n, 2)) * [w, h]
        K[:, :2] *= r.uniform(0.97, 1.03, (n, 2))
    return K


def _scene(case, seed, index, shape):
    """One scene on the GPU: cameras around a cube of 3D line segments, whose visible pixels are the
    edges; records are a uniform subset of them in raster order, with noisy depth."""
    n, w, h, density = shape
    r = np.random.default_rng([int(seed), index, 1])
    g = torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + index) % (1 << 62))
    gt, init = _cameras(r, n)
    K = _intrinsics(case, r, n, w, h)
    target = max(32, int(round(density * w * h)))
    n_seg = max(16, int(2.2 * target / (0.3 * w)))  # a segment covers about 0.3 w pixels of a view
    seg = torch.from_numpy(r.uniform(-5, 5, (n_seg, 2, 3))).cuda()
    s = torch.linspace(0, 1, w, dtype=torch.float64, device="cuda")[None, :, None]
    X = (seg[:, :1] * (1 - s) + seg[:, 1:] * s).reshape(-1, 3)
    M = torch.from_numpy(gt.reshape(n, 3, 4)).cuda()
    records, masks = [], []
    ys, xs = torch.meshgrid(torch.arange(h, device="cuda"), torch.arange(w, device="cuda"), indexing="ij")
    for v in range(n):
        Y = X @ M[v, :, :3].T + M[v, :, 3]
        z = Y[:, 2]
        u = torch.round(K[v, 0] * Y[:, 0] / z + K[v, 2]).long()
        q = torch.round(K[v, 1] * Y[:, 1] / z + K[v, 3]).long()
        ok = (z > 0.1) & (u >= 0) & (u < w) & (q >= 0) & (q < h)
        depth = torch.full((h * w + 1,), math.inf, dtype=torch.float64, device="cuda")
        depth.scatter_reduce_(0, torch.where(ok, q * w + u, h * w), torch.where(ok, z, math.inf), "amin")
        depth = depth[:-1]
        edge = torch.isfinite(depth)
        masks.append(edge.view(h, w).to(torch.uint8))
        pix = torch.nonzero(edge)[:, 0]
        if len(pix) > target:
            pix = pix[torch.randperm(len(pix), generator=g, device="cuda")[:target].sort().values]
        a = torch.from_numpy(r.normal(0, 1, 4)).cuda()
        field = 1 + 0.03 * (a[0] * torch.sin(5.0 * xs / w + a[1]) + a[2] * torch.cos(4.0 * ys / h + a[3])).reshape(-1)
        rec = torch.zeros((len(pix), 4), dtype=torch.float32, device="cuda")
        rec[:, 0], rec[:, 1] = (pix % w).float(), (pix // w).float()
        rec[:, 2] = (depth[pix] * field[pix]).float()
        records.append(rec)
    off = np.concatenate([[0], np.cumsum([len(x) for x in records])]).astype(np.int64)
    fixed = np.zeros(n, dtype=np.uint8)
    fixed[0] = 1
    return dict(W=np.full(n, w, np.int32), H=np.full(n, h, np.int32), K=K, rec_off=off, rec=torch.cat(records),
                masks=masks, pairs=_pairs(gt, case["k"]), fixed=fixed, T=init)


def _scenes(case, seed):
    return [_scene(case, seed, i, s) for i, s in enumerate(_scene_shapes(case))]


def _f16_records(rec):
    out = torch.zeros((len(rec), 4), dtype=torch.int16, device=rec.device)
    out[:, 0], out[:, 1] = rec[:, 0].to(torch.int16), rec[:, 1].to(torch.int16)
    out[:, 2] = rec[:, 2].half().view(torch.int16)
    return out


def _depth_maps(case, seed):
    """Dense depth of every view: spheres inside a large one, with the same smooth noise."""
    n, w, h = case["views"], case["width"], case["height"]
    r = np.random.default_rng([int(seed), 2])
    gt, init = _cameras(r, n)
    K = _intrinsics(case, r, n, w, h)
    ctr = torch.from_numpy(np.concatenate([np.zeros((1, 3)), r.uniform(-5, 5, (10, 3))])).cuda()
    rad = torch.from_numpy(np.concatenate([[25.0], r.uniform(1.0, 2.5, 10)])).cuda()
    ys, xs = torch.meshgrid(torch.arange(h, device="cuda", dtype=torch.float64),
                            torch.arange(w, device="cuda", dtype=torch.float64), indexing="ij")
    maps = []
    for v in range(n):
        M = torch.from_numpy(gt[v].reshape(3, 4)).cuda()
        d = torch.stack([(xs - K[v, 2]) / K[v, 0], (ys - K[v, 3]) / K[v, 1], torch.ones_like(xs)], -1).reshape(-1, 3)
        c = ctr @ M[:, :3].T + M[:, 3]  # sphere centres in the camera's frame
        dd, dc = (d * d).sum(1)[:, None], d @ c.T
        disc = dc * dc - dd * ((c * c).sum(1) - rad * rad)
        root = torch.sqrt(disc.clamp_min(0))
        near, far = (dc - root) / dd, (dc + root) / dd
        t = torch.where(near > 1e-3, near, far)
        t = torch.where((disc > 0) & (t > 1e-3), t, math.inf).min(1).values
        a = r.normal(0, 1, 4)
        field = 1 + 0.004 * (a[0] * torch.sin(5.0 * xs / w + a[1]) + a[2] * torch.cos(4.0 * ys / h + a[3])).reshape(-1)
        maps.append((t * field).float().view(h, w))
    return np.full(n, w, np.int32), np.full(n, h, np.int32), K, init, maps


# ------------------------------------------------------------------------------------------
# a pass
# ------------------------------------------------------------------------------------------
def _options(case):
    o = dict(norm_mode=epo.EPO_NORM_ALL if case["norm_all"] else epo.EPO_NORM_VALID)
    if case["schedule"] != "default":
        gather, block, rpt = case["schedule"].split("/")
        o.update(gather={"ldg": epo.EPO_GATHER_LDG, "tex": epo.EPO_GATHER_TEX}[gather], block_threads=int(block),
                 records_per_thread=int(rpt))
    if case["kind"] == "scheduled":
        o.update(schedule=1, pair_budget=case["budget"], subsample_seed=7)
    if case["kind"] == "refine":
        o.update(refine=1, lr_focal=1e-4, lr_depth=1e-4)
    if case["kind"] == "mlp":
        o.update(pose_param=B.EPO_POSE_MLP)
    return epo.default_options(**o)


def _mlp_init(seed):
    r = np.random.default_rng([int(seed), 3])
    parts = []
    for l, (o, i) in enumerate([(128, 12)] + [(128, 128)] * 4 + [(12, 128)]):
        parts += [np.zeros(o * i) if l == 5 else r.normal(0, math.sqrt(2 / i), o * i), np.zeros(o)]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "viewgraph":
        W, H, K, T, maps = _depth_maps(case, seed)
        return dict(case=case, W=W, H=H, K=K, T=T, depth=torch.cat([m.reshape(-1) for m in maps]))
    scenes = _scenes(case, seed)
    if kind == "maps":
        return dict(case=case, masks=scenes[0]["masks"])
    parts = []
    for sc in scenes:
        maps = [epo.distance_field(m) for m in sc["masks"]]
        if case["mixed"]:
            maps = [epo.round_bf16(m) for m in maps]
        rec = _f16_records(sc["rec"]) if case["mixed"] else sc["rec"]
        parts.append(dict(W=sc["W"], H=sc["H"], K=sc["K"], rec_off=sc["rec_off"], rec=rec, maps=maps,
                          pairs=sc["pairs"], fixed=sc["fixed"]))
    T = np.concatenate([sc["T"] for sc in scenes])
    if kind == "noalloc":
        return _noalloc_state(case, scenes[0], parts[0]["maps"])
    dt = (epo.EPO_F16, epo.EPO_BF16) if case["mixed"] else (epo.EPO_F32, epo.EPO_F32)
    scene = epo.Scene(parts, record_dtype=dt[0], map_dtype=dt[1], options=_options(case), on_device=True)
    if kind == "mlp":
        B.epo_set_pose_mlp(scene.handle, _mlp_init(seed))
    scene.set_poses(T)
    st = dict(case=case, scene=scene, T=T, n_records=sum(len(sc["rec"]) for sc in scenes))
    if kind == "host_step":
        pin = lambda *s: torch.zeros(s, dtype=torch.float64).pin_memory().numpy()
        st.update(T_in=pin(*T.shape), T_out=pin(*T.shape), loss=pin(scene.n_scenes))
        st["T_in"][:] = T
    if kind == "autograd":
        r = np.random.default_rng([int(seed), 4])
        xi = torch.from_numpy(r.normal(0, 0.01, (scene.n_views, 6)))
        st["xi"] = xi.cuda().requires_grad_(True)
        st["weight"] = torch.from_numpy(r.uniform(0.5, 1.5, scene.n_scenes)).cuda()
    return st


def _noalloc_state(case, sc, maps):
    d = lambda a, t: torch.from_numpy(np.ascontiguousarray(np.asarray(a).reshape(-1).astype(t))).cuda()
    size = int(sc["W"][0]) * int(sc["H"][0])
    st = dict(case=case, records=sc["rec"].contiguous(), rec_off=d(sc["rec_off"], np.int64),
              maps=torch.cat([m.reshape(-1) for m in maps]), map_off=d(np.arange(len(maps)) * size, np.int64),
              W=d(sc["W"], np.int32), H=d(sc["H"], np.int32), K=d(sc["K"], np.float64),
              pairs=d(sc["pairs"], np.int32), T=d(sc["T"], np.float64),
              loss=torch.zeros(1, dtype=torch.float64, device="cuda"),
              grad=torch.zeros((case["views"], 6), dtype=torch.float64, device="cuda"))
    p = B.epo_noalloc_problem()
    p.n_views, p.n_pairs = case["views"], len(sc["pairs"])
    p.max_records_per_view = int(np.diff(sc["rec_off"]).max())
    for name in ("records", "rec_off", "maps", "map_off", "W", "H", "K", "pairs", "T"):
        setattr(p, name, st[name].data_ptr())
    p.lam, p.huber_delta, p.eps_z = 10.0, 1.0, 1e-6
    p.norm_mode = epo.EPO_NORM_ALL if case["norm_all"] else epo.EPO_NORM_VALID
    st["problem"] = p
    return st


def _last_loss(scene):
    loss = np.zeros(scene.n_scenes)
    B.epo_last_loss(scene.handle, loss)
    return loss


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "viewgraph":
        frac, pairs = epo.build_viewgraph(state["W"], state["H"], state["K"], state["T"], state["depth"],
                                          stride=case["stride"])
        kept = np.zeros(frac.shape, dtype=np.uint8)
        kept[pairs[:, 0], pairs[:, 1]] = 1
        return dict(frac=frac, kept=kept)
    if kind == "maps":
        maps = [epo.distance_field(m) for m in state["masks"]]
        return [epo.round_bf16(m) for m in maps] if case["mixed"] else maps
    if kind == "noalloc":
        st = B.epo_loss_and_grad_noalloc(state["problem"], state["loss"], state["grad"],
                                         torch.cuda.current_stream().cuda_stream)
        B.check(st)
        return dict(loss=state["loss"], grad=state["grad"])
    scene = state["scene"]
    if kind == "host_step":
        B.epo_step_host(scene.handle, state["T_in"], state["T_out"], state["loss"])
        return dict(T=state["T_out"], loss=state["loss"])
    if kind == "loss_grad":
        loss, grad = scene.loss_and_grad()
        return dict(loss=loss, grad=grad)
    if kind == "autograd":
        xi = state["xi"]
        loss = epo.EdgeLoss.apply(xi, scene)
        (grad,) = torch.autograd.grad((loss * state["weight"]).sum(), xi)
        return dict(loss=loss.detach(), grad=grad)
    if kind in ("optimise", "scheduled"):
        scene.set_poses(state["T"])
        scene.set_state(0)
    scene.step(case["steps"])
    out = dict(T=scene.get_poses(), loss=_last_loss(scene))
    if kind == "scheduled":
        out["theta"], out["phase"] = B.epo_get_schedule(scene.handle, scene.n_scenes)[:2]
    if kind == "refine":
        out["gamma"], out["alpha"], out["beta"] = B.epo_get_refinement(scene.handle, scene.n_views,
                                                                       state["n_records"])
    if kind == "mlp":
        out["theta"], out["delta"] = B.epo_get_pose_mlp(scene.handle, scene.n_scenes, scene.n_views)
    return out


def work(case):
    n = case["views"]
    if case["kind"] == "viewgraph":
        grid = -(-case["width"] // case["stride"]) * -(-case["height"] // case["stride"])
        return dict(bytes=n * grid * 8 + n * n * 8, flops=n * (n - 1) * grid * 80)
    if case["kind"] == "maps":
        px = n * case["width"] * case["height"]
        return dict(bytes=px * (3 if case["mixed"] else 5), flops=px * 10)
    size = 2 if case["mixed"] else 4
    byts = flops = 0
    for v, w, h, d in _scene_shapes(case):
        k = v - 1 if case["k"] == 0 else min(case["k"], v - 1)
        rec = max(32, int(d * w * h))
        pairs = min(v * k, case["budget"] or v * k)
        evals = pairs * rec
        byts += v * rec * (8 if case["mixed"] else 16) + v * w * h * size + pairs * 64 + v * 200
        flops += evals * 85  # transform, projection, bilinear value and slopes, penalty, adjoint
        if case["kind"] == "refine":
            byts += v * rec * 48
            flops += evals * 25
        if case["kind"] == "mlp":
            byts += 69260 * 24
            flops += v * 69260 * 6
    return dict(bytes=byts * case["steps"], flops=flops * case["steps"])


# ------------------------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ------------------------------------------------------------------------------------------
def _exact_edt(masks):
    """Exact Euclidean distance of every pixel to the nearest set pixel (W + H in an empty image)."""
    m = torch.stack(masks).bool()
    n, h, w = m.shape
    x = torch.arange(w, device="cuda", dtype=torch.float64)
    left = torch.where(m, x, -math.inf).cummax(2).values
    right = torch.where(m, x, math.inf).flip(2).cummin(2).values.flip(2)
    f = torch.minimum(x - left, right - x) ** 2
    best = f.clone()
    for d in range(1, h):
        if float(d) ** 2 >= float(best.max()):
            break
        best[:, d:] = torch.minimum(best[:, d:], f[:, :-d] + float(d) ** 2)
        best[:, :-d] = torch.minimum(best[:, :-d], f[:, d:] + float(d) ** 2)
    return torch.where(torch.isinf(best), float(w + h), best.sqrt())


def _exact_inputs(case, sc):
    """The values the scene stores, widened: records (n, 3) and maps (views, H, W)."""
    rec = sc["rec"][:, :3].double()
    maps = _exact_edt(sc["masks"]).float()
    if case["mixed"]:
        rec[:, 2] = sc["rec"][:, 2].half().double()
        maps = maps.bfloat16()
    return rec, maps.double()


def _objective(case, sc, rec, maps, T, lam, active=None, gamma=None, alpha=None, beta=None, scale=1.0):
    """The objective of one scene and its gradients with respect to the leaves among (T, gamma, alpha,
    beta): the backward pass runs per source view, so that no more than one view's samples are held."""
    w, h = int(sc["W"][0]), int(sc["H"][0])
    K = torch.from_numpy(sc["K"]).cuda()
    pairs = sc["pairs"] if active is None else sc["pairs"][active]
    off, total = sc["rec_off"], torch.zeros((), dtype=torch.float64, device="cuda")
    leaves = [x for x in (T, gamma, alpha, beta) if x is not None and x.requires_grad]
    grads = [torch.zeros_like(x) for x in leaves]
    for i in range(len(sc["W"])):
        js = torch.from_numpy(pairs[pairs[:, 0] == i, 1].astype(np.int64)).cuda()
        a, b = int(off[i]), int(off[i + 1])
        if not len(js) or a == b:
            continue
        M = T.view(-1, 3, 4)
        f = K[:, :2] if gamma is None else K[:, :2] * (1 + gamma)[:, None]
        z = rec[a:b, 2] if alpha is None else rec[a:b, 2] * alpha[a:b] + beta[a:b]
        X = torch.stack([(rec[a:b, 0] - K[i, 2]) / f[i, 0] * z, (rec[a:b, 1] - K[i, 3]) / f[i, 1] * z, z], 1)
        world = (X - M[i, :, 3]) @ M[i, :, :3]
        Y = torch.einsum("prc,nc->pnr", M[js, :, :3], world) + M[js, None, :, 3]
        front = Y[..., 2] > 1e-6
        iz = 1 / torch.where(front, Y[..., 2], 1.0)
        u = f[js, 0, None] * Y[..., 0] * iz + K[js, 2, None]
        v = f[js, 1, None] * Y[..., 1] * iz + K[js, 3, None]
        ok = front & (u >= 0) & (u <= w - 1) & (v >= 0) & (v <= h - 1)
        x0 = torch.where(ok, u.detach().floor(), 0).clamp(max=w - 2)
        y0 = torch.where(ok, v.detach().floor(), 0).clamp(max=h - 2)
        ca, cb = u - x0, v - y0
        at = (js[:, None] * (w * h) + y0.long() * w + x0.long())
        flat = maps.reshape(-1)
        m00, m01, m10, m11 = flat[at], flat[at + 1], flat[at + w], flat[at + w + 1]
        d = (1 - cb) * ((1 - ca) * m00 + ca * m01) + cb * ((1 - ca) * m10 + ca * m11)
        d = torch.where(d <= lam, d, lam)
        rho = torch.where(d.abs() <= 1, 0.5 * d * d, d.abs() - 0.5)
        rho = torch.where(ok, rho, 0.0).sum(1)
        n = ok.sum(1).double() if not case["norm_all"] else torch.full_like(rho, float(b - a))
        part = scale * (2.0 / len(pairs)) * torch.where(n > 0, rho / n.clamp(min=1), 0.0).sum()
        if leaves:
            for g, x in zip(grads, torch.autograd.grad(part, leaves, retain_graph=False, allow_unused=True)):
                if x is not None:
                    g += x
        total = total + part.detach()
    return total, grads


def _left_gradient(T, G):
    """dL/dT (n, 12) -> the gradient with respect to a left perturbation Exp(xi) T, xi = (translation, rotation)."""
    M, D = T.view(-1, 3, 4), G.view(-1, 3, 4)
    S = D @ M.transpose(1, 2)
    return torch.cat([D[:, :, 3], torch.stack([S[:, 2, 1] - S[:, 1, 2], S[:, 0, 2] - S[:, 2, 0],
                                               S[:, 1, 0] - S[:, 0, 1]], 1)], 1)


def _exp(xi):
    A = torch.zeros((len(xi), 4, 4), dtype=torch.float64, device="cuda")
    A = A.index_put((torch.arange(len(xi)).cuda()[:, None], torch.tensor([0, 1, 2]).cuda(), torch.tensor([3, 3, 3]).cuda()), xi[:, :3])
    for r, c, k, s in ((0, 1, 5, -1), (0, 2, 4, 1), (1, 0, 5, 1), (1, 2, 3, -1), (2, 0, 4, -1), (2, 1, 3, 1)):
        E = torch.zeros((4, 4), dtype=torch.float64, device="cuda")
        E[r, c] = s
        A = A + xi[:, k, None, None] * E
    return torch.linalg.matrix_exp(A)


def _moved(xi, T):
    """Exp(xi) T."""
    T4 = torch.zeros((len(T), 4, 4), dtype=torch.float64, device="cuda")
    T4[:, :3] = T.view(-1, 3, 4)
    T4[:, 3, 3] = 1
    return (_exp(xi) @ T4)[:, :3].reshape(-1, 12)


def _drawn_pairs(case, n_pairs, step):
    """Algorithm 3's subset: the pairs with the smallest SplitMix64(seed ^ (step << 32 | p))."""
    if not case["budget"] or case["budget"] >= n_pairs:
        return None
    with np.errstate(over="ignore"):
        x = (np.uint64(7) ^ ((np.uint64(step) << np.uint64(32)) | np.arange(n_pairs, dtype=np.uint64)))
        x = x + np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        x = x ^ (x >> np.uint64(31))
    act = np.zeros(n_pairs, dtype=bool)
    act[np.argsort(x, kind="stable")[:case["budget"]]] = True
    return act


def _adam(p, g, lr, t, mom):
    m, v = mom
    m.mul_(0.9).add_(0.1 * g)
    v.mul_(0.999).add_(0.001 * g * g)
    return lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-12)


def _exact_steps(case, scenes):
    """`steps` optimisation steps from the initial poses: poses, loss of the last step and the refinement."""
    out_T, out_loss, extra = [], [], {}
    lr = torch.tensor([2e-2] * 3 + [2e-3] * 3, dtype=torch.float64, device="cuda")
    for sc in scenes:
        rec, maps = _exact_inputs(case, sc)
        T = torch.from_numpy(sc["T"]).cuda()
        mom = [torch.zeros((len(T), 6), dtype=torch.float64, device="cuda") for _ in range(2)]
        ref = None
        if case["kind"] == "refine":
            ref = [torch.zeros(len(T), dtype=torch.float64, device="cuda"),
                   torch.ones(len(rec), dtype=torch.float64, device="cuda"),
                   torch.zeros(len(rec), dtype=torch.float64, device="cuda")]
            rmom = [[torch.zeros_like(x), torch.zeros_like(x)] for x in ref]
        for s in range(case["steps"]):
            leaves = [x.clone().requires_grad_(True) for x in [T] + (ref or [])]
            kw = dict(zip(("gamma", "alpha", "beta"), leaves[1:]))
            loss, grads = _objective(case, sc, rec, maps, leaves[0], 10.0 - 4.0 * s / 1000,
                                     _drawn_pairs(case, len(sc["pairs"]), s), **kw)
            delta = _adam(None, _left_gradient(T, grads[0]), lr, s + 1, mom)
            delta[0] = 0
            T = _moved(-delta, T)
            if ref:
                ref = [x - _adam(None, g, 1e-4, s + 1, m) for x, g, m in zip(ref, grads[1:], rmom)]
        out_T.append(T.cpu().numpy())
        out_loss.append(float(loss))
        if ref:
            extra = dict(gamma=ref[0].cpu().numpy(), alpha=ref[1].cpu().numpy(), beta=ref[2].cpu().numpy())
    return np.concatenate(out_T), np.array(out_loss), extra


def _exact_mlp(case, seed, sc):
    """One AdamW step under the pose MLP from its initial weights (the last layer is zero)."""
    rec, maps = _exact_inputs(case, sc)
    P0 = torch.from_numpy(sc["T"]).cuda()
    M = P0.view(-1, 3, 4)
    C = -(M[:, :, :3] * M[:, :, 3:]).sum(1)
    s = float(((C - C.mean(0)) ** 2).sum(1).mean().sqrt())
    unit = torch.tensor([1, 1, 1, s] * 3, dtype=torch.float64, device="cuda")

    def poses(theta, delta):
        at, layers = 0, []
        for o, i in [(128, 12)] + [(128, 128)] * 4 + [(12, 128)]:
            layers.append((theta[at:at + o * i].view(o, i), theta[at + o * i:at + o * i + o]))
            at += o * i + o
        x = P0 / unit
        for l, (W, b) in enumerate(layers):
            x = x @ W.T + b
            if l < 5:
                x = x.relu()
            if l == 0:
                first = x
            if l == 2:
                x = x + first
        P = (P0 + unit * x).view(-1, 3, 4)
        b1 = P[:, :, 0] / P[:, :, 0].norm(dim=1, keepdim=True)
        u2 = P[:, :, 1] - (b1 * P[:, :, 1]).sum(1, keepdim=True) * b1
        b2 = u2 / u2.norm(dim=1, keepdim=True)
        return torch.stack([b1, b2, torch.linalg.cross(b1, b2), P[:, :, 3] + s * delta], 2).reshape(-1, 12)

    theta = torch.from_numpy(_mlp_init(seed)).cuda().double().requires_grad_(True)
    delta = torch.zeros((len(P0), 3), dtype=torch.float64, device="cuda", requires_grad=True)
    T = poses(theta, delta)
    at = T.detach().requires_grad_(True)
    loss, (G,) = _objective(case, sc, rec, maps, at, 10.0)
    # the objective's gradient in the rotations' tangent only
    g = _left_gradient(at.detach(), G)
    lam, R = g[:, 3:] - torch.linalg.cross(at.detach().view(-1, 3, 4)[:, :, 3], g[:, :3]), at.detach().view(-1, 3, 4)[:, :, :3]
    E = 0.5 * torch.stack([torch.linalg.cross(lam, R[:, :, c]) for c in range(3)], 2)
    D = torch.cat([E, g[:, :3, None]], 2).reshape(-1, 12)
    gt, gd = torch.autograd.grad(T, (theta, delta), D)
    lr = 3e-3 / 25
    new = []
    for p, q, wd in ((theta, gt, 0.01), (delta, gd, 0.1)):
        new.append(p.detach() * (1 - lr * wd) - lr * q / (q.abs() + 1e-8))
    with torch.no_grad():
        T = poses(*new)
    return dict(T=T.cpu().numpy(), loss=np.array([float(loss)]), theta=new[0].cpu().numpy()[None],
                delta=new[1].cpu().numpy())


def _exact_viewgraph(case, seed):
    W, H, K, T, maps = _depth_maps(case, seed)
    n, w, h, s = len(W), int(W[0]), int(H[0]), case["stride"]
    T, K = T.reshape(n, 3, 4), K
    y, x = torch.meshgrid(torch.arange(0, h, s, device="cuda"), torch.arange(0, w, s, device="cuda"), indexing="ij")
    x, y = x.reshape(-1), y.reshape(-1)
    frac = np.zeros((n, n))

    def move(i, j, px, py, z):
        X = [(px - K[i, 2]) / K[i, 0] * z - T[i, 0, 3], (py - K[i, 3]) / K[i, 1] * z - T[i, 1, 3], z - T[i, 2, 3]]
        Wd = [T[i, 0, c] * X[0] + T[i, 1, c] * X[1] + T[i, 2, c] * X[2] for c in range(3)]
        Y = [T[j, r, 0] * Wd[0] + T[j, r, 1] * Wd[1] + T[j, r, 2] * Wd[2] + T[j, r, 3] for r in range(3)]
        ok = Y[2] > 0
        iz = torch.where(ok, Y[2], 1.0)
        return ok, K[j, 0] * Y[0] / iz + K[j, 2], K[j, 1] * Y[1] / iz + K[j, 3]

    depth = [m.double() for m in maps]
    for i in range(n):
        z = depth[i][y, x]
        valid = (z > 0) & torch.isfinite(z)
        for j in range(n):
            if i == j:
                continue
            ok, u, v = move(i, j, x.double(), y.double(), z)
            ok = ok & valid & (u >= 0) & (u <= w - 1) & (v >= 0) & (v <= h - 1)
            un, vn = torch.where(ok, u + 0.5, 0.0).floor().long(), torch.where(ok, v + 0.5, 0.0).floor().long()
            zj = depth[j][vn, un]
            ok = ok & (zj > 0) & torch.isfinite(zj)
            back, a, b = move(j, i, u, v, zj)
            good = ok & back & (((a - x) ** 2 + (b - y) ** 2).sqrt() < 3.0)
            frac[i, j] = float(good.sum()) / max(1.0, float(valid.sum()))
    keep = np.minimum(frac, frac.T) >= 0.125
    np.fill_diagonal(keep, False)
    return dict(frac=frac, kept=keep.astype(np.uint8))


def exact(case, seed):
    kind = case["kind"]
    if kind == "viewgraph":
        return _exact_viewgraph(case, seed)
    scenes = _scenes(case, seed)
    if kind == "maps":
        fields = _exact_edt(scenes[0]["masks"])
        return [None] * len(fields) if case["mixed"] else list(fields)
    if kind == "mlp":
        return _exact_mlp(case, seed, scenes[0])
    if kind in ("host_step", "optimise", "scheduled", "refine"):
        T, loss, extra = _exact_steps(case, scenes)
        if kind == "scheduled":
            extra = dict(theta=None, phase=None)
        return dict(T=T, loss=loss, **extra)
    sc = scenes[0]
    rec, maps = _exact_inputs(case, sc)
    T = torch.from_numpy(sc["T"]).cuda()
    if kind == "autograd":
        r = np.random.default_rng([int(seed), 4])
        xi = torch.from_numpy(r.normal(0, 0.01, (len(T), 6))).cuda().requires_grad_(True)
        weight = float(r.uniform(0.5, 1.5, 1)[0])
        moved = _moved(xi, T)
        at = moved.detach().requires_grad_(True)
        loss, (G,) = _objective(case, sc, rec, maps, at, 10.0)
        (grad,) = torch.autograd.grad(moved, xi, weight * G)
        return dict(loss=loss.reshape(1), grad=grad)
    at = T.clone().requires_grad_(True)
    loss, (G,) = _objective(case, sc, rec, maps, at, 10.0)
    grad, loss = _left_gradient(T, G), loss.reshape(1)
    if kind == "loss_grad":
        grad, loss = grad.cpu().numpy(), loss.cpu().numpy()
    return dict(loss=loss, grad=grad)
