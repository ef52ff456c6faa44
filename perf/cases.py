"""The work that is timed: what a user of the framework has it do, through its
public entry points.

A case is a scene, a set of views and one operation on them:

  query         Index.build + gpf_radiance_fwd: an image from a field
  grad          gpf_radiance (autograd) and its gradient: a step of a loop that
                keeps its own loss and optimiser
  train         one TrainStep (build, forward, MSE, backward, Adam), eager or as
                a replay of the captured graph, from float32 or 16-bit storage
  hybrid_query  a query through the paper's neighbourhood (ball or k_min nearest)
  hybrid_grad   the same with its loss gradient and backward
  kde           the photon density estimate that the field replaces

Scenes: the analytic floor and sphere with a caustic photon map (70 % of the
photons in eight anisotropic 2D blobs on the floor, 30 % uniform by area), one
Gaussian per photon, scaled by the distance to its 8th nearest photon (drawn
from that distance's distribution at the local photon density) and stretched
and rotated at random, as a field is in the middle of its training; or the
unit cube filled with random Gaussians and random hit points. Everything is
drawn on the GPU from the seed alone.
"""

import math

import torch

import paper_2512_12459_gb300 as gpf
from paper_2512_12459_gb300.setup_index import make_index
from paper_2512_12459_gb300.train import TrainStep

R = gpf.PAPER_R                       # falloff, ball and gather radius
EPS = gpf.PAPER_EPS
LR = gpf.PAPER_LR
CUTOFF = 3.0
NEAREST = 8                           # a Gaussian's scale: distance to this neighbour
ANISOTROPY = 0.25                     # spread of the log-scales around it
FLOOR, SPHERE_Z, SPHERE_R = 4.0, 1.0, 1.0
LOOK_AT = (0.0, 0.0, 0.5)
VFOV = 45.0
UNEVEN = (256, 384, 512, 768, 1024)   # sides of the views of an uneven batch

BASE = {"scene": "caustic", "views": "one", "n_views": 1, "width": 1024, "height": 1024,
        "channels": 3, "mode": "sum", "r": R, "albedo": False, "storage": "f32",
        "graph": False, "tuned": True, "cell": 0.02, "k_min": 3}


def _case(name, op, n, **kw):
    return dict(BASE, name=name, op=op, n=n, **kw)


def listed():
    return [
        # the smallest call: a few thousand Gaussians in a cube, planned with
        # the defaults and summed without falloff (the entry points' defaults)
        _case("query_cube_4k", "query", 4096, scene="cube", width=16384, height=1, r=math.inf,
              tuned=False, cell=0.08),
        # a preview-sized fit replayed as a graph: launches and gaps count
        _case("train_small_graph", "train", 10_000, width=128, height=128, graph=True,
              tuned=False, cell=0.05),
        # an image of a mid-sized field, softly normalised as the paper queries it
        _case("query_100k_800", "query", 100_000, width=800, height=800, mode="normalized"),
        # the reference camera's image of a full field
        _case("query_1m_1024", "query", 1_000_000),
        # odd sizes, an albedo, four bins, through autograd, on a default plan
        _case("grad_200k_ragged", "grad", 200_003, width=611, height=907, channels=4,
              mode="normalized", albedo=True, r=0.05, tuned=False),
        # the framework's benchmark: one step at a million Gaussians and one view
        _case("train_1m_1024", "train", 1_000_000),
        # the multi-view fit: eight orbit views as one batch, graph replay
        _case("train_1m_8views_graph", "train", 1_000_000, views="orbit", n_views=8, width=800,
              height=800, graph=True),
        # eight spectral bins in 16-bit storage, full-HD views
        _case("train_bf16_8bins", "train", 1_000_000, views="orbit", n_views=2, width=1920,
              height=1080, channels=8, storage="bf16_mean32"),
        # the largest: many uneven views in one batch
        _case("train_2m_64views", "train", 2_000_000, views="uneven", n_views=64, width=0,
              height=0),
        # the baseline that the field replaces: photons gathered over a view
        _case("kde_1m_1024", "kde", 1_000_000, cell=0.04),
        # the paper's own query and its gradient
        _case("hybrid_query_100k", "hybrid_query", 100_000, mode="normalized", tuned=False),
        _case("hybrid_grad_100k", "hybrid_grad", 100_000, width=800, height=800,
              mode="normalized", tuned=False),
    ]


def draw(rng):
    def spread(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    op = rng.choice(["query", "query", "grad", "grad", "train", "train", "train",
                     "hybrid_query", "hybrid_grad", "kde"])
    c = dict(BASE, op=op, n=spread(2000, 1_500_000))
    c["width"], c["height"] = spread(48, 1400), spread(48, 1100)
    c["mode"] = rng.choice(["sum", "normalized"])
    c["channels"] = rng.choice([1, 3, 3, 3, 4, 8])
    c["albedo"] = rng.random() < 0.3
    c["tuned"] = rng.random() < 0.6
    c["cell"] = rng.choice([0.02, 0.02, 0.04])
    if op in ("query", "grad"):
        c["r"] = rng.choice([R, R, 0.05])
        if rng.random() < 0.3:
            c.update(scene="cube", n=spread(500, 8000), width=spread(500, 40_000), height=1,
                     tuned=False, cell=0.08, r=rng.choice([math.inf, 0.08]))
    elif op == "train":
        c["graph"] = rng.random() < 0.5
        c["storage"] = rng.choice(["f32", "f32", "f32", "bf16_mean32", "bf16"])
        if rng.random() < 0.4:
            c["views"], c["n_views"] = "orbit", rng.randint(2, 8)
            c["width"], c["height"] = min(c["width"], 1000), min(c["height"], 800)
    elif op == "kde":
        c.update(mode="sum", cell=0.04)
    else:
        c.update(n=spread(5000, 250_000), k_min=rng.choice([0, 1, 3, 3, 5, 10]), tuned=False,
                 channels=3)
        c["width"], c["height"] = min(c["width"], 1024), min(c["height"], 1024)
    return c


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 2654435761 % (1 << 31))


def _uni(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _f32(t):
    return t.to(torch.float32).contiguous()


def _caustic_photons(g, n):
    """Positions [n, 3] and the photons per unit area around each."""
    nb = int(round(0.7 * n))
    centre = _uni(g, 8, 2, lo=-2.5, hi=2.5)
    std = torch.exp(_uni(g, 8, 2, lo=math.log(0.02), hi=math.log(0.3)))
    ang = _uni(g, 8, hi=math.pi)
    ca, sa = torch.cos(ang), torch.sin(ang)
    which = torch.randint(0, 8, (nb,), generator=g, device="cuda")
    z = _normal(g, nb, 2) * std[which]
    blob = centre[which] + torch.stack([ca[which] * z[:, 0] - sa[which] * z[:, 1],
                                        sa[which] * z[:, 0] + ca[which] * z[:, 1]], 1)
    blob = blob.clamp(-FLOOR, FLOOR)
    nu = n - nb
    a_floor, a_sphere = (2 * FLOOR) ** 2, 4 * math.pi * SPHERE_R ** 2
    on_sphere = _uni(g, nu) < a_sphere / (a_floor + a_sphere)
    d = _normal(g, nu, 3)
    d = d / d.norm(dim=1, keepdim=True) * SPHERE_R
    d[:, 2] += SPHERE_Z
    flat = torch.cat([_uni(g, nu, 2, lo=-FLOOR, hi=FLOOR), torch.zeros(nu, 1, device="cuda",
                                                                       dtype=torch.float64)], 1)
    uni = torch.where(on_sphere[:, None], d, flat)
    pos = torch.cat([torch.cat([blob, torch.zeros(nb, 1, device="cuda", dtype=torch.float64)], 1),
                     uni])
    # photons per unit area: the uniform part everywhere, the blobs on the floor
    dens = torch.full((n,), nu / (a_floor + a_sphere), device="cuda", dtype=torch.float64)
    floor = torch.cat([torch.ones(nb, dtype=torch.bool, device="cuda"), ~on_sphere])
    for b in range(8):
        e = pos[:, :2] - centre[b]
        u = (ca[b] * e[:, 0] + sa[b] * e[:, 1]) / std[b, 0]
        v = (-sa[b] * e[:, 0] + ca[b] * e[:, 1]) / std[b, 1]
        dens += floor * nb / 8 / (2 * math.pi * std[b, 0] * std[b, 1]) * torch.exp(
            -0.5 * (u * u + v * v))
    perm = torch.randperm(n, generator=g, device="cuda")
    return pos[perm], dens[perm]


def _gaussians(case, g):
    n, ch = case["n"], case["channels"]
    quat = _normal(g, 4, n)
    quat = quat / quat.norm(dim=0)
    if case["scene"] == "cube":
        return [_f32(_uni(g, 3, n)), _f32(quat), _f32(-3.0 + 0.5 * _normal(g, 3, n)),
                _f32(_uni(g, ch, n))]
    pos, dens = _caustic_photons(g, n)
    # the distance r to the 8th neighbour at density p: pi p r^2 ~ Gamma(8)
    gam = -torch.log(_uni(g, NEAREST, n).clamp_min(1e-300)).sum(0)
    s = torch.sqrt(gam / (math.pi * dens)).clamp_min(1e-5)
    lsc = torch.log(s)[None] + ANISOTROPY * _normal(g, 3, n)
    flux = -torch.log(_uni(g, ch, n).clamp_min(1e-300))
    f = [_f32(pos.T), _f32(quat), _f32(lsc), _f32(flux)]
    if case["storage"] != "f32":        # 16-bit storage groups neighbours: Morton order
        q = ((pos + FLOOR) / (2 * FLOOR) * 1023).long().clamp(0, 1023)
        key = torch.zeros(n, dtype=torch.long, device="cuda")
        for b in range(10):
            for a in range(3):
                key |= ((q[:, a] >> b) & 1) << (3 * b + a)
        order = torch.argsort(key, stable=True)
        f = [t[:, order].contiguous() for t in f]
    return f


def _cameras(case, azimuth):
    """(eye, width, height) of every view."""
    w, h, v = case["width"], case["height"], case["n_views"]
    if case["views"] == "one":
        a = -math.pi / 2 + azimuth
        return [((6 * math.cos(a), 6 * math.sin(a), 4.0), w, h)]
    if case["views"] == "orbit":
        return [((6 * math.cos(azimuth + 2 * math.pi * k / v),
                  6 * math.sin(azimuth + 2 * math.pi * k / v), 3.0), w, h) for k in range(v)]
    out = []
    for k in range(v):                  # uneven: side, distance and height cycle
        a = azimuth + 2.39996 * k
        d, z, s = 5 + 3 * ((k * 7) % 16) / 16, 2 + 3 * ((k * 5) % 16) / 16, UNEVEN[k % 5]
        out.append(((d * math.cos(a), d * math.sin(a), z), s, s))
    return out


def _view(eye, width, height, device="cuda"):
    """First hits of a pinhole view with the floor and the sphere: x, normal,
    wo [3, width * height] and valid, in float64."""
    eye = torch.tensor(eye, dtype=torch.float64, device=device)
    up = torch.tensor((0.0, 0.0, 1.0), dtype=torch.float64, device=device)
    fwd = torch.tensor(LOOK_AT, dtype=torch.float64, device=device) - eye
    fwd = fwd / fwd.norm()
    right = torch.linalg.cross(fwd, up)
    right = right / right.norm()
    cup = torch.linalg.cross(right, fwd)
    t = math.tan(math.radians(VFOV) / 2)
    px = (2 * (torch.arange(width, device=device) + 0.5) / width - 1) * t * width / height
    py = (1 - 2 * (torch.arange(height, device=device) + 0.5) / height) * t
    d = (fwd[None, None] + px[None, :, None] * right + py[:, None, None] * cup).reshape(-1, 3)
    d = d / d.norm(dim=1, keepdim=True)
    tf = -eye[2] / d[:, 2]
    p = eye + tf[:, None] * d
    on_floor = (tf > 1e-6) & (p[:, 0].abs() <= FLOOR) & (p[:, 1].abs() <= FLOOR)
    far = torch.full_like(tf, math.inf)
    tb = torch.where(on_floor, tf, far)
    oc = eye - torch.tensor((0.0, 0.0, SPHERE_Z), dtype=torch.float64, device=device)
    b = d @ oc
    disc = b * b - (oc @ oc - SPHERE_R ** 2)
    ts = torch.where(disc >= 0, -b - disc.clamp_min(0).sqrt(), far)
    sphere = (ts > 1e-6) & (ts < tb)
    tb = torch.where(sphere, ts, tb)
    valid = torch.isfinite(tb)
    x = torch.where(valid[:, None], eye + torch.where(valid, tb, 0 * tb)[:, None] * d, 0 * d)
    x[:, 2] = torch.where(on_floor & ~sphere, 0 * tf, x[:, 2])
    nrm = torch.where(sphere[:, None], (x - eye + oc) / SPHERE_R, up.expand_as(d))
    wo = torch.where(valid[:, None], -d, up.expand_as(d))
    return x.T, nrm.T, wo.T, valid


def _points(case, g):
    """x, normal, wo, albedo or None, valid."""
    m_albedo = (lambda m: _f32(_uni(g, case["channels"], m, lo=0.2)) if case["albedo"] else None)
    if case["scene"] == "cube":
        m = case["width"] * case["height"]
        unit = (lambda v: v / v.norm(dim=0))
        return (_f32(_uni(g, 3, m)), _f32(unit(_normal(g, 3, m))), _f32(unit(_normal(g, 3, m))),
                m_albedo(m), torch.ones(m, dtype=torch.uint8, device="cuda"))
    az = float(_uni(g, 1, hi=2 * math.pi))
    parts = [_view(*c) for c in _cameras(case, az)]
    x, nrm, wo = (_f32(torch.cat([p[k] for p in parts], 1)) for k in range(3))
    valid = torch.cat([p[3] for p in parts]).to(torch.uint8)
    return x, nrm, wo, m_albedo(x.shape[1]), valid


def _target(case, g, x):
    """The radiance to fit: a smooth pattern with a path tracer's noise."""
    s = 1.0 if case["mode"] == "normalized" else 8.0
    ph = _uni(g, case["channels"], hi=6.28)
    wave = 1 + 0.5 * torch.sin(2 * x[0].double() + 3 * x[1].double() + ph[:, None])
    return _f32(s * wave * _uni(g, case["channels"], x.shape[1], lo=0.7, hi=1.3))


def _inputs(case, seed):
    g = _gen(seed)
    f = _gaussians(case, g)
    q = _points(case, g)
    m = q[0].shape[1]
    up = None
    if case["op"] in ("train", "hybrid_grad"):
        up = _target(case, g, q[0])
    elif case["op"] == "grad":          # the gradient that the user's loss hands down
        up = _f32(_normal(g, case["channels"], m) / m)
    moments = None
    if case["op"] == "train":           # Adam in the middle of a run, at its gradients' size
        size = 20.0 / case["n"]
        moments = [([_f32(0.1 * size * _normal(g, *t.shape)) for t in f],
                    [_f32((size * torch.exp(0.5 * _normal(g, *t.shape))) ** 2) for t in f])][0]
    return f, q, up, moments


STEP = 100                               # Adam updates before the timed ones


def _mode(case):
    return gpf.GPF_NORMALIZED if case["mode"] == "normalized" else gpf.GPF_SUM


def _plan(case, field, queries, **kw):
    if case["tuned"]:                   # what setup_index.autotune settles on for these scenes
        kw.update(max_span=3, coop_cells=8, split_items=2048 if case["op"] == "kde" else 4096)
    return make_index(field, queries, cutoff_sigma=CUTOFF, query_cell=case["cell"], headroom=1.25,
                      **kw)


def prepare(case, seed):
    f, q, up, moments = _inputs(case, seed)
    queries = gpf.Queries(*q)
    op = case["op"]
    s = {"case": case, "queries": queries, "up": up}
    if op == "kde":
        field = gpf.photon_field(f[0], f[3], R, CUTOFF)
    else:
        field = gpf.Field(*f)
    s["field"] = field
    if op == "train":
        store = None if case["storage"] == "f32" else field.quantized(
            mean32=case["storage"] == "bf16_mean32")
        index = _plan(case, field if store is None else store, queries)
        step = TrainStep(field, queries, up, index, mode=_mode(case), r_max=case["r"], eps=EPS,
                         lr=LR, store=store)
        if case["graph"]:
            first = [t.clone() for t in f]
            step.capture(warmup=1)
            for t, t0 in zip(field.tensors(), first):   # the capture's own step is undone
                t.copy_(t0)
            if store is not None:
                field.quantize_into(store)
        for fields, values in ((step.state.m, moments[0]), (step.state.v, moments[1])):
            for t, v in zip(fields.tensors(), values):
                t.copy_(v)
        step.state.step_counter.fill_(STEP)
        s["step"] = step
        return s
    if op in ("hybrid_query", "hybrid_grad"):
        kw = dict(neighbourhood=gpf.GPF_NB_BALL_KNN, ball_r=R, k_min=case["k_min"])
        if op == "hybrid_grad":         # room for the selected pairs, from a trial
            cap = 64 * queries.m
            for _ in range(2):
                idx = _plan(case, field, queries, ball_radius=R, max_nb_pairs=cap)
                idx.build(field, queries)
                out, z = gpf.gpf_radiance_fwd(idx, field, queries, _mode(case), r_max=case["r"], **kw)
                gpf.gpf_radiance_bwd(idx, field, queries, up, out, z, _mode(case),
                                     r_max=case["r"], **kw)
                cap = int(idx.stats()["n_nb_pairs"] * 1.1) + 1024
            s["index"] = _plan(case, field, queries, ball_radius=R, max_nb_pairs=cap)
        else:
            s["index"] = _plan(case, field, queries, ball_radius=R)
        s["kw"] = kw
    else:
        s["index"] = _plan(case, field, queries)
    if op == "grad":
        for t in field.tensors():
            t.requires_grad_(True)
    return s


def run(s):
    case, field, queries, op = s["case"], s["field"], s["queries"], s["case"]["op"]
    mode, r = _mode(case), case["r"]
    if op == "train":
        step = s["step"]
        step()
        return {"out": step.out, "loss": step.loss, "grads": step.grads.tensors(),
                "params": field.tensors()}
    if op == "grad":
        out = gpf.gpf_radiance(field, s["index"], queries, mode, r, EPS)
        return {"out": out, "grads": list(torch.autograd.grad(out, field.tensors(), s["up"]))}
    idx = s["index"]
    idx.build(field, queries)
    if op == "query":
        out, z = gpf.gpf_radiance_fwd(idx, field, queries, mode, r_max=r)
        return {"out": out, "z": z}
    if op == "kde":
        out, z = gpf.gpf_radiance_fwd(idx, field, queries, gpf.GPF_DISK_KDE, r_max=R)
        return {"out": out, "z": z}
    out, z = gpf.gpf_radiance_fwd(idx, field, queries, mode, r_max=r, **s["kw"])
    if op == "hybrid_query":
        return {"out": out, "z": z}
    loss, gout = gpf.gpf_mse_loss_grad(out, s["up"], queries.valid)
    grads = gpf.gpf_radiance_bwd(idx, field, queries, gout, out, z, mode, r_max=r, **s["kw"])
    return {"out": out, "loss": loss, "grads": grads.tensors()}


# ---------------------------------------------------------------- the least work

def _active(case):
    """Hit points, and how many face the viewer (a coarse raster of each view)."""
    if case["scene"] == "cube":
        m = case["width"] * case["height"]
        return m, m // 2
    m = act = 0
    seen = {}
    for eye, w, h in _cameras(case, 0.0):
        key = (round(math.hypot(eye[0], eye[1]), 6), eye[2], w / h)
        if key not in seen:
            v = _view(eye, max(4, int(48 * w / h)), 48, "cpu")[3]
            seen[key] = float(v.double().mean())
        m += w * h
        act += int(w * h * seen[key])
    return m, act


def work(case):
    """Inputs read once, outputs written once; the flops of the pairs that
    contribute (Q <= 9 for a field; the balls' and disks' means)."""
    n, ch, op = case["n"], case["channels"], case["op"]
    m, act = _active(case)
    bwd = op in ("grad", "train", "hybrid_grad")
    params = n * (10 + ch) * 4
    pts = m * (37 + (4 * ch if case["albedo"] else 0))
    image = m * ch * 4
    b = params + pts + image + (0 if op in ("train", "grad", "hybrid_grad") else 4 * m)
    if bwd:
        b += params + image              # gradients written, the target or upstream read
    if op == "train":
        b += 5 * params                  # moments read and written, parameters written
        if case["storage"] != "f32":
            b += n * 2 * (10 + ch)
    if case["scene"] == "cube":          # the 3-sigma ellipsoids of the mean scale in a unit cube
        per = n * 4 / 3 * math.pi * (3 * math.exp(-3)) ** 3 * math.exp(1.5 * 0.25) * 0.6
    elif op == "kde":                    # photons in the disk, at the mean density over the view
        per = 28e-6 * n
    elif op.startswith("hybrid"):
        per = max(case["k_min"], 5e-5 * n)
    else:                                # pi p (3 r)^2 with pi p r^2 ~ 8
        per = 9 * NEAREST
    flops = per * act * ((8 + ch) if op == "kde" else 25 + 2 * ch + (55 + 4 * ch if bwd else 0))
    return {"bytes": b, "flops": flops}


# ---------------------------------------------------------------- in 64 bits

PAIRS = 3e7                              # (hit point, Gaussian) pairs held at once


def _bf16_values(f, storage):
    """The stored field's values: offsets from the midpoint of each 16
    neighbours' means and log-scales, rounded to bfloat16."""
    mean, quat, lsc, spec = f
    n = mean.shape[1]
    pad = (-n) % 16
    r16 = (lambda t: t.to(torch.bfloat16).to(torch.float32))

    def mid(t):
        hi = torch.nn.functional.pad(t, (0, pad), value=-math.inf).view(t.shape[0], -1, 16)
        lo = torch.nn.functional.pad(t, (0, pad), value=math.inf).view(t.shape[0], -1, 16)
        return lo.amin(2), hi.amax(2)

    l0, l1 = mid(lsc)
    ref = ((l0.amin(0) + l1.amax(0)) * 0.5).repeat_interleave(16)[:n]
    if storage == "bf16":
        m0, m1 = mid(mean)
        org = ((m0 + m1) * 0.5).repeat_interleave(16, dim=1)[:, :n]
        mean = org + r16(mean - org)
    return [mean, r16(quat), ref + r16(lsc - ref), r16(spec)]


def _whiten(quat, lsc):
    """M = S^-1 R^T [n, 3, 3] of quaternions [4, n] and log-scales [3, n]."""
    w, x, y, z = quat / quat.norm(dim=0)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1)
    return rot.view(-1, 3, 3).transpose(1, 2) * torch.exp(-lsc).T[:, :, None]


def _blocks(x):
    """Active hit points [k, 3] in blocks of neighbours."""
    q = ((x - x.amin(0)) / (x.amax(0) - x.amin(0)).amax().clamp_min(1e-9) * 1023).long()
    key = torch.zeros(x.shape[0], dtype=torch.long, device=x.device)
    for b in range(10):
        for a in range(3):
            key |= ((q[:, a] >> b) & 1) << (3 * b + a)
    return torch.split(torch.argsort(key), 1024)


def _gap(pos, lo, hi):
    """Distance from every mean to a box."""
    return torch.clamp(torch.maximum(lo - pos, pos - hi), min=0).norm(dim=1)


def exact(case, seed):
    m, act = _active(case)
    if act * (3 if case["op"] in ("grad", "train", "hybrid_grad") else 1) > 6e6:
        return None                      # takes longer than it is worth
    f32, q, up, moments = _inputs(case, seed)
    if case["op"] == "train" and case["storage"] != "f32":
        f = [t.double() for t in _bf16_values(f32, case["storage"])]
    else:
        f = [t.double() for t in f32]
    x, nrm, wo, alb, valid = q
    ch, op = case["channels"], case["op"]
    hybrid, kde, norm = op.startswith("hybrid"), op == "kde", case["mode"] == "normalized"
    # the falloff radius as the entry points take it, in float32
    r = float(torch.tensor(R if kde else case["r"], dtype=torch.float32))
    ball = float(torch.tensor(R, dtype=torch.float32))
    eps = float(torch.tensor(EPS, dtype=torch.float32))
    ids = torch.nonzero((valid != 0) & ((nrm.double() * wo.double()).sum(0) > 0)).flatten()
    pts = x[:, ids].double().T.contiguous()
    rho = alb[:, ids].double().T if alb is not None else torch.ones(1, ch, device="cuda",
                                                                    dtype=torch.float64)
    pos, phi = f[0].T.contiguous(), f[3].T.contiguous()
    reach = CUTOFF * torch.exp(f[2]).amax(0) * 1.001
    M = _whiten(f[1], f[2])
    Mmu = torch.einsum("njk,nk->nj", M, pos)
    out = torch.zeros(ch, m, device="cuda", dtype=torch.float64)
    zz = torch.zeros(m, device="cuda", dtype=torch.float64)
    n_valid = int((valid != 0).sum())
    gM, gmu, gphi = torch.zeros_like(M), torch.zeros_like(pos), torch.zeros_like(phi)
    loss = torch.zeros((), device="cuda", dtype=torch.float64)
    if up is not None and op != "grad":  # hit points that return nothing still have a target
        dark = valid != 0
        dark = dark.clone()
        dark[ids] = False
        loss = loss + (up[:, dark].double() ** 2).sum()
    for block in _blocks(pts) if len(ids) else []:
        p = pts[block]
        lo, hi = p.amin(0), p.amax(0)
        gap = _gap(pos, lo, hi)
        if hybrid:
            near = _gap(pos, (lo + hi) / 2, (lo + hi) / 2)
            k = min(case["k_min"], case["n"])
            far = float(torch.topk(near, k, largest=False).values[-1]) if k else 0.0
            cand = gap <= max(ball, far + float((hi - lo).norm())) * 1.001
        else:
            cand = gap <= (r * 1.001 if kde else reach)
        cand = torch.nonzero(cand).flatten()
        if not len(cand):
            continue
        for sub in torch.split(torch.arange(len(block), device="cuda"),
                               max(1, int(PAIRS // len(cand)))):
            rows = block[sub]
            p = pts[rows]
            d2 = sum((p[:, k, None] - pos[cand, k]) ** 2 for k in range(3))
            if kde:
                w = (d2 <= r * r).double()
            else:
                u = [p @ M[cand, j].T - Mmu[cand, j] for j in range(3)]
                Q = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
                e = -0.5 * Q
                if math.isfinite(r):
                    d = d2.sqrt()
                    t = ((d - r) / max(r, 1e-6)).clamp_min(0)
                    e = e - 3 * t * t
                if hybrid:
                    sel = d2 <= ball * ball
                    need = sel.sum(1) < min(case["k_min"], case["n"])
                    if bool(need.any()):
                        near = torch.topk(d2[need], min(case["k_min"], len(cand)), largest=False)
                        sel[need] = torch.zeros_like(sel[need]).scatter_(1, near.indices, True)
                else:
                    sel = Q <= CUTOFF * CUTOFF
                w = torch.where(sel, torch.exp(e), 0 * e)
            L, Z = w @ phi[cand], w.sum(1)
            scale = 1 / Z.clamp_min(eps) if norm else torch.ones_like(Z)
            if kde:
                scale = scale / (math.pi * r * r)
            rh = rho[rows] if alb is not None else rho
            o = rh * L * scale[:, None]
            at = ids[rows]
            out[:, at], zz[at] = o.T, Z
            if up is None:
                continue
            g = up[:, at].double().T
            if op != "grad":
                diff = o - g
                loss = loss + (diff ** 2).sum()
                g = 2 * diff / n_valid
            gam = g * rh
            zeta = scale[:, None]
            kappa = ((g * o).sum(1) * (Z > eps))[:, None] if norm else 0.0
            bw = zeta * (gam @ phi[cand].T - kappa) * w
            gphi.index_add_(0, cand, (w * zeta).T @ gam)
            dmu = torch.zeros(len(cand), 3, device="cuda", dtype=torch.float64)
            for j in range(3):
                b = bw * u[j]
                s = b.sum(0)
                dmu += s[:, None] * M[cand, j]
                gM[cand, j] += -(b.T @ p - s[:, None] * pos[cand])
            if math.isfinite(r):
                c = bw * 6 * t / (max(r, 1e-6) * d.clamp_min(1e-30))
                dmu += c.T @ p - c.sum(0)[:, None] * pos[cand]
            gmu.index_add_(0, cand, dmu)
    if up is None:
        return {"out": out, "z": zz}
    quat, lsc = f[1].clone().requires_grad_(True), f[2].clone().requires_grad_(True)
    dq, dl = torch.autograd.grad(_whiten(quat, lsc), (quat, lsc), gM)
    grads = [gmu.T, dq, dl, gphi.T]
    if op == "grad":
        return {"out": out, "grads": grads}
    res = {"out": out, "loss": (loss / max(n_valid, 1)).reshape(1), "grads": grads}
    if op == "train":
        t = STEP + 1
        res["params"] = []
        for p, g, m1, m2 in zip(f32, grads, *moments):
            a = 0.9 * m1.double() + 0.1 * g
            b = 0.999 * m2.double() + 0.001 * g * g
            res["params"].append(p.double() - LR / (1 - 0.9 ** t) * a /
                                 (b.sqrt() / math.sqrt(1 - 0.999 ** t) + 1e-8))
    return res
