"""The work that programs have this library do, as cases that can be timed and compared.

A case is a dict of plain values; `prepare` makes what a training program holds
before the call (attributes, gradients, cameras, an optimizer context with the
moments of earlier steps), `run` is one pass through the public entry points of
`paper_2601_16736_gb300.gsopt`, and `exact` is the same result in 64 bits from
plain torch.

Kinds of case:
  step        one training iteration: gs_step_camera on the current view, with
              gradients on the device; optional terms (position noise, AIU,
              active count) as the case says
  mask        gs_visibility, then gs_step with that mask (a program whose
              renderer needs the mask between the two); `dense`: gs_step over
              every row, without a mask
  host        gs_step_host with the gradients in pinned host memory;
              `noalloc`: gs_step_host_noalloc (at most 65536 rows)
  batch       gs_batch_graph_step over several scenes of uneven sizes
  densify     a densification iteration: gs_active_rows, gs_reindex_state and
              gs_gather_attrs for the new primitive set, then its step
  checkpoint  gs_opt_import_state of a saved state (resume), then
              gs_opt_export_state (save)

Sizes and distributions follow the workloads of bench.py and synth.py: means
uniform in [-5, 5]^3 (most rows visible) or in 64 Gaussian blobs of sigma 0.5
whose centres span [-extent, extent]^3 (the wider, the fewer rows visible),
rows in random order, cameras on circles of radius 10 looking at the origin.
"""
import math

import torch

from paper_2601_16736_gb300 import gsopt as G

GROUPS = (("xyz", 3), ("scale", 3), ("rot", 4), ("opacity", 1), ("sh", 48))
COLS = {"xyz": slice(0, 3), "scale": slice(3, 6), "rot": slice(6, 10), "opacity": slice(10, 11), "sh": slice(11, 59)}
PREC = {"fp32": 0, "bf16": 1, "fp8": 2, "hybrid": 3, "fp16": 4}
# bytes of one moment value in each storage format (hybrid: 45 of 59 columns in 16 bits)
MOMENT_BYTES = {"fp32": 4.0, "bf16": 2.0, "fp8": 1.0, "hybrid": (45 * 2 + 14 * 4) / 59, "fp16": 2.0}
# scene -> (half extent of the blob centres, mean visible fraction over the views)
SCENES = {"uniform": (5.0, 0.88), "room": (12.5, 0.30), "block": (22.0, 0.20), "city": (75.0, 0.10)}
K0 = 2001            # the first pass is this iteration of a running training
N_PIXELS = 800 * 800
LAMBDA_O, LAMBDA_S, CLIP, N_I, EPS = 1e-3, 1e-5, 10.0, 60000.0, 1e-15
B1, B2 = 0.9, 0.999
LR = dict(scale=5e-3, rot=1e-3, opacity=2.5e-2, sh_dc=2.5e-3, sh_rest=2.5e-3 / 20.0)
RESTATE_EVERY, RESTATE_RATIO, SEED = 100, 0.1, 97
NOISE_K, NOISE_T, NOISE_LR, AIU_PROB, AIU_SCALE = 100.0, 0.005, 5e5, 0.1, 0.5


def listed():
    return [
        # the first iterations of a small capture: a few thousand structure-from-motion points
        dict(name="sfm_5k", kind="step", n=5003, scene="uniform", prec="fp32"),
        # an object scan, nearly all of it in every view
        dict(name="object_100k", kind="step", n=100_000, scene="uniform", prec="fp32"),
        # the common room-sized scene in FP32, the library's headline
        dict(name="room_1m", kind="step", n=1_000_000, scene="room", prec="fp32"),
        # a scene at the usual 3 M cap with 16-bit moments
        dict(name="block_3m_fp16", kind="step", n=3_000_000, scene="block", prec="fp16"),
        # a city-sized scene of which a view shows little, hybrid moments
        dict(name="city_6m_hybrid", kind="step", n=6_000_000, scene="city", prec="hybrid"),
        # FP8 moments with block scales, a size that fills no last block
        dict(name="block_2m_fp8", kind="step", n=2_000_003, scene="block", prec="fp8"),
        # 3DGS-MCMC style: noise on every primitive and the active count
        dict(name="mcmc_1m", kind="step", n=1_000_000, scene="room", prec="fp32", noise="all", count=True),
        # the mask made first for the renderer, BF16 moments, an odd size
        dict(name="mask_777k_bf16", kind="mask", n=777_777, scene="room", prec="bf16"),
        # gradients computed on the host side of a pipeline
        dict(name="host_1m", kind="host", n=1_000_000, scene="room", prec="fp32"),
        # sixteen scenes trained side by side
        dict(name="batch_16", kind="batch", n=2_000_000, n_min=50_000, scenes=16, prec="fp32"),
        # a densification event of a large scene
        dict(name="densify_6m_fp16", kind="densify", n=6_000_000, scene="city", prec="fp16"),
        # resume and save
        dict(name="checkpoint_1m_fp16", kind="checkpoint", n=1_234_567, prec="fp16"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["mask", "mask", "host", "batch", "densify", "checkpoint"])
    prec = rng.choice(["fp32", "fp32", "fp16", "fp16", "hybrid", "bf16", "fp8"])
    scene = rng.choice(["uniform", "room", "block", "city"])
    if kind == "step":
        case = dict(kind=kind, n=_log_uniform(rng, 2000, 6_000_000 if scene in ("city", "block") else 2_000_000),
                    scene=scene, prec=prec)
        if prec != "fp8" and rng.random() < 0.4:
            case["noise"] = rng.choice(["off", "visible", "all"])
            case["count"] = rng.random() < 0.5
            case["aiu"] = rng.random() < 0.3
        return case
    if kind == "mask":
        case = dict(kind=kind, n=_log_uniform(rng, 5000, 2_000_000), scene=scene, prec=prec)
        if rng.random() < 0.3:
            case["dense"] = True
        return case
    if kind == "host":
        noalloc = rng.random() < 0.4
        return dict(kind=kind, n=_log_uniform(rng, 5000, 65_536 if noalloc else 1_000_000), scene=scene, prec=prec,
                    noalloc=noalloc)
    if kind == "batch":
        return dict(kind=kind, n=_log_uniform(rng, 50_000, 1_000_000), n_min=_log_uniform(rng, 5000, 50_000),
                    scenes=rng.randint(2, 24), prec="fp16" if prec == "fp8" else prec)
    if kind == "densify":
        return dict(kind=kind, n=_log_uniform(rng, 20_000, 3_000_000), scene=scene, prec=prec)
    return dict(kind=kind, n=_log_uniform(rng, 20_000, 2_000_000), prec=prec)


# ------------------------------------------------------------------- inputs

def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000 + what)
    return g


def _views():
    """The views of a training set in random order, as (R, t, tan_x, tan_y, near, far) rows of 16 values."""
    cams = []
    for el in (-30.0, -15.0, 0.0, 15.0, 30.0):
        for a in range(40):
            e, az = math.radians(el), 2 * math.pi * a / 40
            eye = torch.tensor([10 * math.cos(e) * math.cos(az), 10 * math.cos(e) * math.sin(az), 10 * math.sin(e)],
                               dtype=torch.float64)
            f = -eye / eye.norm()
            x = torch.linalg.cross(f, torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64))
            x = x / x.norm()
            R = torch.stack([x, torch.linalg.cross(f, x), f])
            tan = math.tan(math.radians(30.0))
            cams.append(torch.cat([R.reshape(-1), -R @ eye, torch.tensor([tan, tan, 0.01, 100.0],
                                                                         dtype=torch.float64)]).float())
    return [cams[(37 * i + 11) % len(cams)] for i in range(len(cams))]


def _scene(n, scene, seed):
    """Attributes of n primitives and the gradients of iteration K0."""
    g = _gen(seed, 1)

    def normal(w, mean=0.0, std=1.0):
        return torch.randn(n, w, generator=g, device="cuda") * std + mean

    if scene == "uniform":
        xyz = torch.rand(n, 3, generator=g, device="cuda") * 10.0 - 5.0
    else:
        extent = SCENES[scene][0]
        centres = (torch.rand(64, 3, generator=g, device="cuda") * 2.0 - 1.0) * extent
        xyz = centres[torch.randint(0, 64, (n,), generator=g, device="cuda")] + normal(3, std=0.5)
    rot = torch.nn.functional.normalize(normal(4), dim=1)
    attrs = dict(xyz=xyz, scale=normal(3, -4.0, 0.5), rot=rot, opacity=normal(1), sh=normal(48, std=0.2))
    return attrs, _grads(n, g)


def _grads(n, g):
    return {k: torch.randn(n, w, generator=g, device="cuda") * (1e-4 if k == "xyz" else 1e-3) for k, w in GROUPS}


def _moments(n, seed):
    """m, v [n, 59] and t [n] as earlier steps leave them; one row in fifty was created just now (t = 0)."""
    g = _gen(seed, 2)
    sigma = torch.full((59,), 1e-3, device="cuda")
    sigma[0:3] = 1e-4
    t = torch.randint(1, 2000, (n,), generator=g, device="cuda", dtype=torch.int32)
    t[torch.rand(n, generator=g, device="cuda") < 0.02] = 0
    old = (t > 0).float()[:, None]
    m = torch.randn(n, 59, generator=g, device="cuda") * (0.23 * sigma) * old
    grown = 1.0 - torch.pow(torch.tensor(B2, device="cuda"), t.float())[:, None]
    v = (0.3 + 0.7 * torch.rand(n, 59, generator=g, device="cuda")) * sigma.square() * grown
    return m, v, t


def _event(n, seed):
    """A densification event: 5 % of the rows pruned, as many cloned (fresh state), 2 % relocated (state reset)."""
    g = _gen(seed, 3)
    k = max(1, n // 20)
    keep = torch.randperm(n, generator=g, device="cuda")[k:].sort().values
    moved = torch.randperm(n - k, generator=g, device="cuda")[:max(1, n // 50)]
    src = torch.cat([keep, torch.full((k,), -1, device="cuda")]).int()
    reset = torch.zeros(n, dtype=torch.uint8, device="cuda")
    reset[moved] = 1
    attr_src = torch.cat([keep, keep[torch.randint(0, n - k, (k,), generator=g, device="cuda")]])
    attr_src[moved] = keep[torch.randint(0, n - k, (moved.numel(),), generator=g, device="cuda")]
    return src, reset, attr_src.int()


def _sizes(case, seed):
    """Row counts of a batch's scenes, log-uniform in [n_min, n], and their scene types."""
    g = torch.Generator().manual_seed(4242)       # the sizes belong to the case, not to the inputs
    u = torch.rand(case["scenes"], generator=g).tolist()
    lo, hi = math.log(case["n_min"]), math.log(max(case["n"], case["n_min"] + 1))
    names = ("room", "block", "city", "uniform")
    return [(int(math.exp(lo + (hi - lo) * x)), names[i % 3]) for i, x in enumerate(u)]


# ------------------------------------------------------------------ programs

class Program:
    """What a training program keeps between calls.  The context is freed with it."""

    def __init__(self):
        self.handles, self.batch, self.k, self.views = [], None, K0, None

    def __del__(self):
        if self.batch is not None:
            self.batch.close()
        for h in self.handles:
            G.gs_opt_destroy(h)


def _lr_xyz(k):
    return 1.6e-4 * math.exp(math.log(0.01) * min(1.0, (k - 1) / 30000.0))


def _params(case, n_active=None):
    return G.make_params([_lr_xyz(K0), LR["scale"], LR["rot"], LR["opacity"], LR["sh_dc"], LR["sh_rest"]], K0,
                         restate_ratio=RESTATE_RATIO, seed=SEED,
                         noise={"off": 0, "visible": 1, "all": 2}[case.get("noise") or "off"], noise_lr=NOISE_LR,
                         noise_k=NOISE_K, noise_t=NOISE_T, aiu=bool(case.get("aiu")), aiu_prob=AIU_PROB,
                         aiu_scale=AIU_SCALE, n_active=n_active)


def _context(p, prec, n, seed):
    h = G.gs_opt_init(G.make_config(prec=PREC[prec], n_pixels=N_PIXELS), n)
    p.handles.append(h)
    m, v, t = _moments(n, seed)
    G.gs_opt_import_state(h, m, v, t)
    torch.cuda.synchronize()                     # the imported buffers are released here
    return h


def prepare(case, seed):
    kind, n, prec = case["kind"], case["n"], case["prec"]
    p = Program()
    p.kind, p.n = kind, n
    p.cams = [G.make_camera(c.tolist()) for c in _views()]
    if kind == "checkpoint":
        p.handles.append(G.gs_opt_init(G.make_config(prec=PREC[prec], n_pixels=N_PIXELS), n))
        p.saved = _moments(n, seed)
        p.out = tuple(torch.zeros_like(x) for x in p.saved)
        return p
    p.visible = torch.zeros(1, dtype=torch.int64, device="cuda")
    if kind == "batch":
        sizes = _sizes(case, seed)
        starts, total = [], 0
        for rows, _ in sizes:                     # every scene starts on a multiple of 64 rows of the shared arrays
            starts.append(total)
            total += (rows + 63) // 64 * 64
        p.attrs = {k: torch.zeros(total, w, device="cuda") for k, w in GROUPS}
        p.grads = {k: torch.zeros(total, w, device="cuda") for k, w in GROUPS}
        p.visible = torch.zeros(len(sizes), dtype=torch.int64, device="cuda")
        p.scene_views = []
        for s, (rows, scene) in enumerate(sizes):
            a, g = _scene(rows, scene, seed * 100 + s)
            for k, _ in GROUPS:
                p.attrs[k][starts[s]:starts[s] + rows] = a[k]
                p.grads[k][starts[s]:starts[s] + rows] = g[k]
            _context(p, prec, rows, seed * 100 + s)
        p.batch = G.gs_batch_create(p.handles)
        for s, (rows, _) in enumerate(sizes):
            cut = slice(starts[s], starts[s] + rows)
            p.batch.set(s, attrs=G.make_attrs({k: x[cut] for k, x in p.attrs.items()}),
                        grads=G.make_attrs({k: x[cut] for k, x in p.grads.items()}), params=_params(case))
        return p
    p.attrs, grads = _scene(n, case["scene"], seed)
    p.grads = [grads]
    if kind in ("step", "mask"):
        # successive iterations bring other gradients of mean zero: the moments keep moving and the scene stays put
        p.grads.append(_grads(n, _gen(seed, 4)))
        p.grads += [{k: -x for k, x in g.items()} for g in p.grads]
    if kind == "host":
        p.grads = [{k: x.cpu().pin_memory() for k, x in g.items()} for g in p.grads]
    p.A, p.D = G.make_attrs(p.attrs), [G.make_attrs(g) for g in p.grads]
    p.h = _context(p, prec, n, seed)
    p.mask = torch.zeros(n, dtype=torch.uint8, device="cuda")
    p.active = torch.zeros(1, dtype=torch.int64, device="cuda") if case.get("count") or kind == "densify" else None
    p.params = _params(case, p.active if case.get("count") else None)
    p.dense, p.noalloc = bool(case.get("dense")), bool(case.get("noalloc"))
    if kind == "densify":
        p.src, p.reset, p.attr_src = _event(n, seed)
        p.rows = torch.zeros(n, dtype=torch.int32, device="cuda")
        p.next_attrs = {k: torch.zeros_like(x) for k, x in p.attrs.items()}
        p.B = G.make_attrs(p.next_attrs)
    return p


def run(p):
    kind = p.kind
    if kind == "checkpoint":
        h = p.handles[0]
        G.gs_opt_import_state(h, *p.saved)
        G.gs_opt_export_state(h, *p.out)
        return dict(m=p.out[0], v=p.out[1], t=p.out[2])
    k = p.k
    p.k = k + 1
    cam = p.cams[k % len(p.cams)]
    if kind == "batch":
        b = p.batch
        for s in range(b.n):
            q = b.params[s]
            q.iteration, q.restate = k, k % RESTATE_EVERY == 0
            q.lr[0] = _lr_xyz(k)
            b.cams[s] = p.cams[(k + 7 * s) % len(p.cams)]
        G.gs_batch_graph_step(b, p.visible)
        return dict(p.attrs, visible=p.visible)
    i = k - K0
    grads = p.D[(i + i // len(p.cams)) % len(p.D)]
    q = p.params
    q.iteration, q.restate = k, k % RESTATE_EVERY == 0
    q.lr[0] = _lr_xyz(k)
    if kind == "step":
        G.gs_step_camera(p.h, p.A, grads, cam, q, mask_out=p.mask, n_visible=p.visible)
        out = dict(p.attrs, mask=p.mask, visible=p.visible)
        if p.active is not None:
            out["active"] = p.active
        return out
    if kind == "mask":
        if p.dense:
            G.gs_step(p.h, p.A, grads, None, q)
            return dict(p.attrs)
        G.gs_visibility(p.h, p.attrs["xyz"], cam, p.mask, None, p.visible)
        G.gs_step(p.h, p.A, grads, p.mask, q)
        return dict(p.attrs, mask=p.mask, visible=p.visible)
    if kind == "host":
        step = G.gs_step_host_noalloc if p.noalloc else G.gs_step_host
        return dict(p.attrs, visible=step(p.h, p.A, grads, cam, q))
    G.gs_active_rows(p.h, p.attrs["opacity"], p.rows, p.active)
    G.gs_reindex_state(p.h, p.src, p.reset, p.n)
    G.gs_gather_attrs(p.h, p.A, p.n, p.B, p.attr_src, p.n)
    p.attrs, p.next_attrs, p.A, p.B = p.next_attrs, p.attrs, p.B, p.A
    G.gs_step_camera(p.h, p.A, grads, cam, q, mask_out=p.mask, n_visible=p.visible)
    return dict(p.attrs, mask=p.mask, visible=p.visible, active=p.active, rows=p.rows)


# ---------------------------------------------------------------------- work

def _step_work(case, n, visible):
    row = 59 * (4 * 3 + 4 * MOMENT_BYTES[case["prec"]]) + 8 - 12
    hidden = 44 * (case.get("noise") == "all") + 0.1 * 59 * (8 + 2 * MOMENT_BYTES[case["prec"]]) * bool(case.get("aiu"))
    hidden += 4 * (bool(case.get("count")) and case.get("noise") != "all")
    return n * visible * row + n * 13 + n * (1 - visible) * hidden, n * visible * 59 * 16 + n * 30


def work(case):
    """Bytes and operations of one pass: each visible row's attributes and moments read and written, its
    gradients read, every mean read and mask byte written; the rows an event or a checkpoint moves."""
    kind, n = case["kind"], case["n"]
    mb = MOMENT_BYTES[case["prec"]]
    if kind == "checkpoint":
        b = n * 2 * (59 * 2 * (4 + mb) + 8)
        return {"bytes": b, "flops": n * 59 * 4}
    if kind == "batch":
        got = [_step_work(case, rows, SCENES[scene][1]) for rows, scene in _sizes(case, 0)]
        return {"bytes": sum(b for b, _ in got), "flops": sum(f for _, f in got)}
    b, f = _step_work(case, n, 1.0 if case.get("dense") else SCENES[case["scene"]][1])
    if kind == "mask" and not case.get("dense"):
        b += n
    if kind == "host":
        b -= n
    if kind == "densify":
        b += n * (8 + 4 + 1 + 4 + 2 * 236) + n * (1 + 0.93) * (59 * 2 * mb + 4)
    return {"bytes": b, "flops": f}


# --------------------------------------------------------------------- exact

def _mix(seed, tag, k, rows):
    """Output number tag << 62 | k << 32 | row of the SplitMix64 stream (64-bit wrap-around integers)."""
    def signed(c):
        return c - (1 << 64) if c >= 1 << 63 else c

    def shift(x, s):
        return (x >> s) & ((1 << (64 - s)) - 1)

    counter = rows + signed(((tag << 62) | (k << 32)) & ((1 << 64) - 1))
    z = seed + (counter + 1) * signed(0x9E3779B97F4A7C15)
    z = (z ^ shift(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shift(z, 27)) * signed(0x94D049BB133111EB)
    return z ^ shift(z, 31), shift


def _noise(k, x, rows):
    """What the position noise subtracts from the means of `rows`, from the values before the step."""
    h1, shift = _mix(SEED, 2, k, rows)
    h2, _ = _mix(SEED, 3, k, rows)
    u = [(shift(h, 40) + 1).double() * 2.0 ** -24 for h in (h1, h2)]
    w = [((h >> 16) & 0xFFFFFF).double() * 2.0 ** -24 for h in (h1, h2)]
    r = [torch.sqrt(-2.0 * torch.log(a)) for a in u]
    gamma = torch.stack([r[0] * torch.cos(2 * math.pi * w[0]), r[0] * torch.sin(2 * math.pi * w[0]),
                         r[1] * torch.cos(2 * math.pi * w[1])], 1)
    q = x["rot"][rows]
    q = q / q.norm(dim=1, keepdim=True).clamp_min(1e-12)
    a, b, c, d = q.unbind(1)
    R = torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - a * d), 2 * (b * d + a * c),
                     2 * (b * c + a * d), 1 - 2 * (b * b + d * d), 2 * (c * d - a * b),
                     2 * (b * d - a * c), 2 * (c * d + a * b), 1 - 2 * (b * b + c * c)], 1).reshape(-1, 3, 3)
    y = torch.einsum("nji,nj->ni", R, gamma) * torch.exp(2 * x["scale"][rows])
    gate = torch.sigmoid(-NOISE_K * (torch.sigmoid(x["opacity"][rows]) - NOISE_T))
    return NOISE_LR * _lr_xyz(k) * gate * torch.einsum("nij,nj->ni", R, y)


def _exact_step(case, attrs, grads, m, v, t, cam, dense=False):
    """Attributes after iteration K0, in 64 bits."""
    k = K0
    x = {name: a.double() for name, a in attrs.items()}
    new = {name: a.clone() for name, a in x.items()}
    c = cam.double().cuda()
    pos = x["xyz"] @ c[:9].reshape(3, 3).T + c[9:12]
    z = pos[:, 2]
    vis = (z >= c[14]) & (z <= c[15]) & (pos[:, 0].abs() <= z * c[12]) & (pos[:, 1].abs() <= z * c[13])
    if dense:
        vis = torch.ones_like(vis)
    on, off = vis.nonzero()[:, 0], (~vis).nonzero()[:, 0]

    def rates(name):
        if name == "sh":
            r = torch.full((48,), LR["sh_rest"], dtype=torch.float64, device="cuda")
            r[:3] = LR["sh_dc"]
            return r
        return _lr_xyz(k) if name == "xyz" else LR[name]

    tn = (t[on].double() + 1)[:, None]
    r1, r2 = 1 / (1 - B1 ** tn), 1 / torch.sqrt(1 - B2 ** tn)
    for name, _ in GROUPS:
        cols = COLS[name]
        g = grads[name][on].double()
        mm = B1 * m[on, cols].double() + (1 - B1) * g
        vv = B2 * v[on, cols].double() + (1 - B2) * g * g
        d = torch.sqrt(vv) * r2 + EPS
        step = mm * r1 / d
        if name == "opacity":
            s = torch.sigmoid(x[name][on])
            step += (LAMBDA_O / N_I * s * (1 - s) / d).clamp_max(CLIP)
        elif name == "scale":
            step += (LAMBDA_S / N_I * torch.exp(x[name][on]) / d).clamp_max(CLIP)
        new[name][on] = x[name][on] - rates(name) * step
    if case.get("aiu"):
        h, shift = _mix(SEED, 1, k, off)
        prob = float(torch.tensor(AIU_PROB, dtype=torch.float32))
        rows = off[(shift(h, 11) < math.ceil(prob * 2.0 ** 53)) & (t[off] > 0)]
        tn = t[rows].double()[:, None]
        r1, r2 = 1 / (1 - B1 ** tn), 1 / torch.sqrt(1 - B2 ** tn)
        for name, _ in GROUPS:
            cols = COLS[name]
            step = m[rows, cols].double() * r1 / (torch.sqrt(v[rows, cols].double()) * r2 + EPS)
            new[name][rows] = x[name][rows] - AIU_SCALE * rates(name) * step
    if (case.get("noise") or "off") != "off":
        rows = on if case["noise"] == "visible" else torch.arange(vis.numel(), device="cuda")
        new["xyz"][rows] -= _noise(k, x, rows)
    return new


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "checkpoint":
        m, v, _ = _moments(n, seed)
        return dict(m=m.double(), v=v.double(), t=None)
    views = _views()
    if kind == "batch":
        sizes = _sizes(case, seed)
        out, total = {k: [] for k, _ in GROUPS}, 0
        for s, (rows, scene) in enumerate(sizes):
            new = _exact_step(case, *_scene(rows, scene, seed * 100 + s), *_moments(rows, seed * 100 + s),
                              views[(K0 + 7 * s) % len(views)])
            for k, w in GROUPS:
                out[k] += [new[k], torch.zeros(-rows % 64, w, dtype=torch.float64, device="cuda")]
        return dict({k: torch.cat(x) for k, x in out.items()}, visible=None)
    attrs, grads = _scene(n, case["scene"], seed)
    m, v, t = _moments(n, seed)
    if kind == "densify":
        src, reset, attr_src = _event(n, seed)
        attrs = {k: x[attr_src.long()] for k, x in attrs.items()}
        kept = ((src >= 0) & (reset == 0)).to(m.dtype)[:, None]
        src = src.long().clamp_min(0)
        m, v, t = m[src] * kept, v[src] * kept, t[src] * kept[:, 0].to(t.dtype)
    new = _exact_step(case, attrs, grads, m, v, t, views[K0 % len(views)], bool(case.get("dense")))
    if case.get("dense"):
        return new
    new["visible"] = None
    if kind != "host":
        new["mask"] = None
    if kind == "densify":
        new.update(active=None, rows=None)
    elif case.get("count"):
        new["active"] = None
    return new
