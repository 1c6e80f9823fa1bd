"""What is measured: the work a user of the renderer has it do, through the package's entry points.

A case names a tree (depth, SH degree, leaf type, occupied share of the grid) and one of these uses:

  views   ``render``: pinhole views of one tree, one call
  batch   ``render_batch``: a server's work list, requests of several sizes on several trees
  train   ``render_rays_record``, ``loss_mse``, ``render_backward_recorded``, ``LeafOptimizer.step``:
          one step of the octree optimisation on a batch of rays
  fused   ``render_mse_backward``: colour, loss and gradients of a batch of rays in one call
  filter  ``visibility``: the largest ray weight of every leaf over a set of views

Trees are unions of 8 spheres and boxes in [-1.5, 1.5]^3 filled to the given share of the grid, with
lognormal(3, 1) densities and N(0, 0.5 / (l + 1)) SH coefficients; views look at the origin from a
distance of 4 with a focal length of 1111 / 800 of the image width, as the benchmark's do.
``exact`` integrates the same rays in 64 bits with torch alone.
"""
import math

import numpy as np
import torch

import paper_2103_14024_gb300 as pot

DEV = "cuda"
LO, SIZE = -1.5, 3.0
NEAR, FAR = 2.0, 6.0
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
SERVE_TREES = ((7, 1), (8, 2), (9, 3))
SERVE_SIZES = ((256, 256), (512, 512), (800, 800), (1920, 1080))


def _views(name, depth, degree, dtype, width, height, views, gamma=1e-4, occ=0.03, bg=0.0, arc=0.0, t_final=False):
    return {"name": name, "use": "views", "depth": depth, "degree": degree, "dtype": dtype, "occ": occ,
            "width": width, "height": height, "views": views, "gamma": gamma, "bg": bg, "arc": arc, "t_final": t_final}


def _rays(name, use, depth, degree, rays, gamma=1e-4, occ=0.03, opt="rmsprop", width=800, views=100):
    return {"name": name, "use": use, "depth": depth, "degree": degree, "dtype": "f32", "occ": occ, "rays": rays,
            "gamma": gamma, "opt": opt, "width": width, "height": width, "views": views}


def listed():
    return [
        # the smallest render: one 64 x 64 view of a 32^3 tree (what a test or a thumbnail asks for)
        _views("tiny_64", 5, 0, "f32", 64, 64, 1, gamma=0.0),
        # a preview frame on a white background; a lone request of the server's smallest size
        _views("preview_256_f16", 8, 2, "f16", 256, 256, 1, bg=1.0),
        # one frame of an interactive viewer on the benchmark's tree
        _views("frame_800_f32", 9, 3, "f32", 800, 800, 1, t_final=True),
        # the benchmark's orbit (40 neighbouring views of it) with each leaf type it reports
        _views("orbit_800_f32", 9, 3, "f32", 800, 800, 40, arc=1.8),
        _views("orbit_800_f16", 9, 3, "f16", 800, 800, 40, arc=1.8),
        # full-HD views with the degree-4 basis the paper uses for its large scenes, bfloat16 leaves, early stop 0.01
        _views("hd_sh4_bf16", 9, 4, "bf16", 1920, 1080, 2, gamma=1e-2, arc=90.0),
        # a deep tree (1024^3, brick index) rendered full-HD, as the server's largest tree is
        _views("deep_hd_f16", 10, 2, "f16", 1920, 1080, 1, occ=0.01),
        # a compressed model (SH codebooks) shown at an odd size from views all around
        _views("codebook_601x399", 7, 3, "cb16", 601, 399, 6, arc=60.0),
        # a server's work list under load: 24 requests of mixed sizes on three resident trees
        {"name": "serve_24", "use": "batch", "dtype": "f16", "occ": 0.03, "requests": 24, "largest": 1920, "gamma": 1e-4},
        # one optimisation step on the benchmark's tree and batch
        _rays("train_262144", "train", 9, 3, 1 << 18),
        # a small fine-tuning batch on a small tree, in the one-call form; an odd number of rays
        _rays("fused_20011", "fused", 7, 2, 20011),
        # filtering of a tree against training views
        _rays("filter_800", "filter", 9, 3, 0, views=6),
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    use = rng.choice(["views", "views", "views", "batch", "train", "fused", "filter"])
    depth = rng.choice([5, 6, 7, 7, 8, 8, 9, 9, 10])
    degree = rng.randint(0, 4)
    gamma = rng.choice([0.0, 1e-4, 1e-4, 1e-2])
    occ = round(rng.uniform(0.005, 0.03), 4)
    if depth == 10:
        occ, degree = min(occ, 0.01), min(degree, 2)
    if use == "views":
        dtype = rng.choice(["f32", "f32", "f16", "f16", "bf16", "cb16"])
        if dtype == "cb16":
            depth = min(depth, 7)
        w, h = log_int(40, 1920), log_int(40, 1080)
        most = max(1, min(40, 10_000_000 // (w * h)))
        c = _views("", depth, degree, dtype, w, h, log_int(1, most), gamma, occ, rng.choice([0.0, 0.0, 1.0]),
                   round(rng.uniform(1.0, 60.0), 2), rng.random() < 0.3)
    elif use == "batch":
        c = {"use": "batch", "dtype": rng.choice(["f32", "f16", "bf16"]), "occ": occ, "requests": log_int(1, 24),
             "largest": rng.choice([256, 512, 800, 1920]), "gamma": gamma}
    elif use == "filter":
        c = _rays("", "filter", depth, degree, 0, gamma, occ, width=log_int(100, 800), views=log_int(1, 6))
    else:
        c = _rays("", use, depth, degree, log_int(1000, 1 << 18), gamma, occ, rng.choice(["sgd", "rmsprop", "adam"]),
                  width=rng.choice([400, 641, 800]), views=log_int(4, 100))
    c.pop("name", None)
    return c


# ---- inputs, from the seed alone -------------------------------------------

def _scene(depth, degree, occ, seed):
    """Occupied voxels (Morton order), densities and SH coefficients of a union of 8 shapes, on the GPU."""
    rng = np.random.default_rng([seed, depth, degree])
    centre = rng.uniform(-0.9, 0.9, (8, 3))
    half = np.where(np.arange(8)[:, None] % 2 == 0, rng.uniform(0.2, 0.4, (8, 1)), rng.uniform(0.15, 0.35, (8, 3)))

    def inside(x, y, z, i, scale):
        p = [x - centre[i, 0], y - centre[i, 1], z - centre[i, 2]]
        if i % 2 == 0:
            return p[0] ** 2 + p[1] ** 2 + p[2] ** 2 < (half[i, 0] * scale) ** 2
        return (p[0].abs() < half[i, 0] * scale) & (p[1].abs() < half[i, 1] * scale) & (p[2].abs() < half[i, 2] * scale)

    def axis(d, a):
        v = LO + (torch.arange(1 << d, device=DEV, dtype=torch.float64) + 0.5) * (SIZE / (1 << d))
        return v.view([-1 if k == a else 1 for k in range(3)])

    def occupied(d, scale):
        """Whether each voxel centre lies in some shape, [x][y][z]; each shape looks at its own part of the grid."""
        got = torch.zeros((1 << d,) * 3, dtype=torch.bool, device=DEV)
        g = [axis(d, a).reshape(-1) for a in range(3)]
        for i in range(8):
            ext = half[i] * scale if i % 2 else np.repeat(half[i, 0] * scale, 3)
            lo = [max(0, int((centre[i, a] - ext[a] - LO) / SIZE * (1 << d)) - 1) for a in range(3)]
            hi = [min(1 << d, int((centre[i, a] + ext[a] - LO) / SIZE * (1 << d)) + 2) for a in range(3)]
            if any(h <= l for l, h in zip(lo, hi)):
                continue
            x, y, z = (g[a][lo[a]:hi[a]].view([-1 if k == a else 1 for k in range(3)]) for a in range(3))
            got[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] |= inside(x, y, z, i, scale)
        return got

    # the scale at which the shapes fill the share, from above; the few voxels too many go from the end of the order
    leaves = int(occ * 8 ** depth)
    small, large = 0.1, 4.0
    for _ in range(16):
        mid = 0.5 * (small + large)
        if float(occupied(depth, mid).sum()) < leaves:
            small = mid
        else:
            large = mid
    x, y, z = torch.nonzero(occupied(depth, large), as_tuple=True)
    code = torch.zeros_like(x)
    for b in range(depth):
        code |= ((x >> b) & 1) << (3 * b + 2) | ((y >> b) & 1) << (3 * b + 1) | ((z >> b) & 1) << (3 * b)
    code = torch.sort(code).values[:leaves].contiguous()
    gen = torch.Generator(device=DEV).manual_seed(seed * 1000 + depth * 10 + degree)
    sigma = torch.exp(3.0 + torch.randn(code.shape[0], device=DEV, generator=gen))
    sh = torch.randn((code.shape[0], (degree + 1) ** 2, 3), device=DEV, generator=gen)
    std = [0.5 / (math.isqrt(k) + 1) for k in range((degree + 1) ** 2)]
    sh *= torch.tensor(std, device=DEV).view(1, -1, 1)
    return {"depth": depth, "degree": degree, "morton": code, "sigma": sigma, "sh": sh,
            "centre": centre, "half": half * large}


CAMERA = np.dtype([("c2w", np.float32, (3, 4)), ("fx", np.float32), ("fy", np.float32), ("cx", np.float32),
                   ("cy", np.float32), ("width", np.int32), ("height", np.int32), ("near", np.float32),
                   ("far", np.float32)])


def _cameras(azimuth, elevation, width, height):
    """Cameras at distance 4 looking at the origin; angles in degrees."""
    cams = np.zeros(len(azimuth), CAMERA)
    for c, az, el in zip(cams, np.radians(azimuth), np.radians(elevation)):
        eye = 4.0 * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
        back = eye / np.linalg.norm(eye)
        right = np.cross([0.0, 0.0, 1.0], back)
        right /= np.linalg.norm(right)
        c["c2w"] = np.stack([right, np.cross(back, right), back, eye], axis=1)
        c["fx"] = c["fy"] = 1111.0 * width / 800.0
        c["cx"], c["cy"], c["width"], c["height"] = width * 0.5, height * 0.5, width, height
        c["near"], c["far"] = NEAR, FAR
    return cams


def _pixel_rays(cams, view, row, col):
    """Rays of pixels in float32, one rounding per operation (the pinhole expression of the C header), on the GPU."""
    t = {k: torch.from_numpy(np.ascontiguousarray(cams[k])).to(DEV)[view] for k in ("c2w", "fx", "fy", "cx", "cy")}
    x = (col.to(torch.float32) + 0.5 - t["cx"]) / t["fx"]
    y = -((row.to(torch.float32) + 0.5 - t["cy"]) / t["fy"])
    m = t["c2w"]
    d = (m[:, :, 0] * x[:, None] + m[:, :, 1] * y[:, None]) - m[:, :, 2]
    return m[:, :, 3].contiguous(), d.contiguous()


def _inputs(case, seed):
    """Everything of a case before any call of the package."""
    rng = np.random.default_rng([seed, 77])
    use = case["use"]
    if use == "batch":
        scenes = [_scene(d, k, case["occ"], seed + 1 + i) for i, (d, k) in enumerate(SERVE_TREES)]
        sizes = [s for s in SERVE_SIZES if s[0] <= case["largest"]]
        items = []
        for i in range(case["requests"]):
            # one in four of each size and one in three of each tree, in a mixed order
            w, h = sizes[(i * 7 + 3) % len(sizes)]
            cam = _cameras([rng.uniform(0, 360)], [rng.uniform(10, 50)], w, h)
            items.append(((i * 5 + 1) % len(scenes), cam))
        return {"scenes": scenes, "items": items}
    scene = _scene(case["depth"], case["degree"], case["occ"], seed)
    w, h, n = case["width"], case["height"], case["views"]
    if use == "views":
        first = rng.uniform(0, 360)
        return {"scene": scene, "cams": _cameras([first + case["arc"] * i for i in range(n)], [30.0] * n, w, h)}
    cams = _cameras(rng.uniform(0, 360, n), np.degrees(np.arcsin(rng.uniform(0.02, 0.98, n))), w, h)
    if use == "filter":
        return {"scene": scene, "cams": cams}
    gen = torch.Generator(device=DEV).manual_seed(seed + 5)
    pix = torch.sort(torch.randint(0, n * h * w, (case["rays"],), device=DEV, generator=gen)).values
    o, d = _pixel_rays(cams, pix // (h * w), pix % (h * w) // w, pix % w)
    # colours to fit: random where the ray meets a shape (or passes close by), the background's zero elsewhere
    seen = torch.zeros(case["rays"], dtype=torch.bool, device=DEV)
    for i in range(8):
        c = torch.tensor(scene["centre"][i], dtype=torch.float32, device=DEV)
        r = float(np.linalg.norm(scene["half"][i])) if i % 2 else float(scene["half"][i, 0])
        p = torch.linalg.cross(o - c, d)
        seen |= (p * p).sum(1) < (r + 0.05) ** 2 * (d * d).sum(1)
    target = torch.rand((case["rays"], 3), device=DEV, generator=gen) * seen[:, None]
    return {"scene": scene, "origins": o, "dirs": d, "target": target}


# ---- the package's side ------------------------------------------------------

def _tree(scene, dtype):
    t = pot.Tree.build_sparse(scene["depth"], scene["degree"], (LO,) * 3, SIZE, scene["morton"], scene["sigma"],
                              scene["sh"], dtype="f32" if dtype == "cb16" else dtype)
    if dtype != "cb16":
        return t
    q = t.quantize(16)
    t.free()
    return q


def prepare(case, seed):
    x = _inputs(case, seed)
    s = {"case": case}
    if case["use"] == "batch":
        s["trees"] = [_tree(c, case["dtype"]) for c in x["scenes"]]
        s["items"] = [(s["trees"][t], cam, torch.empty((int(cam["height"][0]), int(cam["width"][0]), 3), device=DEV))
                      for t, cam in x["items"]]
        return s
    s["tree"] = _tree(x["scene"], case["dtype"])
    if "cams" in x:
        s["cams"] = x["cams"]
        return s
    s.update(origins=x["origins"], dirs=x["dirs"], target=x["target"])
    if case["use"] == "train":
        s["records"] = pot.SegmentRecords.for_rays(case["rays"])
        # rates of a fine-tuning run: the tree stays near where it began over many steps
        s["opt"] = pot.LeafOptimizer(s["tree"], case["opt"], lr_sigma=1e-2, lr_sh=1e-4)
    return s


def run(s):
    case = s["case"]
    use, gamma = case["use"], case["gamma"]
    if use == "views":
        return pot.render(s["tree"], s["cams"], bg=(case["bg"],) * 3, gamma=gamma, want_t_final=case["t_final"])
    if use == "batch":
        pot.render_batch([(tree, cam, rgb, (0.0, 0.0, 0.0), gamma, None) for tree, cam, rgb in s["items"]])
        return [rgb for _, _, rgb in s["items"]]
    if use == "filter":
        return pot.visibility(s["tree"], s["cams"], gamma=gamma)
    rays = dict(gamma=gamma, near=NEAR, far=FAR)
    if use == "fused":
        rgb = torch.empty_like(s["origins"])
        loss, gs, gh = pot.render_mse_backward(s["tree"], s["origins"], s["dirs"], s["target"], rgb=rgb, **rays)
        return {"rgb": rgb, "loss": loss, "grad_sigma": gs, "grad_sh": gh}
    rgb = pot.render_rays_record(s["tree"], s["origins"], s["dirs"], s["records"], **rays)
    loss, grad = pot.loss_mse(rgb, s["target"])
    gs, gh = pot.render_backward_recorded(s["tree"], s["origins"], s["dirs"], grad, rgb, s["records"], **rays)
    s["opt"].step(gs, gh)
    return {"rgb": rgb, "loss": loss, "grad_sigma": gs, "grad_sh": gh, "state": s["opt"].state}


# ---- what a pass cannot do without -------------------------------------------

def _one_tree_work(depth, degree, dtype, occ, rays, in_bytes, out_bytes):
    """Every leaf that some ray composites read once, the rays' own inputs and outputs, and the arithmetic of the
    leaf segments.  Counted on the benchmark's scene: 16.5 segments to a ray at depth 9 (in proportion to the grid's
    resolution elsewhere), and 2.46 M of 4.05 M leaves met by one 800 x 800 view."""
    k = (degree + 1) ** 2
    record = {"f32": 4 + 12 * k, "f16": 2 + 6 * k, "bf16": 2 + 6 * k, "cb16": 4 + 2 * k}[dtype]
    leaves = occ * 8.0 ** depth
    met = leaves * (1.0 - math.exp(-6.0 * rays * 2.0 ** (depth - 9) / leaves))
    segments = 16.5 * 2.0 ** (depth - 9) * rays
    return met, met * record + in_bytes + out_bytes, segments * (6 * k + 30)


def work(case):
    use = case["use"]
    if use == "batch":
        sizes = [s for s in SERVE_SIZES if s[0] <= case["largest"]]
        total = [0.0, 0.0]
        for t, (d, k) in enumerate(SERVE_TREES):
            mine = [i for i in range(case["requests"]) if (i * 5 + 1) % len(SERVE_TREES) == t]
            rays = sum(sizes[(i * 7 + 3) % len(sizes)][0] * sizes[(i * 7 + 3) % len(sizes)][1] for i in mine)
            _, b, f = _one_tree_work(d, k, case["dtype"], case["occ"], rays, 80 * len(mine), 12 * rays)
            total = [total[0] + b, total[1] + f]
        return {"bytes": total[0], "flops": total[1]}
    rays = case.get("rays") or case["views"] * case["width"] * case["height"]
    args = (case["depth"], case["degree"], case["dtype"], case["occ"], rays)
    leaves = case["occ"] * 8.0 ** case["depth"]
    values = 1 + 3 * (case["degree"] + 1) ** 2
    if use == "views":
        _, b, f = _one_tree_work(*args, 80 * case["views"], (16 if case["t_final"] else 12) * rays)
    elif use == "filter":
        _, b, f = _one_tree_work(case["depth"], 0, "f32", case["occ"], rays, 80 * case["views"], 4 * leaves)
        b, f = b - 12 * leaves * (1.0 - math.exp(-6.0 * rays * 2.0 ** (case["depth"] - 9) / leaves)), f * 10 / 36
    else:
        # rays and target read, colours and dense gradients written; forward and backward of each segment
        _, b, f = _one_tree_work(*args, 36 * rays, 12 * rays + 4 * leaves * values)
        f *= 3
        if use == "train":
            # the optimiser: values and gradients read, values written, state read and written
            streams = {"sgd": 3, "rmsprop": 5, "adam": 7}[case["opt"]]
            b += 4 * leaves * values * streams
            f += 8 * leaves * values
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits, with torch alone -------------------------------------

def _basis(degree, d):
    """Real spherical harmonics of unit directions [n, 3] (float64), index l^2 + l + m, from the derivatives of the
    Legendre polynomials; cos terms for m > 0, sin terms for m < 0, every sign +."""
    x, y, z = d.unbind(1)
    out = []
    for l in range(degree + 1):
        for m in range(-l, l + 1):
            a = abs(m)
            q = np.polynomial.legendre.leg2poly([0.0] * l + [1.0])
            q = np.polynomial.polynomial.polyder(q, a) if a else q
            n = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - a) / math.factorial(l + a)) * (math.sqrt(2) if a else 1)
            poly = torch.zeros_like(z)
            for c in q[::-1]:
                poly = poly * z + float(c)
            re, im = torch.ones_like(x), torch.zeros_like(x)
            for _ in range(a):
                re, im = re * x - im * y, re * y + im * x
            out.append(n * poly * (im if m < 0 else re))
    return torch.stack(out, 1)


class _Exact:
    """A tree's stored values in float64 and the voxel grid of its leaves."""

    def __init__(self, scene, dtype):
        self.depth, self.degree = scene["depth"], scene["degree"]
        sigma, sh = scene["sigma"], scene["sh"]
        if dtype == "cb16":
            sh = _median_cut(sh)
        else:
            sigma, sh = sigma.to(DTYPES[dtype]), sh.to(DTYPES[dtype])
        self.sigma, self.sh = sigma.double().clamp(min=0), sh
        m, v = scene["morton"], [torch.zeros_like(scene["morton"]) for _ in range(3)]
        for b in range(self.depth):
            for a in range(3):
                v[a] |= ((m >> (3 * b + 2 - a)) & 1) << b
        n = 1 << self.depth
        self.grid = torch.full((n * n * n,), -1, dtype=torch.int32, device=DEV)
        self.grid[(v[0] * n + v[1]) * n + v[2]] = torch.arange(m.shape[0], dtype=torch.int32, device=DEV)

    def segments(self, o, d, near, far, gamma):
        """Per ray of a chunk: the composited leaf segments, as flat lists (ray, leaf, length, T in front, weight, T
        behind) in order along each ray, and each ray's final T."""
        o, d = o.double(), d.double()
        n, h = 1 << self.depth, SIZE / (1 << self.depth)
        length = d.norm(dim=1)
        planes = LO + h * torch.arange(n + 1, device=DEV, dtype=torch.float64)
        t = (planes[None, None, :] - o[:, :, None]) / d[:, :, None]
        still = (d == 0)[:, :, None]
        ends = torch.stack([t[:, :, 0], t[:, :, -1]], 2)
        inf = torch.tensor(math.inf, dtype=torch.float64, device=DEV)
        first = torch.where(still[:, :, 0], -inf, ends.amin(2)).amax(1).clamp(min=0).maximum(near / length)
        last = torch.where(still[:, :, 0], inf, ends.amax(2)).amin(1).minimum(far / length)
        inside = (~still[:, :, 0] | ((o >= LO) & (o < LO + SIZE))).all(1) & (first < last)
        last = torch.where(inside, last, first)
        t = torch.where(still, first[:, None, None], t).reshape(o.shape[0], -1)
        t = torch.cat([first[:, None], t.clamp(first[:, None], last[:, None]), last[:, None]], 1).sort(1).values
        mid, step = 0.5 * (t[:, 1:] + t[:, :-1]), t[:, 1:] - t[:, :-1]
        del t
        cell = torch.zeros(mid.shape, dtype=torch.int64, device=DEV)
        for a in range(3):
            k = torch.addcmul((o[:, a:a + 1] - LO).expand_as(mid), mid, d[:, a:a + 1]).div_(h).floor_().clamp_(0, n - 1)
            cell.mul_(n).add_(k.long())
        del mid, k
        leaf = self.grid[cell]
        del cell
        ray, at = torch.nonzero((leaf >= 0) & (step > 0), as_tuple=True)
        leaf, delta = leaf[ray, at].long(), step[ray, at] * length[ray]
        del step
        # sums along each ray: cumulative over the flat list, less what stood before the ray
        tau = self.sigma[leaf] * delta
        before = torch.cumsum(tau, 0) - tau
        head = torch.searchsorted(ray, torch.arange(o.shape[0], device=DEV))
        base = torch.cat([before, before.new_zeros(1)])[head]
        front = torch.exp(-(before - base[ray]).clamp(min=0))
        keep = front >= gamma
        ray, leaf, delta, tau, front = ray[keep], leaf[keep], delta[keep], tau[keep], front[keep]
        total = torch.zeros(o.shape[0], dtype=torch.float64, device=DEV).index_add_(0, ray, tau)
        return ray, leaf, delta, front, front * -torch.expm1(-tau), front * torch.exp(-tau), torch.exp(-total), d / length[:, None]

    def colours(self, ray, leaf, unit):
        y = _basis(self.degree, unit)
        got = []
        for r, l in zip(ray.split(1 << 20), leaf.split(1 << 20)):
            got.append(torch.sigmoid((self.sh[l].double() * y[r][:, :, None]).sum(1)))
        return (torch.cat(got) if got else torch.zeros((0, 3), dtype=torch.float64, device=DEV)), y

    def chunks(self, rays):
        return torch.arange(rays, device=DEV).split(max(256, (48 << 20) // (3 << self.depth)))

    def render(self, o, d, near, far, gamma, bg):
        rgb, tf = [], []
        for i in self.chunks(o.shape[0]):
            ray, leaf, _, _, w, _, t_end, unit = self.segments(o[i], d[i], near, far, gamma)
            c, _ = self.colours(ray, leaf, unit)
            rgb.append((t_end[:, None] * bg).expand(-1, 3).clone().index_add_(0, ray, w[:, None] * c))
            tf.append(t_end)
        return torch.cat(rgb), torch.cat(tf)

    def weights(self, o, d, near, far, gamma, out):
        for i in self.chunks(o.shape[0]):
            _, leaf, _, _, w, _, _, _ = self.segments(o[i], d[i], near, far, gamma)
            out.scatter_reduce_(0, leaf, w, "amax")

    def gradients(self, o, d, near, far, gamma, upstream):
        """Gradients of sum(upstream(C) . C), where upstream(rays, C) gives dL/dC; the background is zero."""
        gs = torch.zeros_like(self.sigma)
        gh = torch.zeros((self.sh.shape[0], self.sh.shape[1] * 3), dtype=torch.float64, device=DEV)
        for i in self.chunks(o.shape[0]):
            ray, leaf, delta, _, w, behind, _, unit = self.segments(o[i], d[i], near, far, gamma)
            c, y = self.colours(ray, leaf, unit)
            wc = w[:, None] * c
            total = torch.zeros((len(i), 3), dtype=torch.float64, device=DEV).index_add_(0, ray, wc)
            g = upstream(i, total)[ray]
            done = torch.cumsum(wc, 0)
            head = torch.searchsorted(ray, torch.arange(len(i), device=DEV))
            base = torch.cat([done.new_zeros((1, 3)), done])[head]
            rest = total[ray] - (done - base[ray])
            gs.index_add_(0, leaf, torch.where(self.sigma[leaf] > 0, (g * (c * behind[:, None] - rest)).sum(1) * delta, 0.0))
            for r, l, x in zip(ray.split(1 << 20), leaf.split(1 << 20), (g * wc * (1 - c)).split(1 << 20)):
                gh.index_add_(0, l, (y[r][:, :, None] * x[:, None, :]).reshape(len(l), -1))
        return gs, gh.view(self.sh.shape)


def _median_cut(sh, bits=16):
    """The codebook entry of each coefficient: per basis function, boxes of leaves split `bits` times along their
    longest extent at the middle of their order, and the mean of each box in float16."""
    n, k, _ = sh.shape
    pts = sh.transpose(0, 1).contiguous()  # [k, n, 3]
    order = torch.arange(n, device=DEV).expand(k, n).clone()
    edges = np.array([0, n])
    for _ in range(bits):
        size = np.diff(edges)
        box = torch.from_numpy(np.repeat(np.arange(len(size)), size)).to(DEV)
        p = torch.gather(pts, 1, order[:, :, None].expand(-1, -1, 3))
        at = box[None, :, None].expand(k, -1, 3)
        low = torch.full((k, len(size), 3), math.inf, device=DEV).scatter_reduce_(1, at, p, "amin").double()
        high = torch.full((k, len(size), 3), -math.inf, device=DEV).scatter_reduce_(1, at, p, "amax").double()
        ext = torch.where(torch.isfinite(low), high - low, 0.0)
        # the first channel of the largest extent
        axis = torch.where((ext[..., 0] >= ext[..., 1]) & (ext[..., 0] >= ext[..., 2]), 0, torch.where(ext[..., 1] >= ext[..., 2], 1, 2))
        along = torch.gather(p, 2, axis[:, box][:, :, None])[:, :, 0]
        # by leaf, then by value, then by box: stable sorts from the last key to the first; a lone point stays
        by = torch.argsort(order, dim=1, stable=True)
        by = torch.gather(by, 1, torch.argsort(torch.gather(along, 1, by), dim=1, stable=True))
        by = torch.gather(by, 1, torch.argsort(box[by], dim=1, stable=True))
        order = torch.gather(order, 1, by)
        middle = np.where(size >= 2, edges[:-1] + size // 2, edges[1:])
        edges = np.concatenate([np.stack([edges[:-1], middle], 1).reshape(-1), edges[-1:]])
    size = np.diff(edges)
    box = torch.from_numpy(np.repeat(np.arange(len(size)), size)).to(DEV)
    p = torch.gather(pts, 1, order[:, :, None].expand(-1, -1, 3)).double()
    total = torch.zeros((k, len(size), 3), dtype=torch.float64, device=DEV).index_add_(1, box, p)
    mean = (total / torch.from_numpy(np.maximum(size, 1)).to(DEV)[None, :, None]).half()
    got = torch.empty((k, n, 3), dtype=torch.float16, device=DEV)
    got.scatter_(1, order[:, :, None].expand(-1, -1, 3), mean[:, box])
    return got.transpose(0, 1).contiguous()


MOST_CELLS = 1.6e9  # plane crossings that exact() sorts in about ten seconds


def _cells(case):
    if case["use"] == "batch":
        sizes = [s for s in SERVE_SIZES if s[0] <= case["largest"]]
        return sum(3.0 * 2 ** SERVE_TREES[(i * 5 + 1) % 3][0] * sizes[(i * 7 + 3) % len(sizes)][0] * sizes[(i * 7 + 3) % len(sizes)][1]
                   for i in range(case["requests"]))
    return 3.0 * 2 ** case["depth"] * (case.get("rays") or case["views"] * case["width"] * case["height"])


def _view_rays(cams, i):
    w, h = int(cams["width"][i]), int(cams["height"][i])
    pix = torch.arange(w * h, device=DEV)
    return _pixel_rays(cams, torch.full_like(pix, i), pix // w, pix % w)


def exact(case, seed):
    if _cells(case) > MOST_CELLS:
        return None
    x = _inputs(case, seed)
    use, gamma, near, far = case["use"], case["gamma"], float(np.float32(NEAR)), float(np.float32(FAR))
    gamma = float(np.float32(gamma))
    if use == "batch":
        trees = [_Exact(c, case["dtype"]) for c in x["scenes"]]
        return [trees[t].render(*_view_rays(cam, 0), near, far, gamma, 0.0)[0].view(int(cam["height"][0]), int(cam["width"][0]), 3)
                for t, cam in x["items"]]
    e = _Exact(x["scene"], case["dtype"])
    if use == "views":
        got = [e.render(*_view_rays(x["cams"], i), near, far, gamma, case["bg"]) for i in range(case["views"])]
        shape = (case["views"], case["height"], case["width"])
        rgb = torch.stack([r for r, _ in got]).view(*shape, 3)
        return (rgb, torch.stack([t for _, t in got]).view(shape)) if case["t_final"] else rgb
    if use == "filter":
        weight = torch.zeros_like(e.sigma)
        for i in range(case["views"]):
            e.weights(*_view_rays(x["cams"], i), near, far, gamma, weight)
        return weight
    o, d, target = x["origins"], x["dirs"], x["target"].double()
    rgb = torch.empty_like(target)

    def upstream(i, c):
        rgb[i] = c
        return 2.0 * (c - target[i]) / target.numel()

    gs, gh = e.gradients(o, d, near, far, gamma, upstream)
    got = {"rgb": rgb, "loss": ((rgb - target) ** 2).mean().view(1), "grad_sigma": gs, "grad_sh": gh}
    if use == "train":
        g = torch.cat([gs, gh.reshape(-1)])
        square = {"rmsprop": (1 - float(np.float32(0.99))), "adam": (1 - float(np.float32(0.999)))}
        got["state"] = (None if case["opt"] == "sgd" else square["rmsprop"] * g * g if case["opt"] == "rmsprop"
                        else torch.cat([(1 - float(np.float32(0.9))) * g, square["adam"] * g * g]))
    return got
