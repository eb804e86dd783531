"""What a user of the spectral renderer has it do, as cases that can be timed.

A case is a dict of plain values; `kind` names the way the renderer is called:

  render     Renderer.render: spectral and XYZ image in device memory, one band per path
  host       Renderer.render_host: the colour image in host memory (the end-to-end call)
  graph      Renderer.render with use_graph into the caller's buffers: the same views' poses change, the launches replay
  bands4     Renderer.render with four bands per path
  guided     Renderer.render with a trained (frozen) path guide, as after the training passes of a render
  photons    Renderer.render_photons: photon maps and camera pass
  xyz        Renderer.xyz: colour from an accumulated spectral image (progressive renders)
  guide_grad Renderer.guide_grad: loss and gradients of the guide on a batch of training records

Scenes are the package's own seeded workloads, loaded once per process as a user's program does; a seed sets the
camera poses, the Philox key, the records or the image, and nothing else.  Sizes follow the workloads' own
(128 x 128 box, 96 x 72 prism room, 1024 x 768 nave, uneven views of 256 to 1024 pixels, 2M-triangle nave) with
fewer samples where a whole job takes minutes: a job is many such calls.
"""
import math
import random

import numpy as np
import torch

from paper_1912_04000_gb300 import scenes

_BANDS = {"tiny_box": 16, "prism_room": 16, "nave": 81, "crystal_nave": 81, "large_nave": 81}
_TRIS = {"tiny_box": 12, "prism_room": 20, "nave": 197948, "crystal_nave": 199260, "large_nave": 1971228}
_LOG2_TABLE = 19
_LEVELS, _FEATURES = 8, 4
_VIEW_SCALE = (1.0, 0.75, 0.5, 0.875, 0.625, 0.4375)  # uneven views of one batch, as shares of the first


def listed():
    return [
        # the smallest call: a thumbnail of the 12-triangle room, where launches and latency are the cost
        {"name": "box_thumbnail", "kind": "render", "scene": "tiny_box", "width": 32, "height": 24, "views": 1, "spp": 2,
         "depth": 4, "band_first": 0, "bands": 16},
        # the first configuration whole: 128 x 128, 16 bands, 4 spp, depth 4
        {"name": "box_image", "kind": "render", "scene": "tiny_box", "width": 128, "height": 128, "views": 1, "spp": 4,
         "depth": 4, "band_first": 0, "bands": 16},
        # solid dispersive glass, ragged image, a sub-range of the bands (one rank's spectral sub-domain)
        {"name": "prism_ragged", "kind": "render", "scene": "prism_room", "width": 97, "height": 71, "views": 1, "spp": 5,
         "depth": 8, "band_first": 2, "bands": 13},
        # a 256 x 192 view of the church with its colours in host memory: what an interactive or scripted client asks for
        {"name": "nave_view_host", "kind": "host", "scene": "nave", "width": 256, "height": 192, "views": 1, "spp": 2,
         "depth": 8, "band_first": 0, "bands": 81},
        # the 200k-triangle configuration at its full frame, two of its 16 samples
        {"name": "nave_frame", "kind": "render", "scene": "nave", "width": 1024, "height": 768, "views": 1, "spp": 2,
         "depth": 8, "band_first": 0, "bands": 81},
        # batched uneven views, captured once and replayed with other poses
        {"name": "nave_views_graph", "kind": "graph", "scene": "nave", "width": 640, "height": 368, "views": 4, "spp": 1,
         "depth": 8, "band_first": 0, "bands": 81},
        # four bands per path, with refraction that ends the sharing
        {"name": "crystal_bands4", "kind": "bands4", "scene": "crystal_nave", "width": 512, "height": 384, "views": 1,
         "spp": 4, "depth": 8, "band_first": 0, "bands": 81},
        # guided rendering after the training passes: most of a guided job
        {"name": "nave_guided", "kind": "guided", "scene": "nave", "width": 512, "height": 384, "views": 1, "spp": 2,
         "depth": 8, "band_first": 0, "bands": 81},
        # the largest scene: guided and batched views of the 2M-triangle nave, depth 12, one sample pass
        {"name": "large_guided_views", "kind": "guided", "scene": "large_nave", "width": 1024, "height": 768, "views": 2,
         "spp": 1, "depth": 12, "band_first": 0, "bands": 81},
        # photon mapping with its default maps
        {"name": "nave_photons", "kind": "photons", "scene": "nave", "width": 256, "height": 192, "views": 1, "spp": 4,
         "depth": 8, "band_first": 0, "bands": 81, "photons": 65536},
        # colour of a full accumulated frame
        {"name": "xyz_frame", "kind": "xyz", "scene": "nave", "pixels": 786432, "spp": 16, "band_first": 0, "bands": 81},
        # one training batch of the guide: a tenth of the records carry radiance
        {"name": "guide_batch", "kind": "guide_grad", "scene": "nave", "records": 524288, "weighted": 0.1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "host", "graph", "bands4", "guided", "photons", "xyz", "guide_grad"])
    if kind == "xyz":
        bands = rng.choice([81, rng.randint(1, 81)])
        return {"kind": kind, "scene": "nave", "pixels": _log_int(rng, 768, 786432), "spp": rng.randint(1, 64),
                "band_first": rng.randint(0, 81 - bands), "bands": bands}
    if kind == "guide_grad":
        return {"kind": kind, "scene": "nave", "records": _log_int(rng, 500, 1048576),
                "weighted": round(math.exp(rng.uniform(math.log(0.05), 0.0)), 3)}
    scene = {"bands4": ["tiny_box", "prism_room", "nave", "crystal_nave"],
             "guided": ["tiny_box", "nave", "large_nave"],
             "graph": ["tiny_box", "prism_room", "nave", "crystal_nave"],
             "photons": ["tiny_box", "prism_room", "nave", "crystal_nave"]}.get(
                 kind, ["tiny_box", "prism_room", "nave", "nave", "crystal_nave", "large_nave"])
    scene = rng.choice(scene)
    total = _BANDS[scene]
    small = total == 16
    bands = rng.choice([total, rng.randint(1, total)])
    case = {"kind": kind, "scene": scene, "width": _log_int(rng, 16, 160 if small else 1024),
            "height": _log_int(rng, 16, 160 if small else 768), "views": rng.choice([1, 1, 2, 4, 6]),
            "spp": _log_int(rng, 1, 8), "depth": rng.randint(2, 12 if scene == "large_nave" else 8),
            "band_first": rng.randint(0, total - bands), "bands": bands}
    if kind == "photons":
        case["views"] = 1
        case["photons"] = _log_int(rng, 4096, 65536)
        case["width"], case["height"] = min(case["width"], 384), min(case["height"], 288)
    limit = 9e8  # path vertices: below the largest listed frames'
    while _paths(case) * case["depth"] > limit and case["spp"] > 1:
        case["spp"] -= 1
    while _paths(case) * case["depth"] > limit:
        case["width"], case["height"] = max(16, case["width"] // 2 + 1), max(16, case["height"] // 2 + 1)
    return case


def _views(case):
    return [(max(8, int(case["width"] * f)), max(8, int(case["height"] * f))) for f in _VIEW_SCALE[:case["views"]]]


def _pixels(case):
    return case["pixels"] if case["kind"] == "xyz" else sum(w * h for w, h in _views(case))


def _paths(case):
    return _pixels(case) * case["bands"] * case["spp"]


def work(case):
    """Bytes: the scene and its tables once, each output once.  Flops: a closest-hit and a sun ray per path vertex,
    each an ordered descent of a tree over the scene's triangles (about 2.2 log2 n child boxes of 12 flops for a
    closest hit, half of that for a sun ray, two triangles of 55 each), and 150 of shading."""
    if case["kind"] == "guide_grad":
        n_w = case["records"] * case["weighted"]
        grid = _LEVELS * (1 << _LOG2_TABLE) * _FEATURES * 4
        return {"bytes": 48 * case["records"] + min(grid, n_w * 64 * 16) + grid + 2 * 61440, "flops": 92e3 * n_w}
    npix, bands = _pixels(case), case["bands"]
    if case["kind"] == "xyz":
        return {"bytes": npix * (8 * bands + 12), "flops": 6 * npix * bands}
    tris = _TRIS[case["scene"]]
    rays = _paths(case) * case["depth"] / (4.0 if case["kind"] == "bands4" else 1.0)
    slots = 2.2 * math.log2(tris)
    flops = rays * (1.5 * slots * 12 + 4 * 55 + 150)
    if case["kind"] == "guided":
        flops += min(2, case["depth"] - 1) / case["depth"] * rays * 30.7e3
    if case["kind"] == "photons":
        # camera paths end at their first stone vertex; photons take four interactions
        flops = (_paths(case) + 4 * case["photons"] * bands) * (1.5 * slots * 12 + 4 * 55 + 150)
    out = 12 * npix + (0 if case["kind"] == "host" else 8 * npix * bands)
    return {"bytes": tris * 64 + out, "flops": flops}


# ---- what a user's program has in hand -------------------------------------------------------------------------

_workloads, _renderers = {}, {}


def _workload(scene):
    if scene not in _workloads:
        _workloads[scene] = getattr(scenes, scene)()
    return _workloads[scene]


def _loaded(scene):
    from paper_1912_04000_gb300.renderer import Renderer
    return Renderer(0).load(_workload(scene))


def _renderer(scene):
    if scene not in _renderers:
        _renderers[scene] = _loaded(scene)
    return _renderers[scene]


def _guide_weights():
    """Parameters with the spread of a trained guide (fixed: the guide of the scene)."""
    rng = np.random.default_rng(11)
    grid = rng.standard_normal(_LEVELS * (1 << _LOG2_TABLE) * _FEATURES, np.float32) * np.float32(0.1)
    return grid, rng.standard_normal(3 * 64 * 64 + 64 * 48, np.float32) * np.float32(0.2)


def _guided_renderer(scene):
    r = _renderer(scene)
    if not hasattr(r, "guide_log2_table"):
        r.guide_init(seed=11, log2_table=_LOG2_TABLE)
        r.guide_set_params(*_guide_weights())
    return r


def _cameras(case, seed):
    """Poses near the workload's own for the first view, along the aisle (or in the room) for the others."""
    rng = random.Random(seed * 2654435761 + 17)
    base = _workload(case["scene"]).cameras[0]
    room = _BANDS[case["scene"]] == 16
    s = 0.1 if room else 1.0
    cams = []
    for i, (w, h) in enumerate(_views(case)):
        pos = tuple(p + s * rng.uniform(-0.5, 0.5) for p in base.pos)
        look = tuple(p + s * rng.uniform(-2.0, 2.0) for p in base.look)
        if i and not room:
            pos = (rng.uniform(5.0, 40.0), rng.uniform(1.0, 6.0), rng.uniform(8.0, 12.0))
            look = (rng.uniform(50.0, 80.0), rng.uniform(0.0, 25.0), rng.uniform(0.0, 20.0))
        cams.append(scenes.Camera(pos, look, base.up, base.vfov_deg, w, h))
    return cams


def _records(case, seed):
    """Training records on the scene's surfaces (chosen by area): sun samples (directions of the sun cone) and
    continuations (directions of the hemisphere, a tenth of the radiance) in turn, a share of them with exponential
    weights."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    wl, n = _workload(case["scene"]), case["records"]
    v = wl.scene.verts[wl.scene.tris.astype(np.int64)].astype(np.float64)
    nrm = np.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    area = np.linalg.norm(nrm, axis=1)
    share = torch.from_numpy(np.cumsum(area) / area.sum()).cuda()
    tri, nrm = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (v, nrm / area[:, None]))
    u = torch.rand(n, 6, device="cuda", dtype=torch.float64, generator=g)
    pick = torch.searchsorted(share, u[:, 0].contiguous()).clamp(max=len(area) - 1)
    u = u.float()
    su = u[:, 1:2].sqrt()
    bary = torch.cat([1 - su, su * (1 - u[:, 2:3]), su * u[:, 2:3]], 1)
    rec = torch.zeros(n, 12, device="cuda")
    rec[:, 0:3] = (tri[pick] * bary[:, :, None]).sum(1)
    rec[:, 4:7] = nrm[pick]
    rec[:, 7] = (u[:, 3] * 9).floor().clamp(max=8)
    om = torch.randn(n, 3, device="cuda", generator=g)
    om = om / om.norm(dim=1, keepdim=True)
    om = om * torch.where((om * rec[:, 4:7]).sum(1, keepdim=True) < 0, -1.0, 1.0)
    cone = torch.from_numpy(wl.spectra.sun_dir).cuda() + 0.14 * torch.randn(n, 3, device="cuda", generator=g)
    om[::2] = (cone / cone.norm(dim=1, keepdim=True))[::2]
    rec[:, 8:11] = om
    rec[:, 3] = torch.where(u[:, 4] < case["weighted"], -torch.log1p(-0.999999 * u[:, 5]), torch.zeros_like(su[:, 0]))
    rec[1::2, 3] *= 0.1
    return rec


def _image(case, seed):
    """Spectral sums of a partly lit frame: dark pixels among lit ones, sums over the samples."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    p, b = case["pixels"], case["bands"]
    x = torch.rand(p, b, device="cuda", dtype=torch.float64, generator=g) * case["spp"]
    return x * (torch.rand(p, 1, device="cuda", generator=g) < 0.8)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed}
    if kind == "guide_grad":
        s["r"], s["rec"] = _guided_renderer(case["scene"]), _records(case, seed)
        return s
    if kind == "xyz":
        s["r"], s["image"] = _renderer(case["scene"]), _image(case, seed)
        return s
    s["cams"] = _cameras(case, seed)
    if kind == "guided":
        s["r"] = _guided_renderer(case["scene"])
    elif kind == "graph":
        # a handle of its own (it keeps one captured render) and the caller's output buffers
        s["r"] = _loaded(case["scene"])
        npix = _pixels(case)
        s["spectral"] = torch.empty(npix, case["bands"], dtype=torch.float64, device="cuda")
        s["xyz"] = torch.empty(npix, 3, dtype=torch.float32, device="cuda")
    else:
        s["r"] = _renderer(case["scene"])
    return s


def run(s):
    case, r = s["case"], s["r"]
    kind = case["kind"]
    if kind == "xyz":
        return r.xyz(s["image"], case["band_first"], case["spp"])
    if kind == "guide_grad":
        loss, dgrid, dW = r.guide_grad(s["rec"])
        return {"loss": loss, "dgrid": dgrid, "dW": dW}
    args = (s["cams"], case["spp"], case["depth"], s["seed"], case["band_first"], case["bands"])
    if kind == "host":
        return r.render_host(*args)["xyz"]
    if kind == "photons":
        out = r.render_photons(*args, n_photons=case["photons"])
    elif kind == "graph":
        out = r.render(*args, use_graph=True, out_spectral=s["spectral"], out_xyz=s["xyz"])
    else:
        out = r.render(*args, bands_per_path=4 if kind == "bands4" else 1, guided=kind == "guided")
    return {"spectral": out["spectral"], "xyz": out["xyz"]}


# ---- the same in 64 bits ---------------------------------------------------------------------------------------

def exact(case, seed):
    if case["kind"] == "xyz":
        w = torch.from_numpy(_workload(case["scene"]).spectra.cmf_w).double().cuda()
        return _image(case, seed) / case["spp"] @ w[case["band_first"]:case["band_first"] + case["bands"]]
    if case["kind"] == "guide_grad":
        return _guide_gradient(case, seed)
    if case["scene"] == "tiny_box" and case["kind"] in ("render", "host", "graph"):
        spectral, xyz = _box_paths(case, seed)
        return xyz if case["kind"] == "host" else {"spectral": spectral, "xyz": xyz}
    return None  # a path tracer over 10^5 triangles in plain torch takes minutes


def _guide_gradient(case, seed):
    """Loss -sum (w / sum w) log q and its gradients: hash grid, harmonics of the normal and one-hot group through
    a 64-64-64-64-48 ReLU network into eight von Mises-Fisher lobes."""
    sc = _workload(case["scene"]).scene
    grid, W = (torch.from_numpy(a).double().cuda().requires_grad_() for a in _guide_weights())
    rec = _records(case, seed).double()
    rec = rec[rec[:, 3] > 0]
    lo, hi = (torch.from_numpy(f(sc.verts, 0)).double().cuda() for f in (np.min, np.max))
    unit = ((rec[:, 0:3] - lo) / (hi - lo)).clamp(0, 1)
    size, feats = 1 << _LOG2_TABLE, []
    for level in range(_LEVELS):
        res = 16 << level
        pos = unit * res
        cell = torch.minimum(pos.floor(), torch.tensor(res - 1.0, device="cuda", dtype=torch.float64))
        frac, cell, total = pos - cell, cell.long(), 0.0
        for corner in range(8):
            d = [(corner >> a) & 1 for a in range(3)]
            x, y, z = (cell[:, a] + d[a] for a in range(3))
            if (res + 1) ** 3 <= size:
                at = x + y * (res + 1) + z * (res + 1) ** 2
            else:
                at = (x ^ (y * 2654435761) ^ (z * 805459861)) & (size - 1)
            wt = 1.0
            for a in range(3):
                wt = wt * (frac[:, a] if d[a] else 1 - frac[:, a])
            total = total + wt[:, None] * grid.view(-1, _FEATURES)[level * size + at]
        feats.append(total)
    x, y, z = rec[:, 4], rec[:, 5], rec[:, 6]
    c = lambda v: math.sqrt(v / math.pi)  # noqa: E731
    sh = [c(0.25) + 0 * x, -c(0.75) * y, c(0.75) * z, -c(0.75) * x, c(3.75) * x * y, -c(3.75) * y * z,
          c(0.3125) * (3 * z * z - 1), -c(3.75) * x * z, c(0.9375) * (x * x - y * y),
          -c(1.09375) * y * (3 * x * x - y * y), c(26.25) * x * y * z, -c(0.65625) * y * (5 * z * z - 1),
          c(0.4375) * z * (5 * z * z - 3), -c(0.65625) * x * (5 * z * z - 1), c(6.5625) * z * (x * x - y * y),
          -c(1.09375) * x * (x * x - 3 * y * y)]
    group = torch.nn.functional.one_hot(rec[:, 7].long(), 16).double()
    h = torch.cat(feats + [torch.stack(sh, 1), group], 1)
    for layer in range(4):
        n_out = 48 if layer == 3 else 64
        h = h @ W[4096 * layer:4096 * layer + 64 * n_out].view(64, n_out)
        h = h.relu() if layer < 3 else h
    lobes = h[:, :40].view(-1, 8, 5)
    mu = torch.nn.functional.normalize(lobes[:, :, 1:4], dim=2, eps=1e-6)
    kappa = 0.5 + torch.nn.functional.softplus(lobes[:, :, 4])
    cos = (mu * rec[:, None, 8:11]).sum(2)
    log_q = torch.logsumexp(torch.log_softmax(lobes[:, :, 0], 1) + torch.log(kappa / (2 * math.pi))
                            - torch.log(-torch.expm1(-2 * kappa)) + kappa * (cos - 1), 1)
    loss = -(rec[:, 3] / rec[:, 3].sum() * log_q).sum()
    loss.backward()
    return {"loss": float(loss.detach()), "dgrid": grid.grad, "dW": W.grad}


def _philox(c, key):
    """Philox4x32-10 of four int64 tensors holding 32-bit words."""
    def mul(a, x):  # high and low words of a * x
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        return (hi + (lo >> 16)) >> 16, (((hi & 0xFFFF) << 16) + lo) & 0xFFFFFFFF

    k0, k1 = key & 0xFFFFFFFF, key >> 32
    for _ in range(10):
        (h0, l0), (h1, l1) = mul(0xD2511F53, c[0]), mul(0xCD9E8D57, c[2])
        c = (h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [(x >> 8).double() * 2.0 ** -24 for x in c]


def _dot(a, b):
    return (a * b).sum(-1)


def _basis(n):
    sign = torch.copysign(torch.ones_like(n[..., 2]), n[..., 2])
    a = -1 / (sign + n[..., 2])
    b = n[..., 0] * n[..., 1] * a
    return (torch.stack([1 + sign * n[..., 0] ** 2 * a, sign * b, -sign * n[..., 0]], -1),
            torch.stack([b, sign + n[..., 1] ** 2 * a, -n[..., 1]], -1))


def _around(axis, sin, cos, turn):
    """Directions at polar angle (sin, cos) and azimuth 2 pi turn around the axis."""
    t1, t2 = _basis(axis)
    phi = 2 * math.pi * turn
    return (sin * phi.cos())[:, None] * t1 + (sin * phi.sin())[:, None] * t2 + cos[:, None] * axis


def _sheet(c, n, k, lam, thickness):
    """Reflectance and transmittance of an absorbing sheet with incoherent inner reflections."""
    eta = torch.complex(n, k)
    s2 = 1 - c * c
    ct = torch.sqrt(1 - s2 / eta ** 2)
    R = 0.5 * (((c - eta * ct) / (c + eta * ct)).abs() ** 2 + ((eta * c - ct) / (eta * c + ct)).abs() ** 2)
    Ti = torch.exp(-4 * math.pi * k * thickness / (lam * 1e-9) / torch.sqrt(1 - s2 / n ** 2))
    den = 1 - (R * Ti) ** 2
    return R + (1 - R) ** 2 * R * Ti ** 2 / den, (1 - R) ** 2 * Ti / den


def _box_paths(case, seed):
    """Every path of a render of the stone room with its glass wall, by testing all triangles."""
    wl = _workload(case["scene"])
    f64 = lambda a: torch.as_tensor(np.asarray(a, np.float64), device="cuda")  # noqa: E731
    tri = f64(wl.scene.verts)[torch.from_numpy(wl.scene.tris.astype(np.int64)).cuda()]
    mat = torch.from_numpy(wl.scene.mat_id.astype(np.int64)).cuda()
    glass = f64(wl.scene.mat_type == scenes.THIN_GLASS).bool()
    thick = f64(wl.scene.mat_thickness)
    e1, e2 = tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    nrm = torch.stack([e1[:, 1] * e2[:, 2] - e1[:, 2] * e2[:, 1], e1[:, 2] * e2[:, 0] - e1[:, 0] * e2[:, 2],
                       e1[:, 0] * e2[:, 1] - e1[:, 1] * e2[:, 0]], 1)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    sp = wl.spectra
    lam, sunL, n_t, k_t, rho_t = (f64(a) for a in (sp.lambda_nm, sp.sun_L, sp.n, sp.k, sp.rho))
    sun = f64(sp.sun_dir)
    sun = sun / sun.norm()
    omc = 1 - math.cos(sp.sun_half_angle)
    eps = 1e-4 * float(np.linalg.norm(wl.scene.verts.max(0).astype(np.float64) - wl.scene.verts.min(0)))

    def hits(o, d, t_idx):
        """Distance along each ray to one triangle (inf: none), Moeller-Trumbore."""
        p = torch.linalg.cross(d, e2[t_idx].expand_as(d))
        det = _dot(e1[t_idx], p)
        s = o - tri[t_idx, 0]
        u = _dot(s, p) / det
        q = torch.linalg.cross(s, e1[t_idx].expand_as(s))
        v, t = _dot(d, q) / det, _dot(q, e2[t_idx]) / det
        return torch.where((u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0), t, torch.full_like(t, math.inf))

    key, B, b0 = seed, case["bands"], case["band_first"]
    spectral, first = [], 0
    for cam in _cameras(case, seed):
        npix = cam.width * cam.height
        pos, look, up = (f64(np.float32(a)) for a in (cam.pos, cam.look, cam.up))
        f = (look - pos) / (look - pos).norm()
        r = torch.linalg.cross(f, up)
        r = r / r.norm()
        u_ = torch.linalg.cross(r, f)
        th = math.tan(0.5 * float(np.float32(cam.vfov_deg)) * math.pi / 180)
        image = torch.zeros(npix * B, dtype=torch.float64, device="cuda")
        at = torch.arange(npix * B, device="cuda")
        px, band = at // B, b0 + at % B
        for s in range(case["spp"]):
            def rand(call, sel, s=s):
                return _philox((px[sel] + first, torch.full_like(sel, s), band[sel], torch.full_like(sel, call)), key)
            live = at
            u = rand(0, live)
            sx = (2 * ((px % cam.width) + u[0]) / cam.width - 1) * th * cam.width / cam.height
            sy = (1 - 2 * (torch.div(px, cam.width, rounding_mode="floor") + u[1]) / cam.height) * th
            d = f + sx[:, None] * r + sy[:, None] * u_
            d = d / d.norm(dim=1, keepdim=True)
            o, T = pos.expand_as(d), torch.ones_like(sx)
            covered = torch.zeros_like(live, dtype=torch.bool)
            for k in range(1, case["depth"] + 1):
                t, prim = torch.full_like(T, math.inf), torch.zeros_like(live)
                for i in range(tri.shape[0]):
                    ti = hits(o, d, i)
                    prim, t = torch.where(ti < t, i, prim), torch.minimum(t, ti)
                out = torch.isinf(t)
                seen = out & ~covered & (_dot(d, sun) >= math.cos(sp.sun_half_angle))
                image.index_add_(0, live[seen], (T * sunL[band[live]])[seen])
                live, o, d, T, covered, t, prim = (a[~out] for a in (live, o, d, T, covered, t, prim))
                p, ng, m, b = o + t[:, None] * d, nrm[prim], mat[prim], band[live]
                n = torch.where((_dot(ng, d) < 0)[:, None], ng, -ng)
                u, pane = rand(4 * k, live), glass[m]
                # stone: a sun sample through the panes, then a cosine-weighted continuation
                om = u[0] * omc
                w = _around(sun.expand_as(n), torch.sqrt(om * (2 - om)), 1 - om, u[1])
                c = _dot(n, w)
                lit = ~pane & (c > 0)
                so, sd, sb = (p + eps * n)[lit], w[lit], b[lit]
                pass_ = torch.ones_like(c[lit])
                for i in range(tri.shape[0]):
                    hit = ~torch.isinf(hits(so, sd, i))
                    Ts = 0.0
                    if bool(glass[mat[i]]):
                        Ts = _sheet(_dot(sd, nrm[i]).abs(), n_t[mat[i]][sb], k_t[mat[i]][sb], lam[sb], thick[mat[i]])[1]
                    pass_ = torch.where(hit, pass_ * Ts, pass_)
                image.index_add_(0, live[lit], (T * rho_t[m, b] * c * sunL[b] * 2 * omc)[lit] * pass_)
                if k == case["depth"]:
                    break
                nd = _around(n, torch.sqrt(u[2]), torch.sqrt(1 - u[2]), u[3])
                # glass: reflect or pass, the pair's weight kept
                Rs, Ts = _sheet(-_dot(d, n), n_t[m, b], k_t[m, b], lam[b], thick[m])
                mirror = pane & (rand(4 * k + 1, live)[0] < Rs / (Rs + Ts))
                refl = d - 2 * _dot(d, n)[:, None] * n
                d = torch.where(mirror[:, None], refl, torch.where(pane[:, None], d, nd))
                o = torch.where((pane & ~mirror)[:, None], p - eps * n, p + eps * n)
                T = T * torch.where(pane, Rs + Ts, rho_t[m, b])
                covered = torch.where(pane, covered & ~mirror, torch.ones_like(covered))
        first += npix
        spectral.append(image.view(npix, B))
    spectral = torch.cat(spectral)
    return spectral, spectral / case["spp"] @ f64(sp.cmf_w)[b0:b0 + B]
