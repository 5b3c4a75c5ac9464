"""What a program that uses this library has it do, as measurable cases.

A case is a dict of plain values.  `path` names the calls a pass makes:

  frame     hr_render_frame: clusters, thick-hair fit, LoD, BVH and image in one call
  fixed     a fixed LoD setting: hr_build_clusters, hr_build_bvh(lod), hr_render
  render    hr_render alone on a built scene (shadow rays: dual-scattering light paths)
  animated  hr_asset_update from page-locked host memory, hr_render_frame with a BVH
            refit and the deferred LoD, the image back to page-locked host memory
  guided    hr_build_guided_clusters (k-means guides, guide triples, fits, skinning
            weights) with every result read out
  skin      hr_asset_skin with new guide poses, then hr_render_frame on the kept hierarchy
  layers    the single steps: hr_build_clusters, hr_lod_widths, hr_select_lod, and the
            thick hairs read out
  serve     a burst of hr_submit on several resident assets, polled until all are done

The scenes have the shapes of the repository's own configurations (a strand cap, curled
clusters, a full head, long straight hair), made on the GPU from the seed: roots on a
spherical cap, smooth flow, curls whose phase varies smoothly over the scalp, per-vertex
jitter, per-strand materials and elliptical cross-sections.
"""
import math

import numpy as np
import torch

import paper_2405_10565_gb300 as hr

EPS_W = 2.0  # LoD threshold in pixels


def listed():
    return [
        # A material preview: 64 strands, one light, one sample per pixel.  The smallest
        # call there is; launches and latency are all of it.
        dict(name="preview_64", path="frame", hair="cap", n=64, S=16, clusters=0, width=128,
             height=128, spp=1, k=1, lights=0, fill=0.8, ortho=True, precision=0, trt=False),
        # A thumbnail of a small asset, every size odd, with the Marschner lobe.
        dict(name="thumb_odd_3k", path="frame", hair="curls", n=3001, S=23, clusters=131,
             width=211, height=157, spp=3, k=3, lights=2, fill=0.25, ortho=False, precision=0,
             trt=True),
        # A dense close view of curled hair in which half the clusters are thick hairs and
        # composite through the k-buffer.
        dict(name="curls_half_10k", path="fixed", hair="curls", n=10000, S=32, clusters=256,
             width=512, height=512, spp=4, k=4, lights=2, fill=0.8, ortho=False, precision=0,
             trt=False, lod="half"),
        # The benchmark's frame: a full head in a far view, a third of its clusters thick.
        dict(name="head_far_100k", path="frame", hair="head", n=100000, S=64, clusters=4096,
             width=1920, height=1080, spp=8, k=4, lights=8, fill=0.15, ortho=False,
             precision=0, trt=False),
        # The same head close up, every cluster on strands, with the FP16 tables.
        dict(name="head_close_100k", path="frame", hair="head", n=100000, S=64, clusters=4096,
             width=1920, height=1080, spp=8, k=4, lights=8, fill=0.9, ortho=False,
             precision=1, trt=False),
        # Animation: every strand moves each frame, its positions come from the host and the
        # image goes back.
        dict(name="head_animated_100k", path="animated", hair="head", n=100000, S=64,
             clusters=4096, width=1920, height=1080, spp=8, k=4, lights=8, fill=0.45,
             ortho=False, precision=0, trt=False, motion=2e-3),
        # Dual-scattering light paths: a shadow ray per hit and light.
        dict(name="head_shadows_100k", path="render", hair="head", n=100000, S=64,
             clusters=4096, width=1920, height=1080, spp=8, k=4, lights=8, fill=0.15,
             ortho=False, precision=0, trt=False, shadows=True),
        # The largest frame: half a million long strands, 4K, 16 samples, K = 8.
        dict(name="straight_500k_4k", path="frame", hair="straight", n=500000, S=64,
             clusters=16384, width=3840, height=2160, spp=16, k=8, lights=4, fill=0.3,
             ortho=False, precision=1, trt=False),
        # Preparing an asset for skinned animation, once per model.
        dict(name="guided_build_100k", path="guided", hair="head", n=100000, S=64, guides=256,
             iterations=4),
        # Skinned animation: only the guides' poses are new.
        dict(name="skinned_100k", path="skin", hair="head", n=100000, S=64, guides=256,
             iterations=4, width=1920, height=1080, spp=8, k=4, lights=8, fill=0.15,
             ortho=False, precision=0, trt=False, motion=2e-3),
        # The hierarchy, the thick-hair fit and the LoD rule by themselves, ragged sizes.
        dict(name="hierarchy_30k", path="layers", hair="head", n=30011, S=47, clusters=1237,
             width=960, height=540, lights=1, fill=0.15, ortho=False),
        # Serving: a burst of requests on two resident assets, mixed sizes and LoD budgets.
        dict(name="serve_burst_16", path="serve", hair="head", n=50000, n2=10000, S=64,
             clusters=1024, requests=16, width=1280, height=720, spp=4, k=4, lights=8,
             fill=0.15, ortho=False, precision=1, trt=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["frame"] * 5 + ["fixed", "render", "animated", "guided", "skin", "layers",
                                       "serve"])
    hair = rng.choice(["cap", "curls", "head", "head", "straight"])
    n = _log(rng, 64, 200000 if path == "frame" else 60000)
    if path in ("guided", "skin"):
        n = max(n, 600)
    S = rng.randint(7, 64)
    c = dict(path=path, hair=hair, n=n, S=S)
    if path in ("guided", "skin"):
        c.update(guides=_log(rng, 12, max(13, min(256, n // 40))), iterations=rng.randint(1, 6))
    else:
        c["clusters"] = max(1, n // rng.randint(9, 60))
    if path == "guided":
        return c
    width = _log(rng, 64, 1920)
    height = max(33, int(width * rng.uniform(0.5, 0.8)))
    c.update(width=width, height=height, lights=rng.choice([0, 1, 2, 4, 8]),
             fill=round(rng.uniform(0.1, 0.9), 3), ortho=rng.random() < 0.15)
    if path == "layers":
        return c
    c.update(spp=rng.choice([1, 2, 3, 4, 5, 8]), k=rng.randint(1, 8),
             precision=rng.randint(0, 1), trt=rng.random() < 0.3)
    if path == "fixed":
        c["lod"] = rng.choice(["half", "strands", "eth"])
    if path == "render":
        c["shadows"] = rng.random() < 0.6
        if c["shadows"]:  # a shadow ray per hit and light: small images
            c["width"], c["height"] = min(width, 400), min(height, 300)
            c["fill"] = min(c["fill"], 0.3)
    if path in ("animated", "skin"):
        c["motion"] = rng.choice([2e-5, 2e-3])
    if path == "serve":
        c.update(n2=max(64, n // 4), requests=rng.randint(3, 16), width=min(width, 1280),
                 height=min(height, 720))
    return c


# ------------------------------------------------------------------------------ scenes


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


_HAIR = {
    "cap": dict(head=1.0, cap=60.0, length=1.0, jitter=0.02, radius=4e-3),
    "curls": dict(cap=60.0, length=1.0, jitter=0.002, radius=1e-3, curl=0.05, turns=3.0),
    "head": dict(cap=25.0, length=1.0, jitter=4e-4, radius=1e-3, curl=0.02, turns=2.0,
                 hang=0.08, spread=0.3),
    "straight": dict(cap=35.0, length=2.0, jitter=0.0, radius=1e-3, hang=0.05, spread=0.25),
}


def _strands(kind, n, S, g):
    """Vertices [n, S + 1, 4] (x, y, z, r) on the GPU."""
    p = dict(head=0.5, curl=0.0, turns=0.0, hang=0.0, spread=0.35, droop=1.6)
    p.update(_HAIR[kind])
    f64 = dict(dtype=torch.float64, device="cuda")
    cos_t = 1.0 - torch.rand(n, generator=g, **f64) * (1.0 - math.cos(math.radians(p["cap"])))
    sin_t = (1.0 - cos_t * cos_t).clamp_min(0.0).sqrt()
    phi = 2.0 * math.pi * torch.rand(n, generator=g, **f64)
    nrm = torch.stack([sin_t * phi.cos(), cos_t, sin_t * phi.sin()], -1)
    root = p["head"] * nrm
    horiz = nrm * torch.tensor([1.0, 0.0, 1.0], **f64)
    down = torch.tensor([0.0, -1.0, 0.0], **f64)
    s = ((torch.arange(S, **f64) + 0.5) / S)[None, :, None]
    if p["hang"] > 0.0:
        w = torch.exp(-s / p["hang"])
        d = w * nrm[:, None] + (1.0 - w) * (p["spread"] * horiz[:, None] + down)
    else:
        d = (1.0 - s) * nrm[:, None] + s * p["droop"] * (p["spread"] * horiz[:, None] + down)
    verts = torch.empty(n, S + 1, 3, **f64)
    verts[:, 0] = root
    verts[:, 1:] = root[:, None] + torch.cumsum(_unit(d) * (p["length"] / S), 1)
    if p["curl"] > 0.0:
        amp = p["curl"] * (1.0 + 0.2 * torch.sin(7.0 * root[:, 0] + 5.0 * root[:, 2]))
        ph = 2.0 * math.pi * (1.5 * root[:, 0] + 1.1 * root[:, 2])
        ph = (ph + 0.05 * torch.randn(n, generator=g, **f64))[:, None]
        u = _unit(torch.linalg.cross(nrm, torch.tensor([[0.0, 0.0, 1.0]], **f64).expand_as(nrm)) +
                  torch.tensor([1e-6, 0.0, 0.0], **f64))
        v = _unit(torch.linalg.cross(nrm, u))
        sk = torch.arange(S + 1, **f64) / S
        ang = 2.0 * math.pi * p["turns"] * sk[None] + ph
        off = ((ang.cos() - ph.cos())[..., None] * u[:, None] +
               (ang.sin() - ph.sin())[..., None] * v[:, None])
        verts += amp[:, None, None] * (4.0 * sk).clamp_max(1.0)[None, :, None] * off
    if p["jitter"] > 0.0:
        verts[:, 1:] += p["jitter"] * torch.randn(n, S, 3, generator=g, **f64)
    out = torch.full((n, S + 1, 4), p["radius"], dtype=torch.float32, device="cuda")
    out[..., :3] = verts.float()
    return out


def _materials(kind, n, trt, g):
    """Materials [n, 12] and cross-section shapes [n, 2]."""
    r = torch.rand(n, 4, generator=g, device="cuda")
    if kind == "cap":  # one grey fibre, circular cross-section
        fr = ((1.55 - 1.0) / (1.55 + 1.0)) ** 2
        att = (1.0 - fr) ** 2 * math.exp(-0.6)
        row = [fr] * 3 + [att] * 3 + [(1.0 - fr - att) / 2.0] * 3 + [0.2, 0.3, 0.3]
        mat = torch.tensor(row, device="cuda").repeat(n, 1)
        shape = torch.stack([torch.zeros(n, device="cuda"), 2.0 * math.pi * r[:, 3]], -1)
        return mat.contiguous(), shape.contiguous()
    curls = kind == "curls"
    t = torch.full((n, 1), 0.5, device="cuda") if curls else r[:, 0:1]  # melanin
    q = torch.full((n, 1), 0.5, device="cuda") if curls else r[:, 1:2]  # roughness

    def lerp(a, b):
        a, b = torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda")
        return 0.5 * (a + (b - a) * t)

    third = (lerp((0.20, 0.14, 0.08), (0.10, 0.06, 0.03)) if trt
             else lerp((0.20, 0.11, 0.10), (0.40, 0.21, 0.08)))
    mat = torch.cat([lerp((0.03, 0.03, 0.03), (0.25, 0.25, 0.25)),
                     lerp((0.25, 0.17, 0.07), (0.38, 0.25, 0.18)), third,
                     0.08 + 0.07 * q, 0.12 + 0.18 * q, 0.20 + 0.20 * q], 1)
    ecc = {"curls": torch.full((n,), 0.8, device="cuda"),
           "straight": torch.full((n,), 0.9, device="cuda"),
           "head": (0.6 + 0.4 * r[:, 2]).clamp_max(0.99)}[kind]
    return mat.contiguous(), torch.stack([ecc, 2.0 * math.pi * r[:, 3]], -1).contiguous()


def _camera(case, verts):
    """Packed camera record that looks along -z at the hair, whose height (or width) fills
    `fill` of the frame."""
    W, H = case["width"], case["height"]
    p = verts[..., :3].reshape(-1, 3)
    lo, hi = p.amin(0).double().cpu().numpy(), p.amax(0).double().cpu().numpy()
    ctr, ext = 0.5 * (lo + hi), hi - lo
    half = 0.5 * max(ext[1], ext[0] * H / W)
    if case["ortho"]:
        dist, pix = 2.0 + ext[2], 0.5 * H / (half / case["fill"])
    else:
        tan_h = math.tan(math.radians(20.0))
        dist, pix = half / (case["fill"] * tan_h) + 0.5 * ext[2], 0.5 * H / tan_h
    c = np.zeros(20, np.float32)
    c[0:4] = 0 if case["ortho"] else 1, W, H, pix
    c[4:7] = ctr + np.array([0.0, 0.0, dist])
    c[7:10], c[10:13], c[13:16], c[16] = (1, 0, 0), (0, 1, 0), (0, 0, -1), 1e-3
    return c, ctr


def _lights(count, ctr, g):
    if count == 0:  # one directional light
        return np.array([[0.57735, 0.57735, 0.57735, 0.0, 1.0, 1.0, 1.0, 0.0]], np.float32)
    u = torch.rand(count, 2, generator=g, device="cuda").double().cpu().numpy()
    th, ph = np.arccos(0.9 - 1.5 * u[:, 0]), 2.0 * math.pi * u[:, 1]
    d = np.stack([np.sin(th) * np.cos(ph), 0.5 * np.sin(th) * np.sin(ph) + 0.3, np.cos(th)], -1)
    L = np.zeros((count, 8), np.float32)
    L[:, :3] = ctr + 3.0 * d / np.linalg.norm(d, axis=-1, keepdims=True)
    L[:, 3], L[:, 4:7] = 1.0, 9.0 / count
    return L


def _scene(case, seed, n=None):
    g = torch.Generator("cuda").manual_seed(seed)
    n = n or case["n"]
    verts = _strands(case["hair"], n, case["S"], g)
    mat, shape = _materials(case["hair"], n, case.get("trt", False), g)
    cam, lights = None, None
    if "width" in case:
        cam, ctr = _camera(case, verts)
        lights = _lights(case["lights"], ctr, g)
    torch.cuda.synchronize()  # the library reads them on its own stream
    return verts, mat, shape, cam, lights


def _moved(verts, amp):
    """The strands in another pose: a smooth displacement that grows from the roots."""
    v = verts.clone()
    grow = torch.linspace(0.0, amp, v.shape[1], device="cuda")[None]
    v[..., 0] += grow * torch.sin(7.0 * verts[..., 1] + 1.3)
    v[..., 2] += grow * torch.cos(5.0 * verts[..., 0] - 1.3)
    return v


# ---------------------------------------------------------------------------- programs

_shared = {}


def _context():
    """The program's context: one for all its assets, on a stream of its own."""
    if not _shared:
        _shared["stream"] = torch.cuda.Stream()
        _shared["ctx"] = hr.hr_create(0, 0, _shared["stream"].cuda_stream)
    return _shared["ctx"], _shared["stream"]


class State:
    """A program's handles and buffers; gives them back when it is dropped."""

    def __init__(self, ctx, own=False):
        self.ctx, self.own, self.assets, self.i = ctx, own, [], 0

    def __del__(self):
        if self.own:
            hr.hr_serve_stop(self.ctx)
        for a in self.assets:
            hr.hr_asset_destroy(self.ctx, a)
        if self.own:
            hr.hr_destroy(self.ctx)


def _flags(case):
    f = hr.HR_FLAG_TRT if case.get("trt") else 0
    if case.get("shadows"):
        f |= hr.HR_FLAG_SHADOWS
    if case["path"] == "animated":
        f |= hr.HR_FLAG_REFIT | hr.HR_FLAG_DEFERRED_LOD | hr.HR_FLAG_LOD_HYSTERESIS
    if case["path"] == "skin":
        f |= (hr.HR_FLAG_KEEP_HIERARCHY | hr.HR_FLAG_REFIT | hr.HR_FLAG_DEFERRED_LOD |
              hr.HR_FLAG_LOD_HYSTERESIS)
    return f


def _preset(setting, C, L):
    lod = np.full(C, L, np.uint8)
    if setting == "eth":
        lod[:] = 0
    elif setting == "half":
        lod[0::2] = 0
    return lod


def prepare(case, seed):
    path = case["path"]
    if path == "serve":
        return _prepare_serve(case, seed)
    ctx, stream = _context()
    st = State(ctx)
    st.case = case
    verts, mat, shape, st.cam, lights = _scene(case, seed)
    a = hr.hr_asset_create(ctx, verts, mat, shape)
    st.assets.append(a)
    st.asset = a
    st.n_clusters = case.get("clusters", 0)
    dev = dict(device="cuda")
    if path not in ("guided", "layers"):
        st.img = torch.zeros(case["height"], case["width"], 3, **dev)
        st.desc = hr.render_desc(st.cam, lights, case["spp"], case["k"], seed & 0xffffffff,
                                 case["precision"], _flags(case))
    if path == "fixed":
        hr.hr_build_clusters(ctx, a, st.n_clusters)
        st.lod = _preset(case["lod"], *hr.hr_hierarchy_info(ctx, a)[:2])
    elif path == "render":
        hr.hr_build_clusters(ctx, a, st.n_clusters)
        if hr.hr_hierarchy_info(ctx, a)[1]:
            hr.hr_select_lod(ctx, a, st.cam, EPS_W, 0, 0, None)
        hr.hr_build_bvh(ctx, a, None)
    elif path == "animated":
        st.poses = [v.cpu().pin_memory() for v in (_moved(verts, case["motion"]), verts)]
        st.host = torch.zeros(case["height"], case["width"], 3).pin_memory()
        st.stream = stream
    elif path == "guided":
        N = case["n"]
        st.cluster_of = torch.zeros(N, dtype=torch.int32, **dev)
        st.order = torch.zeros(N, dtype=torch.int32, **dev)
        st.guides = torch.zeros(case["guides"], dtype=torch.int32, **dev)
        # the number of thick hairs depends on the hair; it is below the number of strands
        st.xsec = torch.zeros(N, case["S"] + 1, 12, **dev)
        st.mat = torch.zeros(N, 12, **dev)
    elif path == "skin":
        G = case["guides"]
        hr.hr_build_guided_clusters(ctx, a, G, case["iterations"])
        gid = np.zeros(G, np.int32)
        hr.hr_guides_export(ctx, a, gid)
        rows = torch.from_numpy(np.maximum(gid, 0)).long().cuda()
        st.poses = [v[rows].contiguous().cpu().pin_memory()
                    for v in (_moved(verts, case["motion"]), verts)]
    elif path == "layers":
        hr.hr_build_clusters(ctx, a, st.n_clusters)
        C, L, E = hr.hr_hierarchy_info(ctx, a)
        N, S1 = case["n"], case["S"] + 1
        st.cluster_of = torch.zeros(N, dtype=torch.int32, **dev)
        st.order = torch.zeros(N, dtype=torch.int32, **dev)
        st.levels, st.eths = L, E
        st.xsec = torch.zeros(E, S1, 12, **dev)
        st.mat = torch.zeros(E, 12, **dev)
        st.width = torch.zeros(C, L, **dev)
        st.lod = torch.zeros(C, dtype=torch.uint8, **dev)
    torch.cuda.synchronize()
    return st


def _prepare_serve(case, seed):
    ctx = hr.hr_create(0, 0, None)
    st = State(ctx, own=True)
    hr.hr_serve_start(ctx, 16, 1 << 24)
    st.case, st.requests = case, []
    descs = []
    for j, n in enumerate((case["n"], case["n2"])):
        verts, mat, shape, cam, lights = _scene(case, seed + 7 * j, n)
        a = hr.hr_asset_create(ctx, verts, mat, shape)
        st.assets.append(a)
        hr.hr_build_clusters(ctx, a, min(case["clusters"], n))
        descs.append((a, cam, lights))
    for i in range(case["requests"]):
        a, cam, lights = descs[i % 2]
        cam = cam.copy()
        shrink = (1.0, 0.5, 0.25)[i % 3]  # the requests' sizes differ
        W, H = max(16, int(case["width"] * shrink)), max(16, int(case["height"] * shrink))
        cam[3] *= H / cam[2]
        cam[1], cam[2] = W, H
        d = hr.render_desc(cam, lights, max(1, case["spp"] - i % 2), case["k"],
                           (seed + i) & 0xffffffff, case["precision"], _flags(case))
        st.requests.append((a, d, torch.zeros(H, W, 3, device="cuda"), i % 4))
    torch.cuda.synchronize()
    return st


def run(st):
    c, ctx = st.case, st.ctx
    path = c["path"]
    if path == "serve":
        tickets = [hr.hr_submit(ctx, a, d, img, EPS_W, bias) for a, d, img, bias in st.requests]
        for t in tickets:
            status, res = hr.hr_poll(ctx, t, 20000)
            if status != hr.HR_OK or res.status != hr.HR_OK:
                raise RuntimeError("a served request did not finish")
        return [img for _, _, img, _ in st.requests]
    a = st.asset
    if path == "frame":
        hr.hr_render_frame(ctx, a, st.n_clusters, EPS_W, 0, st.desc, st.img)
        return st.img
    if path == "fixed":
        hr.hr_build_clusters(ctx, a, st.n_clusters)
        hr.hr_build_bvh(ctx, a, st.lod)
        hr.hr_render(ctx, a, st.desc, st.img)
        return st.img
    if path == "render":
        hr.hr_render(ctx, a, st.desc, st.img)
        return st.img
    if path == "animated":
        hr.hr_asset_update(ctx, a, st.poses[st.i % 2])
        st.i += 1
        hr.hr_render_frame(ctx, a, st.n_clusters, EPS_W, 0, st.desc, st.img)
        with torch.cuda.stream(st.stream):
            st.host.copy_(st.img, non_blocking=True)
        return st.host
    if path == "skin":
        hr.hr_asset_skin(ctx, a, st.poses[st.i % 2])
        st.i += 1
        hr.hr_render_frame(ctx, a, 0, EPS_W, 0, st.desc, st.img)
        return st.img
    if path == "guided":
        hr.hr_build_guided_clusters(ctx, a, c["guides"], c["iterations"], 0, st.cluster_of,
                                    st.order)
        hr.hr_guides_export(ctx, a, st.guides)
        if hr.hr_hierarchy_info(ctx, a)[2]:
            hr.hr_eth_export(ctx, a, st.xsec, None, st.mat)
        return dict(order=st.order, cluster_of=st.cluster_of, guides=st.guides, xsec=st.xsec,
                    mat=st.mat)
    # layers
    hr.hr_build_clusters(ctx, a, st.n_clusters, 0, st.cluster_of, st.order)
    out = dict(order=st.order, cluster_of=st.cluster_of)
    if st.eths:
        hr.hr_lod_widths(ctx, a, st.cam, st.width)
        hr.hr_select_lod(ctx, a, st.cam, EPS_W, 0, 0, st.lod)
        hr.hr_eth_export(ctx, a, st.xsec, None, st.mat)
        x = st.xsec
        out.update(widths=st.width, lod=st.lod, mat=st.mat, centre=x[..., 0:3], a=x[..., 3],
                   e1=x[..., 4:7], b=x[..., 7], e2=x[..., 8:12])
    return out


def _levels(n, clusters):
    per, k = n // clusters, 0
    if per < 2:
        return 0
    while 4 ** (k + 1) <= per / 2:
        k += 1
    return k + 1


def work(case):
    """Bytes: vertices, materials and shapes read once, results written once.  Operations:
    191 per strand vertex and thick-hair level for the fit, log2(segments) box pairs of 24,
    one primitive test of 60 and 150 per light for each sample that the hair's part of the
    frame holds (a quarter of the framed square), and 8 per vertex pair of a k-means step."""
    total_b = total_f = 0.0
    for n in [case["n"]] + ([case["n2"]] if "n2" in case else []):
        b, f, S1, path = n * (case["S"] + 1) * 16.0 + n * 56.0, 0.0, case["S"] + 1, case["path"]
        if path in ("frame", "fixed", "animated", "layers") and case["clusters"]:
            f += 191.0 * n * S1 * _levels(n, case["clusters"])
        if path == "guided":
            f += 8.0 * n * S1 * case["guides"] * (case["iterations"] + 2)
            b += n * S1 * 16.0
        if path == "layers":
            E = sum(case["clusters"] * 4 ** k for k in range(_levels(n, case["clusters"])))
            b += E * (S1 * 48.0 + 48.0) + 8.0 * n
        if "spp" in case:
            px = case["width"] * case["height"] * (
                sum((1.0, 0.25, 0.0625)[i % 3] for i in range(case["requests"])) / 2
                if path == "serve" else 1.0)
            b += px * 12.0
            side = case["fill"] * case["height"]
            rays = (px * case["spp"] * 0.25 * min(1.0, side * side / (case["width"] * case["height"])))
            f += rays * (math.log2(n * case["S"]) * 24.0 + 60.0 + 150.0 * max(1, case["lights"]))
        total_b, total_f = total_b + b, total_f + f
    return {"bytes": total_b, "flops": max(total_f, 1.0)}


# ------------------------------------------------------------------- 64-bit references


def exact(case, seed):
    if case["path"] == "frame" and case["n"] * case["S"] <= 3000 and not case["clusters"] and \
            case["width"] * case["height"] * case["spp"] <= 40000:
        return _exact_strands(case, seed)
    if case["path"] == "layers":
        return _exact_layers(case, seed)
    return None


def _splitmix(seed, idx):
    """Outputs number `idx` of the SplitMix64 stream of `seed` (numpy uint64)."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (idx + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _gauss(beta, x):
    return torch.exp(-0.5 * (x / beta) ** 2) / (math.sqrt(2.0 * math.pi) * beta)


def _exact_strands(case, seed):
    """The image of a scene of plain strands: every sample against every segment."""
    verts, mat, shape, cam, lights = _scene(case, seed)
    P, mat, shape = verts.double(), mat.double(), shape.double()
    W, H, spp = case["width"], case["height"], case["spp"]
    sid = np.arange(W * H * spp, dtype=np.uint64)
    jit = [(_splitmix(seed & 0xffffffff, np.uint64(2) * sid + np.uint64(j)) >> np.uint64(40))
           .astype(np.float64) / 16777216.0 for j in (0, 1)]
    pix = (sid // np.uint64(spp)).astype(np.int64)
    sx = torch.from_numpy((pix % W + jit[0] - 0.5 * W) / float(cam[3])).cuda()
    sy = torch.from_numpy((0.5 * H - pix // W - jit[1]) / float(cam[3])).cuda()
    eye, right, up, fwd = (torch.tensor(cam[i:i + 3].astype(np.float64), device="cuda")
                           for i in (4, 7, 10, 13))
    plane = sx[:, None] * right + sy[:, None] * up
    if case["ortho"]:
        o, d = eye + plane, fwd.expand(len(sid), 3)
    else:
        o, d = eye.expand(len(sid), 3), fwd + plane
    d = _unit(d)
    # segment frames: the ellipse of the circle's area in the basis of Duff et al. 2017
    n, S = case["n"], case["S"]
    c0, ax = P[:, :-1, :3].reshape(-1, 3), (P[:, 1:, :3] - P[:, :-1, :3]).reshape(-1, 3)
    length = ax.norm(dim=-1)
    t = ax / length[:, None]
    sgn = torch.where(t[:, 2] >= 0, 1.0, -1.0).double()
    qa = -1.0 / (sgn + t[:, 2])
    qb = t[:, 0] * t[:, 1] * qa
    b1 = torch.stack([1 + sgn * t[:, 0] ** 2 * qa, sgn * qb, -sgn * t[:, 0]], -1)
    b2 = torch.stack([qb, sgn + t[:, 1] ** 2 * qa, -t[:, 1]], -1)
    ecc, psi = (shape[:, j].repeat_interleave(S) for j in (0, 1))
    e1 = psi.cos()[:, None] * b1 + psi.sin()[:, None] * b2
    e2 = torch.linalg.cross(t, e1)
    rad = P[:, 0, 3].repeat_interleave(S)
    q = (1 - ecc ** 2) ** 0.25
    e1, e2, t = e1 / (rad / q)[:, None], e2 / (rad * q)[:, None], t / length[:, None]
    out = torch.zeros(len(sid), 3, dtype=torch.float64, device="cuda")
    for i in range(0, len(sid), 2048):
        oo, dd = o[i:i + 2048], d[i:i + 2048]
        uvw = [((oo @ e.T) - (c0 * e).sum(-1), dd @ e.T) for e in (e1, e2, t)]
        (u0, du), (v0, dv), (w0, dw) = uvw
        A = du * du + dv * dv
        tc = -(u0 * du + v0 * dv) / A
        disc = 1 - (u0 + tc * du) ** 2 - (v0 + tc * dv) ** 2
        half = (disc.clamp_min(0) / A).sqrt()
        best = torch.full_like(tc, math.inf)
        for root in (tc + half, tc - half):  # the nearer root in range wins
            w = w0 + root * dw
            best = torch.where((disc >= 0) & (root > 0) & (w >= 0) & (w <= 1), root, best)
        th, j = best.min(1)
        hit = torch.isfinite(th)
        out[i:i + 2048][hit] = _shade(oo[hit] + th[hit, None] * dd[hit], -dd[hit],
                                      _unit(t[j[hit]]), mat[j[hit] // S], lights,
                                      case.get("trt", False))
    return out.reshape(H, W, spp, 3).mean(2)


def _shade(x, wo, t, m, lights, trt):
    """Sum over the lights of f_single E cos(theta_i)."""
    so = (wo * t).sum(-1).clamp(-1, 1)
    wop = wo - so[:, None] * t
    rgb = torch.zeros_like(x)
    for L in lights.astype(np.float64):
        pos = torch.tensor(L[:3], device="cuda")
        if L[3] == 0:
            wi, E = _unit(pos).expand_as(x), 1.0
        else:
            dd = ((pos - x) ** 2).sum(-1)
            wi, E = (pos - x) / dd.sqrt()[:, None], 1.0 / dd
        si = (wi * t).sum(-1).clamp(-1, 1)
        wip = wi - si[:, None] * t
        cphi = ((wip * wop).sum(-1) / (wip.norm(dim=-1) * wop.norm(dim=-1))).clamp(-1, 1)
        th = 0.5 * (torch.asin(si) + torch.asin(so))
        lobe_r = _gauss(m[:, 9], th) / (2 * math.pi)
        lobe_t = _gauss(m[:, 10], th) * _gauss(m[:, 11], torch.acos(cphi) - math.pi)
        third = (_gauss(2 * m[:, 9], th) / (2 * math.pi) if trt
                 else torch.full_like(th, 1 / (2 * math.pi ** 2)))
        f = m[:, 0:3] * lobe_r[:, None] + m[:, 3:6] * lobe_t[:, None] + m[:, 6:9] * third[:, None]
        rgb += f * (E * (1 - si * si).clamp_min(0).sqrt())[:, None] * torch.tensor(L[4:7], device="cuda")
    return rgb


def _jacobi(A):
    """Eigenvalues (last axis) and vectors (columns) of symmetric 3x3 matrices."""
    A, V = A.clone(), torch.eye(3, dtype=A.dtype, device=A.device).expand_as(A).clone()
    for _ in range(8):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            apq = A[:, p, q]
            th = (A[:, q, q] - A[:, p, p]) / (2 * torch.where(apq == 0, torch.ones_like(apq), apq))
            tt = torch.where(th >= 0, 1.0, -1.0) / (th.abs() + (th * th + 1).sqrt())
            tt = torch.where(apq == 0, torch.zeros_like(tt), tt)
            c = (1 / (tt * tt + 1).sqrt())[:, None]
            s = tt[:, None] * c
            for M, rows in ((A, False), (A, True), (V, False)):
                x, y = (M[:, p].clone(), M[:, q].clone()) if rows else (M[:, :, p].clone(),
                                                                        M[:, :, q].clone())
                if rows:
                    M[:, p], M[:, q] = c * x - s * y, s * x + c * y
                else:
                    M[:, :, p], M[:, :, q] = c * x - s * y, s * x + c * y
    return torch.diagonal(A, dim1=1, dim2=2), V


def _exact_layers(case, seed):
    """Centres and semi-axes of the thick hairs' cross-sections, their materials and the
    clusters' widths.  The axes' signs are free, so e1 and e2 have no value here."""
    verts, mat, _, cam, _ = _scene(case, seed)
    N, S1, C = case["n"], case["S"] + 1, case["clusters"]
    L = _levels(N, C)
    none = dict(order=None, cluster_of=None)
    if not L:
        return none
    # Morton order of the roots: 10 bits per axis in the bounding cube, FP32 as stated
    root = verts[:, 0, :3].cpu().numpy()
    lo = root.min(0)
    ext = (root.max(0) - lo).max()
    scale = np.float32(1024.0) / ext if ext > 0 else np.float32(0.0)
    q = np.clip(np.floor((root - lo) * scale), 0, 1023).astype(np.int64)
    code = np.zeros(N, np.int64)
    for bit in range(10):
        for axis in range(3):
            code |= ((q[:, axis] >> bit) & 1) << (3 * bit + 2 - axis)
    order = torch.from_numpy(np.argsort(code, kind="stable")).cuda()
    rank = torch.arange(N, device="cuda")
    cl = rank * C // N
    first = (torch.arange(C + 1, device="cuda") * N + C - 1) // C
    in_cl, size = rank - first[cl], (first[1:] - first[:-1])[cl]
    P, M = verts.double()[order], mat.double()[order]
    tang = P[:, :, :3].clone()
    tang[:, 1:-1] = P[:, 2:, :3] - P[:, :-2, :3]
    tang[:, 0], tang[:, -1] = P[:, 1, :3] - P[:, 0, :3], P[:, -1, :3] - P[:, -2, :3]
    tang = _unit(tang)
    P, r = P[..., :3], P[:, 0, 3]
    eye, right, up, fwd = (torch.tensor(cam[i:i + 3].astype(np.float64), device="cuda")
                           for i in (4, 7, 10, 13))
    out = dict(centre=[], a=[], b=[], mat=[], widths=[])
    for k in range(L):
        sub = 4 ** k
        e = cl * sub + in_cl * sub // size
        nb = C * sub

        def total(v):
            return torch.zeros((nb,) + v.shape[1:], dtype=torch.float64, device="cuda").index_add_(0, e, v)

        def most(v):
            return torch.zeros((nb,) + v.shape[1:], dtype=torch.float64, device="cuda").index_reduce_(
                0, e, v, "amax")

        cnt = total(torch.ones(N, dtype=torch.float64, device="cuda"))
        ctr = total(P) / cnt[:, None, None]
        tan = _unit(total(tang))
        off = P - ctr[e]
        cov = total(off[..., :, None] * off[..., None, :]) / cnt[:, None, None, None]
        val, vec = _jacobi(cov.reshape(-1, 3, 3))
        drop = torch.einsum("nij,ni->nj", vec, tan.reshape(-1, 3)).abs().argmax(1)
        keep = val.scatter(1, drop[:, None], -1.0).argmax(1)
        e1 = vec.gather(2, keep[:, None, None].expand(-1, 3, 1))[..., 0].reshape(nb, S1, 3)
        e1 = _unit(e1 - (e1 * tan).sum(-1, keepdim=True) * tan)
        e2 = torch.linalg.cross(tan, e1)
        u, v = (off * e1[e]).sum(-1), (off * e2[e]).sum(-1)
        a, b = most(u.abs() + r[:, None]), most(v.abs() + r[:, None])
        grow = most((u / a[e]) ** 2 + (v / b[e]) ** 2).sqrt().clamp_min(1.0)
        a, b = a * grow, b * grow
        corners = []
        for p in (ctr + a[..., None] * e1, ctr - a[..., None] * e1, ctr + b[..., None] * e2,
                  ctr - b[..., None] * e2):
            rel = p - eye
            z = rel @ fwd if cam[0] == 1 else torch.ones((), dtype=torch.float64, device="cuda")
            corners.append(torch.stack([rel @ right / z, rel @ up / z], -1) * float(cam[3]))
        w = torch.stack([(corners[i] - corners[j]).norm(dim=-1)
                         for i in range(4) for j in range(i + 1, 4)]).amax(0)
        out["widths"].append(w.reshape(C, -1).amax(1))
        out["centre"].append(ctr)
        out["a"].append(a)
        out["b"].append(b)
        out["mat"].append(total(M) / cnt[:, None])
    res = {name: torch.cat(out[name]) for name in ("centre", "a", "b", "mat")}
    res.update(widths=torch.stack(out["widths"], 1), e1=None, e2=None, lod=None, **none)
    return res
