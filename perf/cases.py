"""What a program has this library do, as timed cases: one pass of each is one call sequence through
the public binding (paper_2605_11536_gb300.tof), on the scenes of paper_2605_11536_gb300.scenes.

Kinds of a case:
  gated      one frame of a time-gated view: tof_bvh_build with the frame's transforms, then
             tof_render_gated (or its allocation-free form).  With temporal reuse, prepare() renders
             the frames that come before, and every pass renders the next one.
  transient  a capture of a few frames of a confocal scan: the view's history is forgotten, then
             each frame is built and rendered; the last histogram comes back.
  pt         plain gated path tracing, the method that ToF ReSTIR is compared with.
  batch      many small and large gated views as one tof_render_batch.
  served     several streams' next frames through the request server until all are done.

The images are seeded Monte Carlo estimates.  exact() gives their 64-bit values where a frame is a
plain sum over its path trees (no reuse: a reservoir's f(y) W is the sum of its candidates' weights;
plain path tracing is that sum by definition) in the closed box, which is small enough to trace every
ray against every triangle.  With reuse, a value depends on which samples the selections kept, and
there is no such sum.
"""
import math

import numpy as np
import torch

from paper_2605_11536_gb300 import scenes, tof

NF = 32  # frames of a moving scene's sequence; later frames start over


def listed():
    return [
        # the smallest call: one frame of a static interior, a few thousand pixels; launches and latency
        dict(name="box_64", kind="gated", scene="box", W=64, H=64, depth=3, trees=4, nb=1, radius=8, temporal=0, dL=0.05,
             flags=0, entry="gated"),
        # a first frame, or a still image without reuse: path trees alone
        dict(name="box_trees_240x160", kind="gated", scene="box", W=240, H=160, depth=4, trees=16, nb=0, radius=8, temporal=0,
             dL=0.25, flags=0, entry="gated"),
        # a fixed-memory loop (frames recorded or run under a memory pool) at its size limit
        dict(name="noalloc_128", kind="gated", scene="box", W=128, H=128, depth=3, trees=4, nb=5, radius=6, temporal=1, dL=0.25,
             flags=0, entry="noalloc"),
        # a ragged view with the real-time reuse setting (3 neighbours), long paths and a wider gate
        dict(name="dynamic_301x203", kind="gated", scene="dynamic", W=301, H=203, depth=5, trees=4, nb=3, radius=10, temporal=1,
             dL=0.077, flags=0, entry="gated"),
        # the dynamic proximity-sensor sequence at the size that the benchmark renders
        dict(name="dynamic_512", kind="gated", scene="dynamic", W=512, H=512, depth=4, trees=4, nb=5, radius=30, temporal=1,
             dL=0.03, flags=0, entry="gated"),
        # the same with the ellipsoidal connection, pairwise MIS and the cross-triangle walk
        dict(name="dynamic_512_ell", kind="gated", scene="dynamic", W=512, H=512, depth=4, trees=4, nb=5, radius=30, temporal=1,
             dL=0.03, flags=324, entry="gated"),
        # the largest view
        dict(name="dynamic_1024", kind="gated", scene="dynamic", W=1024, H=1024, depth=4, trees=4, nb=5, radius=30, temporal=1,
             dL=0.03, flags=0, entry="gated"),
        # a navigation sensor: small histograms, temporal reuse only
        dict(name="transient_64x64", kind="transient", W=64, H=64, B=64, trees=4, nb=0, frames=2, flags=0),
        # a confocal scan with full histograms and per-bin temporal and spatial reuse
        dict(name="transient_128x1024", kind="transient", W=128, H=128, B=1024, trees=8, nb=3, frames=3, flags=0),
        # the comparison method, with as many samples as fit a frame's time
        dict(name="pt_box_200x150", kind="pt", scene="box", W=200, H=150, depth=3, spp=32, dL=0.25),
        # views of many sizes over scenes of many sizes in one call
        dict(name="batch_32", kind="batch", n=32, res=512),
        # requests of several streams served together
        dict(name="served_4", kind="served", n=4, res=512),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["gated", "gated", "gated", "transient", "pt", "batch", "served"])
    if kind == "gated":
        scene = rng.choice(["box", "dynamic", "dynamic"])
        H = _log(rng, 48, 900)
        W = max(48, min(1024, int(H * rng.uniform(0.75, 1.5))))
        trees = rng.randint(2, 8)
        while W * H * trees > 4 * 1024 * 1024 // (1 if scene == "dynamic" else 2):
            trees = max(1, trees // 2)
            if trees == 1:
                break
        flags = rng.choice([0, 0, 0, 4, 324]) if W * H <= 640 * 640 else 0
        nb = rng.choice([0, 1, 3, 5])
        small = W * H <= 16384
        return dict(kind="gated", scene=scene, W=W, H=H, depth=rng.randint(2, 5), trees=trees, nb=nb, radius=rng.randint(4, 30),
                    temporal=rng.randint(0, 1), dL=round(rng.uniform(0.02, 0.2), 4), flags=flags,
                    entry=rng.choice(["gated", "noalloc"]) if small else "gated")
    if kind == "transient":
        B = rng.choice([48, 64, 200, 512, 1000, 1024])
        H = _log(rng, 32, 120)
        return dict(kind="transient", W=max(32, min(128, int(H * rng.uniform(0.75, 1.3)))), H=H, B=B, trees=rng.randint(2, 8),
                    nb=rng.choice([0, 0, 2, 3]), frames=rng.randint(1, 3), flags=0)
    if kind == "pt":
        H = _log(rng, 40, 300)
        return dict(kind="pt", scene=rng.choice(["box", "dynamic"]), W=max(40, int(H * rng.uniform(0.75, 1.4))), H=H,
                    depth=rng.randint(2, 4), spp=rng.randint(4, 32), dL=round(rng.uniform(0.05, 0.3), 4))
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(3, 31), res=_log(rng, 100, 500))
    return dict(kind="served", n=rng.randint(2, 4), res=_log(rng, 100, 500))


class _State:
    """A context with what lives in it; destroyed with the state."""

    def __init__(self, case, seed):
        self.case, self.seed, self.frame = case, int(seed), 0
        self.ctx = tof.tof_create(torch.cuda.current_device())
        self.stream = torch.cuda.current_stream().cuda_stream
        self.srv = None

    def upload(self, sc):
        return tof.tof_scene_upload(self.ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)

    def __del__(self):
        if getattr(self, "srv", None) is not None:
            tof.tof_server_destroy(self.srv)
        if getattr(self, "ctx", None) is not None:
            tof.tof_destroy(self.ctx)


def _f32(sc):
    return [np.ascontiguousarray(sc.xforms[f].reshape(-1), dtype=np.float32) for f in range(sc.n_frames)]


def _scene(case, seed):
    if case["scene"] == "box":
        sc = scenes.box_icosphere(W=case["W"], H=case["H"], seed=seed)
        gate = (5.0, case["dL"])
    else:
        sc = scenes.heightfield_spheres(W=case["W"], H=case["H"], frames=NF, seed=seed)
        gate = (8.0, case["dL"])
    p = sc.params
    p.depth, p.n_cand = case["depth"], case.get("trees", 1)
    p.n_spatial, p.radius, p.temporal = case.get("nb", 0), case.get("radius", 8), case.get("temporal", 0)
    p.flags = case.get("flags", 0)
    return sc, gate


def prepare(case, seed):
    st = _State(case, seed)
    kind = case["kind"]
    if kind in ("gated", "pt"):
        st.sc, st.gate = _scene(case, seed)
        st.xf = _f32(st.sc)
        st.sid = st.upload(st.sc)
        st.out = torch.zeros(case["H"], case["W"], device="cuda")
        if kind == "gated":
            st.vid = tof.tof_view_create(st.ctx, st.sid, case["W"], case["H"], 0)
        if case.get("temporal"):
            for _ in range(3):   # the frames before
                run(st)
        else:
            tof.tof_bvh_build(st.ctx, st.sid, st.xf[0], stream=st.stream)
    elif kind == "transient":
        B = case["B"]
        sc = scenes.confocal_nlos(W=case["W"], H=case["H"], frames=case["frames"], seed=seed, B=B)
        p = sc.params
        p.n_cand, p.n_spatial, p.flags = case["trees"], case["nb"], case["flags"]
        st.sc, st.xf, st.bins = sc, _f32(sc), (1.35, 1.024 / B, B)
        st.sid = st.upload(sc)
        st.vid = tof.tof_view_create(st.ctx, st.sid, case["W"], case["H"], B)
        st.out = torch.zeros(case["H"], case["W"], B, device="cuda")
    elif kind == "batch":
        shapes = [(50, 40, 10), (100, 100, 20), (200, 150, 40), (300, 250, 60)]   # 12k .. 198k triangles
        st.scs = [scenes.heightfield_spheres(W=64, H=64, frames=8, seed=seed + i, nx=nx, ny=ny, n_spheres=ns)
                  for i, (nx, ny, ns) in enumerate(shapes)]
        st.xf = [_f32(sc) for sc in st.scs]
        st.sids = [st.upload(sc) for sc in st.scs]
        # the sizes, gates and depths belong to the case, the scenes and random numbers to the seed
        st.inst = scenes.batch_instances(n=case["n"], seed=case["n"] + case["res"], max_res=case["res"], min_res=min(64, case["res"]))
        st.views, st.outs, st.params = [], [], []
        for it in st.inst:
            st.views.append(tof.tof_view_create(st.ctx, st.sids[it["scene"]], it["W"], it["H"], 0))
            st.outs.append(torch.zeros(it["H"], it["W"], device="cuda"))
            p = type(st.scs[0].params)(**vars(st.scs[0].params))
            p.depth = it["depth"]
            st.params.append(p)
        for _ in range(2):   # the frames before
            run(st)
    else:
        sizes = [case["res"], case["res"] // 2, case["res"] * 7 // 10, case["res"]][:case["n"]]
        st.scs = [scenes.heightfield_spheres(W=r, H=r, frames=NF, seed=seed + 10 * k) for k, r in enumerate(sizes)]
        st.xf = [_f32(sc) for sc in st.scs]
        st.sids = [st.upload(sc) for sc in st.scs]
        for sid, xf in zip(st.sids, st.xf):
            tof.tof_bvh_build(st.ctx, sid, xf[0], stream=st.stream)
        st.outs = [torch.zeros(r, r, device="cuda") for r in sizes]
        st.srv = tof.tof_server_create(st.ctx, 120 << 30)
        st.streams = [tof.tof_server_open_stream(st.srv, st.sids[k], r, r, 0) for k, r in enumerate(sizes)]
        for _ in range(2):   # the streams are admitted, and have history
            run(st)
    return st


def run(st):
    case, f = st.case, st.frame
    kind = case["kind"]
    if kind == "gated":
        sc, k = st.sc, f % st.sc.n_frames
        call = tof.tof_render_gated_noalloc if case["entry"] == "noalloc" else tof.tof_render_gated
        tof.tof_bvh_build(st.ctx, st.sid, st.xf[k], stream=st.stream)
        call(st.ctx, st.sid, st.vid, sc.sensors[k], sc.emitters[k], st.gate, sc.params, st.seed, f, st.out.data_ptr(), st.stream)
        st.frame += 1
        return st.out
    if kind == "transient":
        sc = st.sc
        tof.tof_reservoirs_reset(st.ctx, st.vid)
        for k in range(case["frames"]):
            tof.tof_bvh_build(st.ctx, st.sid, st.xf[k], stream=st.stream)
            tof.tof_render_transient(st.ctx, st.sid, st.vid, sc.sensors[k], sc.emitters[k], st.bins, sc.params, st.seed, f + k,
                                     st.out.data_ptr(), st.stream)
        st.frame += case["frames"]
        return st.out
    if kind == "pt":
        sc = st.sc
        tof.tof_render_pt(st.ctx, st.sid, sc.sensors[0], sc.emitters[0], st.gate, None, sc.params, st.seed, f, case["spp"],
                          st.out.data_ptr(), st.stream)
        st.frame += 1
        return st.out
    if kind == "batch":
        for s, sc in enumerate(st.scs):
            tof.tof_bvh_build(st.ctx, st.sids[s], st.xf[s][f % sc.n_frames], stream=st.stream)
        jobs = []
        for i, it in enumerate(st.inst):
            sc = st.scs[it["scene"]]
            k = f % sc.n_frames
            jobs.append(tof.job(st.sids[it["scene"]], st.views[i], dict(sc.sensors[k], W=it["W"], H=it["H"]), sc.emitters[k],
                                st.params[i], st.seed + i, f, st.outs[i].data_ptr(), gate=(sc.gates[k][0], it["dL"])))
        tof.tof_render_batch(st.ctx, jobs, st.stream)
        st.frame += 1
        return st.outs
    tickets = []
    for k, sc in enumerate(st.scs):
        j = f % sc.n_frames
        job = tof.job(st.sids[k], 0, sc.sensors[j], sc.emitters[j], sc.params, st.seed + k, f, st.outs[k].data_ptr(), gate=sc.gates[j])
        tickets.append(tof.tof_server_submit(st.srv, st.streams[k], job, st.xf[k][j]))
    while tickets:   # a server's loop: launch what can be launched, take what is done
        tof.tof_server_step(st.srv, st.stream)
        tickets = [t for t in tickets if tof.tof_server_poll(st.srv, t)[0] != 2]
    st.frame += 1
    return st.outs


def work(case):
    """Bytes: the triangles (three corners each) that a frame's hierarchy is built from, a view's
    reservoirs (104 B) and primary hits (16 B) read where a frame has a predecessor and written, and
    the image or histogram.  Operations: per ray one root-to-leaf walk (two boxes a level, 24 operations)
    and one triangle (40); per shift 600."""
    def gated(px, nt, depth, trees, nb, temporal):
        slots = (1 + nb) * (1 if nb else 0)
        shifts = px * 0.5 * (2 * temporal + nb + nb * nb)
        rays = px * (1 + trees * (depth - 1)) + 2 * shifts * 0.5
        return (36 * nt + px * (120 + 4 + (120 if temporal or slots else 0)), rays * (24 * math.log2(nt) + 40) + 600 * shifts)

    kind = case["kind"]
    if kind in ("gated", "pt"):
        px, nt = case["W"] * case["H"], 332 if case["scene"] == "box" else 66000
        if kind == "pt":
            return {"bytes": 36 * nt + 4 * px, "flops": px * case["spp"] * case["depth"] * (24 * math.log2(nt) + 40)}
        b, f = gated(px, nt, case["depth"], case["trees"], case["nb"], case["temporal"])
    elif kind == "transient":
        px, nt = case["W"] * case["H"], 100000
        b, f = 0.0, 0.0
        for k in range(case["frames"]):
            bb, ff = gated(px, nt, 4, case["trees"], 0, 0)
            # per pixel at most one occupied bin per candidate and frame, and a reservoir in each
            bins = min(case["B"], 3 * case["trees"] * (k + 1) * (1 + case["nb"]))
            shifts = 0.25 * px * bins * (2 * (k > 0) + case["nb"] + case["nb"] ** 2)
            b += bb + px * (96 * bins + case["B"] / 8) + (4 * px * case["B"] if k + 1 == case["frames"] else 0)
            f += ff + shifts * (600 + 24 * math.log2(nt) + 40)
    elif kind == "batch":
        nts = [12000, 36000, 92000, 198000]
        b, f = 36.0 * sum(nts), 0.0
        for it in scenes.batch_instances(n=case["n"], seed=case["n"] + case["res"], max_res=case["res"], min_res=min(64, case["res"])):
            bb, ff = gated(it["W"] * it["H"], nts[it["scene"]], it["depth"], 4, 5, 1)
            b, f = b + bb - 36 * nts[it["scene"]], f + ff
    else:
        b, f = 0.0, 0.0
        for r in [case["res"], case["res"] // 2, case["res"] * 7 // 10, case["res"]][:case["n"]]:
            bb, ff = gated(r * r, 66000, 4, 4, 5, 1)
            b, f = b + bb, f + ff
    return {"bytes": float(b), "flops": float(f)}


# ---- 64-bit values: path trees in the closed box, every ray against every triangle ---------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    M = 0xFFFFFFFF

    def mul(a, b):
        p1, p2 = (a & 0xFFFF) * b, (a >> 16) * b
        return (p2 + (p1 >> 16)) >> 16, (p1 + ((p2 & 0xFFFF) << 16)) & M
    k0, k1 = seed & M, (seed >> 32) & M
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    return [(c >> 8).double() / 16777216.0 for c in (c0, c1)]


def exact(case, seed):
    if case.get("scene") != "box" or not (case["kind"] == "pt" or (case["kind"] == "gated" and not case["nb"] and not case["temporal"]
                                                                   and not case["flags"])):
        return None
    sc, gate = _scene(case, seed)
    W, H, depth = case["W"], case["H"], case["depth"]
    pt = case["kind"] == "pt"
    n = case["spp"] if pt else case["trees"]
    dev, d64 = "cuda", torch.float64
    if W * H * n * depth > 6_000_000:   # over the time that a value may take
        return None
    f32 = lambda x: torch.tensor(np.asarray(x, dtype=np.float32).astype(np.float64), device=dev)   # the call takes 32-bit values
    V = f32(sc.verts)[torch.tensor(sc.tris.astype(np.int64), device=dev)]
    v0, e1, e2 = V[:, 0], V[:, 1] - V[:, 0], V[:, 2] - V[:, 0]
    nrm = torch.linalg.cross(e1, e2)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    alb = f32(sc.materials[sc.object_material[sc.tri_object].astype(np.int64), 1])
    sensor, em = sc.sensors[0], sc.emitters[0]
    eye, lamp, power = f32(sensor["pos"]), f32(em["pos"]), float(np.float32(em["power"]))
    L0, dL, eps = float(np.float32(gate[0])), float(np.float32(gate[1])), float(np.float32(sc.params.ray_eps))
    dot = lambda a, b: (a * b).sum(-1)
    unit = lambda a: a / a.norm(dim=-1, keepdim=True)

    def hits(o, d, tmax):
        """Nearest triangle along each ray within tmax, or -1, and its distance."""
        if not len(o):
            return torch.zeros(0, dtype=torch.int64, device=dev), torch.zeros(0, dtype=d64, device=dev)
        tri, tt = [], []
        for a in range(0, len(o), 8192):
            oo, dd = o[a:a + 8192, None], d[a:a + 8192, None]
            pv = torch.linalg.cross(dd.expand(-1, len(v0), -1), e2[None].expand(len(dd), -1, -1))
            det = dot(e1[None], pv)
            inv = 1.0 / torch.where(det.abs() < 1e-20, torch.ones_like(det), det)
            tv = oo - v0[None]
            u = dot(tv, pv) * inv
            qv = torch.linalg.cross(tv, e1[None].expand_as(tv))
            w, t = dot(dd, qv) * inv, dot(e2[None], qv) * inv
            ok = (det.abs() >= 1e-20) & (u >= -1e-6) & (u <= 1 + 1e-6) & (w >= -1e-6) & (u + w <= 1 + 1e-6) & (t > 0) & (t < tmax[a:a + 8192, None])
            t, k = torch.where(ok, t, torch.full_like(t, math.inf)).min(1)
            tri.append(torch.where(t < math.inf, k, torch.full_like(k, -1)))
            tt.append(t)
        return torch.cat(tri), torch.cat(tt)

    def off(p, m, d):
        return p + m * torch.where(dot(m, d) >= 0, eps, -eps)[:, None]

    pix = torch.arange(W * H, device=dev).repeat_interleave(n)
    tree = torch.arange(n, device=dev).repeat(W * H)
    zero = torch.zeros_like(pix)
    u0, u1 = _philox(pix, zero, tree if pt else zero, zero + 1, seed)
    fwd = unit(f32(sensor["fwd"]))
    right = unit(torch.linalg.cross(fwd, f32(sensor["up"])))
    up = torch.linalg.cross(right, fwd)
    th = math.tan(0.5 * float(np.float32(sensor["fov_y"])))
    sx = (2 * ((pix % W) + u0) / W - 1) * th * W / H
    sy = (1 - 2 * ((pix // W) + u1) / H) * th
    d = unit(fwd + right * sx[:, None] + up * sy[:, None])
    tri, t = hits(eye.expand_as(d), d, torch.full_like(u0, math.inf))
    live = tri >= 0
    img = torch.zeros(W * H, dtype=d64, device=dev)
    pix, tree, d, tri, t = pix[live], tree[live], d[live], tri[live], t[live]
    p, wi, length = eye + d * t[:, None], -d, t
    beta = torch.ones_like(length)
    for k in range(1, depth + 1):
        m = nrm[tri]
        if k >= 2:
            wl = lamp - p
            dist = wl.norm(dim=1)
            wl = wl / dist[:, None]
            tau = length + dist
            c = beta * alb[tri] / math.pi * power * dot(m, wl).abs() / dist ** 2
            ok = (dot(m, wi) * dot(m, wl) > 0) & (tau >= L0) & (tau < L0 + dL)
            o = off(p, m, wl)[ok]
            s = lamp - o
            far = s.norm(dim=1)
            ok = ok.clone()
            ok[ok.nonzero()[:, 0]] = hits(o, s / far[:, None], far)[0] < 0
            img.index_add_(0, pix[ok], c[ok] / n)
        if k == depth:
            break
        u0, u1 = _philox(pix, torch.zeros_like(pix), (tree << 8) | k, torch.zeros_like(pix) + 2, seed)
        m = torch.where((dot(m, wi) < 0)[:, None], -m, m)
        a1 = torch.tensor([0.4140355211239282, 0.731736150464251, 0.5414210869105452], dtype=d64, device=dev)
        a2 = torch.tensor([0.0, 0.5947978113475719, -0.8038753408434284], dtype=d64, device=dev)
        ax = torch.where((dot(m, a1).abs() < 0.6)[:, None], a1, a2)
        tx = unit(torch.linalg.cross(ax, m))
        ty = torch.linalg.cross(m, tx)
        r, ph = u0.sqrt(), 2 * math.pi * u1
        wo = tx * (r * ph.cos())[:, None] + ty * (r * ph.sin())[:, None] + m * (1 - u0).clamp(min=0).sqrt()[:, None]
        nt, t = hits(off(p, nrm[tri], wo), wo, torch.full_like(u0, math.inf))
        live = (nt >= 0) & (dot(m, wo) > 0)
        q = off(p, nrm[tri], wo) + wo * t[:, None]
        beta = beta * alb[tri]
        length = length + (q - p).norm(dim=1)
        pix, tree, wi, p, beta, length, tri = pix[live], tree[live], -wo[live], q[live], beta[live], length[live], nt[live]
    return img.reshape(H, W)
