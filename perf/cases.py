"""What a user of the renderer has it do, as timed cases.

A scene is a box room of the kinds that ``ltinputs`` describes (made here on the GPU
from the seed, because the host ray caster takes seconds on the larger rooms); the
parameters are those of the workload presets.  Every case goes through
``Renderer`` and the ``lt`` binding, as a program does.  The kinds:

* ``frame``      one whole frame: pass 1, pass 2, evaluation, completion, image, by
                 the one-call form or as a replayed graph, with or without the learned
                 pass-2 pdf;
* ``sample``     the sampling half of a frame (pass 1 with coarsening, pass 2, entry
                 evaluation), what an occluded scene spends most on;
* ``evaluate``   the evaluation of a frame's pass-2 entries (shadow rays);
* ``complete``   masked ALS completion of a frame's samples and the image from it;
* ``adm``        the nonnegative completion of the same samples;
* ``colour``     the three channels of every sample, the stacked completion, the image;
* ``setup``      a new scene or camera: tree, global cut, forest, slices, point order;
* ``targets``    training data of the proposal: features, full slice matrices,
                 leverage targets;
* ``train``      one training step of the proposal: loss, gradient, Adam;
* ``brute``      the image over all VPLs (the reference images of a study).

The buffers of samples and factors are a program's own; here they are laid out once
per case for the largest cut and slice count that its parameters allow.
"""
import math

import numpy as np
import torch

from ltinputs import Scene, get_config
from ltinputs import scenes
from paper_2202_12567_gb300 import lt, proposal
from paper_2202_12567_gb300.renderer import Renderer

_ROOM = dict(kind="frame", width=256, height=256, vpls=16384, big=2, small=0, meshes=0, glossy=0.0, slices=64,
             lo=0, hi=0, rate=0.18, rate1=0.002, rank=16, cols=0, sweeps=10, cut=8192, tau=5e-4, d_min=0.1,
             graph=False, learned=False)


def _case(name=None, **kw):
    c = dict(_ROOM, **kw)
    if name:
        c["name"] = name
    return c


_OCCLUDED = dict(big=0, small=200, rate=0.10, rate1=0.015, cut=4096)


def listed():
    return [
        # the smallest frame (preview size), by the plain one-call form: launches and read-backs count
        _case("frame_64", width=64, height=64, vpls=1024, slices=16, rate=0.10, rate1=0.03, rank=8, cut=1024, tau=0.02,
              d_min=0.01),
        # the headline: a scene's frame replayed as a graph with the learned pdf, another seed each frame
        _case("frame_256_learned", graph=True, learned=True),
        # a large, occluded, partly glossy scene with uneven slices: where sampling dominates
        _case("sample_512_glossy", kind="sample", width=512, height=512, vpls=65536, big=0, small=1000, glossy=0.3,
              slices=128, lo=128, hi=4096, rate=0.10, rate1=0.015, cut=4096),
        # shadow rays against triangle meshes
        _case("evaluate_256_mesh", kind="evaluate", meshes=6, rate=0.15),
        # the completion at the usual rank, and with per-slice ranks up to the largest
        _case("complete_256", kind="complete"),
        _case("complete_256_rank32", kind="complete", **dict(_OCCLUDED, rank=32, cols=512)),
        # the paper's own nonnegative completion
        _case("adm_256", kind="adm", rate=0.15, sweeps=100),
        # a coloured frame from its samples on: three times the rows of the scalar completion
        _case("colour_256", kind="colour", rate=0.15),
        # a moved camera or a new scene: everything that comes before its first frame
        _case("setup_256", kind="setup"),
        # training of the learned pdf: one scene's data, one step
        _case("targets_256", kind="targets"),
        _case("train_256", kind="train"),
        # a reference image
        _case("brute_256", kind="brute"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["frame", "frame", "sample", "evaluate", "complete", "complete", "adm", "colour", "setup",
                       "targets", "train", "brute"])
    big = kind in ("frame", "sample", "setup")
    side = int(_log(rng, 48, 400 if big else 256))
    width, height = side, max(40, int(side * rng.uniform(0.6, 1.0)))  # odd and even, not square
    vpls = int(_log(rng, 700, 40000 if big else 16384))
    boxes = rng.choice(["two", "two", "few", "many"])
    c = dict(_ROOM, kind=kind, width=width, height=height, vpls=vpls)
    if boxes != "two":
        c.update(big=rng.choice([0, 1, 3]), small=int(_log(rng, 5, 60 if boxes == "few" else 500)))
    if rng.random() < 0.3 and kind != "colour":
        c["glossy"] = round(rng.uniform(0.1, 0.5), 2)
    if rng.random() < 0.2 and kind in ("frame", "sample", "evaluate"):
        c["meshes"] = rng.randint(1, 6)
    c["slices"] = max(4, int(width * height / _log(rng, 250, 2500)))
    if rng.random() < 0.25:
        c.update(lo=128, hi=4096)
    c.update(rate=round(rng.uniform(0.05, 0.25), 3), rate1=rng.choice([0.002, 0.015, 0.03]),
             cut=rng.choice([1024, 4096, 8192, 16384]), tau=rng.choice([5e-4, 2e-3, 0.02]))
    c["rank"] = rng.choice([5, 8, 10, 12, 16, 16, 16, 24, 32])
    if c["rank"] > 16 and rng.random() < 0.5:
        c["cols"] = 512
    if kind == "adm":
        c.update(sweeps=rng.randint(20, 100), cols=0)
    if kind == "targets":
        c["rank"] = min(c["rank"], 16)
    if kind == "frame":
        c["graph"] = rng.random() < 0.5
        c["learned"] = c["graph"] and rng.random() < 0.5
    return c


# ------------------------------------------------------------------ scenes
def _config(case, seed):
    over = dict(width=case["width"], height=case["height"], n_vpl=case["vpls"], n_big_boxes=case["big"],
                n_small_boxes=case["small"], glossy_frac=case["glossy"], n_meshes=case["meshes"], mesh_subdiv=3,
                n_slices=case["slices"], rate=case["rate"], rate1=case["rate1"], rank=case["rank"],
                rank_cols=case["cols"], als_iters=case["sweeps"], adm_iters=case["sweeps"], max_cut=case["cut"],
                tau=case["tau"], d_min=case["d_min"], scene_seed=seed, frame_seed=_frame_seed(seed),
                completion="adm" if case["kind"] == "adm" else "als", rgb=case["kind"] == "colour")
    if case["lo"]:
        over["slice_bounds"] = (case["lo"], case["hi"])
    return get_config("room256_vpl16k_2box", **over)


def _frame_seed(seed):
    return 7 + int(seed) % 1000003


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _cast(org, d, boxes, tris, spheres):
    """Nearest hit (float64, on the GPU) in the room: (t, face, normal); faces as in ltinputs.scenes."""
    inv = 1.0 / d
    far = torch.where(d > 0, (1.0 - org) * inv, torch.where(d < 0, -org * inv, math.inf))
    t, ax = far.min(1)
    pos = d.gather(1, ax[:, None])[:, 0] > 0
    face = torch.where(ax == 1, pos.long(), torch.where(ax == 0, 3 - (~pos).long(), torch.where(pos, 4, -1)))
    walls = torch.tensor([[0, 1, 0], [0, -1, 0], [1, 0, 0], [-1, 0, 0], [0, 0, -1], [0, 0, 0]], dtype=org.dtype,
                         device=org.device)
    nrm = walls[face]
    nb = boxes.shape[0]
    for s in range(0, org.shape[0], 32768) if nb else ():
        o, iv = org[s:s + 32768, None], inv[s:s + 32768, None]
        ta, tb = (boxes[None, :, :3] - o) * iv, (boxes[None, :, 3:] - o) * iv
        near, nax = torch.minimum(ta, tb).nan_to_num(-math.inf).max(2)
        ok = (near <= torch.maximum(ta, tb).nan_to_num(math.inf).amin(2)) & (near > 1e-7)
        tn, b = torch.where(ok, near, math.inf).min(1)
        a = nax.gather(1, b[:, None])[:, 0]
        neg = d[s:s + 32768].gather(1, a[:, None])[:, 0] <= 0
        c = (tn < t[s:s + 32768]).nonzero()[:, 0]
        t[s + c] = tn[c]
        face[s + c] = 5 + 6 * b[c] + 2 * a[c] + neg[c].long()
        n = torch.zeros(c.numel(), 3, dtype=org.dtype, device=org.device)
        n.scatter_(1, a[c, None], (2.0 * neg[c].double() - 1.0)[:, None])
        nrm[s + c] = n
    per = tris.shape[0] // len(spheres) if tris is not None else 0
    for k, (centre, r) in enumerate(spheres if tris is not None else ()):
        oc = org - torch.as_tensor(centre, device=org.device)
        b = (oc * d).sum(1)
        ids = (b * b - (d * d).sum(1) * ((oc * oc).sum(1) - (1.001 * r) ** 2) >= 0).nonzero()[:, 0]
        T = tris[k * per:(k + 1) * per]
        for s in range(0, ids.numel(), 16384):
            i = ids[s:s + 16384]
            tt = _triangles(org[i], d[i], T)
            tt, j = torch.where(tt > 1e-7, tt, math.inf).min(1)
            c = (tt < t[i]).nonzero()[:, 0]
            t[i[c]] = tt[c]
            face[i[c]] = 5 + 6 * nb + k
            v = T[j[c]]
            n = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
            n = n / n.norm(dim=1, keepdim=True)
            nrm[i[c]] = torch.where((n * d[i[c]]).sum(1, keepdim=True) > 0, -n, n)
    return t, face, nrm


def _triangles(org, d, T):
    """t of every (ray, triangle) pair, NaN where the closed triangle is not met."""
    v0, e1, e2 = T[None, :, 0], (T[:, 1] - T[:, 0])[None], (T[:, 2] - T[:, 0])[None]
    o, D = org[:, None], d[:, None]
    p = torch.linalg.cross(D, e2)
    det = (e1 * p).sum(2)
    sv = o - v0
    q = torch.linalg.cross(sv, e1.expand_as(sv))
    u, v, t = (sv * p).sum(2) / det, (D * q).sum(2) / det, (e2 * q).sum(2) / det
    return torch.where((det != 0) & (u >= 0) & (u <= 1) & (v >= 0) & (u + v <= 1), t, math.nan)


def _scene(cfg, seed):
    rng, dev = np.random.default_rng(seed), _dev()
    boxes = scenes._make_boxes(cfg, rng)
    nb = boxes.shape[0]
    tris, spheres = scenes._make_meshes(cfg, np.random.default_rng(seed + 104729), boxes)
    faces = 5 + 6 * nb + len(spheres)
    albedo, gloss = scenes._materials(faces, cfg["glossy_frac"], rng)
    rgb = None
    if cfg["rgb"]:
        face_rgb = rng.uniform(0.2, 0.8, size=(faces, 3))
        albedo = face_rgb @ scenes.LUMINANCE
    bx = torch.from_numpy(boxes).to(dev).double()
    tr = None if tris is None else torch.from_numpy(tris).to(dev).double()
    org, d = (torch.from_numpy(x).to(dev) for x in scenes._camera_rays(cfg["width"], cfg["height"]))
    t, face, nrm = _cast(org, d, bx, tr, spheres)
    al, gl = torch.from_numpy(albedo).to(dev), torch.from_numpy(gloss).to(dev)

    def planes(pos, face, nrm, third, w):
        p = torch.zeros(3, pos.shape[0], 4, device=dev)
        p[0, :, :3], p[0, :, 3], p[1, :, :3], p[1, :, 3], p[2, :, :3], p[2, :, 3] = pos, al[face], nrm, gl[face], third, w
        return p.cpu().numpy()

    points = planes(org + t[:, None] * d, face, nrm, -d, 0.0)
    # one cosine-weighted bounce from the ceiling light; rays that leave through the front deposit nothing
    n = cfg["n_vpl"]
    r = torch.from_numpy(rng.uniform(size=(2 * n + 1024, 4))).to(dev)
    lo = torch.stack([0.4 + 0.2 * r[:, 0], torch.ones_like(r[:, 0]), 0.4 + 0.2 * r[:, 1]], 1)
    phi, sin = 2 * math.pi * r[:, 2], r[:, 3].sqrt()
    dd = torch.stack([sin * phi.cos(), -(1 - r[:, 3]).sqrt(), sin * phi.sin()], 1)
    vt, vf, vn = _cast(lo, dd, bx, tr, spheres)
    k = (vf >= 0).nonzero()[:n, 0]
    flux = 1.0 / float(k[-1] + 1)
    light = np.asarray(cfg["light_rgb"]) if cfg["rgb"] else None
    scalar = flux if light is None else flux * float(light @ scenes.LUMINANCE)
    vpls = planes(lo[k] + vt[k, None] * dd[k], vf[k], vn[k], -dd[k], scalar)
    if light is not None:
        rgb = dict(point_albedo=face_rgb[face.cpu().numpy()].astype(np.float32),
                   vpl_albedo=face_rgb[vf[k].cpu().numpy()].astype(np.float32),
                   vpl_flux=np.broadcast_to(flux * light, (n, 3)).astype(np.float32))
    return Scene(cfg=cfg, boxes=boxes, points=points, vpls=vpls, width=cfg["width"], height=cfg["height"],
                 n_emitted=int(k[-1]) + 1, rgb=rgb, tris=tris)


# ------------------------------------------------------------------ buffers
def _most(case):
    """Largest slice count and cut."""
    m = case["width"] * case["height"]
    return case["slices"] + (m // 2048 + 2 if case["lo"] else 0), min(case["cut"], case["vpls"])


def _samples_size(case):
    S, C = _most(case)
    m = case["width"] * case["height"]
    return int(S * (9.1 * C + 128) + (2.1 * case["rate1"] + case["rate"]) * m * C)


def _lay_out(st):
    """The frame's samples and factors in the case's buffers."""
    R, case = st["R"], st["case"]
    (S, C), n, r = _most(case), _samples_size(case), case["rank"]
    i32, f32 = dict(dtype=torch.int32, device=R.dev), dict(dtype=torch.float32, device=R.dev)
    buf = dict(ncol=torch.zeros(S, **i32), col_node=torch.zeros(S * C, **i32), g=torch.zeros(S * C, **f32),
               n1=torch.zeros(S, **i32), cnt=torch.zeros(S, **i32), key=torch.zeros(n, **i32),
               val=torch.zeros(n, **f32), V=torch.zeros(S * C * r, **f32))
    s, uv = R.smp, R.uv
    for k in ("ncol", "col_node", "g", "n1", "cnt", "key", "val"):
        setattr(s, k, buf[k][:getattr(s, k).numel()])
    uv.V = buf["V"][:uv.V.numel()]
    s._s = lt.lt_samples(*(t.data_ptr() for t in (s.ncol, s.col_node, s.g, s.off, s.key, s.val, s.n1, s.cnt)))
    uv._s = lt.lt_factors(r, uv.U.data_ptr(), uv.V.data_ptr(), None if uv.rank is None else uv.rank.data_ptr())
    st["buf"] = buf


def _lay_out_colour(st):
    G, b = st["R"].rgb, st["buf"]
    full = dict(key=torch.zeros(3 * b["key"].numel(), dtype=torch.int32, device=G.key.device),
                val=torch.zeros(3 * b["val"].numel(), device=G.key.device), V=torch.zeros_like(b["V"]))
    for k, t in full.items():
        setattr(G, k, t[:getattr(G, k).numel()])
    s = G._smp3
    G._smp3 = lt.lt_samples(s.ncol, s.col_node, s.g, s.off, G.key.data_ptr(), G.val.data_ptr(), s.n1, s.cnt)
    G._uv3 = lt.lt_factors(G.r, G.U.data_ptr(), G.V.data_ptr(), None if G.rank is None else G.rank.data_ptr())
    st["buf3"] = full


# ------------------------------------------------------------------ the cases
def prepare(case, seed):
    kind = case["kind"]
    cfg = _config(case, seed)
    if kind == "colour":
        cfg["light_rgb"] = (1.0, 0.85, 0.7)
    R = Renderer(_scene(cfg, seed), cfg, device=torch.cuda.current_device())
    st = dict(case=case, R=R, seed=cfg["frame_seed"])
    if kind == "brute":
        return st
    S, C = _most(case)
    if kind == "setup":
        st.update(cut=torch.zeros(C, dtype=torch.int32, device=R.dev),
                  forest=torch.zeros((2 * C - 1) * 8, dtype=torch.int32, device=R.dev),
                  nodes=torch.zeros(max(C - 1, 1), dtype=torch.int32, device=R.dev))
        return st
    R.setup()
    _lay_out(st)
    if kind == "colour":
        R.setup_rgb()
        _lay_out_colour(st)
    if kind == "frame" and case["graph"]:
        theta = proposal.load_theta(device=R.dev.index) if case["learned"] else None
        st["theta"] = theta
        st["graph"] = lt.lt_frame_graph_capture(R.ctx, R.frame, lt.params(cfg, proposal=theta, mix=0.8), R.smp, R.uv,
                                                R.row_perm, R.img, keep=(theta,))
    if kind in ("evaluate", "complete", "adm", "colour", "targets", "train"):
        R.pass1(st["seed"])
    if kind in ("evaluate", "complete", "adm", "colour"):
        R.pass2(st["seed"])
    if kind in ("complete", "adm", "colour"):
        R.evaluate()
    if kind in ("targets", "train"):
        ncol = R.smp.ncol.cpu().numpy().astype(np.int64)
        st["cap"] = max(int(np.sum(R.frame.sizes * ncol)),
                        R.frame.m * min(C, max(1024, int(10 * math.sqrt(case["vpls"])))))
        st["n"] = int(ncol.sum())
        st["feat"] = torch.zeros(S * C, lt.MLP_FEATURES, device=R.dev)
        st["goff"] = torch.zeros(S + 1, dtype=torch.int32, device=R.dev)
        st["target"] = torch.zeros(S * C, device=R.dev)
    if kind == "train":
        feat, goff, M, target = _targets(st)
        st.update(feat=feat[:st["n"]].clone(), target=target[:st["n"]].clone(), step=0)
        st["theta"] = lt.lt_proposal_init(R.ctx, 1 + int(seed) % 97)
        st["m"], st["v"] = torch.zeros_like(st["theta"]), torch.zeros_like(st["theta"])
    lt.lt_sync(R.ctx)
    return st


def _targets(st):
    R = st["R"]
    feat, goff = lt.lt_proposal_features(R.ctx, R.frame, R.smp, st["feat"], st["goff"])
    M, moff = lt.lt_slice_matrices(R.ctx, R.frame, R.smp, R.cfg["d_min"], st["cap"])
    target = lt.lt_leverage_targets(R.ctx, R.frame, R.smp, M, moff, goff, R.cfg["rank"], proposal.TARGET_ITERS,
                                    st["seed"], st["target"])
    return feat, goff, M, target


def run(st):
    R, kind, seed = st["R"], st["case"]["kind"], st["seed"]
    if kind == "frame":
        if "graph" in st:
            lt.lt_frame_graph_launch(st["graph"], seed)
        else:
            R.render_frame(seed, sync=False)
        return dict(img=R.img, **_samples(st))
    if kind == "sample":
        R.pass1(seed)
        R.pass2(seed)
        R.evaluate()
        return _samples(st)
    if kind == "evaluate":
        R.evaluate()
        return dict(val=st["buf"]["val"])
    if kind in ("complete", "adm"):
        R.complete(seed)
        R.render_image()
        return dict(img=R.img, U=R.uv.U, V=st["buf"]["V"])
    if kind == "colour":
        c, G = R.cfg, R.rgb
        lt.lt_expand_rgb(R.ctx, R.frame, R.smp, G)
        if G.rank is not None:
            lt.lt_slice_ranks(R.ctx, R.frame, R.smp, c["rank"], c["rank_cols"], G.rank)
        lt.lt_complete_rgb(R.ctx, G, c["als_iters"], c["lam_rel"], seed)
        lt.lt_render_rgb(R.ctx, G)
        return dict(img=G.img, U=G.U, **st["buf3"])
    if kind == "setup":
        R.setup()
        t = R.tree
        for k, v in (("cut", R.cut), ("forest", R.frame.forest), ("nodes", R.frame.level_nodes)):
            st[k][:v.numel()].copy_(v)
        return dict(order=t.order, child=t.child, parent=t.parent, range=t.range, rep=t.rep, I=t.I, B=t.B, aabb=t.aabb,
                    cut=st["cut"], forest=st["forest"], nodes=st["nodes"], perm=R.row_perm, off=R.slice_off,
                    points=R.pts_s)
    if kind == "targets":
        feat, goff, M, target = _targets(st)
        return dict(feat=feat, goff=goff, M=M, target=target)
    if kind == "train":
        st["step"] += 1
        grad, loss = lt.lt_proposal_grad(R.ctx, st["theta"], st["feat"], st["target"], st["goff"], R.frame.S, st["n"])
        lt.lt_proposal_adam(R.ctx, st["theta"], st["m"], st["v"], grad, st["step"], 3e-3)
        return dict(loss=loss, grad=grad, theta=st["theta"], m=st["m"], v=st["v"])
    return dict(img=R.bruteforce())


def _samples(st):
    return {k: st["buf"][k] for k in ("ncol", "col_node", "g", "n1", "cnt", "key", "val")}


def work(case):
    """Inputs and outputs once; columns per slice as the usual tau leaves them (about 5 sqrt(VPLs))."""
    m, n, r, kind = case["width"] * case["height"], case["vpls"], case["rank"], case["kind"]
    cols = min(5 * math.sqrt(n), case["cut"])
    entries = case["rate"] * m * cols
    ray = 40 + 40 + 6 * 8 + 24 * min(10, case["big"] + case["small"] + 1) + (24 * 24 if case["meshes"] else 0)
    ends = 48 * (m + n)
    lines = m + case["slices"] * cols
    solve = 2 * case["sweeps"] * (entries * r * (r + 3) + lines * r ** 3 / 6)
    if kind == "brute":
        return dict(bytes=ends + 4 * m, flops=float(m) * n * ray)
    if kind == "setup":
        return dict(bytes=ends + 48 * m + 2 * n * 72, flops=(m / 64) * cols * 100 + 10 * m * case["slices"] * 18)
    if kind == "sample":
        return dict(bytes=ends + 8 * entries, flops=entries * ray)
    if kind == "evaluate":
        return dict(bytes=ends + 8 * entries, flops=entries * ray)
    if kind == "complete":
        return dict(bytes=8 * entries + 4 * r * lines + 4 * m, flops=solve)
    if kind == "adm":
        return dict(bytes=8 * entries + 4 * r * lines + 4 * m,
                    flops=case["sweeps"] * (entries * 6 * r + lines * 4 * r * r))
    if kind == "colour":
        return dict(bytes=8 * entries + 24 * entries + 4 * r * (3 * m + case["slices"] * cols) + 12 * m,
                    flops=2 * case["sweeps"] * (3 * entries * r * (r + 3) / 2 + 3 * entries * r * (r + 3) / 2))
    if kind == "targets":
        dense = m * cols
        return dict(bytes=ends + 4 * dense + case["slices"] * cols * 132,
                    flops=dense * ray + dense * cols + case["slices"] * 30 * (2 * cols * cols * r + 2 * cols * r * r))
    if kind == "train":
        rows = case["slices"] * cols
        return dict(bytes=rows * 136 + 7 * 4 * 10497, flops=rows * 6 * 10304.0)
    return dict(bytes=ends + 8 * entries + 4 * m, flops=entries * ray + solve)


# ------------------------------------------------------------------ the same in 64 bits
def _philox(c0, c1, c2, c3, seed):
    """First word of Philox4x32-10 (numpy uint64 lanes)."""
    u, mask = np.uint64, np.uint64(0xFFFFFFFF)
    x = [np.asarray(v, dtype=u) for v in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1 = u(seed & 0xFFFFFFFF), u(seed >> 32)
    for _ in range(10):
        p0, p1 = u(0xD2511F53) * x[0], u(0xCD9E8D57) * x[2]
        x = [(p1 >> u(32)) ^ x[1] ^ k0, p1 & mask, (p0 >> u(32)) ^ x[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + u(0x9E3779B9)) & mask, (k1 + u(0xBB67AE85)) & mask
    return x[0].astype(np.float64)


def _start(s, count, r, tag, mu, seed):
    w = _philox(np.arange(r)[None, :], np.arange(count)[:, None], s, tag, seed)
    return torch.from_numpy(math.sqrt(max(mu, 0.0) / r) * (0.5 + w * 2.0 ** -32)).to(_dev())


def _brdf(alb, gloss, n, wi, wo):
    ni, no, io = (n * wi).sum(-1), (n * wo).sum(-1), (wi * wo).sum(-1)
    cm1 = 2 * ni * no - io - 1
    lobe = torch.where(cm1 > -1, torch.exp(gloss * torch.log1p(cm1.clamp(min=-1 + 1e-15))), torch.zeros_like(cm1))
    g = 0.5 * alb / math.pi + 0.5 * alb * (gloss + 2) / (2 * math.pi) * lobe
    return torch.where(gloss > 0, g, alb / math.pi)


def _entries(P, L, d_min, boxes, tris, spheres):
    """A of broadcast point and VPL planes ([..., 3, 4], float64)."""
    d = L[..., 0, :3] - P[..., 0, :3]
    d2 = (d * d).sum(-1)
    w = d / d2.clamp(min=1e-300).sqrt()[..., None]
    cp, cq = (P[..., 1, :3] * w).sum(-1), -(L[..., 1, :3] * w).sum(-1)
    G = cp.clamp(min=0) * cq.clamp(min=0) / d2.clamp(min=d_min * d_min)
    v = (L[..., 2, 3] * G * _brdf(P[..., 0, 3], P[..., 1, 3], P[..., 1, :3], w, P[..., 2, :3])
         * _brdf(L[..., 0, 3], L[..., 1, 3], L[..., 1, :3], L[..., 2, :3], -w))
    o = P[..., 0, :3] + 1e-4 * P[..., 1, :3]
    D = L[..., 0, :3] + 1e-4 * L[..., 1, :3] - o
    inv = 1.0 / D
    for b in boxes:
        ta, tb = (b[:3] - o) * inv, (b[3:] - o) * inv
        near = torch.minimum(ta, tb).nan_to_num(-math.inf).amax(-1).clamp(min=1e-4)
        far = torch.maximum(ta, tb).nan_to_num(math.inf).amin(-1).clamp(max=1 - 1e-4)
        v = torch.where(near <= far, 0.0, v)
    per = tris.shape[0] // len(spheres) if tris is not None else 0
    for k, (centre, r) in enumerate(spheres if tris is not None else ()):
        oc = o - torch.as_tensor(centre, device=o.device)
        b = (oc * D).sum(-1)
        disc = b * b - (D * D).sum(-1) * ((oc * oc).sum(-1) - (1.001 * r) ** 2)
        ids = ((disc >= 0) & (v > 0)).nonzero()[:, 0]
        for s in range(0, ids.numel(), 16384):
            i = ids[s:s + 16384]
            t = _triangles(o[i], D[i], tris[k * per:(k + 1) * per])
            v[i] = torch.where(((t > 1e-4) & (t < 1 - 1e-4)).any(1), 0.0, v[i])
    return v


def _node_side(R, nodes):
    """VPL planes and scale of light-tree nodes (float64)."""
    L = R.vpls.double()[:, R.tree.rep.long()[nodes]].transpose(0, 1)
    return L, R.tree.I.double()[nodes] / (L[:, 2, 3] * L[:, 0, 3])


def _occluders(R):
    boxes = [b for b in R.boxes.double()]
    if getattr(R.scene, "tris", None) is None:
        return boxes, None, []
    _, spheres = scenes._make_meshes(R.cfg, np.random.default_rng(R.cfg["scene_seed"] + 104729), R.scene.boxes)
    return boxes, R.tris.double().view(-1, 3, 3), spheres


def _slices(R, key, val, off, cnt):
    for s in range(R.frame.S):
        o, k = int(off[s]), int(cnt[s])
        kk = key[o:o + k].long() & 0xFFFFFFFF
        yield s, kk >> 16, kk & 0xFFFF, val[o:o + k].double()


def _half(mask, M, F, lam_rel):
    r = F.shape[1]
    G = (mask @ (F[:, :, None] * F[:, None, :]).reshape(-1, r * r)).view(-1, r, r)
    tr = G.diagonal(dim1=1, dim2=2).sum(1)
    eye = torch.eye(r, dtype=F.dtype, device=F.device)
    G = G + torch.where(tr > 0, lam_rel * tr / r, 1.0)[:, None, None] * eye
    return torch.cholesky_solve((M @ F)[:, :, None], torch.linalg.cholesky(G))[:, :, 0]


def _als(R, key, val, off, cnt, ncol, bounds, U, V, sweeps, cols, seed):
    """U, V [S][C][r] in 64 bits (rows beyond a slice's columns as they were)."""
    S, C, Rk = R.frame.S, R.frame.C, R.cfg["rank"]
    U, Vall = torch.zeros_like(U, dtype=torch.float64).view(-1, Rk), V.double().clone()
    V = Vall[:S * C * Rk].view(S, C, Rk)
    img = torch.zeros(U.shape[0], dtype=torch.float64, device=U.device)
    for s, i, j, v in _slices(R, key, val, off, cnt):
        a, b, n = int(bounds[s]), int(bounds[s + 1]), int(ncol[s])
        r = min(Rk, max(8, 8 * -(-n // cols))) if cols else Rk
        mask = torch.zeros(b - a, n, dtype=torch.float64, device=v.device)
        M = torch.zeros_like(mask)
        mask[i, j] = 1.0
        M[i, j] = v
        F = _start(s, n, r, 3, float(v.mean()) if v.numel() else 0.0, seed)
        W = torch.zeros(b - a, r, dtype=torch.float64, device=v.device)
        for _ in range(sweeps):
            W = _half(mask, M, F, R.cfg["lam_rel"])
            F = _half(mask.T, M.T, W, R.cfg["lam_rel"])
        U[a:b, :r] = W
        V[s, :n] = 0.0
        V[s, :n, :r] = F
        img[a:b] = (W @ F.sum(0)).clamp(min=0)
    return U.reshape(-1), Vall, img


def _adm(R, Vbuf, seed):
    c, C, q = R.cfg, R.frame.C, R.cfg["rank"]
    U, Vall = torch.zeros(R.frame.m, q, dtype=torch.float64, device=R.dev), Vbuf.double().clone()
    V = Vall[:R.frame.S * C * q].view(-1, C, q)
    img, off = torch.zeros(R.frame.m, dtype=torch.float64, device=R.dev), R.frame.slice_off_host
    eye = torch.eye(q, dtype=torch.float64, device=R.dev)
    for s, i, j, v in _slices(R, R.smp.key, R.smp.val, R.smp.off_host, R.smp.cnt.cpu()):
        a, b, n = int(off[s]), int(off[s + 1]), int(R.smp.ncol[s])
        mu = float(v.mean()) if v.numel() else 0.0
        V[s, :n] = 0.0
        if mu <= 0:
            continue
        mask = torch.zeros(b - a, n, dtype=torch.bool, device=v.device)
        M = torch.zeros(b - a, n, dtype=torch.float64, device=v.device)
        mask[i, j] = True
        M[i, j] = v
        X, Y = _start(s, b - a, q, 6, mu, seed), _start(s, n, q, 3, mu, seed).T.contiguous()
        al, be = (c["adm_alpha_rel"] * float((F * F).sum()) / q for F in (Y, X))
        A, B, La, Pi = X.clone(), Y.clone(), torch.zeros_like(X), torch.zeros_like(Y)
        Z = torch.where(mask, M, X @ Y)
        for _ in range(c["adm_iters"]):
            X = (Z @ Y.T + al * A - La) @ torch.linalg.inv(Y @ Y.T + al * eye)
            Y = torch.linalg.inv(X.T @ X + be * eye) @ (X.T @ Z + be * B - Pi)
            Z = torch.where(mask, M, X @ Y)
            A, B = (X + La / al).clamp(min=0), (Y + Pi / be).clamp(min=0)
            La, Pi = La + c["adm_gamma"] * al * (X - A), Pi + c["adm_gamma"] * be * (Y - B)
        U[a:b], V[s, :n], img[a:b] = X, Y.T, (X @ Y.sum(1)).clamp(min=0)
    return U.reshape(-1), Vall, img


def _leverage(R, M, s, n, r, seed):
    w = _philox(np.arange(min(r, n))[None, :], np.arange(n)[:, None], s, 4, seed)
    Q = torch.from_numpy(w * 2.0 ** -32 - 0.5).to(R.dev)
    G = M.T @ M
    Q = torch.linalg.qr(Q)[0]
    for _ in range(proposal.TARGET_ITERS):
        Q = torch.linalg.qr(G @ Q)[0]
    t = (Q * Q).sum(1) + 1.0 / n
    return t / t.sum()


def _round(x):
    return x + (x.to(torch.bfloat16).double() - x).detach()


def _gradient(st, S):
    """Loss and its gradient through the rounded network (the rounding taken as the identity)."""
    th = st["theta"].double().requires_grad_(True)
    at, x = 0, st["feat"].to(torch.bfloat16).double()
    for out, inp in ((64, 32), (64, 64), (64, 64), (1, 64)):
        W, b = th[at:at + out * inp].view(out, inp), th[at + out * inp:at + out * inp + out]
        at += out * inp + out
        h = x @ _round(W).T + b
        x = _round(torch.nn.functional.silu(h)) if out > 1 else h[:, 0]
    off, loss = st["goff"][:S + 1].cpu().tolist(), 0.0
    for a, b in zip(off[:-1], off[1:]):
        if b > a:
            loss = loss - (st["target"][a:b].double() * torch.log_softmax(x[a:b], 0)).sum() / S
    loss.backward()
    return loss.detach().reshape(1), th.grad


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("evaluate", "complete", "adm", "colour", "targets", "train", "brute"):
        return None  # draws, cuts and orders are whole numbers; the values follow from them
    st = prepare(case, seed)
    R = st["R"]
    if kind == "brute":
        P, L, occ = R.pts.double().transpose(0, 1), R.vpls.double().transpose(0, 1), _occluders(R)
        if float(P.shape[0]) * L.shape[0] * (len(occ[0]) + 4) > 1.2e10:
            return None
        step = max(1, 8_000_000 // L.shape[0])
        return dict(img=torch.cat([_entries(p[:, None], L[None], case["d_min"], *occ).sum(1) for p in P.split(step)]))
    if kind == "train":
        loss, grad = _gradient(st, R.frame.S)
        return dict(loss=loss, grad=grad, theta=None, m=None, v=None)
    bounds = R.frame.slice_off_host
    if kind == "targets":
        off, occ = st["R"].frame.slice_off_host, _occluders(R)
        ncol = R.smp.ncol.cpu().tolist()
        if st["cap"] * (len(occ[0]) + 4) > 4e9:
            return None
        P, Ms, ts = R.pts_s.double().transpose(0, 1), [], []
        for s, n in enumerate(ncol):
            nodes = R.smp.col_node.view(-1, R.frame.C)[s, :n].long()
            L, scale = _node_side(R, nodes)
            Ms.append(_entries(P[off[s]:off[s + 1], None], L[None], case["d_min"], *occ) * scale)
            ts.append(_leverage(R, Ms[-1], s, n, case["rank"], st["seed"]))
        target, M = st["target"].double().clone(), torch.zeros(st["cap"], dtype=torch.float64, device=R.dev)
        for out, parts in ((target, ts), (M, [x.reshape(-1) for x in Ms])):
            x = torch.cat(parts)
            out[:x.numel()] = x
        return dict(feat=None, goff=None, M=M, target=target)
    cnt = R.smp.cnt.cpu()
    if kind == "evaluate":
        occ, val = _occluders(R), st["buf"]["val"].double().clone()
        P, n1 = R.pts_s.double().transpose(0, 1), R.smp.n1.cpu()
        for s, i, j, v in _slices(R, R.smp.key, R.smp.val, R.smp.off_host, cnt):
            a, o = int(n1[s]), int(R.smp.off_host[s])
            L, scale = _node_side(R, R.smp.col_node.view(-1, R.frame.C)[s].long()[j[a:]])
            for b in range(0, L.shape[0], 1 << 20):
                e = slice(b, b + (1 << 20))
                val[o + a + b:o + a + b + L[e].shape[0]] = scale[e] * _entries(P[bounds[s] + i[a:][e]], L[e],
                                                                             case["d_min"], *occ)
        return dict(val=val)
    if kind == "adm":
        U, V, im = _adm(R, st["buf"]["V"], st["seed"])
        img = torch.zeros_like(im)
        img[R.row_perm.long()] = im
        return dict(img=img, U=U, V=V)
    if kind == "complete":
        U, V, im = _als(R, R.smp.key, R.smp.val, R.smp.off_host, cnt, R.smp.ncol.cpu(), bounds, R.uv.U, st["buf"]["V"],
                        case["sweeps"], case["cols"], st["seed"])
        img = torch.zeros_like(im)
        img[R.row_perm.long()] = im
        return dict(img=img, U=U, V=V)
    # colour: every sample's three channels from the tables, then the stacked completion
    G = R.rgb
    key, val = torch.zeros_like(G.key).long(), st["buf3"]["val"].double().clone()
    pr, nr = G.pt_ratio.view(-1, 4).double(), G.node_ratio.view(-1, 4).double()
    for s, i, j, v in _slices(R, R.smp.key, R.smp.val, R.smp.off_host, cnt):
        o = int(G.off_host[s])
        node = R.smp.col_node.view(-1, R.frame.C)[s].long()[j]
        x = v[:, None] * pr[int(bounds[s]) + i, :3] * nr[node, :3]
        k = torch.arange(3, device=v.device)
        key[o:o + 3 * v.numel()] = (((3 * i[:, None] + k) << 16) | j[:, None]).reshape(-1)
        val[o:o + 3 * v.numel()] = x.reshape(-1)
    U, V, im = _als(R, key, val, G.off_host, 3 * cnt, R.smp.ncol.cpu(), 3 * bounds, G.U, st["buf3"]["V"], case["sweeps"],
                    case["cols"], st["seed"])
    img = torch.zeros_like(im)
    img[G.row_perm3.long()] = im
    return dict(img=img, U=U, V=V, key=None, val=val)
