"""Forms of the calls that the parity tests do not reach: sizes, orders and refusals at which
a layout, a launch or a check of the library decides.  Tolerances are those of the parity tests.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from ltinputs import get_config, make_scene
from oracle import adm as o_adm, pipeline, proposal as o_prop, shading, slices as o_slices

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lt():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2202_12567_gb300 import lt as _lt
    _lt.load()
    return _lt


def _targets_renderer(**over):
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", **{**dict(width=24, height=24, eps_cut=1e-4, rate1=0.002), **over})
    R = Renderer(make_scene(cfg), cfg, device=0).setup()
    R.pass1(3)
    return R


def _check_targets(R, M, moff, goff, ncol, t, rank, iters, seed):
    M, moff, goff, t = (x.cpu().numpy() for x in (M, moff, goff, t))
    for s in range(R.frame.S):
        A = M[moff[s]:moff[s + 1]].reshape(-1, ncol[s]).astype(np.float64)
        want = o_prop.targets(o_prop.leverage(A, rank, iters, seed, s))
        got = t[goff[s]:goff[s + 1]]
        assert np.linalg.norm(got - want) <= 1e-3 * np.linalg.norm(want), (s, ncol[s])


@pytest.mark.parametrize("slices,cut,rank,iters", [(17, 631, 5, 0), (17, 631, 1, 1), (3, 257, 7, 0)])
def test_targets_odd_layout(lt, slices, cut, rank, iters):
    """Slices, cut and rank all odd: the parts of the scratch hold an odd number of floats."""
    R = _targets_renderer(n_slices=slices, max_cut=cut, rank=rank)
    assert R.frame.C == cut and R.frame.S == slices
    _, goff = lt.lt_proposal_features(R.ctx, R.frame, R.smp)
    ncol = R.smp.ncol.cpu().numpy()
    M, moff = lt.lt_slice_matrices(R.ctx, R.frame, R.smp, R.cfg["d_min"], int(np.sum(R.frame.sizes * ncol)))
    t = lt.lt_leverage_targets(R.ctx, R.frame, R.smp, M, moff, goff, rank, iters, 9)
    lt.lt_sync(R.ctx)
    _check_targets(R, M, moff, goff, ncol, t, rank, iters, 9)


def test_targets_after_refused_matrices(lt):
    """Matrices beyond the caller's capacity are refused at the next sync; the targets queued
    behind them read nothing of the buffer and write nothing."""
    R = _targets_renderer(n_slices=4, max_cut=256, rank=4)
    _, goff = lt.lt_proposal_features(R.ctx, R.frame, R.smp)
    M, moff = lt.lt_slice_matrices(R.ctx, R.frame, R.smp, R.cfg["d_min"], 1000)
    t = torch.full((R.frame.S * R.frame.C,), -7.0, device="cuda")
    lt.lt_leverage_targets(R.ctx, R.frame, R.smp, M, moff, goff, 4, 2, 9, t)
    with pytest.raises(lt.LtError):
        lt.lt_sync(R.ctx)
    assert int(moff[-1]) > 1000 and torch.all(t == -7.0) and torch.all(M == 0)
    ncol = R.smp.ncol.cpu().numpy()  # the sync cleared the status: the same calls with room
    M, moff = lt.lt_slice_matrices(R.ctx, R.frame, R.smp, R.cfg["d_min"], int(np.sum(R.frame.sizes * ncol)))
    lt.lt_leverage_targets(R.ctx, R.frame, R.smp, M, moff, goff, 4, 0, 9, t)
    lt.lt_sync(R.ctx)
    _check_targets(R, M, moff, goff, ncol, t, 4, 0, 9)


def _wide_slices(lt, ncol):
    """Slices of ncol columns each, all of one coarsened cut of more than 4096 nodes."""
    S, most = len(ncol), max(ncol)
    R = _targets_renderer(n_slices=S, n_vpl=8192, max_cut=8192, target_cut=most, rank=2, width=20, height=16)
    assert R.smp.ncol.cpu().tolist() == [most] * S
    R.smp.ncol.copy_(torch.tensor(ncol, dtype=torch.int32))
    goff = torch.tensor(np.concatenate([[0], np.cumsum(ncol)]).astype(np.int32), device="cuda")
    M, moff = lt.lt_slice_matrices(R.ctx, R.frame, R.smp, R.cfg["d_min"], int(np.sum(R.frame.sizes * np.array(ncol))))
    t = torch.full((R.frame.S * R.frame.C,), -7.0, device="cuda")
    lt.lt_leverage_targets(R.ctx, R.frame, R.smp, M, moff, goff, 2, 1, 9, t)
    return R, M, moff, goff, t


def test_targets_within_capacity(lt):
    """Above 4096 columns in one slice, the squares of all within two times 4096 squared, though
    not with every row of the products padded to four floats."""
    ncol = [5001, 2923]
    assert sum(n * n for n in ncol) <= 2 * 4096 ** 2 < sum(n * ((n + 3) & ~3) for n in ncol)
    R, M, moff, goff, t = _wide_slices(lt, ncol)
    lt.lt_sync(R.ctx)
    _check_targets(R, M, moff, goff, ncol, t, 2, 1, 9)


def test_targets_beyond_capacity(lt):
    """Products that do not fit are an error, not targets left as they were."""
    R, _, _, _, t = _wide_slices(lt, [4200])
    with pytest.raises(lt.LtError):
        lt.lt_sync(R.ctx)
    assert torch.all(t == -7.0)


def test_pass1_many_slices(lt):
    """More slices than a grid has in its second dimension: 66560 of no rows, then 1024 of one."""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", width=32, height=32, n_vpl=64, max_cut=8)
    sc = make_scene(cfg)
    st = pipeline.setup(sc, cfg, slicing=(np.arange(sc.m), np.maximum(np.arange(66560 + sc.m + 1) - 66560, 0)))
    R = Renderer(sc, cfg, device=0).setup(cut=st["cut"], row_perm=st["row_perm"], slice_off=st["slice_off"])
    assert R.frame.S == 67584
    R.pass1(11)
    lt.lt_sync(R.ctx)
    assert int(R.smp.cnt[:66560].abs().max()) == 0 and int(R.smp.ncol[:66560].abs().max()) == 0
    for s in (66560, 67000, 67583):
        rows, cols, vals, col_node, _ = R.smp.slice(s)
        o = pipeline.run_slice(st, sc, cfg, s, 11).p1
        assert np.array_equal(col_node, o.col_node) and np.array_equal(rows, o.rows) and np.array_equal(cols, o.cols)
        assert np.all(np.abs(vals - o.vals) <= 1e-5 * np.abs(o.vals) + 1e-12)


@pytest.mark.parametrize("n,eps", [(1, 0.02), (64, 1e9), (1024, 1e9)])
def test_cut_that_ends_at_once(lt, n, eps):
    """The cut is the root after one round; the rounds that are launched before the host hears
    of it are few (four kernels each)."""
    sc = make_scene(get_config("room64_vpl1k_2box", n_vpl=n))
    ctx = lt.Context(0)
    vp, pts = torch.from_numpy(sc.vpls).cuda(), torch.from_numpy(np.ascontiguousarray(sc.points)).cuda()
    tree = lt.lt_build_tree(ctx, vp)
    rows = torch.arange(0, sc.m, 64, dtype=torch.int32, device="cuda")
    launches = []
    for _ in range(5):  # the first call also loads the kernels
        before = lt.lt_launch_count(ctx)
        cut = lt.lt_build_global_cut(ctx, tree, pts, vp, rows, eps, 8192, 0.5, 0.1)
        launches.append(lt.lt_launch_count(ctx) - before)
        assert cut.tolist() == [0]
    assert sorted(launches)[2] <= 42, launches


def test_cut_of_a_tree_with_children_exchanged(lt):
    """The cut is in leaf order whichever child a tree names first."""
    sc = make_scene(get_config("room64_vpl1k_2box", n_vpl=1000))
    ctx = lt.Context(0)
    vp, pts = torch.from_numpy(sc.vpls).cuda(), torch.from_numpy(np.ascontiguousarray(sc.points)).cuda()
    tree = lt.lt_build_tree(ctx, vp)
    rows = torch.arange(0, sc.m, 64, dtype=torch.int32, device="cuda")
    cut = lt.lt_build_global_cut(ctx, tree, pts, vp, rows, 0.02, 300, 0.5, 0.1)
    child = tree.child.view(-1, 2)
    swap = torch.arange(child.shape[0], device="cuda") % 3 != 0
    child[swap] = child[swap].flip(1)
    again = lt.lt_build_global_cut(ctx, tree, pts, vp, rows, 0.02, 300, 0.5, 0.1)
    assert cut.numel() > 200 and torch.equal(cut, again)
    first = tree.range.view(-1, 2)[cut.long(), 0]
    assert torch.all(first[1:] > first[:-1])


@pytest.mark.parametrize("kind", ["repeated", "negative", "past_the_tree", "short", "nested", "too_many", "levels"])
def test_forest_refusals_write_nothing(lt, kind):
    """A cut that is no partition, or higher than the caller's levels, is an error and leaves the
    caller's arrays as they were; the cut itself is accepted with room for exactly its levels."""
    import ctypes
    n = 300
    sc = make_scene(get_config("room64_vpl1k_2box", n_vpl=n, width=16, height=16))
    ctx = lt.Context(0)
    tree = lt.lt_build_tree(ctx, torch.from_numpy(sc.vpls).cuda())
    child = tree.child.cpu().numpy().reshape(-1, 2)
    good = [0]
    for _ in range(100):  # the first internal node is split
        i = next(k for k, x in enumerate(good) if x < n - 1)
        good[i:i + 1] = child[good[i]].tolist()
    _, _, _, H = lt.lt_cut_forest(ctx, tree, torch.tensor(good, dtype=torch.int32, device="cuda"))
    assert H > 1
    cut, levels = list(good), H
    if kind == "repeated":
        cut[5] = cut[50]
    elif kind == "negative":
        cut[5] = -1
    elif kind == "past_the_tree":
        cut[5] = 2 * n - 1
    elif kind == "short":
        del cut[5]
    elif kind == "nested":
        i = next(k for k, x in enumerate(cut) if x < n - 1)
        cut.insert(i, int(child[cut[i]][0]))
    elif kind == "too_many":
        cut = list(range(n + 1))
    else:
        levels = H - 1

    def call(cut, levels):
        C = len(cut)
        c = torch.tensor(cut, dtype=torch.int32, device="cuda")
        out = [torch.full((k,), -7, dtype=torch.int32, device="cuda") for k in (8 * (2 * C - 1), levels + 2, C)]
        h, s = ctypes.c_int32(-7), tree.struct()
        status = ctx.lib.lt_cut_forest(ctx.h, ctypes.byref(s), c.data_ptr(), C, out[0].data_ptr(), out[1].data_ptr(),
                                       levels, out[2].data_ptr(), ctypes.byref(h))
        return status, h.value, all(bool(torch.all(x == -7)) for x in out)

    assert call(cut, levels) == (1, -7, True)  # LT_EINVAL
    assert call(good, H) == (0, H, False)


@pytest.mark.parametrize("nb,extra", [(2, 0), (2, 15), (0, 0)])
def test_counters_follow_the_path(lt, nb, extra):
    """Up to 16 boxes every ray of the evaluation and of the brute force tests every box and visits
    no cell; more boxes (here: outside the room) are found through the grid by the same rays."""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", n_vpl=300, max_cut=128)
    sc = make_scene(cfg)
    R = Renderer(sc, cfg, device=0).setup()
    far = np.array([[9, 9, 9, 9.5, 9.5, 9.5]], np.float32)
    lt.lt_scene_upload(R.ctx, torch.from_numpy(np.concatenate([sc.boxes[:nb], np.repeat(far, extra, 0)])).cuda())
    R.pass1(5)
    R.pass2(5)
    R.evaluate()
    lt.lt_sync(R.ctx)
    ev = lt.lt_eval_stats(R.ctx, R.frame, R.smp, cfg["d_min"])
    bf = lt.lt_bruteforce_stats(R.ctx, R.pts, R.vpls, cfg["d_min"])
    assert bf["entries"] == sc.m * sc.n and ev["entries"] == int((R.smp.cnt - R.smp.n1).sum())
    assert bf["rays"] > 0 and (ev["rays"] > 0 or ev["entries"] == 0)  # (a coarse cut leaves pass 2 nothing)
    for st in (ev, bf):
        assert st["rays"] <= st["entries"]
        if extra == 0:
            assert st["cells"] == 0 and st["boxes"] == nb * st["rays"]
        else:
            assert st["cells"] > 0 or st["entries"] == 0
    lt.lt_scene_upload(R.ctx, torch.from_numpy(np.repeat(far, 17, 0)).cuda())
    assert lt.lt_bruteforce_stats(R.ctx, R.pts, R.vpls, cfg["d_min"])["rays"] == bf["rays"]


@pytest.mark.parametrize("slices,rank,least", [(40, 16, 45_000), (80, 8, 27_000), (20, 10, 102_000)])
def test_adm_clusters_in_turns(lt, slices, rank, least):
    """Slices of many entries on clusters of twice the Gram parts that run in two turns: 8 CTAs over 4
    parts, 4 over 2, 16 over 8.  (Smaller slices keep to clusters of the parts.)"""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", width=96, height=96, n_vpl=4096, max_cut=1024, eps_cut=1e-4, n_slices=slices,
                     rank=rank, rate=0.7, rate1=0.002, tau=1e-4, completion="adm", adm_iters=5)
    R = Renderer(make_scene(cfg), cfg, device=0).setup()
    R.render(seed=4)
    assert float(R.smp.cnt.double().mean()) >= least
    img = R.img.clone()
    for s in range(0, slices, 13):
        rows, cols, vals, col_node, _ = R.smp.slice(s)
        a, b, n = int(R.frame.slice_off_host[s]), int(R.frame.slice_off_host[s + 1]), int(R.smp.ncol[s])
        Xo, Yo = o_adm.complete_slice_adm(rows, cols, vals.astype(np.float64), b - a, n, rank, 5, cfg["adm_alpha_rel"],
                                          cfg["adm_gamma"], 4, s)
        U = R.uv.U.cpu().numpy().reshape(-1, rank)[a:b].astype(np.float64)
        V = R.uv.V.cpu().numpy().reshape(R.frame.S, R.frame.C, rank)[s, :n].astype(np.float64)
        assert np.linalg.norm(U @ V.T - Xo @ Yo.T) <= 1e-3 * np.linalg.norm(Xo @ Yo.T), s
    R.complete(4)
    R.render_image()
    lt.lt_sync(R.ctx)
    assert torch.equal(R.img, img)


@pytest.mark.parametrize("order", ["image", "random"])
@pytest.mark.parametrize("S", [5, 64, 500])
def test_slices_of_points_in_any_order(lt, S, order):
    """A warp's points in one cluster, in a few and in 32 clusters: the oracle's labels."""
    pts = np.ascontiguousarray(make_scene(get_config("room64_vpl1k_2box", width=63, height=61)).points)
    if order == "random":
        pts = np.ascontiguousarray(pts[:, np.random.default_rng(S).permutation(pts.shape[1])])
    perm, off = lt.lt_make_slices(lt.Context(0), torch.from_numpy(pts).cuda(), S, 10, 0.3)
    perm, off = perm.cpu().numpy(), off.cpu().numpy()
    lab = np.empty(pts.shape[1], np.int64)
    lab[perm] = np.repeat(np.arange(S), np.diff(off))
    assert np.mean(lab == o_slices.kmeans_slices(pts, S, 10, 0.3)[2]) >= 0.99


@pytest.mark.parametrize("nr,C", [(1, 1), (33, 7), (64, 1215), (64, 1300), (64, 5000)])
def test_cut_errors_of_every_row(lt, nr, C):
    """One round's errors at cuts on both sides of the rules for warps per node, on rows that the
    cut lights (each is compared) and with a row that it leaves dark (every bound infinite)."""
    n = 8192
    sc = make_scene(get_config("room256_vpl16k_200box", n_vpl=n, width=16, height=16))
    ctx, vp = lt.Context(0), torch.from_numpy(sc.vpls).cuda()
    t = lt.lt_build_tree(ctx, vp)
    rng = np.random.default_rng(C)
    I, B, rep, bb = (x.cpu().numpy() for x in (t.I, t.B, t.rep, t.aabb))
    cut = np.sort(rng.choice(2 * n - 1, C, replace=False)).astype(np.int32) if C > 1 else np.zeros(1, np.int32)
    rc, pts = rep[cut], sc.points.copy()
    scale = I[cut].astype(np.float64) / (sc.vpls[2, rc, 3].astype(np.float64) * sc.vpls[0, rc, 3])
    rr, cc = np.repeat(np.arange(sc.m), C), np.tile(np.arange(C), sc.m)
    est = (shading.unoccluded(pts, sc.vpls, rr, rc[cc], 0.1) * scale[cc]).reshape(sc.m, C).sum(1)
    rows = np.argsort(-est, kind="stable")[rng.permutation(np.arange(max(nr, 64)))[:nr]].astype(np.int32)
    assert (est[rows] > 0).all()

    def errors(pts, rows):
        p, r = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (pts, rows))
        return lt.lt_cut_errors(ctx, t, p, vp, r, torch.from_numpy(cut).cuda(), 0.1).cpu().numpy()

    P = pts[0, rows].astype(np.float64)
    lo, hi = bb.reshape(-1, 6)[cut, :3].astype(np.float64), bb.reshape(-1, 6)[cut, 3:].astype(np.float64)
    gap = np.maximum(0, np.maximum(lo[None] - P[:, None, :3], P[:, None, :3] - hi[None]))
    bound = (I * B)[cut].astype(np.float64) * (P[:, 3] / np.pi)[:, None] / np.maximum((gap ** 2).sum(2), 0.01)
    np.testing.assert_allclose(errors(pts, rows), (bound / est[rows][:, None]).max(0), rtol=1e-4)
    dark = pts.copy()
    dark[0, rows[0], :3], dark[1, rows[0], :3] = (0.5, 2.0, 0.5), (0.0, 1.0, 0.0)  # above the room, facing up
    assert np.all(np.isinf(errors(dark, rows)))


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("rate1,slices", [(0.002, 2), (0.03, 1)])
def test_pass1_decides_as_the_oracle(lt, rate1, slices, form):
    """Every pair whose children both coarsenings reached: merged by both or by neither, unless its
    cost is within 1e-4 of the threshold."""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", max_cut=256, n_slices=slices, rate1=rate1, tau=0.2)
    sc = make_scene(cfg)
    st = pipeline.setup(sc, cfg)
    fo = st["forest"]
    R = Renderer(sc, cfg, device=0).setup(cut=st["cut"], row_perm=st["row_perm"], slice_off=st["slice_off"])
    lt.lt_set_tuning(R.ctx, p1_form=form)
    R.pass1(11)
    lt.lt_sync(R.ctx)
    for s in range(slices):
        col_node = set(R.smp.slice(s)[3].tolist())
        ours = np.zeros(len(fo.node), bool)  # the node is a column or lies under one
        for x in range(len(fo.node)):
            y = x
            while y >= 0 and int(fo.node[y]) not in col_node:
                y = int(fo.parent[y])
            ours[x] = y >= 0
        o = pipeline.run_slice(st, sc, cfg, s, 11).p1
        reached = lambda x: x < fo.C or ours[x]
        ties = [f for f, _, cf, thr, merged, *_ in o.log
                if ours[f] != merged and reached(fo.child[f, 0]) and reached(fo.child[f, 1]) and
                abs(cf - thr) <= 1e-4 * thr]
        wrong = [f for f, _, cf, thr, merged, *_ in o.log
                 if ours[f] != merged and reached(fo.child[f, 0]) and reached(fo.child[f, 1]) and f not in ties]
        assert len(o.log) > 50 and not wrong, (s, wrong)
        assert ties or col_node == set(o.col_node.tolist())


@pytest.mark.parametrize("rank,slices,side,rate,K,parts",
                         [(8, 40, 64, 0.3, 4, 4), (16, 40, 64, 0.3, 4, 4), (20, 80, 64, 0.3, 2, 2), (12, 3, 64, 0.3, 16, 8),
                          (24, 12, 64, 0.3, 8, 8), (16, 20, 64, 0.3, 8, 8), (16, 40, 96, 0.7, 8, 4), (8, 80, 96, 0.7, 4, 2),
                          (10, 20, 96, 0.7, 16, 8)])
def test_adm_shapes(lt, rank, slices, side, rate, K, parts):
    """The clusters that the cases of the ADM tests run on (with fewer entries a slice those of the
    Gram parts, with more twice as many CTAs), as the kernel itself reports them."""
    from paper_2202_12567_gb300.renderer import Renderer
    over = dict(max_cut=128) if side == 64 else dict(n_vpl=4096, max_cut=1024, eps_cut=1e-4, tau=1e-4)
    cfg = get_config("room64_vpl1k_2box", width=side, height=side, n_slices=slices, rank=rank, rate=rate, rate1=0.002,
                     completion="adm", adm_iters=2, **over)
    R = Renderer(make_scene(cfg), cfg, device=0).setup()
    R.render(seed=4)
    assert lt.lt_debug_scratch(R.ctx, 14)[:8].view(torch.int32).tolist() == [K, parts]
