"""Sizes at which the kernels and their dispatch rules change path.

* shadow rays: 16 boxes (tested one by one) and 17 (grid walk), one and few triangles;
* brute force: points and lights around the 32-point CTA, the 256-light tile and the
  16-warp rule, against the float64 oracle;
* sorts around one 4096-key chunk, and the cut errors of small and large cuts;
* pass 1 with slices of thousands of rows: pairs of 8 lanes, of a warp and of a CTA, nodes
  drawn by a thread and by a warp, in both forms, against the oracle's coarsening;
* pass 2 at a rate where most draws repeat a key;
* leverage targets around 512 columns, above rank 16 and above 2048 columns;
* completion of slices larger than the stage (ranks read by 16-byte and by scalar loads),
  ranks above 16 that are no multiple of 4, and the ADM with clusters of twice the Gram parts.

Tolerances are those of the parity tests: draws, cuts and trees exact, entries 1e-5, images
and slice matrices 1e-3, at most 1e-4 of the shadow rays, targets 1e-3 normwise.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from ltinputs import get_config, make_scene
from oracle import adm as o_adm, als as o_als, bruteforce, pass2 as o_pass2, pipeline, proposal as o_prop, shading
from oracle import tree as o_tree

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lt():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2202_12567_gb300 import lt as _lt
    _lt.load()
    return _lt


@pytest.fixture(scope="module")
def ctx(lt):
    return lt.Context(0)


def _cuda(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t if dtype is None else t.to(dtype)).cuda()


def _segments(k, seed):
    rng = np.random.default_rng(seed)
    o, e = rng.uniform(0, 1, (2, k, 3)).astype(np.float32)
    o[: k // 8, 0] = e[: k // 8, 0]  # axis-parallel ones among them
    o[: k // 16, 1] = e[: k // 16, 1]
    return o, e


@pytest.mark.parametrize("nb", [1, 8, 16, 17])
def test_few_boxes(lt, ctx, nb):
    cfg = get_config("room256_vpl16k_200box", n_small_boxes=nb, width=8, height=8, n_vpl=8)
    boxes = make_scene(cfg).boxes
    o, e = _segments(100_000, nb)
    lt.lt_scene_upload(ctx, _cuda(boxes))
    got = lt.lt_shadow_test(ctx, _cuda(o), _cuda(e)).cpu().numpy().astype(bool)
    exp = shading.segment_blocked(o.astype(np.float64), e.astype(np.float64), boxes)
    assert np.mean(got != exp) <= 1e-4
    # the other path on the same boxes: copies of the first box change no answer
    n = 17
    if n > nb:
        lt.lt_scene_upload(ctx, _cuda(np.concatenate([boxes, np.repeat(boxes[:1], n - nb, 0)])))
        again = lt.lt_shadow_test(ctx, _cuda(o), _cuda(e)).cpu().numpy().astype(bool)
        assert np.mean(again != got) <= 1e-4


@pytest.mark.parametrize("nt", [1, 2, 3, 33])
def test_few_triangles(lt, ctx, nt):
    rng = np.random.default_rng(nt)
    tris = rng.uniform(0, 1, (nt, 3, 3)).astype(np.float32)
    o, e = _segments(50_000, nt)
    lt.lt_scene_upload(ctx, torch.zeros(0, 6, device="cuda"))
    lt.lt_mesh_upload(ctx, _cuda(tris))
    got = lt.lt_shadow_test(ctx, _cuda(o), _cuda(e)).cpu().numpy().astype(bool)
    lt.lt_mesh_upload(ctx, None)
    exp = shading.segment_hits_triangles(o, e, tris)
    assert np.mean(got != exp) <= 1e-4


@pytest.mark.parametrize("m,n", [(1, 1), (31, 255), (32, 256), (33, 257), (1000, 513)])
def test_bruteforce_sizes(lt, ctx, m, n):
    sc = make_scene(get_config("room64_vpl1k_2box", n_vpl=n))
    pts = np.ascontiguousarray(sc.points[:, ::4][:, :m])
    lt.lt_scene_upload(ctx, _cuda(sc.boxes))
    img = lt.lt_bruteforce(ctx, _cuda(pts), _cuda(sc.vpls), 0.1).cpu().numpy()
    ref = bruteforce.render(pts, sc.vpls, sc.boxes, 0.1)
    assert np.linalg.norm(img - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("nb,glossy,d_min", [(0, 0.0, 0.1), (2, 0.5, 0.0), (16, 0.3, 0.01)])
def test_bruteforce_forms(lt, ctx, nb, glossy, d_min):
    """Few boxes (diffuse pairs without a unit direction, box planes relative to the points)
    against the walk, which copies of a box, or of one outside the room, select.  A sum of n
    positive float32 values that differ by a few roundings: (n + 40) 2^-24 relative."""
    n = 257
    cfg = get_config("room256_vpl16k_200box", n_small_boxes=max(nb, 1), glossy_frac=glossy, width=16, height=9, n_vpl=n)
    sc = make_scene(cfg)
    boxes = sc.boxes[:nb].astype(np.float32)
    vpls = sc.vpls.copy()
    vpls[0, :3, :3] = sc.points[0, :3, :3]  # lights at points: no distance, no direction
    vpls[0, 3:6, 0] = sc.points[0, 3:6, 0]  # axis-parallel rays
    far = np.array([[9, 9, 9, 9.5, 9.5, 9.5]], np.float32)
    imgs = []
    for b in (boxes, np.concatenate([boxes, np.repeat(far, 17, 0)])):
        lt.lt_scene_upload(ctx, _cuda(b))
        imgs.append(lt.lt_bruteforce(ctx, _cuda(sc.points), _cuda(vpls), d_min).cpu().numpy().astype(np.float64))
    assert np.isfinite(imgs[0]).all()
    assert np.all(np.abs(imgs[0] - imgs[1]) <= (n + 40) * 2.0 ** -24 * np.abs(imgs[1]))


@pytest.mark.parametrize("n", [2048, 4095, 4096, 4097, 8193])
def test_sort_chunks(lt, ctx, n):
    sc = make_scene(get_config("room256_vpl16k_200box", n_vpl=n, width=8, height=8), seed=n)
    ref = o_tree.build(sc.vpls)
    t = lt.lt_build_tree(ctx, _cuda(sc.vpls))
    assert np.array_equal(t.order.cpu().numpy(), ref.order)
    assert np.array_equal(t.child.cpu().numpy().reshape(-1, 2), ref.child)


@pytest.mark.parametrize("nr,C", [(1, 1), (33, 7), (64, 1215), (64, 1300), (64, 5000)])
def test_cut_errors_sizes(lt, ctx, nr, C):
    """One round's errors at cuts on both sides of the rules for warps per node."""
    sc = make_scene(get_config("room256_vpl16k_200box", n_vpl=8192, width=16, height=16))
    vp = _cuda(sc.vpls)
    t = lt.lt_build_tree(ctx, vp)
    n = 8192
    rng = np.random.default_rng(C)
    cut = np.sort(rng.choice(2 * n - 1, C, replace=False)).astype(np.int32)
    rows = rng.choice(sc.m, nr, replace=False).astype(np.int32)
    err = lt.lt_cut_errors(ctx, t, _cuda(sc.points), vp, _cuda(rows), _cuda(cut), 0.1).cpu().numpy()
    bb = t.aabb.cpu().numpy().astype(np.float64)[cut]
    I, B, rep = (x.cpu().numpy()[cut] for x in (t.I, t.B, t.rep))
    P = sc.points[:, rows].astype(np.float64)
    rr, cc = np.repeat(np.arange(nr), C), np.tile(np.arange(C), nr)
    L = sc.vpls.astype(np.float64)
    scale = I.astype(np.float64) / (L[2, rep, 3] * L[0, rep, 3])
    est = (shading.unoccluded(sc.points, sc.vpls, rows[rr], rep[cc], 0.1) * scale[cc]).reshape(nr, C).sum(1)
    gap = np.maximum(0, np.maximum(bb[None, :, :3] - P[0][:, None, :3], P[0][:, None, :3] - bb[None, :, 3:]))
    bound = (I * B).astype(np.float64) * (P[0, :, 3] / np.pi)[:, None] / np.maximum((gap ** 2).sum(2), 0.01)
    ok = est > 1e-9 * est.max()
    if ok.all():
        ref = (bound / est[:, None]).max(0)
        np.testing.assert_allclose(err, ref, rtol=1e-4)


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("rate1,slices", [(0.002, 2), (0.03, 1)])
def test_pass1_pair_classes(lt, rate1, slices, form):
    """Slices of 2048 and 4096 rows: unions from four rows to a thousand."""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", max_cut=256, n_slices=slices, rate1=rate1, tau=0.2)
    sc = make_scene(cfg)
    st = pipeline.setup(sc, cfg)
    R = Renderer(sc, cfg, device=0).setup(cut=st["cut"], row_perm=st["row_perm"], slice_off=st["slice_off"])
    lt.lt_set_tuning(R.ctx, p1_form=form)
    R.pass1(11)
    lt.lt_sync(R.ctx)
    for s in range(slices):
        rows, cols, vals, col_node, g = R.smp.slice(s)
        o = pipeline.run_slice(st, sc, cfg, s, 11).p1
        if not np.array_equal(col_node, o.col_node):
            margins = [abs(cf - thr) / max(thr, 1e-30) for (_, _, cf, thr, *_rest) in o.log]
            assert min(margins) < 1e-4, f"slice {s}: coarsened cut differs without a near tie"
            continue
        got = dict(zip((rows * 65536 + cols).tolist(), vals.tolist()))
        exp = dict(zip((o.rows * 65536 + o.cols).tolist(), o.vals.tolist()))
        assert got.keys() == exp.keys()
        k = sorted(exp)
        gv, ev = np.array([got[x] for x in k]), np.array([exp[x] for x in k])
        assert np.all(np.abs(gv - ev) <= 1e-5 * np.abs(ev) + 1e-12)


@pytest.mark.parametrize("rate", [0.2, 0.6, 0.9])
def test_pass2_repeated_keys(lt, rate):
    """Slices of some thousand cells: a round of 16384 draws repeats most of its keys."""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", max_cut=64, n_slices=24, rate=rate, rate1=0.002, tau=0.05)
    sc = make_scene(cfg)
    R = Renderer(sc, cfg, device=0).setup()
    R.pass1(5)
    lt.lt_sync(R.ctx)
    p1 = [R.smp.slice(s) for s in range(R.frame.S)]
    R.pass2(5)
    lt.lt_sync(R.ctx)
    for s, (rows, cols, _, col_node, g) in enumerate(p1):
        r, c, *_ = R.smp.slice(s)
        r2, c2, _, _ = o_pass2.draw_pass2(5, s, int(R.frame.sizes[s]), g.astype(np.float32),
                                          rows * col_node.size + cols, rate)
        assert np.array_equal(r[rows.size:], r2) and np.array_equal(c[rows.size:], c2), f"slice {s}"


@pytest.mark.parametrize("target,rank,iters", [(1, 5, 0), (63, 16, 0), (513, 16, 0), (600, 20, 0), (2200, 16, 0),
                                               (1, 1, 1), (129, 2, 1), (513, 2, 1), (600, 2, 2), (2200, 2, 1)])
def test_targets_sizes(lt, target, rank, iters):
    """Without a product: the Gram-Schmidt of the (well-conditioned) random start.  With
    one: two columns, which the largest singular values keep apart."""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", width=24, height=24, n_vpl=4096, n_slices=2, max_cut=4096, eps_cut=1e-4,
                     rank=rank, target_cut=target, rate1=0.002)
    R = Renderer(make_scene(cfg), cfg, device=0).setup()
    R.pass1(3)
    feat, goff = lt.lt_proposal_features(R.ctx, R.frame, R.smp)
    ncol = R.smp.ncol.cpu().numpy()
    M, moff = lt.lt_slice_matrices(R.ctx, R.frame, R.smp, cfg["d_min"], int(np.sum(R.frame.sizes * ncol)))
    t = lt.lt_leverage_targets(R.ctx, R.frame, R.smp, M, moff, goff, rank, iters, 9).cpu().numpy()
    lt.lt_sync(R.ctx)
    M, moff, goff = M.cpu().numpy().astype(np.float64), moff.cpu().numpy(), goff.cpu().numpy()
    for s in range(R.frame.S):
        A = M[moff[s]:moff[s + 1]].reshape(-1, ncol[s])
        want = o_prop.targets(o_prop.leverage(A, rank, iters, 9, s))
        got = t[goff[s]:goff[s + 1]]
        assert np.linalg.norm(got - want) <= 1e-3 * np.linalg.norm(want), (s, ncol[s])


def _completed(lt, R, s, Uo, Vo):
    r = R.cfg["rank"]
    a, b = int(R.frame.slice_off_host[s]), int(R.frame.slice_off_host[s + 1])
    n = int(R.smp.ncol[s])
    U = R.uv.U.cpu().numpy().reshape(-1, r)[a:b].astype(np.float64)
    V = R.uv.V.cpu().numpy().reshape(R.frame.S, R.frame.C, r)[s, :n].astype(np.float64)
    return np.linalg.norm(U @ V.T - Uo @ Vo.T) / np.linalg.norm(Uo @ Vo.T)


@pytest.mark.parametrize("rank,slices", [(16, 1), (10, 1), (8, 1), (5, 3), (17, 8), (20, 2), (31, 8), (32, 5)])
def test_completion_sizes(lt, rank, slices):
    """One slice of 4096 rows is more than the stage holds at rank 16 (about 3000 rows of
    64 bytes) and at rank 8 (as many of 32 bytes, two CTAs per SM)."""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", max_cut=128, n_slices=slices, rank=rank, als_iters=2, rate=0.3, rate1=0.002)
    R = Renderer(make_scene(cfg), cfg, device=0).setup()
    R.render(seed=4)
    for s in range(R.frame.S):
        rows, cols, vals, col_node, _ = R.smp.slice(s)
        Uo, Vo = o_als.complete_slice(rows, cols, vals.astype(np.float64), int(R.frame.sizes[s]), col_node.size, rank, 2,
                                      cfg["lam_rel"], 4, s)
        assert _completed(lt, R, s, Uo, Vo) <= 1e-3, s


@pytest.mark.parametrize("rank,slices", [(8, 40), (16, 40), (20, 80), (12, 3), (24, 12), (16, 20)])
def test_adm_clusters(lt, rank, slices):
    """More than 38 slices: clusters of 8 CTAs over 4 Gram parts (80: 4 over 2); few: clusters of
    16 over 8 where all of them can run at once, else of 8."""
    from paper_2202_12567_gb300.renderer import Renderer
    cfg = get_config("room64_vpl1k_2box", max_cut=128, n_slices=slices, rank=rank, rate=0.3, rate1=0.002,
                     completion="adm", adm_iters=7)
    R = Renderer(make_scene(cfg), cfg, device=0).setup()
    R.render(seed=4)
    for s in range(0, R.frame.S, 7):
        rows, cols, vals, col_node, _ = R.smp.slice(s)
        Xo, Yo = o_adm.complete_slice_adm(rows, cols, vals.astype(np.float64), int(R.frame.sizes[s]), col_node.size,
                                          rank, 7, cfg["adm_alpha_rel"], cfg["adm_gamma"], 4, s)
        assert _completed(lt, R, s, Xo, Yo) <= 1e-3, s
