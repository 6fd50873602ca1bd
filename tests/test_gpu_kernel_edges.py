"""Kernels at the edges of their blocks, batches and dispatch rules, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from oracle import sched as osc
from paper_2505_24796_gb300 import scenes

from .helpers import f32, margin_mask, scene64, to_torch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def tc():
    import paper_2505_24796_gb300 as m
    m._lib.load()
    return m


@pytest.mark.parametrize("width,height", [(60, 40), (800, 400)])
def test_tile_features_list_lengths(tc, width, height):
    """Lists around the multiples of a block's threads and of its entries in flight, in a view of few tiles
    (512 threads a tile) and one of many (128).  FP32 sums of at most 2049 terms: 1e-4 as for the
    workload's lists."""
    cam = scenes.pinhole(width, height, fx=100.0)
    gw, gh = oracle.grid(cam)
    rng = np.random.default_rng(3)
    P = 4000
    lens = np.resize([0, 1, 31, 127, 128, 129, 511, 512, 513, 2047, 2048, 2049], gw * gh)
    ends = np.cumsum(lens)
    a, c = rng.uniform(0.05, 1.0, (2, P))
    inp = dict(mean2d=f32(rng.uniform(0, width, (P, 2))),
               conic=f32(np.stack([a, 0.9 * rng.uniform(-1, 1, P) * np.sqrt(a * c), c], 1)),
               opacity=f32(rng.uniform(0.01, 1, P)), depth=f32(rng.uniform(1, 9, P)),
               radius=rng.integers(1, 30, P).astype(np.int32))
    b = dict(ids=rng.integers(0, P, int(ends[-1])), ranges=np.stack([ends - lens, ends], 1), n=int(ends[-1]))
    ref = osc.tile_features(cam, b, inp["mean2d"], inp["conic"], inp["opacity"], inp["depth"], inp["radius"])
    d = {k: to_torch(v, DEV) for k, v in inp.items()}
    got = tc.tcgs_tile_features(cam, to_torch(b["ranges"].astype(np.int32), DEV), to_torch(b["ids"].astype(np.int32), DEV),
                                d["mean2d"], d["conic"], d["opacity"], d["depth"], d["radius"])
    torch.cuda.synchronize()
    np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=1e-4, atol=1e-4)


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 300])
def test_mlp_block_edges(tc, n):
    """Item counts around the block's 128.  The targets lie 2 to 4 from the outputs, so that an FP16 rounding
    that falls the other way (2e-3 (1 + |y|) of the output, as in the workload's test) moves a gradient by
    at most about 0.5% of the largest."""
    rng = np.random.default_rng(n)
    p = osc.unpack(rng.normal(0, 0.3, osc.NPARAMS))
    p["b1"], p["b2"] = np.abs(p["b1"]) + 0.05, np.abs(p["b2"]) + 0.05
    params, X = f32(osc.pack(p)), f32(rng.normal(0, 2, (n, 8)) + 1.0)
    norm = f32(np.concatenate([np.full(8, 1.0), np.full(8, 0.5)]))
    yr, _ = osc.mlp_forward(params.astype(np.float64), norm.astype(np.float64), X, fp16=True)
    t = f32(yr + rng.uniform(2, 4, n) * rng.choice([-1, 1], n))
    d = [to_torch(v, DEV) for v in (params, norm, X)]
    y = tc.tcgs_mlp_fwd(*d).cpu().numpy()
    assert (np.abs(y - yr) <= 2e-3 * (1 + np.abs(yr))).all()
    loss = torch.zeros(1, device=DEV)
    grad, _ = tc.tcgs_mlp_bwd(*d, to_torch(t, DEV), loss=loss)
    gr, lr = osc.mlp_backward(params.astype(np.float64), norm.astype(np.float64), X, t, fp16=True)
    assert np.abs(grad.cpu().numpy() - gr).max() <= 1e-2 * np.abs(gr).max()
    assert abs(float(loss.item()) - lr) <= 1e-2 * lr


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_project_backward_rows_and_alignment(tc, degree, aligned):
    """Gaussian counts around a warp's 32 rows and a block's 128, every SH degree, coefficient arrays on and off
    a 16-byte boundary: the oracle's gradients (bounds as for the workloads), rows of unseen Gaussians
    untouched, and a second call adds the same again."""
    for P in (1, 31, 32, 33, 127, 161):
        cam, sc = scenes.plain_forward(P=P, seed=40 + P)
        rng = np.random.default_rng(P)
        K = (degree + 1) ** 2
        sc = dict(sc, sh=f32(rng.normal(0, 0.3, (P, K, 3))), sh_degree=degree)
        sc["means3"] = sc["means3"].copy()
        sc["means3"][::5, 2] = -1.0     # behind the camera
        pr = oracle.project(cam, scene64(sc))
        w = [f32(rng.normal(size=(P, k))) for k in (2, 3, 3)]
        ref = oracle.project_bwd(cam, scene64(sc), pr["radius"], *w)
        off = 0 if aligned else 1

        def place(a):
            buf = torch.zeros(a.size + off, device=DEV)
            v = buf[off:].view(a.shape)
            v.copy_(torch.from_numpy(a))
            return v

        d = tc.scene_to_device(sc, DEV)
        grads = dict(dmeans3=torch.zeros(P, 3, device=DEV), dscales=torch.zeros(P, 3, device=DEV),
                     dquats=torch.zeros(P, 4, device=DEV), dsh=place(np.zeros((P, K, 3), np.float32)))
        args = (cam, d["means3"], d["scales"], d["quats"], place(sc["sh"]), degree,
                to_torch(pr["radius"].astype(np.int32), DEV), *(to_torch(v, DEV) for v in w))
        tc.tcgs_project_bwd(*args, grads=grads)
        once = {k: v.cpu().numpy().astype(np.float64) for k, v in grads.items()}
        tc.tcgs_project_bwd(*args, grads=grads)
        seen = pr["radius"] > 0
        for k, v in once.items():
            assert (v[~seen] == 0).all()
            np.testing.assert_allclose(grads[k].cpu().numpy(), 2 * v, rtol=1e-6, atol=0)
            if seen.any():
                r = ref[k].reshape(P, -1)[seen]
                scale = np.abs(r).max(axis=1) + 1e-6 * (np.abs(r).max() + 1e-30)
                err = np.abs(v.reshape(P, -1)[seen] - r).max(axis=1) / scale
                assert err.max() <= 2e-3, (P, k, err.max())


def _pair_case(rng, lens, wide):
    """A 40 x 40 view (9 tiles) whose tiles' lists have the given lengths; wide: footprints of many tiles."""
    cam = scenes.pinhole(40, 40, fx=50.0)
    n = int(np.sum(lens))
    ends = np.cumsum(lens)
    t = np.repeat(np.arange(9), lens)
    a, c = rng.uniform(*((0.0005, 0.005) if wide else (0.02, 1.5)), (2, n))
    inp = dict(mean2d=f32(np.stack([t % 3 * 16 + rng.uniform(-4, 20, n), t // 3 * 16 + rng.uniform(-4, 20, n)], 1)),
               conic=f32(np.stack([a, 0.95 * rng.uniform(-1, 1, n) * np.sqrt(a * c), c], 1)),
               opacity=f32(rng.uniform(0.002, 0.5, n)), rgb=f32(rng.uniform(0, 1, (n, 3))))
    b = dict(ids=np.arange(n), ranges=np.stack([ends - lens, ends], 1).astype(np.int64), n=n)
    return cam, inp, b


def _render(tc, cam, inp, b, bg=(0, 0, 0), **kw):
    d = {k: to_torch(v, DEV) for k, v in inp.items()}
    lists = (to_torch(b["ranges"].astype(np.int32), DEV), to_torch(b["ids"].astype(np.int32), DEV))
    return d, lists, tc.tcgs_render_fwd(cam, tc.render_opts("fp32", **kw), *lists, d["mean2d"], d["conic"], d["opacity"],
                                        d["rgb"], bg=bg)


LENGTHS = np.array([0, 1, 3, 4, 5, 127, 128, 129, 260])   # around the group (4) and the batch (128)


@pytest.mark.parametrize("early", [False, True])
def test_fp32_blending_list_lengths(tc, early):
    """Forward and backward against the oracle, a view whose last row and column of tiles are partly outside.
    Footprints of a few pixels, whose transmittance stays above 0.05: the image to 1e-5, as for the workloads,
    and the gradients to 2e-4 of the Gaussian's largest component + 1e-3 of the array's, as at full size."""
    rng = np.random.default_rng(5)
    cam, inp, b = _pair_case(rng, LENGTHS, False)
    bg = (0.25, 0.5, 0.75)
    d, lists, f = _render(tc, cam, inp, b, bg, early_cull=early)
    i64 = {k: v.astype(np.float64) for k, v in inp.items()}
    o = oracle.render(cam, b, i64["mean2d"], i64["conic"], i64["opacity"], i64["rgb"], bg=bg)
    G = f32(rng.standard_normal((3, 40, 40)))
    margin = margin_mask(o)
    G[:, margin] = 0
    assert margin.mean() < 0.01
    assert np.abs(f["img"].cpu().numpy() - o["img"]).max(axis=0)[~margin].max() <= 1e-5
    ref = oracle.render_bwd(cam, b, i64["mean2d"], i64["conic"], i64["opacity"], i64["rgb"], G.astype(np.float64), bg=bg)
    g = tc.tcgs_render_bwd(cam, tc.render_opts("fp32", early_cull=early), *lists, d["mean2d"], d["conic"], d["opacity"],
                           d["rgb"], f["img"], f["T_final"], f["n_contrib"], to_torch(G, DEV), bg=bg)
    for k, v in g.items():
        a, r = v.cpu().numpy().reshape(b["n"], -1), ref[k].reshape(b["n"], -1)
        scale = np.abs(r).max(axis=1) + 1e-3 * np.abs(r).max()
        assert (np.abs(a - r).max(axis=1) / scale).max() <= 2e-4, k


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("early", [False, True])
def test_fp32_blending_does_not_depend_on_what_is_not_blended(tc, wide, early):
    """The same fragments with others between them that no pixel blends, half of which pass the block test (a
    footprint between the pixel centres): batches and groups fall elsewhere, image, transmittance and every
    gradient stay the same bit for bit.  So do they without the block tests."""
    rng = np.random.default_rng(7 + wide)
    cam, inp, b = _pair_case(rng, LENGTHS, wide)
    n, m = b["n"], 300
    tile = rng.integers(1, 9, m)
    pad = dict(mean2d=f32(np.stack([tile % 3 * 16 + rng.integers(1, 16, m), tile // 3 * 16 + rng.integers(1, 16, m)], 1)),
               conic=f32(np.tile([3.3, 0.0, 3.3], (m, 1))), opacity=f32(np.where(np.arange(m) % 2, 0.005, 0.002)),
               rgb=f32(rng.uniform(0, 1, (m, 3))))
    both = {k: np.concatenate([inp[k], pad[k]]) for k in inp}
    ids, ranges = [], np.zeros((9, 2), np.int64)
    for t in range(9):
        own = list(range(*b["ranges"][t]))
        for k in n + np.nonzero(tile == t)[0]:
            own.insert(int(rng.integers(0, len(own) + 1)), int(k))
        ranges[t] = len(ids), len(ids) + len(own)
        ids += own
    bp = dict(ids=np.array(ids), ranges=ranges, n=n + m)
    G = to_torch(f32(rng.standard_normal((3, 40, 40))), DEV)
    res = []
    for c, lists_of, cull in ((inp, b, True), (inp, b, False), (both, bp, True)):
        d, lists, f = _render(tc, cam, c, lists_of, early_cull=early, tile_cull=cull)
        g = tc.tcgs_render_bwd(cam, tc.render_opts("fp32", early_cull=early), *lists, d["mean2d"], d["conic"], d["opacity"],
                               d["rgb"], f["img"], f["T_final"], f["n_contrib"], G)
        res.append((f, g))
    (f0, g0), (f1, _), (f2, g2) = res
    for k in ("img", "T_final", "n_contrib"):
        assert torch.equal(f0[k], f1[k]), k
    for k in ("img", "T_final"):
        assert torch.equal(f0[k], f2[k]), k
    for k in g0:
        assert torch.equal(g0[k], g2[k][:n]), k
        assert (g2[k][n:] == 0).all()


def test_fp32_blending_keeps_infinities_where_they_are(tc):
    """An infinite colour or a NaN in dL/dimg reaches only the pixels that blend it and the Gaussians that the
    pixel blends; conics that are not positive definite or hold a NaN are evaluated at every pixel."""
    rng = np.random.default_rng(9)
    cam, inp, b = _pair_case(rng, np.full(9, 40), False)
    d, lists, clean = _render(tc, cam, inp, b)
    odd = {k: v.copy() for k, v in inp.items()}
    odd["rgb"][b["ranges"][4, 0] + 7] = np.inf
    _, _, f = _render(tc, cam, odd, b)
    finite = torch.isfinite(f["img"])
    assert not finite.all() and torch.equal(f["img"][finite], clean["img"][finite])
    assert torch.equal(f["T_final"], clean["T_final"])
    for bad in ((np.nan, 0.1, 0.2), (0.01, 0.5, 0.01), (-0.01, 0.0, 0.02)):
        odd = {k: v.copy() for k, v in inp.items()}
        odd["conic"][b["ranges"][4, 0] + 7] = f32(bad)
        _, _, f = _render(tc, cam, odd, b)
        _, _, every = _render(tc, cam, odd, b, tile_cull=False)
        for k in ("img", "T_final", "n_contrib"):
            assert torch.equal(f[k], every[k]), (bad, k)

    G = to_torch(f32(rng.standard_normal((3, 40, 40))), DEV)
    run = lambda dl: tc.tcgs_render_bwd(cam, tc.render_opts("fp32"), *lists, d["mean2d"], d["conic"], d["opacity"],  # noqa: E731
                                        d["rgb"], clean["img"], clean["T_final"], clean["n_contrib"], dl)
    G[:, 20, 20] = 0
    ref = run(G)
    lit = torch.zeros_like(G)
    lit[:, 20, 20] = 1
    blends = (run(lit)["drgb"] != 0).any(dim=1)
    G[:, 20, 20] = float("nan")
    got = run(G)
    assert blends.any() and not blends.all()
    for k in ref:
        assert torch.equal(got[k][~blends], ref[k][~blends]), k
        assert torch.isnan(got[k][blends]).any()


@pytest.mark.parametrize("P", [1, 31, 32, 33, 1023, 1025, 3000])
def test_small_view_depth_order_edges(tc, P):
    """Counts around the ranking kernel's 32 Gaussians a block and 1024 keys a tile, with depth ties and culled
    Gaussians: the oracle's lists; N and the status when the capacity is N and N - 1."""
    cam = scenes.pinhole(100, 70, fx=100.0)
    rng = np.random.default_rng(P)
    mean2d = f32(rng.uniform(-10, 110, (P, 2)))
    radius = rng.integers(0, 12, P).astype(np.int32)
    depth = f32(rng.integers(1, max(2, P // 3), P))
    b = oracle.bin_sort(cam, mean2d, radius, depth)
    d = [to_torch(v, DEV) for v in (mean2d, radius, depth)]
    for cap in (b["n"], max(b["n"] - 1, 0)):
        assert cap <= 32768
        o = tc.tcgs_bin_sort(cam, *d, cap)
        assert int(o["n_splats"].item()) == b["n"]
        if cap == b["n"]:
            assert int(o["status"].item()) == 0
            assert (o["ids_sorted"].cpu().numpy()[:cap] == b["ids"]).all()
            got, ref = o["tile_ranges"].cpu().numpy(), b["ranges"]
            assert ((got == ref) | (ref[:, :1] == ref[:, 1:]) & (got[:, :1] == got[:, 1:])).all()
        else:
            assert int(o["status"].item()) == 3


def _tile_lists(o, gw, cols):
    """Lengths [rows, cols] and the concatenated ids of the lists of the first `cols` columns."""
    r = o["tile_ranges"].cpu().numpy().astype(np.int64).reshape(-1, gw, 2)[:, :cols]
    lens = r[..., 1] - r[..., 0]
    at = np.repeat(r[..., 0].ravel() - (np.cumsum(lens) - lens.ravel()), lens.ravel()) + np.arange(int(lens.sum()))
    return lens, o["ids_sorted"].cpu().numpy()[at]


@pytest.mark.parametrize("height", [640, 4096])
@pytest.mark.parametrize("mode", ["rectangles", "tiles", "rows"])
def test_row_lists_equal_radix_lists(tc, height, mode):
    """A view of 256 tile columns (sorted by row lists) against the same Gaussians in one of 257 (sorted by
    radix passes): every list of the common columns is the same.  Narrow and wide footprints, blocks of
    256 Gaussians with more runs than the kernels keep in shared memory, rows and columns of many chunks, and
    (exact coverage) conics that are not positive definite or hold a NaN, whose rows are reached in parts."""
    rng = np.random.default_rng(len(mode) + height)
    P = 3000
    wide = np.arange(P) % 3 == 0
    sigma = np.where(wide, rng.uniform(*((5, 20) if mode == "tiles" else (60, 220)), P), rng.uniform(0.5, 6, P))
    mean2d = np.stack([rng.uniform(-30, 3500, P), rng.uniform(-30, height + 30, P)], 1)
    mean2d[1500:2200] = rng.uniform(0, 300, (700, 2))       # long lists in a corner
    c = 0.9 * rng.uniform(-1, 1, P)
    conic = np.stack([1 / sigma ** 2, c / sigma ** 2, 1 / sigma ** 2], 1) / (1 - c * c)[:, None]
    odd = rng.choice(np.nonzero(mean2d[:, 0] < 2500)[0], 60, replace=False)
    conic[odd[:20], 1] = 2 * conic[odd[:20], 0]             # hyperbolic
    conic[odd[20:40], 0] *= -1
    conic[odd[40:]] = np.nan
    opacity = rng.uniform(0.003, 1, P)
    radius = np.ceil(3 * sigma).astype(np.int32)
    radius[rng.choice(P, 100, replace=False)] = 0
    mean2d, conic, opacity = f32(mean2d), f32(conic), f32(opacity)
    depth = f32(rng.integers(1, 500, P))
    d = [to_torch(v, DEV) for v in (mean2d, radius, depth)]
    exact = dict(conic=to_torch(conic, DEV), opacity=to_torch(opacity, DEV)) if mode != "rectangles" else {}
    n = int(oracle.bin_sort(scenes.pinhole(4112, height, fx=500.0), mean2d, radius, depth)["n"])
    # the capacity chooses the coverage by tiles or by rows in both paths
    cap = max(n, 32 * P) if mode != "tiles" else 32 * P - 1
    res = [tc.tcgs_bin_sort(scenes.pinhole(16 * gw, height, fx=500.0), *d, cap, **exact) for gw in (256, 257)]
    assert n <= cap
    assert int(res[0]["status"].item()) == int(res[1]["status"].item()) == 0
    (la, ia), (lb, ib) = _tile_lists(res[0], 256, 256), _tile_lists(res[1], 257, 256)
    assert (la == lb).all() and (ia == ib).all()
    assert la.sum() == int(res[0]["n_splats"].item())
    again = tc.tcgs_bin_sort(scenes.pinhole(4096, height, fx=500.0), *d, int(la.sum()) - 1, **exact)
    assert int(again["status"].item()) == 3
    if mode == "rectangles":
        assert int(again["n_splats"].item()) == la.sum()


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_project_backward_store_equals_accumulate(tc, degree):
    """Stored gradients are those added to zeroed arrays, unseen Gaussians' and whole unseen warps' included."""
    for P, behind in ((1, 1), (33, 5), (161, 2), (100, 100)):
        cam, sc = scenes.plain_forward(P=P, seed=50 + P)
        rng = np.random.default_rng(P)
        sc = dict(sc, sh=f32(rng.normal(0, 0.3, (P, (degree + 1) ** 2, 3))), sh_degree=degree)
        sc["means3"] = sc["means3"].copy()
        sc["means3"][::behind, 2] = -1.0
        if P == 161:
            sc["means3"][32:64, 2] = -1.0
        d = tc.scene_to_device(sc, DEV)
        pr = tc.tcgs_project(cam, d["means3"], d["scales"], d["quats"], d["sh"], degree)
        w = [to_torch(f32(rng.normal(size=(P, k))), DEV) for k in (2, 3, 3)]
        args = (cam, d["means3"], d["scales"], d["quats"], d["sh"], degree, pr["radius"], *w)
        zeros = {"d" + k: torch.zeros_like(d[k]) for k in ("means3", "scales", "quats", "sh")}
        added = tc.tcgs_project_bwd(*args, grads=zeros)
        for _ in range(2):      # fresh memory is not zero
            torch.full((P, 400), float("nan"), device=DEV)
            stored = tc.tcgs_project_bwd(*args)
            for k in added:
                assert torch.equal(stored[k], added[k]), (P, k)
