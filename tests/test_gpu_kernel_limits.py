"""Inputs at the limits of what the kernels' shortcuts may assume: needles, conics that are no ellipse, infinities,
oversized arrays, ill-formed lists."""
import numpy as np
import pytest

import oracle
from paper_2505_24796_gb300 import scenes

from .helpers import f32, to_torch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def tc():
    import paper_2505_24796_gb300 as m
    m._lib.load()
    return m


def _needle_conics(rng, sigma_long, n):
    """FP32 conics of needles `sigma_long` pixels long (n values) and under two wide, with the 0.3 px dilation, and the
    unit vectors along them."""
    s, th = rng.uniform(0.3, 2.0, n), rng.uniform(0, np.pi, n)
    c, d = np.cos(th), np.sin(th)
    A, B, C = ((c * sigma_long) ** 2 + (d * s) ** 2 + 0.3, c * d * (sigma_long ** 2 - s ** 2),
               (d * sigma_long) ** 2 + (c * s) ** 2 + 0.3)
    return f32(np.stack([C, -B, A], 1) / (A * C - B * B)[:, None]), np.stack([c, d], 1)


@pytest.mark.parametrize("kind", ["needles_100_400", "needles_500_1500", "hyperbolic", "nan"])
@pytest.mark.parametrize("early", [False, True])
def test_backward_replays_what_the_forward_blended(tc, kind, early):
    """One Gaussian a tile, of colour 1: the image is its alpha, and with dL/dimg = 1 in one channel its colour
    gradient is the sum of the tile's pixels (256 positive terms added by a tree of at most 12 roundings: 1e-6).
    Needles whose means lie 2 to 3.4 sigma along their axis from the tile, where the conic form cancels, and
    conics that are no ellipse."""
    rng = np.random.default_rng(len(kind))
    gw = gh = 64
    n = gw * gh
    cam = scenes.pinhole(16 * gw, 16 * gh, fx=500.0)
    centre = np.stack([np.arange(n) % gw, np.arange(n) // gw], 1) * 16.0 + 8.0
    if kind.startswith("needles"):
        lo, hi = (float(v) for v in kind.split("_")[1:])
        L = rng.uniform(lo, hi, n)
        conic, axis = _needle_conics(rng, L, n)
        mean2d = f32(centre + axis * (rng.choice([-1, 1], n) * rng.uniform(2, 3.4, n) * L)[:, None] + rng.uniform(-6, 6, (n, 2)))
    else:
        mean2d = f32(centre + rng.uniform(-40, 40, (n, 2)))
        conic = f32(np.tile([0.01, 0.5, 0.01] if kind == "hyperbolic" else [np.nan, 0.1, 0.2], (n, 1)))
    t = {k: to_torch(v, DEV) for k, v in dict(mean2d=mean2d, conic=conic, opacity=f32(rng.uniform(0.5, 0.99, n)),
                                              rgb=np.ones((n, 3), np.float32)).items()}
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    ranges = torch.stack([ids, ids + 1], 1).contiguous()
    opts = tc.render_opts("fp32", early_cull=early)
    args = (t["mean2d"], t["conic"], t["opacity"], t["rgb"])
    o = tc.tcgs_render_fwd(cam, opts, ranges, ids, *args)
    dl = torch.zeros_like(o["img"])
    dl[0] = 1
    g = tc.tcgs_render_bwd(cam, opts, ranges, ids, *args, o["img"], o["T_final"], o["n_contrib"], dl)
    alpha = o["img"][0].double().view(gh, 16, gw, 16).sum(dim=(1, 3)).view(-1)
    assert int((alpha > 0).sum()) > n // 20
    torch.testing.assert_close(g["drgb"][:, 0].double(), alpha, rtol=1e-6, atol=0)


@pytest.mark.parametrize("conic,mean", [((1e38, 0, 1e38), None), ((np.inf, 0, np.inf), None), ((np.nan, 0.1, 0.2), None),
                                        (None, (np.inf, 4)), (None, (4, -np.inf)), (None, (np.nan, 4)), (None, (3e38, 3e38))])
def test_backward_keeps_odd_geometry_where_it_is_not_blended(tc, conic, mean):
    """A conic that overflows at a pixel's offset, an infinity or a NaN in a conic or a mean: a pixel that does not
    blend the Gaussian, or blends it with a clamped alpha, adds nothing to the gradients of its geometry, and every
    other Gaussian's gradients stay finite."""
    rng = np.random.default_rng(2)
    n, cam = 24, scenes.pinhole(16, 16, fx=50.0)
    s = rng.uniform(2, 6, n)
    inp = dict(mean2d=f32(rng.uniform(0, 16, (n, 2))), conic=f32(np.stack([1 / s ** 2, 0 * s, 1 / s ** 2], 1)),
               opacity=f32(rng.uniform(0.05, 0.3, n)), rgb=f32(rng.uniform(0, 1, (n, 3))))
    inp["mean2d"][9] = 4    # between the pixel centres of the first block
    if conic is not None:
        inp["conic"][9] = f32(conic)
    if mean is not None:
        inp["mean2d"][9] = f32(mean)
    t = [to_torch(inp[k], DEV) for k in ("mean2d", "conic", "opacity", "rgb")]
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    ranges = torch.tensor([[0, n]], dtype=torch.int32, device=DEV)
    o = tc.tcgs_render_fwd(cam, tc.render_opts("fp32"), ranges, ids, *t)
    g = tc.tcgs_render_bwd(cam, tc.render_opts("fp32"), ranges, ids, *t, o["img"], o["T_final"], o["n_contrib"],
                           to_torch(f32(rng.standard_normal((3, 16, 16))), DEV))
    assert int(o["n_contrib"].max()) > 10
    for k, v in g.items():
        assert torch.isfinite(v).all(), k
    for k in ("dmean2d", "dconic", "dopacity"):
        assert (g[k][9] == 0).all(), k


@pytest.mark.parametrize("extra", ["sh", "scales", "quats"])
def test_project_backward_zeroes_rows_beyond_its_gaussians(tc, monkeypatch, extra):
    """Arrays with more rows than there are Gaussians: the rows that belong to none get a gradient of 0, whatever
    the memory held."""
    cam, sc = scenes.plain_forward(P=40, seed=3)
    d = tc.scene_to_device(sc, DEV)
    pr = tc.tcgs_project(cam, d["means3"], d["scales"], d["quats"], d["sh"], d["sh_degree"])
    d[extra] = torch.cat([d[extra], torch.ones_like(d[extra])])
    w = [torch.randn(40, k, device=DEV) for k in (2, 3, 3)]
    monkeypatch.setattr(torch, "empty_like", lambda t: torch.full_like(t, float("nan")))
    g = tc.tcgs_project_bwd(cam, d["means3"], d["scales"], d["quats"], d["sh"], d["sh_degree"], pr["radius"], *w)
    assert (g["d" + extra][40:] == 0).all()
    for k, v in g.items():
        assert torch.isfinite(v).all() and (v[:40] != 0).any(), k


def _lists(o, gw, cols):
    """Lengths and concatenated ids of the lists of the first `cols` of `gw` tile columns."""
    r = o["tile_ranges"].long().view(-1, gw, 2)[:, :cols].reshape(-1, 2)
    lens = r[:, 1] - r[:, 0]
    at = torch.repeat_interleave(r[:, 0] - (lens.cumsum(0) - lens), lens) + torch.arange(int(lens.sum()), device=DEV)
    return lens, o["ids_sorted"][at]


@pytest.mark.parametrize("P,seen", [(500_000, 60_000), (200_000, 20_000)])   # more and fewer than 10 blocks of 256 an SM
@pytest.mark.parametrize("kind", ["needles", "undilated", "axis", "round"])
def test_row_lists_of_needles_equal_radix_lists(tc, kind, P, seen):
    """Exact coverage tile by tile (fewer than 32 splats of capacity a Gaussian): a view of 256 tile columns, sorted by
    row lists, keeps the tiles of one of 257, whose radix passes test every tile of every rectangle, also for needles
    whose conic form cancels and whose rows are reached in parts."""
    rng = np.random.default_rng(len(kind))
    H = 1024
    L = np.exp(rng.uniform(*np.log([20, 60] if kind == "round" else [100, 1500]), seen))
    s = dict(needles=rng.uniform(0.3, 2, seen), undilated=rng.uniform(1e-3, 0.2, seen), axis=rng.uniform(0.3, 2, seen),
             round=0.8 * L)[kind]
    th = rng.uniform(-0.01, 0.01, seen) + np.pi / 2 * rng.integers(0, 2, seen) if kind == "axis" else rng.uniform(0, np.pi, seen)
    c, d, dil = np.cos(th), np.sin(th), 0.0 if kind == "undilated" else 0.3
    A, B, C = f32((c * L) ** 2 + (d * s) ** 2 + dil), f32(c * d * (L * L - s * s)), f32((d * L) ** 2 + (c * s) ** 2 + dil)
    det = A * C - B * B
    pad = lambda a, v: np.concatenate([f32(a), np.full((P - seen,) + a.shape[1:], v, np.float32)])  # noqa: E731
    conic = pad(np.stack([C, -B, A], 1) / np.where(det > 0, det, 1)[:, None], 1.0)
    mean2d = pad(np.stack([rng.uniform(-50, 3000, seen), rng.uniform(-50, H + 50, seen)], 1), 0.0)
    radius = np.zeros(P, np.int32)
    radius[:seen] = np.where(det > 0, np.minimum(np.ceil(3 * L), 1000), 0)
    t = [to_torch(v, DEV) for v in (mean2d, radius, f32(rng.integers(1, 500, P)))]
    exact = dict(conic=to_torch(conic, DEV), opacity=to_torch(pad(rng.uniform(0.003, 1, seen), 1.0), DEV))
    res = [tc.tcgs_bin_sort(scenes.pinhole(16 * gw, H, fx=500.0), *t, 32 * P - 1, **exact) for gw in (256, 257)]
    assert [int(o["status"].item()) for o in res] == [0, 0]
    (la, ia), (lb, ib) = _lists(res[0], 256, 256), _lists(res[1], 257, 256)
    assert int(la.sum()) == int(res[0]["n_splats"].item())
    assert int((la != lb).sum()) == 0 and torch.equal(ia, ib)


def test_inverted_ranges_are_empty_lists(tc):
    """A range whose end lies before its start holds no entry: background, no gradient, an empty list's features."""
    cam = scenes.pinhole(48, 32, fx=50.0)
    n = 40
    rng = np.random.default_rng(1)
    t = [to_torch(f32(v), DEV) for v in (rng.uniform(0, 48, (n, 2)), np.tile([0.1, 0, 0.1], (n, 1)), np.full(n, 0.5),
                                         np.ones((n, 3)), np.ones(n))]
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    empty = torch.zeros(6, 2, dtype=torch.int32, device=DEV)
    inverted = torch.tensor([[n, 0], [1, 0], [n - 1, 3], [0, 0], [7, 6], [n, n - 1]], dtype=torch.int32, device=DEV)
    radius = torch.full((n,), 5, dtype=torch.int32, device=DEV)
    res = []
    for r in (empty, inverted):
        o = tc.tcgs_render_fwd(cam, tc.render_opts("fp32"), r, ids, *t[:4], bg=(0.25, 0.5, 0.75))
        g = tc.tcgs_render_bwd(cam, tc.render_opts("fp32"), r, ids, *t[:4], o["img"], o["T_final"], o["n_contrib"],
                               torch.ones_like(o["img"]))
        res.append((*o.values(), *g.values(), tc.tcgs_tile_features(cam, r, ids, t[0], t[1], t[2], t[4], radius)))
    for a, b in zip(*res):
        assert torch.equal(a, b)


def test_fp32_paths_take_their_order_from_their_own_entry_points(tc):
    """The tensor-core renderer's order in the options, here one that names a tile twice and leaves one out, is not
    read by TCGS_FP32 and the backward; a permutation given to their ordered entry points changes neither image
    nor gradients (a Gaussian lies in one tile here, so that its sums do not depend on the tiles' order)."""
    cam = scenes.pinhole(64, 48, fx=50.0)
    rng = np.random.default_rng(4)
    n, nt = 240, 12
    tile = np.arange(n) // 20
    t = [to_torch(f32(v), DEV) for v in (np.stack([tile % 4 * 16, tile // 4 * 16], 1) + rng.uniform(0, 16, (n, 2)),
                                         np.tile([0.05, 0.01, 0.05], (n, 1)), rng.uniform(0.1, 0.6, n), rng.uniform(0, 1, (n, 3)))]
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    ranges = torch.stack([torch.arange(nt) * 20, torch.arange(1, nt + 1) * 20], 1).int().to(DEV)
    bad = torch.arange(nt, dtype=torch.int32, device=DEV)
    bad[3] = 5
    perm = torch.arange(nt - 1, -1, -1, dtype=torch.int32, device=DEV)
    counter = torch.zeros(1, dtype=torch.int32, device=DEV)
    dl = torch.randn(3, 48, 64, device=DEV)
    res = []
    for opts, order in ((tc.render_opts("fp32"), None), (tc.render_opts("fp32", tile_order=bad, work_counter=counter), None),
                        (tc.render_opts("fp32"), perm)):
        kw = ({}, {}) if order is None else (dict(fp32_order=order), dict(tile_order=order))
        o = dict(img=torch.full((3, 48, 64), -1.0, device=DEV), T_final=torch.full((48, 64), -1.0, device=DEV),
                 n_contrib=torch.full((48, 64), -1, dtype=torch.int32, device=DEV))
        tc.tcgs_render_fwd(cam, opts, ranges, ids, *t, out=o, **kw[0])
        g = tc.tcgs_render_bwd(cam, opts, ranges, ids, *t, o["img"], o["T_final"], o["n_contrib"], dl, **kw[1])
        res.append((*o.values(), *g.values()))
        for a, b in zip(res[0], res[-1]):
            assert torch.equal(a, b)
    with pytest.raises(tc.TcgsError):
        tc.tcgs_render_fwd(cam, tc.render_opts("tc_fp16_split"), ranges, ids, *t, fp32_order=perm)


@pytest.mark.parametrize("exact", [False, True])
def test_packed_tile_sort_of_wide_views(tc, exact):
    """A view of 257 x 40 tiles is sorted by radix passes: as key-value pairs below a capacity of 2^23 splats, from
    there on as packed (tile >> 8, id) words.  The same lists and ranges either way, the oracle's for rectangles, and
    in the common columns those of a view of 256 columns (row lists)."""
    rng = np.random.default_rng(6)
    P, H = 30_000, 640
    sigma = np.exp(rng.uniform(np.log(1), np.log(25), P))
    mean2d = f32(np.stack([rng.uniform(-30, 4140, P), rng.uniform(-30, H + 30, P)], 1))
    radius = np.where(rng.random(P) < 0.1, 0, np.ceil(3 * sigma)).astype(np.int32)
    depth = f32(rng.integers(1, 2000, P))
    conic = f32(np.stack([1 / sigma ** 2, 0.5 / sigma ** 2 * rng.uniform(-1, 1, P), 1 / sigma ** 2], 1))
    cams = {gw: scenes.pinhole(16 * gw, H, fx=500.0) for gw in (256, 257)}
    b = oracle.bin_sort(cams[257], mean2d, radius, depth)
    t = [to_torch(v, DEV) for v in (mean2d, radius, depth)]
    kw = dict(conic=to_torch(conic, DEV), opacity=to_torch(f32(rng.uniform(0.003, 1, P)), DEV)) if exact else {}
    assert b["n"] + 17 < 32 * P < 1 << 23
    res = [tc.tcgs_bin_sort(cams[gw], *t, cap, **kw) for gw, cap in ((257, b["n"] + 17), (257, 1 << 23), (256, b["n"] + 17))]
    assert [int(o["status"].item()) for o in res] == [0, 0, 0]
    n = int(res[0]["n_splats"].item())
    assert n == int(res[1]["n_splats"].item()) and (n < b["n"] if exact else n == b["n"])
    assert torch.equal(res[0]["ids_sorted"][:n], res[1]["ids_sorted"][:n])
    assert torch.equal(res[0]["tile_ranges"], res[1]["tile_ranges"])
    if not exact:
        np.testing.assert_array_equal(res[1]["ids_sorted"].cpu().numpy()[:n], b["ids"])
        np.testing.assert_array_equal(res[1]["tile_ranges"].cpu().numpy(), b["ranges"])
    for x, y in zip(_lists(res[1], 257, 256), _lists(res[2], 256, 256)):
        assert torch.equal(x, y)
