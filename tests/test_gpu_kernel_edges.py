"""Kernels at the edges of their blocks, batches and dispatch rules, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from oracle import sched as osc
from paper_2505_24796_gb300 import scenes

from .helpers import f32, scene64, to_torch

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
