"""Calls whose launches are chained (each may start before its predecessor has completed): captured by
the caller into a CUDA graph and replayed, and interleaved on two streams, they give what the same
calls give one after the other."""
import numpy as np
import pytest
import torch

from paper_2312_06827_gb300 import scene, svgf

pytestmark = pytest.mark.gpu

KEYS = ("noisy", "gbuf_nz", "motion", "roughness")


def frames_of(w, h, n, seed=5):
    sc = scene.SceneConfig(w, h, n_spheres=8, moving_sphere=True, seed=seed)
    out, prev = [], None
    for t in range(n):
        f = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in scene.render_frame(sc, t, KEYS).items()}
        out.append(svgf.make_frame(f["noisy"], f["gbuf_nz"], f["motion"], f["roughness"], prev))
        prev = f["gbuf_nz"]
    return out


@pytest.mark.parametrize("mode", [svgf.ATROUS_5X5, svgf.SEPARABLE])
def test_captured_frame_equals_direct_frame(mode):
    w, h = 333, 140
    cfg = svgf.default_config(w, h)
    cfg.spatial_mode = mode
    frames = frames_of(w, h, 3)
    a, b = svgf.Denoiser(cfg), svgf.Denoiser(cfg)
    side = torch.cuda.Stream()
    for t, f in enumerate(frames):
        oa, ob = torch.empty(h, w, 4, device="cuda"), torch.zeros(h, w, 4, device="cuda")
        a.denoise_frame(f, oa)
        torch.cuda.synchronize()
        if t == 0:
            b.denoise_frame(f, ob)
        else:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                b.denoise_frame(f, ob)
            g.replay()
        torch.cuda.synchronize()
        assert torch.equal(oa, ob), t


def test_captured_forward_equals_direct_forward():
    B, H, W = 2, 37, 150
    k = svgf.KPN(B * H * W)
    k.init_params(seed=1, last_scale=1.0)
    rng = np.random.default_rng(2)
    feats = torch.from_numpy(rng.standard_normal((B, H, W, 16)).astype(np.float32)).cuda().bfloat16().view(torch.int16)
    c0 = torch.from_numpy(rng.random((B, H, W, 4)).astype(np.float32)).cuda()
    oa, ob = torch.empty(B, H, W, 4, device="cuda"), torch.zeros(B, H, W, 4, device="cuda")
    k.forward(feats, c0, oa)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        k.forward(feats, c0, ob)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(oa, ob) and k.check_device() == 0


def test_two_streams_interleaved_equal_one_after_the_other():
    w, h = 260, 200
    cfg = svgf.default_config(w, h)
    seqs = [frames_of(w, h, 4, seed=s) for s in (5, 6)]
    want = []
    for fs in seqs:
        d = svgf.Denoiser(cfg)
        outs = [torch.empty(h, w, 4, device="cuda") for _ in fs]
        for f, o in zip(fs, outs):
            d.denoise_frame(f, o)
        torch.cuda.synchronize()
        want.append(outs)
    ds, streams = [svgf.Denoiser(cfg) for _ in seqs], [torch.cuda.Stream() for _ in seqs]
    got = [[torch.empty(h, w, 4, device="cuda") for _ in fs] for fs in seqs]
    torch.cuda.synchronize()
    for t in range(4):
        for i in range(2):
            ds[i].denoise_frame(seqs[i][t], got[i][t], stream=streams[i])
    torch.cuda.synchronize()
    for i in range(2):
        for t in range(4):
            assert torch.equal(want[i][t], got[i][t]), (i, t)


@pytest.mark.parametrize("fresh", [True, False])
def test_captured_learned_frame_equals_direct_frame(fresh):
    """The longest chain: ten launches, and on a handle's first use a memset between two of them."""
    w, h = 333, 140
    frames = frames_of(w, h, 2)
    albedo = torch.from_numpy(np.random.default_rng(3).random((h, w, 3)).astype(np.float32)).cuda()
    outs = []
    for captured in (False, True):
        d, k = svgf.Denoiser(svgf.default_config(w, h)), svgf.KPN(w * h, train=False)
        k.init_params(seed=4, last_scale=1.0)
        o = torch.zeros(h, w, 4, device="cuda")
        if fresh:
            d.denoise_frame(frames[0], o)
        else:
            k.denoise_frame(d, frames[0], albedo, o)
        torch.cuda.synchronize()
        o.zero_()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=torch.cuda.Stream()):
                k.denoise_frame(d, frames[1], albedo, o)
            g.replay()
        else:
            k.denoise_frame(d, frames[1], albedo, o)
        torch.cuda.synchronize()
        assert k.check_device() == 0
        outs.append(o)
    assert float(outs[0][..., :3].abs().max()) > 0
    assert torch.equal(*outs)


@pytest.mark.parametrize("fresh", [True, False])
def test_captured_training_step_equals_direct_step(fresh):
    """One block adds up each sum here, so that the order of its additions is the same on every run."""
    B, H, W = 1, 1, 30
    rng = np.random.default_rng(7)
    feats = torch.from_numpy(rng.standard_normal((B, H, W, 16)).astype(np.float32)).cuda().bfloat16().view(torch.int16)
    c0, target = (torch.from_numpy(rng.random((B, H, W, 4)).astype(np.float32)).cuda() for _ in range(2))
    got = []
    for captured in (False, True):
        k = svgf.KPN(B * H * W)
        k.init_params(seed=1, last_scale=1.0)
        if not fresh:
            k.train_step(feats, c0, target)
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=torch.cuda.Stream()):
                loss = k.train_step(feats, c0, target)
            g.replay()
        else:
            loss = k.train_step(feats, c0, target)
        torch.cuda.synchronize()
        assert k.check_device() == 0
        got.append([x.clone() for x in (loss, k.grad, k.params, k.adam_m, k.adam_v)])
    assert float(got[0][1].abs().max()) > 0
    for a, b in zip(*got):
        assert torch.equal(a, b)
