"""The 7x7 variance estimate of short histories where its weights change form: normals so close
that log(1 - t) takes the power series, around the switch to log1pf at t = 1/32, far apart and
opposed, in images smaller than the window and across tile edges.

The reference is the estimate's definition in FP64, E_w[S] + Var_w[mu1] on a first frame (S = 0),
with the variance formed from deviations: the oracle's difference of moments cancels to 0 where
all but the centre's weight is below 1e-16, which these normals reach."""
import numpy as np
import pytest
import torch

from paper_2312_06827_gb300 import svgf
from parity import VAR_TOL

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
LUMA = np.array([0.2126, 0.7152, 0.0722])


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def first_frame_variance(luma, gbuf, sigma_z, sigma_n, eps, r=3):
    h, w = luma.shape
    z = gbuf[..., 3]
    gx, gy = (np.gradient(z, axis=1) if w > 1 else 0 * z), (np.gradient(z, axis=0) if h > 1 else 0 * z)
    out = np.zeros((h, w))
    for y in range(h):
        for x in range(w):
            ys, xs = slice(max(0, y - r), y + r + 1), slice(max(0, x - r), x + r + 1)
            dy, dx = np.mgrid[ys, xs][:, :h - ys.start, :w - xs.start] - np.array([y, x])[:, None, None]
            q = gbuf[ys, xs]
            t = np.minimum(0.5 * ((q[..., :3] - gbuf[y, x, :3]) ** 2).sum(-1), 1.0)
            with np.errstate(divide="ignore"):
                e = sigma_n * np.log1p(-t) - np.abs(q[..., 3] - z[y, x]) / (
                    sigma_z * np.abs(gx[y, x] * dx + gy[y, x] * dy) + eps)
            wt, m = np.exp(e), luma[ys, xs]
            mean = (wt * m).sum() / wt.sum()
            out[y, x] = (wt * (m - mean) ** 2).sum() / wt.sum()
    return out


@pytest.mark.parametrize("w,h", [(1, 1), (3, 9), (33, 8), (40, 21), (97, 35)])
@pytest.mark.parametrize("spread", [0.02, 0.18, 1.5])
@pytest.mark.parametrize("sigma_n", [2.0, 128.0])
def test_weights_around_the_series_switch(w, h, spread, sigma_n):
    rng = np.random.default_rng([w, h, int(100 * spread)])
    n = np.array([0.0, 0.0, 1.0]) + spread * rng.standard_normal((h, w, 3))
    n /= np.linalg.norm(n, axis=-1, keepdims=True)
    z = 5.0 + 0.02 * np.arange(w)[None, :] + 0.01 * rng.standard_normal((h, w))
    gbuf = np.concatenate([n, z[..., None]], -1).astype(np.float32)
    noisy = rng.exponential(1.0, (h, w, 3)).astype(np.float32)
    motion, rough = np.zeros((h, w, 2), np.float32), np.full((h, w), 0.5, np.float32)
    cfg = svgf.default_config(w, h)
    cfg.sigma_n = sigma_n
    d = svgf.Denoiser(cfg)
    cv = torch.empty(h, w, 4, device="cuda")
    d.reproject_accumulate(svgf.make_frame(dev(noisy), dev(gbuf), dev(motion), dev(rough)), cv)
    got = cv[..., 3].cpu().numpy().astype(np.float64)
    l = noisy.astype(np.float64) @ LUMA
    l = l / (1.0 + l)
    ref = first_frame_variance(l, gbuf.astype(np.float64), cfg.sigma_z, sigma_n, float(np.float32(cfg.eps)))
    # the stage's bar: 1e-5 of the value, and the rounding that FP32 luminances carry
    tol = VAR_TOL * ref + 8 * U * l.max() * np.sqrt(ref)
    assert np.all(np.abs(got - ref) <= tol), np.abs(got - ref).max()


@pytest.mark.parametrize("radius", [2, 3])
def test_large_luminances_without_tone_map(radius):
    """Linear radiances whose square is past FP32's range but whose variance is not: the estimate is
    formed from deviations and stays finite."""
    w, h = 35, 10
    rng = np.random.default_rng(radius)
    gbuf = np.zeros((h, w, 4), np.float32)
    gbuf[..., 2], gbuf[..., 3] = 1.0, 5.0
    noisy = (3e19 * (1.0 + 1e-3 * rng.standard_normal((h, w, 3)))).astype(np.float32)
    cfg = svgf.default_config(w, h)
    cfg.tonemap, cfg.spatial_var_radius = 0, radius
    d = svgf.Denoiser(cfg)
    cv = torch.empty(h, w, 4, device="cuda")
    d.reproject_accumulate(svgf.make_frame(dev(noisy), dev(gbuf), dev(np.zeros((h, w, 2))), dev(np.full((h, w), 0.5))), cv)
    got = cv[..., 3].cpu().numpy().astype(np.float64)
    l = noisy.astype(np.float64) @ LUMA
    ref = first_frame_variance(l, gbuf.astype(np.float64), cfg.sigma_z, cfg.sigma_n, float(np.float32(cfg.eps)), radius)
    tol = VAR_TOL * ref + 8 * U * l.max() * np.sqrt(ref)
    assert np.all(np.abs(got - ref) <= tol), np.abs(got / ref - 1).max()


def first_frame(noisy, gbuf, cfg):
    """The temporal stage's colour + variance and the luminances it estimated the variance from."""
    h, w = gbuf.shape[:2]
    d = svgf.Denoiser(cfg)
    cv, hist, mom = (torch.empty(h, w, 4, device="cuda") for _ in range(3))
    d.reproject_accumulate(svgf.make_frame(dev(noisy), dev(gbuf), dev(np.zeros((h, w, 2))), dev(np.full((h, w), 0.5))), cv)
    d.history_export(hist, mom)
    return cv[..., 3].cpu().numpy().astype(np.float64), mom[..., 0].cpu().numpy().astype(np.float64)


def test_small_noise_on_a_large_mean():
    """Noise of 0.1 % of the luminance: the estimate's rounding is of the size of the deviations, not of
    the luminance.  Against the definition in FP64 from the FP32 luminances themselves.

    The bar, u = 2^-24: depth is constant and |e| < 1, so a weight is off by at most 40 u (the bound
    of one tap), which moves a weighted variance by at most twice that; the deviations, sums, quotients
    and merges 48 u."""
    w, h = 90, 40
    rng = np.random.default_rng(11)
    n = np.array([0.0, 0.0, 1.0]) + 0.1 * rng.standard_normal((h, w, 3))
    n /= np.linalg.norm(n, axis=-1, keepdims=True)
    gbuf = np.concatenate([n, np.full((h, w, 1), 5.0)], -1).astype(np.float32)
    cfg = svgf.default_config(w, h)
    cfg.sigma_n = 2.0
    got, l = first_frame(0.7 * (1.0 + 1e-3 * rng.standard_normal((h, w, 3))), gbuf, cfg)
    ref = first_frame_variance(l, gbuf.astype(np.float64), cfg.sigma_z, cfg.sigma_n, float(np.float32(cfg.eps)))
    assert np.all(np.abs(got - ref) <= 128 * U * ref), np.abs(got / ref - 1.0).max() / U


@pytest.mark.parametrize("radius", [1, 3, 7])
@pytest.mark.parametrize("sigma_n,what", [(1.0, "depth"), (1.0, "normal"), (128.0, "normal")])
def test_one_tap_weight_against_fp64(radius, sigma_n, what):
    """The weight w of a single tap, read off the variance of two samples 0 and m, w m^2 / (1 + w)^2:
    pairs of pixels of one row, so far apart (opposed normals between them) that nothing else has
    weight.  `depth` sweeps exp(e) over e = 0 .. -85, `normal` (1 - t)^sigma_n through t = 0 .. 1/32,
    where log(1 - t) is a series, and on to 0.2.

    The bar, u = 2^-24, to first order.  Of w: exp 6 u (ex2.approx 4 u, the correction 2 u); an
    exponent e that is off by some k u |e| moves w by k u |e|: the FP32 depth or t 4 u, the
    logarithm 3 u, their product 1 u.  Of the variance from w: the two sums and the mean 2 u each, the
    deviation twice, the products, the merge of the rows and the final quotients 12 u.  In all
    8 u |e| + 24 u; taken as 8 u |e| + 32 u.

    Roundings have no sign, and the exponential unit's bias (-0.85 u over most of `depth`'s range) is put
    back by half a unit: that leaves 0.35 u, and the mean of 500 roundings of 1 u rms another 0.05 u, of
    which five are allowed: 0.6 u."""
    n, step = 500, 2 + radius
    w = n * step
    s = np.linspace(0.0, 1.0, n)
    gbuf = np.zeros((1, w, 4), np.float32)
    gbuf[..., 2] = -1.0                                    # between the pairs
    a, b = np.arange(n) * step, np.arange(n) * step + 1
    gbuf[0, a, 2] = 1.0
    if what == "depth":
        gbuf[0, b, 2] = 1.0
        gbuf[0, b, 3] = 85.0 * s                          # eps = 1, sigma_z = 0: e = -|dz|
    else:
        t = np.where(s < 0.8, s / 0.8 / 32.0, 1 / 32.0 + (s - 0.8) / 0.2 * (0.2 - 1 / 32.0))
        gbuf[0, b, 0], gbuf[0, b, 2] = np.sqrt(t * (2.0 - t)), 1.0 - t
    noisy = np.zeros((1, w, 3), np.float32)
    noisy[0, b] = 1.0
    cfg = svgf.default_config(w, 1)
    cfg.tonemap, cfg.spatial_var_radius = 0, radius
    cfg.sigma_z, cfg.sigma_n, cfg.eps = 0.0, sigma_n, 1.0
    got, l = (x[0] for x in first_frame(noisy, gbuf, cfg))
    g = gbuf[0].astype(np.float64)
    t = 0.5 * ((g[a, :3] - g[b, :3]) ** 2).sum(-1)
    e = sigma_n * np.log1p(-t) - np.abs(g[a, 3] - g[b, 3])
    wt = np.exp(e)
    ref = wt * l[b] ** 2 / (1.0 + wt) ** 2
    for p in (a, b):
        rel = np.abs(got[p] / ref - 1.0)
        assert np.all(rel <= U * (8.0 * np.abs(e) + 32.0)), (rel / U / (8.0 * np.abs(e) + 32.0)).max()
        if what == "depth":
            assert abs(np.mean(got[p] / ref - 1.0)) <= 0.6 * U


@pytest.mark.parametrize("radius", [2, 3])
def test_infinite_depth_tolerance(radius):
    """sigma_z = infinity: along a depth gradient the depth term is 0; where there is none its denominator,
    infinity times 0, is not a number and the tap, the centre among them, has weight 0."""
    w, h = 40, 20
    rng = np.random.default_rng(5)
    gbuf = np.zeros((h, w, 4), np.float32)
    gbuf[..., 2] = 1.0
    gbuf[..., 3] = 5.0 + 0.25 * np.arange(w)               # no gradient along y, exactly representable
    gbuf[:, 30:, 3] = 9.0                                  # none at all
    cfg = svgf.default_config(w, h)
    cfg.sigma_z, cfg.sigma_n, cfg.spatial_var_radius = np.inf, 2.0, radius
    got, l = first_frame(rng.exponential(1.0, (h, w, 3)), gbuf, cfg)
    ref = np.zeros((h, w))
    gx, gy = np.gradient(gbuf[..., 3].astype(np.float64), axis=1), np.gradient(gbuf[..., 3].astype(np.float64), axis=0)
    for y in range(h):
        for x in range(w):
            ys, xs = slice(max(0, y - radius), min(h, y + radius + 1)), slice(max(0, x - radius), min(w, x + radius + 1))
            dy, dx = np.mgrid[ys, xs] - np.array([y, x])[:, None, None]
            wt = (gx[y, x] * dx + gy[y, x] * dy != 0.0).astype(np.float64)
            if wt.sum() > 0:
                m = (wt * l[ys, xs]).sum() / wt.sum()
                ref[y, x] = (wt * (l[ys, xs] - m) ** 2).sum() / wt.sum()
    tol = VAR_TOL * ref + 8 * U * l.max() * np.sqrt(ref)
    assert np.all(np.abs(got - ref) <= tol), np.abs(got - ref).max()
