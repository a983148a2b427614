"""A launch that the runtime refuses is reported by the call that made it and by no other: the
library's later calls and the program's own work on the device go on as before.

The refused launch is the kernel application over 65,536 crops, one more than a grid's z extent
holds: the runtime returns an error and nothing of it runs."""
import pytest
import torch

from paper_2312_06827_gb300 import svgf

pytestmark = pytest.mark.gpu


def test_refused_launch_leaves_no_error_behind():
    B, H, W = 65536, 1, 3
    k = svgf.KPN(B * H * W)
    k.init_params(seed=1)
    feats = torch.zeros(B, H, W, 16, dtype=torch.int16, device="cuda")
    c0, out = torch.rand(B, H, W, 4, device="cuda"), torch.empty(B, H, W, 4, device="cuda")
    d = svgf.Denoiser(svgf.default_config(40, 24))
    cv, rgb = torch.rand(24, 40, 4, device="cuda"), torch.empty(24, 40, 4, device="cuda")
    torch.cuda.synchronize()
    for call in (lambda: k.forward(feats, c0, out), lambda: k.compute_grad(feats, c0, c0)):
        with pytest.raises(svgf.SvgfError):
            call()
        d.inverse_tonemap(cv, rgb)                      # a launcher that reads the last error
        with pytest.raises(svgf.SvgfError):
            call()
        assert float((rgb + 1.0).isfinite().float().mean()) == 1.0   # so does the program's own launch
    assert k.check_device() == 0
    half = B // 2
    k.forward(feats[:half], c0[:half], out[:half])      # the handle works on
    assert bool(out[:half, ..., :3].isfinite().all())
