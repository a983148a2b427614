"""The weight and bias gradients at the edges of the tensor-core kernel's tiles: images of a few pixels,
around the 16-pixel product and the 128-pixel column, of a few rows and of more chunks than one
block takes, against the oracle with BF16 values where the kernels keep them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2312_06827_gb300 import svgf

pytestmark = pytest.mark.gpu


def bits(x):
    return torch.from_numpy(x).cuda().bfloat16()


@pytest.mark.parametrize("B,H,W", [(1, 1, 3), (2, 3, 15), (1, 2, 16), (3, 5, 17), (1, 40, 127), (2, 7, 129), (1, 9, 300),
                                   (40, 3, 260)])
def test_gradients_at_tile_edges(B, H, W):
    rng = np.random.default_rng([B, H, W])
    k = svgf.KPN(B * H * W)
    k.init_params(seed=3, last_scale=1.0)
    feats = np.zeros((B, H, W, 16), np.float32)
    feats[..., :10] = rng.standard_normal((B, H, W, 10))
    fb = bits(feats)
    c0 = rng.random((B, H, W, 4)).astype(np.float32)
    target = rng.random((B, H, W, 4)).astype(np.float32)
    k.compute_grad(fb.view(torch.int16), torch.from_numpy(c0).cuda(), torch.from_numpy(target).cuda())
    assert k.check_device() == 0
    got = k.grad.cpu().numpy().astype(np.float64)
    _, ref = oracle.kpn_grad(fb.float().cpu().numpy()[..., :10], c0[..., :3], target[..., :3],
                             k.params.cpu().numpy().astype(np.float64), quant=True)
    off = 0
    for ci, co in zip(svgf.KPN_CIN, svgf.KPN_COUT):
        for n in (co * 9 * ci, co):                      # the layer's weights, then its biases
            g, o = got[off:off + n], ref[off:off + n]
            off += n
            # the bar of the per-layer gradient tests: 1 % of the norm (BF16 rounding boundaries that
            # FP32 and FP64 sums fall on either side of)
            assert np.linalg.norm(g - o) <= 0.01 * np.linalg.norm(o), (ci, co, n)


@pytest.mark.parametrize("B,H,W", [(700, 2, 20), (330, 9, 40), (110, 2, 300), (1300, 1, 17)])
def test_gradients_of_more_chunks_than_blocks(B, H, W):
    """More 128-pixel columns than the grid's blocks, so that the blocks take several chunks one after
    the other and carry their rings' slots and phases from one to the next."""
    blocks = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert B * -(-W // 128) > blocks                     # a chunk is then a whole column
    test_gradients_at_tile_edges(B, H, W)
