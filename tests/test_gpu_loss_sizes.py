"""The loss kernels' tiles are 32 x 8 pixels and their partial sums 1,024 blocks:
images of one pixel, one row or column, a tile's size and one more, and more
tiles than blocks, against the oracle; the adjoint may be written into the
image's own buffer.  Loss within 1e-6, blurred image and adjoint within 1e-6
of their largest entry (nine FP32 products), except where a residual is within
that rounding of zero, whose sign may differ."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2101_05356_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("w,h", [(1, 1), (1, 9), (33, 1), (2, 2), (32, 8), (33, 9), (64, 7), (1025, 300)])
def test_loss_matches_oracle(w, h):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    rng = np.random.default_rng(w * 1000 + h)
    img, tgt = (rng.uniform(0.0, 1.0, (h, w, 3)).astype(np.float32) for _ in range(2))
    r = facert.Renderer(dataclasses.replace(synth.make_scene("tiny"), width=w, height=h))
    di, dt = torch.as_tensor(img).cuda(), torch.as_tensor(tgt).cuda()
    loss, adj, bl = r.loss(di, dt)
    lo, blo, ado = oracle.loss(img.astype(np.float64), tgt)
    assert abs(loss.item() - lo) <= 1e-6 * lo
    assert np.max(np.abs(bl.cpu().numpy() - blo)) <= 1e-6
    unsure = np.abs(blo - tgt) <= 1e-6
    far = ~unsure
    for y in range(3):
        for x in range(3):
            far &= ~np.pad(unsure, ((1, 1), (1, 1), (0, 0)))[y:y + h, x:x + w]
    assert np.max(np.abs(adj.cpu().numpy() - ado)[far], initial=0.0) <= 1e-6
    own = di.clone()
    facert.fr_loss(r.ctx, own, dt, loss, own, None)          # the adjoint into the image's buffer
    assert torch.equal(own, adj)
