"""Launches of few blocks share a sample's shadow rays over a block's warps
(csrc/api.cu, split_lights); larger ones, and images above 32 samples a pixel,
do not.  A batch of copies of a small face crosses the line that the face alone
stays under, for the forward and for the primary edges, so the images must be
bitwise the single render's and the gradients its own (their sums are fixed
point: equal too); ragged sizes, light counts that leave a warp without a
light, two visibility words, environment blocks."""
import numpy as np
import pytest

from paper_2101_05356_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SCENES = {
    "1 light": dict(n_lights=1),
    "3 lights": dict(n_lights=3),
    "40 lights": dict(n_lights=40),
    "66 lights": dict(n_lights=66),
    "environment": dict(env=(8, 2)),
}


@pytest.mark.parametrize("w,h,spp", [(24, 24, 2), (37, 29, 16), (50, 41, 32)])
@pytest.mark.parametrize("name", list(SCENES))
def test_split_equals_unsplit(name, w, h, spp):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    sc = synth.make_scene("tiny", width=w, height=h, spp=spp, **SCENES[name])
    n = 64
    r = facert.Renderer(sc, max_batch=n, edge_spp=2)
    p = r.device_params(synth.random_params(sc, 1))
    tgt = torch.rand(h, w, 3, generator=torch.Generator().manual_seed(0)).cuda()
    image, loss, grads = r.render(p, tgt, iteration=2)
    items = [dict(width=w, height=h, spp=spp, edge_spp=2, iteration=2, face_id=0, params=p, target=tgt,
                  image=torch.zeros(h, w, 3, device="cuda"), loss=torch.zeros(1, dtype=torch.float64, device="cuda"),
                  grads=r.zero_grads(p)) for _ in range(n)]
    facert.fr_render_batch(r.ctx, items)
    for it in (items[0], items[n // 2], items[-1]):
        assert torch.equal(it["image"], image) and torch.equal(it["loss"], loss)
        for k, g in grads.items():
            if k in ("coef", "rot", "trans"):        # FP64 sums of the vertex gradients, not fixed point
                assert torch.allclose(it["grads"][k], g, rtol=1e-5, atol=1e-5 * float(g.abs().max()))
            else:
                assert torch.equal(it["grads"][k], g), k
    assert r.status() == 0
