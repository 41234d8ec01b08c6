"""Images and losses are stored whole, whatever their buffers held: buffers full
of NaN give bitwise what zeroed ones do, at the sample counts where the pixel's
sum changes hands (lanes of a warp, warps of a block, two blocks), with light
splitting (the small image) and without, and for a face that covers few pixels."""
import pytest

from paper_2101_05356_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("w,h", [(1, 1), (37, 29), (130, 65)])
@pytest.mark.parametrize("spp", [1, 16, 32, 64, 128, 256])
def test_outputs_are_stored(w, h, spp):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    sc = synth.make_scene("tiny", width=w, height=h, spp=spp)
    r = facert.Renderer(sc)
    p = r.device_params(synth.random_params(sc, 1))
    tgt = torch.rand(h, w, 3, generator=torch.Generator().manual_seed(0)).cuda()
    out = []
    for fill in (0.0, float("nan")):
        img, fwd = (torch.full((h, w, 3), fill, device="cuda") for _ in range(2))
        loss, alone = (torch.full((1,), fill, dtype=torch.float64, device="cuda") for _ in range(2))
        facert.fr_forward(r.ctx, p, fwd, 2)
        facert.fr_render(r.ctx, p, tgt, img, loss, None, 2)
        facert.fr_loss(r.ctx, img, tgt, alone)
        out.append((img, fwd, loss, alone))
    for a, b in zip(*out):
        assert torch.isfinite(b).all() and torch.equal(a, b)
    assert r.status() == 0
