"""A face's gradients do not depend on whether its launches share a sample's
shadow rays over a block's warps (csrc/api.cu, split_lights).  The focal length's
is a sum over all edge samples in units of 2^-32; under lights of intensity 1e-5
it is so small that FP32 holds every unit of it, so a sum rounded at different
places would show.  The face alone stays under the line for the split and the
batch is above it, for the forward and the primary edges, on any GPU of 64 to 256
multiprocessors (the lines lie between 1 and 14 blocks of 128 threads for each)."""
import pytest

from paper_2101_05356_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_lights", [8, 20, 40, 66])
def test_focal_gradient_alone_and_in_a_batch(n_lights):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    w, h, spp, n = 48, 40, 16, 64
    sc = synth.make_scene("tiny", width=w, height=h, spp=spp, n_lights=n_lights)
    r = facert.Renderer(sc, max_batch=n, edge_spp=2)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edge_blocks, blocks = 2 * 2 * w * h // 128, w * h * spp // 128
    assert edge_blocks <= 1 * sms and n * edge_blocks > 6 * sms
    assert blocks <= 5 * sms and n * blocks > 16 * sms
    pr = synth.random_params(sc, 1)
    pr.light_i = pr.light_i * 1e-5
    p = r.device_params(pr)
    tgt = torch.rand(h, w, 3, generator=torch.Generator().manual_seed(0)).cuda()
    for iteration in range(4):
        image, _, grads = r.render(p, tgt, iteration=iteration)
        items = [dict(width=w, height=h, spp=spp, edge_spp=2, iteration=iteration, face_id=0, params=p, target=tgt,
                      image=torch.zeros(h, w, 3, device="cuda"), loss=torch.zeros(1, dtype=torch.float64, device="cuda"),
                      grads=r.zero_grads(p)) for _ in range(n)]
        facert.fr_render_batch(r.ctx, items)
        for it in (items[0], items[-1]):
            assert torch.equal(it["image"], image)
            assert float(grads["focal"].abs()) > 0.0
            assert torch.equal(it["grads"]["focal"], grads["focal"]), (it["grads"]["focal"], grads["focal"])
    assert r.status() == 0


@pytest.mark.parametrize("width,height", [(48, 40), (331, 290)])
def test_focal_gradient_is_linear_in_the_lights(width, height):
    """The primary edges' focal gradient under lights dimmed by 2^-20 is 2^-20 of the gradient (every product scales
    exactly): sums kept to 2^-32 would be off by 1e-4 of it, kept to 2^-64 the FP32 result's rounding is left."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    sc = synth.make_scene("tiny", width=width, height=height, n_lights=40)
    r = facert.Renderer(sc, flags=facert.FLAG_NO_INTERIOR | facert.FLAG_NO_SHADOW_EDGE | facert.FLAG_NO_SPECULAR_EDGE)
    pr = synth.random_params(sc, 1)
    adj = torch.randn(height, width, 3, generator=torch.Generator().manual_seed(0)).cuda()
    g = []
    for scale in (1.0, 2.0 ** -20):
        p = r.device_params(pr)
        p["light_i"] = p["light_i"] * scale
        g.append(float(r.backward(p, adj, iteration=1)["focal"]) / scale)
    assert abs(g[0]) > 0.0 and abs(g[1] - g[0]) <= 2e-7 * abs(g[0]), g


@pytest.mark.parametrize("spp", [1, 2, 4, 32])
@pytest.mark.parametrize("n_lights", [2, 5, 11, 40, 66])
def test_image_alone_and_in_a_batch(n_lights, spp):
    """One sample a pixel (32 pixels a block of the split form) to 32, with light counts from every part of the lines."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    n = 64
    w, h = {1: (83, 75), 2: (61, 56), 4: (45, 41), 32: (17, 15)}[spp]
    sc = synth.make_scene("tiny", width=w, height=h, spp=spp, n_lights=n_lights)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = (w * h * spp + 127) // 128
    assert blocks <= sms and n * blocks > 16 * sms
    r = facert.Renderer(sc, max_batch=n)
    p = r.device_params(synth.random_params(sc, 2))
    tgt = torch.zeros(h, w, 3, device="cuda")
    image, _, _ = r.render(p, tgt, iteration=3, with_grad=False)
    items = [dict(width=w, height=h, spp=spp, edge_spp=1, iteration=3, face_id=0, params=p, target=tgt,
                  image=torch.full((h, w, 3), -1.0, device="cuda"), loss=torch.zeros(1, dtype=torch.float64, device="cuda"),
                  grads=None) for _ in range(n)]
    facert.fr_render_batch(r.ctx, items)
    for it in (items[0], items[n // 2], items[-1]):
        assert torch.equal(it["image"], image)
    assert float(image.abs().sum()) > 0.0 and r.status() == 0
