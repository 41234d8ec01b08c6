"""fr_backward forks the part that needs only the geometry onto the context's
stream and joins it before the call's last work on the caller's, so it can be
recorded into a CUDA graph like the fused step; each replay equals the eager call bit
for bit, with records of the whole image in one pass, in tiles, and re-traced."""
import pytest

from paper_2101_05356_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("name,flags,tile", [("area", 0, 0), ("area", 0, 256), ("area", "recompute", 0), ("env", 0, 0)])
def test_backward_replays_from_a_cuda_graph(name, flags, tile):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    flags = facert.FLAG_RECOMPUTE if flags == "recompute" else flags
    sc = synth.make_scene("tiny", **(dict(env=(8, 2)) if name == "env" else {}))
    r = facert.Renderer(sc, flags=flags)
    if tile:
        facert.fr_debug_record_tile(r.ctx, tile)
    p = r.device_params(synth.random_params(sc, 4))
    adj = torch.randn(sc.height, sc.width, 3, generator=torch.Generator().manual_seed(1)).cuda()
    want = r.backward(p, adj, iteration=2)
    torch.cuda.synchronize()

    g = r.zero_grads(p)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.zero_()
        facert.fr_backward(r.ctx, p, adj, g, 2, 0)
    for _ in range(2):
        g.flat.fill_(7.0)
        graph.replay()
        torch.cuda.synchronize()
        for k in want:
            assert torch.equal(g[k], want[k]), k
    assert any(float(v.abs().max()) > 0.0 for v in want.values())
    assert r.status() == 0
