"""Plane bounds of the per-call tree (FLAG_LBVH; csrc/lbvh.cu, k_planes) where the
launch changes: trees around the 512 and the 1,024 triangles a bound may span, trees whose nodes
get a warp each and trees with many to a warp, alone and as a batch (fewer blocks a
face).  Bounds only cull, so images are bitwise those of the static tree, whose
camera hits and visibility do not depend on the tree."""
import pytest

from tests.test_gpu_plane_bounds import _soup

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,faces", [(2, 3), (511, 1), (512, 1), (513, 1), (514, 40), (1100, 2), (9000, 1), (16383, 1), (16384, 1), (20011, 64)])
def test_images_equal_the_static_trees(n, faces):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    sc, pr = _soup(n, 1.0, False)
    images = []
    for flags in (0, facert.FLAG_LBVH):
        r = facert.Renderer(sc, flags=flags, max_batch=faces)
        p = r.device_params(pr)
        tgt = torch.zeros(sc.height, sc.width, 3, device="cuda")
        items = [dict(width=sc.width, height=sc.height, spp=sc.spp, edge_spp=1, flags=flags, iteration=k, face_id=k,
                      params=p, target=tgt, image=torch.zeros_like(tgt),
                      loss=torch.zeros(1, dtype=torch.float64, device="cuda"), grads=None) for k in range(faces)]
        facert.fr_render_batch(r.ctx, items)
        images.append(torch.stack([it["image"] for it in items]))
        assert r.status() == 0
    assert float(images[0].abs().sum()) > 0.0
    assert torch.equal(images[0], images[1])
