"""The any-hit traversal culls a BVH node whose plane bound the ray stays above
(csrc/refit.cu; csrc/lbvh.cu, k_planes).  A bound that cut off a triangle would
lose shadows, so every sample's visibility words are compared with the oracle's
brute force on triangle soups of the sizes where the bounds change hands: one
and two triangles, the 8 a thread takes and one more, the 256 of a refit block
and one more, the 4,096 a bound may span and more, at the face's scale and 50
times it, for both trees.  At most two samples may disagree (FP32 and FP64 flips
at triangle edges).  Overlapping
triangles of one plane tie for the camera ray's closest hit, which FP32 and
FP64 rounding then pick differently, so the flat soups compare the visibility
where the two sides' hits are the same triangle."""
import numpy as np
import pytest

import oracle
from tests import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _soup(n, scale, flat, seed=0):
    """n separate triangles facing the camera around z = -4, randomly tilted or
    all in two parallel planes (every mean normal equal), under three quads: one
    over the camera, one at the side, one grazing along the soup."""
    rng = np.random.default_rng(seed)
    size = 1.2 / np.sqrt(n) + 0.05
    c = rng.uniform([-1.5, -1.5, -4.4], [1.5, 1.5, -3.6], (n, 1, 3))
    if flat:
        c[..., 2] = np.where(rng.uniform(size=(n, 1)) < 0.3, -3.7, -4.3)
    off = rng.uniform(-size, size, (n, 3, 3))
    if flat:
        off[..., 2] = 0.0
    p = c + off
    nz = np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
    back = (nz * p[:, 0]).sum(1) > 0
    p[back] = p[back][:, ::-1]
    lights = [scenes.quad_light([0.2, 0.1, -1.0], [0.8, 0.0, 0.0], [0.0, -0.8, 0.0]),
              scenes.quad_light([2.5, 0.3, -3.0], [0.0, 0.6, 0.0], [0.0, 0.0, -0.6]),
              scenes.quad_light([0.0, 3.0, -3.9], [0.5, 0.0, 0.0], [0.0, 0.0, 0.5])]
    for r in lights:
        n_l = np.cross(r[4:7], r[7:10])
        if np.dot(n_l, np.array([0.0, 0.0, -4.0]) - r[1:4]) < 0:        # emit towards the soup
            r[4:7], r[7:10] = r[7:10].copy(), r[4:7].copy()
        r[1:10] *= scale
    sc, pr = scenes.make(p.reshape(-1, 3) * scale, np.arange(3 * n).reshape(n, 3), np.zeros((1, 3 * n, 3)),
                         lights, width=24, height=24, spp=4)
    pr.focal = np.array([24.0], np.float32)
    return sc, pr


@pytest.mark.parametrize("flat", [False, True])
@pytest.mark.parametrize("scale", [1.0, 50.0])
@pytest.mark.parametrize("n", [1, 2, 8, 9, 256, 257, 300, 4096, 5003])
def test_visibility_equals_brute_force(n, scale, flat):
    from paper_2101_05356_gb300 import facert
    sc, pr = _soup(n, scale, flat)
    _, ot, om = oracle.render(sc, pr, records=True)
    for flags in (0, facert.FLAG_LBVH):
        r = facert.Renderer(sc, flags=flags)
        _, tri, mask = r.records(r.device_params(pr))
        same = tri.cpu().numpy() == ot
        vis = (mask.cpu().numpy().view(np.uint64) == om).all(axis=1)
        agree = (vis | ~same) if flat else (vis & same)
        assert np.sum(~agree) <= 2, int(np.sum(~agree))
        assert r.status() == 0


def _with_far_chain(n, steps):
    """The soup with single triangles outside the view at distances 8^k along +-x, +-y and behind the camera: each
    split of the tree takes off few of them, so the soup's leaves lie deep."""
    sc, pr = _soup(n, 1.0, False)
    far = []
    for k in range(steps):
        d = 6.0 * 8.0 ** k
        for ax, sg in ((0, 1), (0, -1), (1, 1), (1, -1), (2, 1)):
            c = np.zeros(3)
            c[ax] = sg * d
            c[2] += 1.0
            far.append(c + 0.05 * d * np.array([[0, 0, 0], [1, 0, 0.3], [0, 1, 0.6]]))
    v = np.concatenate([sc.mean, np.concatenate(far)])
    m = len(v)
    return scenes.make(v, np.arange(m).reshape(-1, 3), np.zeros((1, m, 3)), sc.lights, width=24, height=24, spp=4)[0], pr


@pytest.mark.parametrize("n,steps", [(40, 3), (3000, 12), (3000, 14)])
def test_cover_of_deep_leaves(n, steps):
    """A warp's shadow rays start from the siblings of a leaf's ancestors, at most 23 of them; deeper leaves keep the
    topmost ones and the path's node below them."""
    from paper_2101_05356_gb300 import facert
    sc, pr = _with_far_chain(n, steps)
    _, ot, om = oracle.render(sc, pr, records=True)
    r = facert.Renderer(sc)
    dp = r.device_params(pr)
    out = torch.zeros(3, dtype=torch.int32, device="cuda")
    facert.fr_debug_bvh(r.ctx, dp, out)
    assert (out.cpu().tolist()[2] > 24) == (n > 1000)
    _, tri, mask = r.records(dp)
    agree = (tri.cpu().numpy() == ot) & (mask.cpu().numpy().view(np.uint64) == om).all(axis=1)
    assert np.sum(~agree) <= 2, int(np.sum(~agree))
    assert r.status() == 0
