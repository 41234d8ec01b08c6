"""Plane bounds and rays from far away: a floor at depth `depth` lit by an
emitter near the camera, half of whose light a small screen parallel to the floor
takes.  The rays start at coordinates far above the screen's, and their height
over its plane is rounded there, while the bound's pad is only its own
magnitude's.  Every sample's visibility words against the oracle's brute force;
the screen's edges are met within about 2^-22 depth, 1e-3 of the emitter's width
at the farthest, so one sample in a hundred may differ."""
import numpy as np
import pytest

import oracle
from tests import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _scene(depth, by_coefficient):
    # (rays run from the floor to the emitter beside the view; the screen covers its left half)
    w = 0.6 * depth
    floor = [[-w, -w, -depth], [w, -w, -depth], [w, w, -depth], [-w, w, -depth]]
    screen = [[1.0, -1.0, -0.5], [1.5, -1.0, -0.5], [1.5, 1.0, -0.5], [1.0, 1.0, -0.5]]
    faces = [[0, 1, 2], [0, 2, 3], [4, 5, 6], [4, 6, 7]]
    light = scenes.quad_light([1.2, -0.3, -0.2], [0.0, 0.6, 0.0], [0.6, 0.0, 0.0])
    if np.cross(light[4:7], light[7:10])[2] > 0:
        light[4:7], light[7:10] = light[7:10].copy(), light[4:7].copy()
    move = np.zeros((1, 8, 3))
    if by_coefficient:                          # the mean's floor is near; the basis takes it to its depth
        move[0, :4] = np.asarray(floor) * (1.0 - 4.0 / depth) / 0.75
        floor = (np.asarray(floor) * (4.0 / depth)).tolist()
    sc, pr = scenes.make(floor + screen, faces, move, [light], width=24, height=24, spp=4)
    pr.coef = np.array([0.75 if by_coefficient else 0.0], np.float32)
    pr.focal = np.array([24.0], np.float32)
    return sc, pr


@pytest.mark.parametrize("by_coefficient", [False, True])
@pytest.mark.parametrize("depth", [4.0, 100.0, 300.0, 1000.0])
def test_screen_before_a_far_floor(depth, by_coefficient):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    sc, pr = _scene(depth, by_coefficient)
    _, ot, om = oracle.render(sc, pr, records=True)
    lit = (om[:, 0] != 0)
    assert 0.2 < np.mean(lit) < 0.8                   # the screen takes some of the light and leaves some
    for flags in (0, facert.FLAG_LBVH):
        r = facert.Renderer(sc, flags=flags)
        _, tri, mask = r.records(r.device_params(pr))
        same = (tri.cpu().numpy() == ot) & (mask.cpu().numpy().view(np.uint64) == om).all(axis=1)
        assert np.sum(~same) <= len(same) // 100, (flags, int(np.sum(~same)), len(same))
        assert r.status() == 0
