"""The facing classes behind the shadow-edge candidates (csrc/render.cu,
k_face_class) where the kernel changes path: environment blocks narrower than half
a turn (whose range comes from cross products), half a turn wide and wider (from
angles), area emitters alone (the kernel without the blocks' code) and both
together.  Candidate lists equal the oracle's."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2101_05356_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _scene(env, block, area):
    sc = synth.make_scene("tiny", n_lights=max(area, 1))
    if env:
        rec, d, a = synth.env_blocks(env, block)
        keep = slice(0, area)
        sc = dataclasses.replace(sc, lights=np.concatenate([sc.lights[keep], rec]),
                                 light_d=np.concatenate([sc.light_d[keep], d]),
                                 light_a=np.concatenate([sc.light_a[keep], a]), env_size=env)
    return sc


@pytest.mark.parametrize("env,block,area", [(0, 0, 1), (0, 0, 9), (8, 2, 0), (8, 4, 0), (8, 8, 0), (12, 6, 0), (12, 4, 3),
                                            (32, 16, 9), (30, 15, 0), (9, 3, 7)])
def test_candidates_equal_the_oracles(env, block, area):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    sc = _scene(env, block, area)
    pr = synth.random_params(sc, 3)
    r = facert.Renderer(sc)
    n, e = sc.lights.shape[0], r.n_edges
    prim, n_prim = torch.empty(e, dtype=torch.int32, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda")
    per, counts = torch.empty((n, e), dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
    facert.fr_debug_silhouettes(r.ctx, r.device_params(pr), prim, n_prim, per, counts)
    _, want = oracle.silhouettes(sc, pr)
    c, got = counts.cpu().numpy(), per.cpu().numpy()
    for j in range(n):
        assert np.array_equal(got[j, :c[j]], want[j]), j
