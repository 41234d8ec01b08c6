"""The linear models' kernels for one face and for a batch give a face bitwise
the same values, at the sizes where they change path: fewer rows than a chunk of
1,024, a chunk and a ragged rest, an odd number of columns (the transpose takes
two a warp), column counts around the 12 and 36 loads kept in flight, and
textures of 227^2 and 228^2 texels (the one-face morph keeps fewer loads in
flight above 4 blocks per SM).  Against FP64: the morph within (K + 2) 2^-24 of
the terms' magnitudes, the transpose within 1e-5 of them (FP32 sums of 1,024
rows in 13 additions at most, then FP64)."""
import dataclasses

import numpy as np
import pytest

from paper_2101_05356_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,k", [(4, 1), (18, 3), (19, 20), (37, 13), (64, 37), (227, 13), (228, 13), (228, 36)])
def test_one_face_equals_batch(m, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_05356_gb300 import facert
    rng = np.random.default_rng(m + k)
    basis = [rng.normal(size=(k, m, m, 3)).astype(np.float32) for _ in range(2)]
    mean = [rng.uniform(0.3, 0.7, (m, m, 3)).astype(np.float32) for _ in range(2)]
    sc = dataclasses.replace(synth.make_scene("tiny"), tex_size=m,
                             albedo=synth.AlbedoModel(mean[0], basis[0], mean[1], basis[1]))
    r = facert.Renderer(sc, max_batch=2)
    coef = torch.as_tensor(rng.normal(size=(2, 2, k)), dtype=torch.float32).cuda()
    grad = torch.as_tensor(rng.normal(size=(2, 2, m, m, 3)), dtype=torch.float32).cuda()

    def run(faces):
        tex = torch.empty(2, len(faces), m, m, 3, device="cuda")
        g = torch.zeros(2, len(faces), k, device="cuda")
        # (whole tensors per face: each must start on a 16-byte boundary)
        t = [[torch.empty(m, m, 3, device="cuda") for _ in faces] for _ in range(2)]
        gr = [[grad[q, f].clone() for f in faces] for q in range(2)]
        co = [[coef[q, f].clone() for f in faces] for q in range(2)]
        facert.fr_albedo_morph(r.ctx, co[0], co[1], t[0], t[1])
        facert.fr_albedo_adjoint(r.ctx, gr[0], gr[1], list(g[0]), list(g[1]))
        for q in range(2):
            for i in range(len(faces)):
                tex[q, i] = t[q][i]
        return tex, g

    tex, g = run([0, 1])
    for f in range(2):
        t1, g1 = run([f])
        assert torch.equal(t1[:, 0], tex[:, f]) and torch.equal(g1[:, 0], g[:, f])
        for q in range(2):
            b = basis[q].reshape(k, -1).astype(np.float64)
            c, gg = coef[q, f].cpu().numpy().astype(np.float64), grad[q, f].cpu().numpy().astype(np.float64).ravel()
            mag = np.abs(mean[q].ravel()) + np.abs(c) @ np.abs(b)
            err = np.abs(tex[q, f].cpu().numpy().ravel() - (mean[q].ravel().astype(np.float64) + c @ b))
            assert np.max(err / mag) <= (k + 2) * 2.0 ** -24
            assert np.max(np.abs(g[q, f].cpu().numpy() - b @ gg) / (np.abs(b) @ np.abs(gg))) <= 1e-5
