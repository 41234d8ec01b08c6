"""fr_adam's texture groups at the sizes where their kernels change path, and
the energy's arithmetic: sides of one texel up, an odd side (the middle column
has no mirror image), arrays that are not 16-byte aligned (the update then goes
element by element), no energy wanted, and texels whose squares overflow FP32.
Moments and parameters against the FP64 definitions of oracle/optim.py within
1e-5 (relative to the largest entry: FP32 differences of numbers near one, some
ten roundings of 6e-8 each, times the weights); the energy within 1e-6 (the
FP32 differences that are squared).  The chromaticity divides by a texel's
channel sum twice, so texels whose sum is under 0.3 (the random textures have
sums near zero) amplify the roundings beyond that estimate and are left out of
the moments' comparison."""
import numpy as np
import pytest

from oracle import optim as ora

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
W = dict(w_smooth=0.0002, w_sym=0.3, w_chroma=0.3, w_box=1.0)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _dev(a, shift):
    """Device copy that starts `shift` elements past an aligned address."""
    buf = torch.zeros(a.size + 4, dtype=torch.float32, device="cuda")
    v = buf[shift:shift + a.size].view(a.shape)
    v.copy_(torch.as_tensor(a))
    return v


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("energy", [True, False])
@pytest.mark.parametrize("m", [1, 2, 15, 16, 33])
def test_texture_groups(m, energy, shift):
    from paper_2101_05356_gb300 import facert
    rng = np.random.default_rng(m)
    groups, want, e_want = [], [], 0.0
    for c in (3, 1):
        shp = (m, m, 3) if c == 3 else (m, m)
        x, g, mo = (rng.uniform(-0.2, 1.2, shp), rng.normal(size=shp), 0.1 * rng.normal(size=shp))
        v, ref = 0.01 * rng.uniform(0.1, 1.0, shp), rng.uniform(0.2, 0.8, shp)
        x, g, mo, v, ref = (a.astype(np.float32) for a in (x, g, mo, v, ref))
        d = [_dev(a, shift) for a in (x, mo, v, g, ref)]
        kw = dict(W) if c == 3 else dict(w_smooth=W["w_smooth"], w_box=1.0)
        groups.append((facert.opt_group(d[0], d[1], d[2], d[3], aux=d[4] if c == 3 else None, width=m, lr=5e-3, step=7,
                                        kind=facert.GROUP_TEX_RGB if c == 3 else facert.GROUP_TEX_MONO, **kw), d))
        f = [a.astype(np.float64) for a in (x, g, mo, v, ref)]
        wk = [kw["w_smooth"], kw.get("w_sym", 0.0), kw.get("w_chroma", 0.0), kw["w_box"]]
        r0 = f[4] if c == 3 else None
        fine = np.broadcast_to(np.abs(f[0].sum(axis=-1, keepdims=True)) >= 0.3, shp) if c == 3 else np.ones(shp, bool)
        want.append((fine,) + ora.adam(f[0], f[1] + ora.tex_grad(f[0], *wk, r0), f[2], f[3], 7, 5e-3))
        e_want += ora.tex_energy(f[0], *wk, r0)
    reg = torch.zeros(1, dtype=torch.float64, device="cuda")
    facert.fr_adam([g for g, _ in groups], reg_energy=reg if energy else None)
    for (_, d), w in zip(groups, want):
        fine = w[0]
        for got, ref in zip(d[:3], w[1:]):
            err = np.abs(got.cpu().numpy() - ref)[fine]
            assert np.max(err, initial=0.0) <= 1e-5 * max(1.0, np.abs(ref[fine]).max(initial=0.0))
    if energy:
        assert abs(reg.item() - e_want) <= 1e-6 * max(e_want, 1e-3)


def test_energy_of_texels_whose_squares_overflow():
    from paper_2101_05356_gb300 import facert
    x = torch.zeros(4, 4, device="cuda")
    x[1, 2] = 3e25
    z = [torch.zeros(4, 4, device="cuda") for _ in range(3)]
    reg = torch.zeros(1, dtype=torch.float64, device="cuda")
    facert.fr_adam([facert.opt_group(x, z[0], z[1], z[2], kind=facert.GROUP_TEX_MONO, width=4, lr=0.0, w_smooth=0.5,
                                     w_box=1.0, step=1)], reg_energy=reg)
    big = float(np.float32(3e25)) ** 2
    assert abs(reg.item() - (0.5 * 8 * big + big)) <= 1e-6 * 5 * big        # 4 neighbours, each pair twice; the box
