"""The energy of fr_adam's texture groups, an FP64 number, against the exact sum
(rational arithmetic) of its FP32 terms' squares and magnitudes times the weights.

Up to 32 texels (one warp) are summed in more bits than FP64 has and rounded once
into it: 2^-52 of the total bounds that.  Near the ends of FP32's range (texels
whose energies are finite one by one but not when a warp's 32 are added; squares
that underflow) the terms are FP64, some forty additions a texel: 2^-45."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _energy(x, width, **weights):
    from paper_2101_05356_gb300 import facert
    z = [torch.zeros_like(x) for _ in range(3)]
    reg = torch.zeros(1, dtype=torch.float64, device="cuda")
    kind = facert.GROUP_TEX_MONO if x.dim() == 2 else facert.GROUP_TEX_RGB
    facert.fr_adam([facert.opt_group(x, z[0], z[1], z[2], kind=kind, width=width, lr=0.0, step=1, **weights)],
                   reg_energy=reg)
    return reg.item()


@pytest.mark.parametrize("value", [2e18, 3e18, 1e19, 1.8e19])
@pytest.mark.parametrize("m", [5, 16, 33])
def test_energy_whose_warp_sum_overflows(m, value):
    got = _energy(torch.full((m, m), value, device="cuda"), m, w_box=1.0)
    want = m * m * float(np.float32(value)) ** 2
    assert abs(got - want) <= 2.0 ** -45 * want
    got = _energy(torch.full((m, m, 3), -value / 2, device="cuda"), m, w_box=1.0)
    want = 3 * m * m * float(np.float32(-value / 2)) ** 2
    assert abs(got - want) <= 2.0 ** -45 * want


def _exact(x, ref, w_smooth, w_sym, w_chroma, w_box):
    """The energy of texture x [m, m, c] as a rational number; differences and quotients are the kernel's FP32 ones."""
    f = np.float32
    def total(terms, power):
        return sum((Fraction(float(v)) ** power for v in np.abs(terms).ravel()), Fraction(0))
    e = 2 * Fraction(float(f(w_smooth))) * (total(x[1:] - x[:-1], 2) + total(x[:, 1:] - x[:, :-1], 2))
    e += Fraction(float(f(w_sym))) * total(x - x[:, ::-1], 1)
    if w_chroma:
        s, s0 = (((q[..., 0] + q[..., 1]) + q[..., 2]) + f(1e-6) for q in (x, ref))
        e += Fraction(float(f(w_chroma))) * total(x / s[..., None] - ref / s0[..., None], 1)
    return e + Fraction(float(f(w_box))) * (total(np.minimum(x, f(0)), 2) + total(np.maximum(x - f(1), f(0)), 2))


@pytest.mark.parametrize("scale,bound", [(1.0, 2.0 ** -52), (1e-9, 2.0 ** -52), (1e6, 2.0 ** -52), (1e-17, 2.0 ** -45),
                                         (1e-21, 2.0 ** -45), (1e-25, 2.0 ** -45), (1e20, 2.0 ** -45)])
@pytest.mark.parametrize("c", [1, 3])
@pytest.mark.parametrize("m", [2, 3, 4, 5])
def test_energy_is_as_exact_as_fp64(m, c, scale, bound):
    for seed in range(8):
        rng = np.random.default_rng(100 * m + 10 * c + seed)
        x = (scale * rng.uniform(-0.2, 1.2, (m, m, c))).astype(np.float32)
        ref = rng.uniform(0.2, 0.8, (m, m, c)).astype(np.float32)
        # (the chromaticity is of order one at any scale: it would hide the small squares and, like the box, large ones)
        w = dict(w_smooth=0.0123, w_sym=0.3 if scale == 1.0 else 0.0, w_chroma=0.3 if c == 3 and scale == 1.0 else 0.0,
                 w_box=0.7)
        from paper_2101_05356_gb300 import facert
        d = torch.as_tensor(x if c == 3 else x[..., 0]).cuda()
        z = [torch.zeros_like(d) for _ in range(3)]
        reg = torch.zeros(1, dtype=torch.float64, device="cuda")
        facert.fr_adam([facert.opt_group(d, z[0], z[1], z[2], aux=torch.as_tensor(ref).cuda() if c == 3 else None,
                                         kind=facert.GROUP_TEX_RGB if c == 3 else facert.GROUP_TEX_MONO, width=m, lr=0.0,
                                         step=1, **w)], reg_energy=reg)
        want = _exact(x, ref, **w)
        assert abs(Fraction(reg.item()) - want) <= Fraction(bound) * want, seed
