"""The energy of fr_adam's texture groups near the end of FP32's range: texels
whose energies are finite in FP32 one by one but not when a warp's 32 are added.
The sums behind the kernel's exact terms are FP64, some forty additions a texel,
so 2^-45 of the total bounds their rounding."""
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
