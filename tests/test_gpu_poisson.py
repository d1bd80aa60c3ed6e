"""The Hartree energy from the spectrum of the density (no potential asked
for) against the grid sum of the potential, on even and odd transform lengths."""
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_2108_13478_gb300 as dft  # noqa: E402


@pytest.mark.parametrize("name", ["tiny2", "tiny8"])     # 54 and 75 points along x
@pytest.mark.parametrize("model", [dft.DFT_MODEL_NEUTRAL, 0])
def test_energies_without_the_potential(name, model):
    ctx = dft.Context(w.config_system(name), model=model, xc=dft.DFT_XC_PW92)
    n = ctx.initial_density()
    n *= 1.0 + 0.3 * torch.rand(n.shape, dtype=n.dtype, device=n.device, generator=torch.Generator("cuda").manual_seed(1))
    v, with_v = ctx.hartree_xc(n)
    without = dft.dft_hartree_xc(ctx.ctx, n, None)
    ctx.close()
    # both are sums of 1e5 .. 1e6 FP64 terms after FP64 transforms (sqrt(N) eps of their
    # size); the neutral Hartree terms have both signs on the grid side and are ~1e-2 of their sum of moduli
    for a, b in zip(with_v, without):
        assert abs(a - b) < 1e-11 * max(1.0, abs(a))
