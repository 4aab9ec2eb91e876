"""Forces with fitted series coefficients at high order and many frequencies: c_n = s_n / rho^n grows by
2^100 and more between the lowest and the highest frequency, while the Krylov vectors it multiplies fall.
The sliced products (series adjoint with digit planes up to 32 frequencies, sliced FP64 P and Q beyond, the
tcgen05 and the warp-level products) against the same library's FP64 products, with the tolerances of
the parity suite: 1e-10 relative for energies, 1e-8 eV/Angstrom for forces."""
import pytest
import torch

from paper_2407_06409_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lm():
    from paper_2407_06409_gb300 import build, lmbd
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lmbd


@pytest.mark.parametrize("warp", [False, True])
@pytest.mark.parametrize("n_freq,order", [(12, 6), (12, 10), (24, 10), (32, 3), (32, 8), (40, 8)])
def test_forces_match_fp64_products(lm, n_freq, order, warp):
    s = inputs.cluster(40, radius=8.0, min_sep=1.2, seed=40)
    args = (torch.tensor(s.positions, device="cuda"), None,
            torch.tensor(s.species, dtype=torch.int32, device="cuda"), torch.tensor(s.hirshfeld, device="cuda"))

    def run(**kw):
        m = lm.LMBD(s.table, lm.default_params(), n_freq, order)
        m.set_series_fit(12)
        if kw.get("fp64"):
            m.set_precision(lm.PREC_FP64)
        if kw.get("warp"):
            m.set_mma_path(lm.MMA_WARP)
        return m.energy_forces(*args)

    e0, f0 = run(fp64=True)
    e, f = run(warp=warp)
    assert (e - e0).abs().max().item() <= 1e-10 * e0.abs().max().item()
    assert (f - f0).abs().max().item() < 1e-8
