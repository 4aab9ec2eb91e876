"""T_LR, W, P and Q digit planes written as tile images, the persistent chain kernel and the series
adjoint at the edges of their shapes: frequency counts around the 16-column and 32-frequency limits,
every series order with its own mix of 5- and 6-digit steps, products of one K step, a partial
one and several chunks, and more tiles than blocks.  Compared with the same library's FP64 products
at the tolerances of the parity suite: 1e-10 relative for energies, 1e-8 eV/Angstrom for forces."""
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


def _compare(lm, s, n_freq, order):
    p = lm.default_params(r_scs=3.0, r_mbd1=30.0, r_mbd2=6.0, r_sphere=30.0)
    args = (torch.tensor(s.positions, device="cuda"), None,
            torch.tensor(s.species, dtype=torch.int32, device="cuda"), torch.tensor(s.hirshfeld, device="cuda"))
    ref = lm.LMBD(s.table, p, n_freq, order)
    ref.set_precision(lm.PREC_FP64)
    e0, f0 = ref.energy_forces(*args)
    e, f = lm.LMBD(s.table, p, n_freq, order).energy_forces(*args)
    assert (e - e0).abs().max().item() <= 1e-10 * e0.abs().max().item()
    assert (f - f0).abs().max().item() < 1e-8


@pytest.mark.parametrize("n_freq", [1, 2, 5, 10, 11, 15, 16, 17, 31, 32, 33, 64])
@pytest.mark.parametrize("n", [5, 47])
def test_frequency_counts(lm, n, n_freq):
    _compare(lm, inputs.cluster(n, radius=2.2 * n ** (1.0 / 3.0), min_sep=1.2, seed=n), n_freq, 6)


@pytest.mark.parametrize("order", [3, 4, 5, 7, 8, 9, 10])
@pytest.mark.parametrize("n", [11, 86, 171])
def test_series_orders(lm, n, order):
    # 171 atoms: 513 rows, five row tiles a centre, more tiles than SMs
    _compare(lm, inputs.cluster(n, radius=2.2 * n ** (1.0 / 3.0), min_sep=1.2, seed=n), 12, order)
