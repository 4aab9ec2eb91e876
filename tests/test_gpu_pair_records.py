"""Pair records, T_LR digit planes and the tcgen05 pair adjoint at the edges of their tiles: sphere
sizes around 16 / 42 sites (pair tiles), 64 / 128 sites (partner chunks) and single pairs, all pairs
coupled and split cutoffs, against the same library's FP64 products (which read FP64 blocks and
coefficients instead of the records).  Tolerances of the parity suite: 1e-10 relative for
energies, 1e-8 eV/Angstrom for forces."""
import numpy as np
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


def _case(lm, n, r_mbd2):
    s = inputs.cluster(n, radius=2.2 * n ** (1.0 / 3.0), min_sep=1.2, seed=n)
    p = lm.default_params(r_scs=3.0, r_mbd1=30.0, r_mbd2=r_mbd2, r_sphere=30.0)
    args = (torch.tensor(s.positions, device="cuda"), None,
            torch.tensor(s.species, dtype=torch.int32, device="cuda"), torch.tensor(s.hirshfeld, device="cuda"))
    return s, args, lambda: lm.LMBD(s.table, p, 4, 5)


@pytest.mark.parametrize("n", [1, 2, 3, 16, 17, 42, 43, 64, 65, 128, 129, 205])
@pytest.mark.parametrize("r_mbd2", [30.0, 4.0])
def test_sphere_sizes_match_fp64_products(lm, n, r_mbd2):
    s, args, model = _case(lm, n, r_mbd2)
    ref = model()
    ref.set_precision(lm.PREC_FP64)
    e0, f0 = ref.energy_forces(*args)
    m = model()
    e, f = m.energy_forces(*args)
    assert m.site_counts(n)[:, 1].min() == n           # every sphere holds every atom
    assert (e - e0).abs().max().item() <= 1e-10 * e0.abs().max().item()
    assert (f - f0).abs().max().item() < 1e-8
    e1, _ = model().energy_forces(*args, forces=False)
    assert torch.equal(e1, e)


@pytest.mark.parametrize("power", [-200, -60, 60, 200])
def test_weights_of_any_magnitude(lm, power):
    s, args, model = _case(lm, 43, 30.0)
    w = torch.linspace(0.5, 1.5, 43, device="cuda", dtype=torch.float64)
    _, f0 = model().energy_forces(*args, weights=w)
    _, f = model().energy_forces(*args, weights=w * 2.0 ** power)
    assert (f * 2.0 ** -power - f0).abs().max().item() < 1e-12
