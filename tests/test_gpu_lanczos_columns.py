"""Lanczos intervals of the polynomial-fit coefficients at the edges of their kernel: one row tile
and a ragged one, more rows than threads, products shorter than one summation chunk, and
frequency counts around the 4, 8 and 12 columns of a pass, against the oracle at the parity
tolerance for energies (1e-10 relative)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2407_06409_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lm():
    from paper_2407_06409_gb300 import build, lmbd
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lmbd


@pytest.mark.parametrize("n, n_freq", [(2, 12), (3, 4), (11, 5), (11, 1), (22, 8), (22, 9), (43, 13), (86, 3), (172, 2)])
def test_energies_match_oracle(lm, n, n_freq):
    s = inputs.cluster(n, radius=2.2 * n ** (1.0 / 3.0), min_sep=1.2, seed=n)
    p = lm.default_params(r_scs=3.0, r_mbd1=30.0, r_mbd2=30.0, r_sphere=30.0)
    model = lm.LMBD(s.table, p, n_freq, 5)
    model.set_series_fit(9)
    e, _ = model.energy_forces(torch.tensor(s.positions, device="cuda"), None,
                               torch.tensor(s.species, dtype=torch.int32, device="cuda"),
                               torch.tensor(s.hirshfeld, device="cuda"), forces=False)
    po = oracle.Params(r_scs=p.r_scs, r_mbd1=p.r_mbd1, r_mbd2=p.r_mbd2, r_sphere=p.r_sphere, r_buf=p.r_buf,
                       r_inner=p.r_inner, beta=p.beta, d=p.d, n_freq=n_freq, series_order=5,
                       omega_scale=p.omega_scale, lanczos_steps=9)
    ref = oracle.System(s.positions, None, s.species, s.hirshfeld, s.table, po).energies()
    assert np.abs(e.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
