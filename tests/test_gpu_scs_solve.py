"""Screening solves and their adjoint at the edges of their kernels: one, two and three warps of
sites per system (|K1| = 32 / 33, 64 / 65, 96), a group of warps per right-hand side (few systems)
and all three right-hand sides together (many), and the adjoint contraction with its frequencies
split over blocks and taken in chunks.

Every atom of these free clusters lies within r_SCS of every other, so |K1| = n for every centre.
Central polarisabilities within 1e-12 relative of the oracle, forces within 1e-8 eV/Angstrom of the
oracle or of central differences of the library's energies (4-point stencil, h = 2e-3 Angstrom:
truncation ~1e-10, rounding ~1e-10 eV/Angstrom).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2407_06409_gb300 import inputs

pytestmark = pytest.mark.gpu

TABLE = np.array([[3.0, 8.0, 3.3], [2.5, 6.0, 3.1], [3.5, 10.0, 3.6]])


@pytest.fixture(scope="module")
def lm():
    from paper_2407_06409_gb300 import build, lmbd
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lmbd


def _case(lm, n, n_freq):
    s = inputs.cluster(n, radius=4.0, min_sep=1.1, seed=n)
    p = lm.default_params(r_scs=9.0, r_mbd1=9.0, r_mbd2=9.0, r_sphere=9.0)
    model = lm.LMBD(TABLE, p, n_freq, 3)
    args = [None, torch.tensor(s.species, dtype=torch.int32, device="cuda"), torch.tensor(s.hirshfeld, device="cuda")]
    op = oracle.Params(r_scs=9.0, r_mbd1=9.0, r_mbd2=9.0, r_sphere=9.0, n_freq=n_freq, series_order=3)
    return s, model, args, oracle.System(s.positions, None, s.species, s.hirshfeld, TABLE, op)


def _check_alpha(model, so, n, atoms):
    a = model.central_polarizabilities(n).numpy()[atoms]
    ref = np.stack([v.numpy() for v in so.central_alpha(atoms).values()])
    assert model.site_counts(n)[:, 0].min() == n          # |K1| = n everywhere
    assert model.stats()["scs_lu_systems"] == 0
    assert np.allclose(a, ref, rtol=1e-12, atol=0)


@pytest.mark.parametrize("n", [1, 2, 32, 33, 64, 65])
def test_few_systems_match_the_oracle(lm, n):
    s, model, args, so = _case(lm, n, 3)
    w = np.zeros(n)
    w[0] = 1.0
    _, f = model.energy_forces(torch.tensor(s.positions, device="cuda"), *args,
                               weights=torch.tensor(w, device="cuda"))
    _check_alpha(model, so, n, list(range(min(n, 8))))
    _, f_ref = so.energies_forces(centres=[0])
    assert np.abs(f.cpu().numpy() - f_ref).max() < 1e-8


@pytest.mark.parametrize("n,n_freq", [(30, 63), (64, 30), (96, 40)])
def test_many_systems_match_central_differences(lm, n, n_freq):
    s, model, args, so = _case(lm, n, n_freq)
    pos = torch.tensor(s.positions, device="cuda")
    _, f = model.energy_forces(pos, *args)
    _check_alpha(model, so, n, [0, n - 1])
    h = 2e-3
    for atom, d in ((0, 0), (n - 1, 2)):
        def total(shift):
            x = pos.clone()
            x[atom, d] += shift
            return float(model.energy_forces(x, *args, forces=False)[0].sum())
        ref = -(8.0 * (total(h) - total(-h)) - (total(2 * h) - total(-2 * h))) / (12.0 * h)
        assert abs(float(f[atom, d]) - ref) < 1e-8
