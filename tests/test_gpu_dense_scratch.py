"""Scratch of the modes that store T_LR in FP64 (fitted coefficients, the paper's forces): a memory budget
that fits the FP64 matrix, its digit planes and the pair coefficients is enough, whatever other
layout the default mode has.  The arena is the need and an eighth."""
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


def test_no_records_beside_fp64_blocks(lm):
    s = inputs.cluster(40, radius=8.0, min_sep=1.2, seed=40)
    args = (torch.tensor(s.positions, device="cuda"), None,
            torch.tensor(s.species, dtype=torch.int32, device="cuda"), torch.tensor(s.hirshfeld, device="cuda"))

    def need(setup, forces):
        m = lm.LMBD(s.table, lm.default_params(), 12, 6)
        setup(m)
        m.energy_forces(*args, forces=forces)
        return m.stats()["bytes_arena"] * 8 / 9, m

    series, m = need(lambda m: None, False)
    ns2 = int((m.site_counts(40)[:, 1].astype(int) ** 2).sum())
    # energies: 72 n_s^2 bytes of FP64 T_LR in the place of 32 of pair records
    fit, _ = need(lambda m: m.set_series_fit(12), False)
    assert abs(fit - series - 40 * ns2) < 4096
    # forces with FP64 products: 32 n_s^2 of pair coefficients (the paper's forces hold the same ones), and per
    # site 13 + 1 + 9 doubles, two more Krylov blocks of 3 x 36 and P and Q of 3 x 144
    ns = int(m.site_counts(40)[:, 1].sum())
    energies, _ = need(lambda m: m.set_precision(lm.PREC_FP64), False)
    forces, _ = need(lambda m: m.set_precision(lm.PREC_FP64), True)
    assert abs(forces - energies - 32 * ns2 - 8 * ns * (23 + 2 * 108 + 2 * 432)) < 8192
