"""Weights (upstream gradients) at the ends of the FP64 range or not finite, and polarisabilities that turn negative: the call
returns, the forces that depend on them are NaN, and all others are those of the same call without them.

Two clusters 200 Angstrom apart share no site list, so the weights of one never reach the other.  Once
with few screening systems (a group of warps per right-hand side) and once with many (63 frequencies:
three right-hand sides together); on the LU fallback (a polarisation catastrophe); and with the digit
planes of the warp-level path.  Finite weights scaled by a power of two scale the forces, to 1e-12
eV/Angstrom of the unscaled ones (rounding is relative; the smallest scale leaves 2^-60 of a force)."""
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


def _args(pos, species, nu):
    return (torch.tensor(pos, device="cuda"), None, torch.tensor(species, dtype=torch.int32, device="cuda"),
            torch.tensor(nu, device="cuda"))


def _two_clusters():
    a, b = inputs.cluster(24, seed=1), inputs.cluster(24, seed=2)
    pos = np.concatenate([a.positions, b.positions + [200.0, 0.0, 0.0]])
    return a.table, _args(pos, np.concatenate([a.species, b.species]), np.concatenate([a.hirshfeld, b.hirshfeld])), pos


def _check(f, ref, pos, k, r):
    """Atom k and its neighbours within r have NaN forces, the second cluster its own."""
    near = np.flatnonzero(np.linalg.norm(pos - pos[k], axis=1) < r)
    assert len(near) > 3
    assert torch.isnan(f[near]).all()
    assert (f[24:] - ref[24:]).abs().max().item() < 1e-12


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n_freq", [12, 63])
@pytest.mark.parametrize("path", ["tc05", "warp", "fp64"])
def test_weights_that_are_not_finite(lm, bad, n_freq, path):
    table, args, pos = _two_clusters()
    model = lm.LMBD(table, lm.default_params(r_scs=5.0, r_mbd1=5.0, r_mbd2=5.0, r_sphere=5.0), n_freq, 6)
    if path == "warp":
        model.set_mma_path(lm.MMA_WARP)
    elif path == "fp64":
        model.set_precision(lm.PREC_FP64)
    w = torch.linspace(0.5, 1.5, 48, device="cuda", dtype=torch.float64)
    e0, ref = model.energy_forces(*args, weights=w)
    w[3] = bad
    e, f = model.energy_forces(*args, weights=w)
    assert torch.equal(e, e0)
    _check(f, ref, pos, 3, 5.0)


def test_backward_of_an_overflowed_loss(lm):
    table, args, pos = _two_clusters()
    model = lm.LMBD(table, lm.default_params(r_scs=5.0, r_mbd1=5.0, r_mbd2=5.0, r_sphere=5.0), 12, 6)
    x = args[0].clone().requires_grad_(True)
    e = lm.lmbd_energy(x, model, *args[1:])
    w = torch.ones_like(e)
    w[3] = float("inf")
    (e * w).sum().backward()
    ref = model.energy_forces(*args)[1]
    _check(-x.grad, ref, pos, 3, 5.0)


def test_lu_fallback(lm):
    n = 6
    rng = np.random.default_rng(7)
    pos = np.zeros((n, 3))
    pos[:, 2] = 1.4 * np.arange(n)
    pos += rng.normal(scale=0.03, size=pos.shape)
    cell = torch.tensor(np.diag([20.0, 20.0, 1.4 * n]), device="cuda")
    model = lm.LMBD(np.array([[90.0, 30.0, 3.0]]), lm.default_params(r_scs=4.0, r_mbd1=5.0, r_mbd2=5.0, r_sphere=5.0), 4, 4)
    args = (torch.tensor(pos, device="cuda"), cell, torch.zeros(n, dtype=torch.int32, device="cuda"),
            torch.ones(n, dtype=torch.float64, device="cuda"))
    w = torch.ones(n, dtype=torch.float64, device="cuda")
    w[0] = float("nan")
    e, f = model.energy_forces(*args, weights=w)
    assert model.stats()["scs_lu_systems"] == n
    assert torch.isfinite(e).all() and torch.isnan(f).all()


def test_negative_polarisabilities(lm):
    s = inputs.box(64, seed=6, jitter=0.05)
    table = s.table.copy()
    table[:, 0] *= 3.0
    model = lm.LMBD(table, lm.default_params(), 12, 6)
    e, f = model.energy_forces(torch.tensor(s.positions, device="cuda"), torch.tensor(s.cell, device="cuda"),
                               torch.tensor(s.species, dtype=torch.int32, device="cuda"),
                               torch.tensor(s.hirshfeld, device="cuda"))
    assert (model.central_polarizabilities(64).numpy() < 0).any()
    assert torch.isnan(e).all() and torch.isnan(f).all()


@pytest.mark.parametrize("path", ["tc05", "warp"])
@pytest.mark.parametrize("power", [-1000, -950, 920, 990])
def test_weights_at_the_ends_of_the_range(lm, power, path):
    table, args, _ = _two_clusters()
    model = lm.LMBD(table, lm.default_params(r_scs=5.0, r_mbd1=5.0, r_mbd2=5.0, r_sphere=5.0), 12, 6)
    if path == "warp":
        model.set_mma_path(lm.MMA_WARP)
    w = torch.linspace(0.5, 1.5, 48, device="cuda", dtype=torch.float64)
    f0 = model.energy_forces(*args, weights=w)[1]
    f = model.energy_forces(*args, weights=w * 2.0 ** power)[1]
    assert (f * 2.0 ** -power - f0).abs().max().item() < 1e-12
