"""Edges of the W-form reconstruction's fixed-point sums (Euler, FP64 paths).

The halo states of a tile become integers of one power-of-two unit, so the
kernel is run where that unit leaves the ranges it is computed in, and where it
does not exist: states scaled by powers of two (the linear scheme's residual
scales exactly, so only rounding may differ: the parity bar of 1e-11 per
variable), tiles that mix magnitudes, and states with an infinity or a NaN,
whose residual must be non-finite in the cells where the kernels without the
fixed-point sums (variant 1) say so and equal to theirs elsewhere."""
import numpy as np
import pytest

from paper_2105_02127_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

BAR = 1e-11


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_02127_gb300 import build, teno
    build.build()
    return teno


def _state(mesh, jump):
    c = mesh.unwrapped_vertices().mean(axis=1)
    k = 2.0 * np.pi / 10.0
    box = jump * ((np.abs(c[:, 0] - 5.0) < 2.0) & (np.abs(c[:, 1] - 5.0) < 2.0))
    rho = 1.0 + 0.1 * np.sin(k * c[:, 0]) + box
    p = 1.0 + 0.1 * np.cos(k * c[:, 1]) + 2.0 * box
    return inputs.prim_to_cons(rho, 0.3 + 0.1 * np.sin(k * c[:, 1]), 0.1 * np.cos(k * c[:, 0]), p)


def _residual(T, mesh, U, order, precision, variant=2, linear=0):
    t = T.Teno(device=0).load(mesh)
    t.precompute_stencils(order=order, n_var=4, flux=T.FLUX_HLL, precision=precision,
                          recon_variant=variant, linear=linear)
    t.set_state(U)
    return t.residual(want_sel=True)


@pytest.mark.parametrize("order", [3, 4, 5, 6])
@pytest.mark.parametrize("precision,exps", [(0, (-96, -40, 30)), (2, (-400, -96, 30, 200))],
                         ids=["pairs", "native"])
def test_scaled_states(T, order, precision, exps):
    mesh = inputs.jittered_mesh(13, 14, 10.0, 10.0, seed=1021)  # 364 cells: a ragged last tile
    U = _state(mesh, 0.4)
    R, _ = _residual(T, mesh, U, order, precision, linear=1)
    for e in exps:
        Rs, _ = _residual(T, mesh, np.ldexp(U, e), order, precision, linear=1)
        err = np.abs(np.ldexp(Rs, -e) - R).max(axis=1) / np.abs(R).max(axis=1)
        assert err.max() <= BAR, (e, err)


@pytest.mark.parametrize("order", [3, 4, 5, 6])
@pytest.mark.parametrize("precision", [0, 2], ids=["pairs", "native"])
def test_mixed_magnitudes(T, order, precision):
    """A jump of 10^4 inside the tiles: small and large states share units."""
    mesh = inputs.jittered_mesh(24, 23, 10.0, 10.0, seed=1022)
    U = _state(mesh, 1e4)
    R, sel = _residual(T, mesh, U, order, precision)
    R1, sel1 = _residual(T, mesh, U, order, precision, variant=1)
    assert np.array_equal(sel, sel1)
    assert (np.abs(R - R1).max(axis=1) <= BAR * np.abs(R1).max(axis=1)).all()


@pytest.mark.parametrize("order", [3, 6])
@pytest.mark.parametrize("precision", [0, 2], ids=["pairs", "native"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_state(T, order, precision, bad):
    mesh = inputs.jittered_mesh(24, 23, 10.0, 10.0, seed=1023)
    U = _state(mesh, 0.4)
    U[0, 137] = bad
    U[3, 900] = -bad
    R, _ = _residual(T, mesh, U, order, precision)
    R1, _ = _residual(T, mesh, U, order, precision, variant=1)
    ok, ok1 = np.isfinite(R).all(axis=0), np.isfinite(R1).all(axis=0)
    assert np.array_equal(ok, ok1) and 0 < ok.sum() < ok.size
    scale = np.abs(R1[:, ok1]).max(axis=1)
    assert (np.abs(R[:, ok] - R1[:, ok]).max(axis=1) <= BAR * scale).all()
