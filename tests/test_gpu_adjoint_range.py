"""Residual adjoint (pairs, W form) with cotangents of very different size in a
tile, far below one, and not finite.

The tile kernel adds its contributions in one unit per tile and variable or, where
that is too coarse for some cell, in pairs.  Its result is compared cell by cell
with that of the kernel that keeps pairs throughout (variant 1): cell j takes part
in the faces of the cells whose stencils hold it, so its scale is the largest
|w| of these cells and their neighbours, times the largest entry that the same
adjoint gives for cotangents near one; the bar of 1e-11 of it is the parity bar."""
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


def _setup(T, order):
    mesh = inputs.jittered_mesh(24, 23, 10.0, 10.0, seed=1061)  # 1,104 cells: a ragged last tile
    c = mesh.unwrapped_vertices().mean(axis=1)
    box = 0.4 * ((np.abs(c[:, 0] - 5.0) < 2.0) & (np.abs(c[:, 1] - 5.0) < 2.0))
    U = inputs.prim_to_cons(1.0 + box, 0.3 + 0.1 * np.sin(c[:, 1]), 0.1 * np.cos(c[:, 0]),
                            1.0 + 1.5 * box)
    solvers = []
    for variant in (1, 2):
        t = T.Teno(device=0).load(mesh)
        t.precompute_stencils(order=order, n_var=4, flux=T.FLUX_HLL, recon_variant=variant)
        t.set_state(U)
        solvers.append(t)
    # the same selection on both sides, cut cells among them
    sel = solvers[0].residual(want_sel=True)[1]
    assert (sel != 8).any() and (sel == 8).any()
    for t in solvers:
        t.set_selection_override(sel)
    return mesh, c, solvers


def _reach(mesh, t, x):
    """largest x over the cells whose cotangent reaches cell j, per j"""
    edges = {}
    for c, (a, b, d) in enumerate(mesh.tri.tolist()):
        for e in ((a, b), (b, d), (d, a)):
            edges.setdefault(frozenset(e), []).append(c)
    y = x.copy()
    for p, q in edges.values():
        y[p], y[q] = max(y[p], x[q]), max(y[q], x[p])
    large, small = t.stencils()
    out = y.copy()
    for ids in (large, small.reshape(mesh.n_cell, -1)):
        np.maximum.at(out, np.where(ids >= 0, ids, np.arange(mesh.n_cell)[:, None]), y[:, None])
    return out


@pytest.mark.parametrize("order", [3, 4, 5, 6])
@pytest.mark.parametrize("small", [2.0 ** -10, 2.0 ** -40, 2.0 ** -70, 0.0])
def test_mixed_magnitudes(T, order, small):
    mesh, c, (t1, t2) = _setup(T, order)
    w = np.random.default_rng(1062).standard_normal((4, mesh.n_cell))
    J = np.abs(t1.residual_vjp(w)).max()
    size = np.where(c[:, 0] < 5.0, 1.0, small)
    v1, v2 = t1.residual_vjp(w * size), t2.residual_vjp(w * size)
    scale = _reach(mesh, t1, size)
    assert small == 0.0 or (scale == small).sum() > 100
    assert (np.abs(v2 - v1) <= BAR * J * scale).all()


@pytest.mark.parametrize("order", [3, 6])
@pytest.mark.parametrize("exp", [-60, -100, 60])
def test_scaled(T, order, exp):
    mesh, _, (t1, t2) = _setup(T, order)
    w = np.ldexp(np.random.default_rng(1063).standard_normal((4, mesh.n_cell)), exp)
    v1, v2 = t1.residual_vjp(w), t2.residual_vjp(w)
    assert np.abs(v2 - v1).max() <= BAR * np.abs(v1).max()


@pytest.mark.parametrize("order", [3, 6])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite(T, order, bad):
    mesh, _, (t1, t2) = _setup(T, order)
    w = np.random.default_rng(1064).standard_normal((4, mesh.n_cell))
    w[0, 137] = bad
    w[2, 900] = -bad
    v1, v2 = t1.residual_vjp(w), t2.residual_vjp(w)
    ok = np.isfinite(v1)
    assert np.array_equal(ok, np.isfinite(v2)) and 0 < ok.sum() < ok.size
    assert np.abs(v2 - v1)[ok].max() <= BAR * np.abs(v1[ok]).max()
