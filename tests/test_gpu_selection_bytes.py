"""Selection overrides with bits above the low nibble: a byte acts as its low
nibble (bits 0-2 the kept directional stencils, bit 3 the large one) in the
residual and its adjoint, and is returned as it was given."""
import numpy as np
import pytest

from paper_2105_02127_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_02127_gb300 import build, teno
    build.build()
    return teno


@pytest.mark.parametrize("order", [3, 6])
@pytest.mark.parametrize("variant", [1, 2])
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["pairs", "mixed", "native"])
def test_high_bits(T, precision, variant, order):
    mesh = inputs.jittered_mesh(13, 14, 10.0, 10.0, seed=1041)  # 364 cells: a ragged last tile
    c = mesh.unwrapped_vertices().mean(axis=1)
    box = ((np.abs(c[:, 0] - 5.0) < 2.0) & (np.abs(c[:, 1] - 5.0) < 2.0)).astype(np.float64)
    U = inputs.prim_to_cons(1.0 + 2.0 * box, 0.3 + 0.1 * np.sin(c[:, 1]), 0.1 * np.cos(c[:, 0]),
                            1.0 + 3.0 * box)
    t = T.Teno(device=0).load(mesh)
    t.precompute_stencils(order=order, n_var=4, flux=T.FLUX_HLL, precision=precision,
                          recon_variant=variant)
    t.set_state(U)
    _, sel = t.residual(want_sel=True)
    assert (sel != 8).any()
    r = np.random.default_rng(1042)
    sel = np.where(r.random(sel.shape) < 0.1, 0, sel).astype(np.uint8)  # no stencil kept
    high = (sel | (r.integers(0, 16, sel.shape) << 4)).astype(np.uint8)
    w = r.standard_normal(U.shape)
    out = []
    for s in (sel, high):
        t.set_selection_override(s)
        R, got = t.residual(want_sel=True)
        assert np.array_equal(got, s)
        out.append((t.edge_values(), R, t.residual_vjp(w) if precision != T.FP32_MIXED else R))
    assert np.isfinite(out[0][0]).all()
    for a, b in zip(*out):  # (mixed selections leave the physical range at some faces: NaN)
        assert np.array_equal(a, b, equal_nan=True)
