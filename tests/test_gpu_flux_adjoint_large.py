"""Flux adjoint (HLL, pairs) on a mesh above the line where a thread takes a face's
points in turn (524,288 faces): the whole mesh's adjoint against that of its two parts, each
below the line (one thread per point).  The per-face arithmetic is the same and
the parts sum the same terms in another order: the bar of 1e-13 of a variable's
largest entry is that of the partition tests."""
import numpy as np
import pytest

from paper_2105_02127_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [3, 5])
def test_points_in_turn(order):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_02127_gb300 import build, teno
    build.build()
    mesh = inputs.jittered_mesh(421, 419, 10.0, 10.0, seed=1081)  # 352,798 cells, 529,197 faces
    c = mesh.unwrapped_vertices().mean(axis=1)
    box = 0.4 * ((np.abs(c[:, 0] - 5.0) < 2.0) & (np.abs(c[:, 1] - 5.0) < 2.0))
    U = inputs.prim_to_cons(1.0 + box, 0.3 + 0.1 * np.sin(c[:, 1]), 0.1 * np.cos(c[:, 0]),
                            1.0 + 1.5 * box)
    w = np.random.default_rng(1082).standard_normal(U.shape)
    kw = dict(order=order, n_var=4, flux=teno.FLUX_HLL)
    whole = teno.Teno(device=0).load(mesh)
    whole.precompute_stencils(**kw)
    whole.set_state(U)
    v = whole.residual_vjp(w)
    whole.close()
    parts = [teno.Teno(device=0).load(mesh).precompute_partition(2, p, **kw) for p in range(2)]
    for t in parts:
        t.set_state(U)
    vp = teno.group_residual_vjp(parts, w)
    assert np.isfinite(v).all()
    assert (np.abs(vp - v).max(axis=1) <= 1e-13 * np.abs(v).max(axis=1)).all()
