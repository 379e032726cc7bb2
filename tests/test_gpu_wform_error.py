"""Rounding error of the W form on the pair path: its residuals are no further from
the FP64 oracle's than those of the kernels that form every product in pairs
(variant 1), root mean square over a smooth state and one with jumps.  (The pairs'
rounding stands far above the oracle's own.)"""
import numpy as np
import pytest

from paper_2105_02127_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("state", ["vortex", "box"])
@pytest.mark.parametrize("order", [3, 4, 5, 6])
def test_error_against_oracle(oracle_mod, order, state):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_02127_gb300 import build, teno
    build.build()
    sq = [0.0, 0.0]
    for seed in (1111, 1112):
        mesh = inputs.jittered_mesh(48, 45, 10.0, 10.0, seed=seed)
        if state == "vortex":
            U = inputs.cell_average(mesh, inputs.isentropic_vortex)
        else:
            c = mesh.unwrapped_vertices().mean(axis=1)
            k = 0.2 * np.pi
            box = 0.5 * ((np.abs(c[:, 0] - 5.0) < 2.0) & (np.abs(c[:, 1] - 5.0) < 2.0))
            U = inputs.prim_to_cons(1.0 + 0.1 * np.sin(k * c[:, 0]) + box,
                                    0.3 + 0.1 * np.sin(k * c[:, 1]), 0.1 * np.cos(k * c[:, 0]) - 0.2,
                                    1.0 + 0.1 * np.cos(k * c[:, 1]) + 1.5 * box)
        o = oracle_mod.Oracle(mesh, order=order, n_var=4, flux=1)
        Ro, sel, _ = o.residual(U)
        for i, variant in enumerate((1, 2)):
            t = teno.Teno(device=0).load(mesh)
            t.precompute_stencils(order=order, n_var=4, flux=teno.FLUX_HLL, recon_variant=variant)
            t.set_state(U)
            t.set_selection_override(sel)
            sq[i] += float(((t.residual()[0] - Ro) ** 2).sum())
            t.close()
    assert sq[1] <= sq[0]
