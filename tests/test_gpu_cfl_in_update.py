"""The CFL maximum that the last update of a step takes for the next one: n steps
in one call equal n calls of one step (whose maximum is its own kernel's) bit for
bit, on a ragged last block, for every precision and both equations; and a state
that turns non-physical is reported either way."""
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


def _solver(T, n_var, precision):
    mesh = inputs.jittered_mesh(13, 14, 10.0, 10.0, seed=1031)  # 364 cells: 256 + 108
    c = mesh.unwrapped_vertices().mean(axis=1)
    s = np.sin(0.2 * np.pi * c[:, 0]) * np.cos(0.2 * np.pi * c[:, 1])
    t = T.Teno(device=0).load(mesh)
    t.precompute_stencils(order=3, n_var=n_var, flux=T.FLUX_UPWIND if n_var == 1 else T.FLUX_HLL,
                          precision=precision)
    U = s[None] if n_var == 1 else inputs.prim_to_cons(1 + 0.1 * s, 0.5 + 0.3 * s, 0.2 - s, 1 - 0.2 * s)
    return t, U


@pytest.mark.parametrize("n_var", [1, 4])
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["pairs", "mixed", "native"])
def test_steps_equal_single_steps(T, n_var, precision):
    t, U = _solver(T, n_var, precision)
    t.set_state(U)
    t.rk3_steps(5)
    a = t.get_state()
    t.set_state(U)
    for _ in range(5):
        t.rk3_steps(1)
    b = t.get_state()
    assert np.isfinite(a).all() and not np.array_equal(a, U)
    assert np.array_equal(a, b)


@pytest.mark.parametrize("precision", [0, 2], ids=["pairs", "native"])
def test_nonphysical_state_is_reported(T, precision):
    t, U = _solver(T, 4, precision)
    U[3, 200] = 0.0
    for n in (1, 3):
        t.set_state(U)
        with pytest.raises(T.TenoError):
            t.rk3_steps(n)
            t.check_state()
