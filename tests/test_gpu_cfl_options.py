"""The CFL maximum that a step's last update takes for the next step, with the
options that change a cell's speed or its update: the rotating velocity field,
positivity scaling, boundaries with an outflow layer, higher orders.  n steps in
one call equal n calls of one step bit for bit (the latter reduce the maximum in
its own kernel); and a state that is physical at first and turns non-physical in
the third of the steps is reported either way."""
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


def _mesh(bounded):
    return inputs.jittered_mesh(13, 14, 10.0, 10.0, seed=1071, periodic=not bounded)  # 256 + 108


def _both(T, mesh, U, **kw):
    t = T.Teno(device=0).load(mesh)
    t.precompute_stencils(**kw)
    out = []
    for calls in ((4,), (1, 1, 1, 1)):
        t.set_state(U)
        for n in calls:
            t.rk3_steps(n)
        out.append(t.get_state())
        t.check_state()
    assert np.isfinite(out[0]).all() and not np.array_equal(out[0], U)
    assert np.array_equal(*out)


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["pairs", "mixed", "native"])
def test_rotation(T, precision):
    mesh = _mesh(False)
    c = mesh.unwrapped_vertices().mean(axis=1)
    U = np.sin(0.2 * np.pi * c[:, 0])[None] * np.cos(0.2 * np.pi * c[:, 1])
    _both(T, mesh, U, order=5, n_var=1, flux=T.FLUX_UPWIND, precision=precision,
          rotation=(5.0, 5.0, 1.0, 4.0, 4.8))


@pytest.mark.parametrize("bounded", [False, True], ids=["periodic", "outflow"])
@pytest.mark.parametrize("order,positivity", [(4, 1), (6, 0)])
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["pairs", "mixed", "native"])
def test_euler(T, precision, order, positivity, bounded):
    mesh = _mesh(bounded)
    c = mesh.unwrapped_vertices().mean(axis=1)
    s = np.sin(0.2 * np.pi * c[:, 0]) * np.cos(0.2 * np.pi * c[:, 1])
    U = inputs.prim_to_cons(1 + 0.3 * s, 0.5 + 0.3 * s, 0.2 - s, 1 - 0.2 * s)
    _both(T, mesh, U, order=order, n_var=4, flux=T.FLUX_HLLC, precision=precision,
          positivity=positivity)


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["pairs", "mixed", "native"])
def test_state_that_turns_nonphysical(T, precision):
    mesh = inputs.jittered_mesh(13, 14, 10.0, 10.0, seed=1031)
    c = mesh.unwrapped_vertices().mean(axis=1)
    o = np.ones(len(c))
    U = inputs.prim_to_cons(o, np.sign(c[:, 0] - 5.0), 0 * o, 0.05 * o)  # two streams part
    t = T.Teno(device=0).load(mesh)
    t.precompute_stencils(order=3, n_var=4, flux=T.FLUX_HLL, precision=precision)
    t.set_state(U)
    t.rk3_steps(1)
    t.check_state()
    for calls in ((5,), (1,) * 5):
        t.set_state(U)
        with pytest.raises(T.TenoError):
            for n in calls:
                t.rk3_steps(n)
            t.check_state()
