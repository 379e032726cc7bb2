"""The FP64 Riemann solver's own form, branch by branch, against the oracle: flow
supersonic along an axis and across it (faces of every orientation: left state,
right state and star region), gas at rest (signed zeros, equal states), a
contact at rest (HLLC's middle wave at zero speed), cold gas (sound speed zero:
HLLC without a middle wave), random states, and scales near both ends of the
exponent range.  Bar: 1e-13 of (perimeter / area) times the largest |u| + c and the
flux it carries (rho, rho (|u| + c) for a momentum, E): some hundred roundings,
and a factor of ten for the kinetic energy taken out of E; the same cells finite."""
import numpy as np
import pytest

from paper_2105_02127_gb300 import inputs

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


def _states(c):
    n = len(c)
    o, z = np.ones(n), np.zeros(n)
    s = 1.0 + 0.1 * np.sin(0.2 * np.pi * c[:, 0])
    r = np.random.default_rng(1101)
    rand = inputs.prim_to_cons(r.uniform(0.5, 2.0, n), r.normal(size=n), r.normal(size=n),
                               r.uniform(0.5, 2.0, n))
    return {"supersonic": inputs.prim_to_cons(s, 3.5 * o, z, o),
            "oblique": inputs.prim_to_cons(s, 2.6 * o, -2.9 * o, s),
            "rest": inputs.prim_to_cons(o, -z, z, o),
            "contact": inputs.prim_to_cons(np.where(c[:, 0] < 5.0, 1.0, 4.0), z, z, o),
            "cold": inputs.prim_to_cons(o, o, z, z),
            "random": rand, "small": np.ldexp(rand, -480), "large": np.ldexp(rand, 480)}


@pytest.mark.parametrize("flux", [1, 2], ids=["hll", "hllc"])
def test_branches(oracle_mod, flux):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_02127_gb300 import build, teno
    build.build()
    mesh = inputs.jittered_mesh(16, 15, 10.0, 10.0, seed=1102)
    t = teno.Teno(device=0).load(mesh)
    t.precompute_stencils(order=3, n_var=4, flux=flux, precision=teno.FP64_NATIVE, linear=1)
    o = oracle_mod.Oracle(mesh, order=3, n_var=4, flux=flux, linear=True)
    V = mesh.unwrapped_vertices()
    e = np.roll(V, -1, axis=1) - V
    per = np.hypot(e[..., 0], e[..., 1]).sum(axis=1)
    area = 0.5 * np.abs(e[:, 0, 0] * e[:, 1, 1] - e[:, 0, 1] * e[:, 1, 0])
    for name, U in _states(mesh.unwrapped_vertices().mean(axis=1)).items():
        t.set_state(U)
        R = t.residual()[0]
        Ro = o.residual(U)[0]
        assert np.isfinite(Ro).all() and np.isfinite(R).all(), name
        u = np.hypot(U[1], U[2]) / U[0]
        p = 0.4 * (U[3] - 0.5 * U[0] * u * u)
        a = (u + np.sqrt(1.4 * np.maximum(p, 0.0) / U[0])).max()
        rho, E = U[0].max(), U[3].max()
        f = np.array([rho * a, rho * a * a, rho * a * a, max(E, rho * a * a) * a])
        assert (np.abs(R - Ro) <= 1e-13 * f[:, None] * (per / area)).all(), name
