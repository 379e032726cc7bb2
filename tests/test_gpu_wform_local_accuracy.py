"""Gauss-point values of cells on the small side of a jump (Euler, FP64 paths).

The W form's differences are integers of one unit per tile and variable, set by
the tile's largest difference.  A cell whose own stencil is smooth keeps its own
accuracy although its tile holds a jump: the values are compared cell by cell
with those of the kernels without the fixed-point sums (variant 1) against a bar
of rounding errors at the cell's own scale,

  u (4 |U_0| a + K sum_s A_s |U_s - U_0|),   A_s = max_p sum_l |Psi'_pl| |G_ls|

(Psi', G in a basis in which the smoothness indicator is the sum of squares),
over the stencil (or the kept directional ones) that the cell takes: K = 2 (n +
m + 8) roundings of the two n-term sums, m coefficients and their evaluation;
u = 2^-53 and a = 1 in FP64, u = 2^-48 and a = 1 + sum_s A_s in pairs, whose
states are rounded to pairs before the difference is formed."""
import numpy as np
import pytest

from oracle import oracle as orc
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


@pytest.fixture(scope="module")
def mesh():
    return inputs.jittered_mesh(24, 23, 10.0, 10.0, seed=1051)  # 1,104 cells: a ragged last tile


@pytest.fixture(scope="module")
def matrices(mesh):
    """per order, for the large and the directional stencils: A_s and the cells s, [cell][n]"""
    out = {}

    def get(order):
        if order not in out:
            o = orc.Oracle(mesh, order=order, n_var=4, flux=1)
            o.prepare()
            r = o.reference_data()
            t, z = r["gt"], np.zeros_like(r["gt"])
            x, y = np.concatenate([t, 1.0 - t, z]), np.concatenate([z, t, 1.0 - t])
            psi = np.stack([x ** a * y ** b for a, b in r["ex"]], axis=1) - r["mean0"]
            out[order] = []
            for k, B in enumerate([r["Br"]] + [r["B2"]] * 3):
                L, n = np.linalg.cholesky(B), len(B)
                q = np.abs(psi[:, :n] @ np.linalg.inv(L).T)
                M = [o.recon_matrix(c, k) for c in range(mesh.n_cell)]
                G = np.array([Ah * vol for _, Ah, vol, _ in M])
                out[order].append(((q @ np.abs(L.T @ G)).max(axis=1), np.array([m[3] for m in M])))
        return out[order]

    return get


def _state(mesh, jump):
    c = mesh.unwrapped_vertices().mean(axis=1)
    k = 2.0 * np.pi / 10.0
    box = jump * ((np.abs(c[:, 0] - 5.0) < 2.0) & (np.abs(c[:, 1] - 5.0) < 2.0))
    rho = 1.0 + 0.1 * np.sin(k * c[:, 0]) + box
    p = 1.0 + 0.1 * np.cos(k * c[:, 1]) + 2.0 * box
    return inputs.prim_to_cons(rho, 0.3 + 0.1 * np.sin(k * c[:, 1]), 0.1 * np.cos(k * c[:, 0]), p)


@pytest.mark.parametrize("jump", [0.0, 1e2, 1e4, 1e6, 1e8])
@pytest.mark.parametrize("order", [3, 4, 5, 6])
@pytest.mark.parametrize("precision", [0, 2], ids=["pairs", "native"])
def test_small_side_of_a_jump(T, mesh, matrices, precision, order, jump):
    U = _state(mesh, jump)
    got = []
    for variant in (1, 2):
        t = T.Teno(device=0).load(mesh)
        t.precompute_stencils(order=order, n_var=4, flux=T.FLUX_HLL, precision=precision,
                              recon_variant=variant)
        t.set_state(U)
        sel = t.residual(want_sel=True)[1]
        got.append((t.edge_values(), sel))
    A = matrices(order)
    d = [np.abs(U[:, s] - U[:, :, None]) for _, s in A]  # [var][cell][slot]
    sum_a = [a.sum(axis=1)[None] for a, _ in A]
    sum_d = [np.einsum("vcs,cs->vc", x, a) for x, (a, _) in zip(d, A)]
    (e1, s1), (e2, s2) = got
    same = s1 == s2
    assert same.mean() > 0.99
    keep = [(s1 & 8) != 0] + [((s1 >> k) & 1 != 0) & ((s1 & 8) == 0) for k in range(3)]
    sa = sum(np.where(k, x, 0.0) for k, x in zip(keep, sum_a))
    sd = sum(np.where(k, x, 0.0) for k, x in zip(keep, sum_d))
    u, a = (2.0 ** -53, 1.0) if precision == T.FP64_NATIVE else (2.0 ** -48, 1.0 + sa)
    bar = u * (4.0 * np.abs(U) * a + 2.0 * (t.ns + t.m + 8) * sd)
    err = np.abs(e2 - e1).max(axis=(1, 2)).T  # [var][cell]
    ratio = np.where(same, err / bar, 0.0)
    assert ratio.max() <= 1.0, (ratio.max(), np.unravel_index(ratio.argmax(), ratio.shape))
    if jump > 1.0:  # such cells are there: a smooth stencil in a tile that holds the jump
        calm = d[0][0].max(axis=1) < 0.1 * jump
        perm = t.permutation()
        tiles = [perm[i:i + 32] for i in range(0, mesh.n_cell, 32)]
        shared = sum(int(calm[c].sum()) for c in tiles if d[0][0][c].max() > 0.5 * jump)
        assert shared > 20
