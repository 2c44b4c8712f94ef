"""The FP32 grid adjoint as rows times columns against the oracle's analytic
gradient for given maps: every column axis, one pair, odd and even numbers of
columns around the 16-pair chunks, rows around the 16-row stages, symmetric, uneven
and unsorted axes, species, occupancies, off-centre crystals, and no atoms of a
species.  Tolerance 1e-5 (L2): MUFU sin/cos (2^-21 absolute) per row, FP32 sums per
16 rows, on sums that partly cancel."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


def _t(v):
    return torch.tensor(v, device="cuda:0")


def _axis(n, centre, kind, rng):
    if n == 1:
        return np.array([centre + 0.01])
    a = W.linspace_axis(centre, n, step=0.02)
    if kind == "uneven":
        a = a + rng.uniform(-0.006, 0.006, n)
    if kind == "unsorted":
        a = rng.permutation(a)
    return a


@pytest.mark.parametrize("shape, kind, n_sp, offset", [
    ((5, 7, 64), "even", 1, (0, 0, 0)), ((4, 33, 6), "even", 2, (17.3, -8.0, 40.4)), ((65, 3, 5), "even", 3, (0, 0, 0)),
    ((17, 1, 16), "uneven", 2, (0.4, 0.3, -0.4)), ((3, 6, 31), "unsorted", 1, (0, 0, 0)), ((16, 16, 32), "even", 2, (0, 0, 0)),
    ((2, 2, 200), "uneven", 1, (0, 0, 0)), ((31, 17, 1), "even", 2, (0, 0, 0)),
])
def test_gradient(shape, kind, n_sp, offset):
    c = W.fcc_sphere(radius_cells=4.3, seed=501)
    rng = np.random.default_rng(502)
    xyz = c.xyz + np.array(offset, dtype=np.float64)
    coef = np.concatenate([c.coef, c.coef[:1] * 0.8, c.coef[:1] * 1.3])[:n_sp]
    sp = rng.integers(0, n_sp, len(xyz)).astype(np.int32) if n_sp < 3 else np.where(rng.random(len(xyz)) < 0.5, 0, 2).astype(np.int32)
    occ = rng.uniform(0.5, 1.0, len(xyz)).astype(np.float32)
    axes = [_axis(n, ct, kind, rng) for n, ct in zip(shape, (0.0, 0.0, 4.0))]
    S = W.grid_points(axes)
    A = (oracle.amplitude(xyz, S, coef, A_LAT, species=sp, occ=occ) * np.exp(0.3j * rng.normal(size=len(S)))).astype(np.complex64)
    I_obs = (np.abs(A) ** 2 * rng.uniform(0.6, 1.3, len(S))).astype(np.float32)
    plan = api.Plan(coef, A_LAT, len(xyz), axes=axes, atom_species=sp, path="generic", radius_hint=1e5)
    loss, g = plan.backward(_t(xyz), _t(A), _t(I_obs), _t(occ))
    plan.check()
    sel = rng.choice(len(xyz), 200, replace=False)
    L_ref, ref = oracle.loss_grad_atoms(xyz, S, A, I_obs, coef, A_LAT, sel, species=sp, occ=occ)
    g = g.cpu().numpy().astype(np.float64)
    assert abs(loss.item() - L_ref) < 1e-5 * L_ref
    assert np.linalg.norm(g[sel] - ref) / np.linalg.norm(ref) < 1e-5
    again = plan.backward(_t(xyz), _t(A), _t(I_obs), _t(occ))[1].cpu().numpy()
    assert np.array_equal(g.astype(np.float32), again)
