"""Positions in other units than cells: coordinates times 2^-k and S times 2^k (and
with them the lattice parameter of |S| / 2a) have the same phases to the last place, so
maps and gradients are those of the crystal in cells.  2^-30 stands for crystals
in metres (S of 1e9, positions of 1e-8).  Tolerances: the FP32 sums' 1e-5, the
tensor cores' 1e-4."""
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


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.complex128), np.asarray(b, dtype=np.complex128)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("k", [0, 8, 10, 14, 20, 30])
@pytest.mark.parametrize("kind, tol", [("list", 1e-5), ("batch", 1e-5), ("generic", 1e-5), ("separable", 1e-4)])
def test_scaled_crystal(kind, tol, k):
    u = 2.0 ** -k
    # four thousand atoms and more: the folded form of the separable path
    c = W.fcc_sphere(radius_cells=6.3 if kind == "separable" else 4.0, seed=501)
    rng = np.random.default_rng(502)
    n, sp = len(c.xyz), c.species
    if kind in ("list", "batch"):
        S = np.array([0.0, 1.0, 4.0]) + rng.uniform(-0.2, 0.2, (400, 3))
        kw = dict(s_list=S / u)
        if kind == "batch":
            kw.update(atom_off=[0, n // 2, n], s_off=[0, 150, 400])
    else:
        axes = [W.linspace_axis(x, m, step=0.03) for x, m in zip((0.0, 1.0, 4.0), (18, 13, 12))]
        S = W.grid_points(axes)
        kw = dict(axes=[a / u for a in axes], path=kind)
    plan = api.Plan(c.coef, A_LAT / u, n, atom_species=sp, **kw)
    x = _t(c.xyz * u)
    A = plan.amplitude(x).cpu().numpy()
    plan.check()
    parts = [(0, n, 0, len(S))] if kind != "batch" else [(0, n // 2, 0, 150), (n // 2, n, 150, 400)]
    for a0, a1, s0, s1 in parts:
        ref = oracle.amplitude(c.xyz[a0:a1], S[s0:s1], c.coef, A_LAT, species=sp[a0:a1])
        assert _rel(A[s0:s1], ref) < tol
    if kind == "batch":
        return
    I_obs = (np.abs(A) ** 2 * rng.uniform(0.7, 1.2, len(A))).astype(np.float32)
    _, g = plan.backward(x, _t(A), _t(I_obs))
    sel = rng.choice(n, 60, replace=False)
    _, gref = oracle.loss_grad_atoms(c.xyz, S, A, I_obs, c.coef, A_LAT, sel, species=sp)
    assert _rel(g.cpu().numpy()[sel], gref / u) < tol
