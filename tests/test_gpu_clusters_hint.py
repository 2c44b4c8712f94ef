"""Radius hints at the ends of what a float holds, with crystals of one point (every
atom at the same place) and of many: every point of the map and every gradient is
written.  Tolerance 1e-5, the FP32 sums'."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


@pytest.mark.parametrize("hint", [1e-300, 1e-30, 1e18, 1e300])
@pytest.mark.parametrize("spread", [0.0, 3.0])
def test_every_output_is_written(hint, spread):
    rng = np.random.default_rng(571)
    n = 4000
    # one point: a cell's corner, its centring leaves no distance at all
    xyz = (np.array([0.2, -0.1, 0.3]) if spread else np.array([7.0, -2.0, 0.0])) + rng.uniform(-spread, spread, (n, 3))
    S = W.ewald_slice(60001, rocking_deg=0.02, seed=572)
    plan = api.Plan(W.unit_species()[None], A_LAT, n, s_list=S, radius_hint=hint)
    x = torch.tensor(xyz, device="cuda:0")
    out = torch.full((len(S),), complex(np.nan, np.nan), dtype=torch.complex64, device="cuda:0")
    A = plan.amplitude(x, out=out).cpu().numpy()
    sel = rng.choice(len(S), 300, replace=False)
    ref = oracle.amplitude(xyz, S[sel], W.unit_species()[None], A_LAT)
    assert np.all(np.isfinite(A.view(np.float32)))
    assert np.linalg.norm(A[sel] - ref) < 1e-5 * np.linalg.norm(ref)
    A = (A * np.exp(1j * rng.uniform(0.3, 1.0, len(A)))).astype(np.complex64)  # at its own phases a point's gradient vanishes
    I_obs = (np.abs(A) ** 2 * rng.uniform(0.7, 1.2, len(A))).astype(np.float32)
    _, g = plan.backward(x, torch.tensor(A, device="cuda:0"), torch.tensor(I_obs, device="cuda:0"))
    plan.check()
    at = rng.choice(n, 20, replace=False)
    _, gref = oracle.loss_grad_atoms(xyz, S, A, I_obs, W.unit_species()[None], A_LAT, at)
    assert np.linalg.norm(g.cpu().numpy()[at] - gref) < 1e-5 * np.linalg.norm(gref)
