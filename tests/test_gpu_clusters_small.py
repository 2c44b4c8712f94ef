"""Gradients of clustered lists for crystals much smaller than the radius that the
clusters were made for, down to a single point: a column may not matter for the sum
and yet for its derivative.  Tolerance 1e-5, the FP32 gradients'."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


@pytest.mark.parametrize("hkl", [(1.0, 1.0, 1.0), (0.0, 0.0, 0.0)])
@pytest.mark.parametrize("spread", [0.0, 1e-6, 1e-4, 3e-3, 0.03, 0.1, 0.3, 1.0, 4.0])
def test_small_crystals(spread, hkl):
    rng = np.random.default_rng(581)
    n = 4000
    u = rng.normal(size=(n, 3))
    u *= np.cbrt(rng.uniform(0.0, 1.0, (n, 1))) / np.linalg.norm(u, axis=1, keepdims=True)
    xyz = np.array([7.0, -2.0, 0.0]) + spread * u
    S = np.array(hkl) + rng.uniform(-0.05, 0.05, (60001, 3)) * np.array([1.0, 1.0, 0.02])
    plan = api.Plan(W.unit_species()[None], A_LAT, n, s_list=S)
    bare = api.Plan(W.unit_species()[None], A_LAT, n, s_list=S, split_k=1)
    assert plan.info()["workspace_bytes"] > bare.info()["workspace_bytes"] + 1000000  # its clusters
    x = torch.tensor(xyz, device="cuda:0")
    A = (plan.amplitude(x).cpu().numpy() * np.exp(1j * rng.uniform(0.3, 1.0, len(S)))).astype(np.complex64)
    I_obs = (np.abs(A) ** 2 * rng.uniform(0.7, 1.2, len(A))).astype(np.float32)
    _, g = plan.backward(x, torch.tensor(A, device="cuda:0"), torch.tensor(I_obs, device="cuda:0"))
    plan.check()
    at = rng.choice(n, 20, replace=False)
    _, ref = oracle.loss_grad_atoms(xyz, S, A, I_obs, W.unit_species()[None], A_LAT, at)
    assert np.linalg.norm(g.cpu().numpy()[at] - ref) < 1e-5 * np.linalg.norm(ref)
