"""FP32 gradients on grids whose long axis has as many pairs of columns as the
rows-times-columns form's launch grid has room for, and a few more (the other
forms take those).  Tolerance 1e-5, the FP32 gradients'."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


@pytest.mark.parametrize("n", [16 * 65535, 16 * 65535 + 1, 1 << 20])
def test_longest_uneven_axis(n):
    rng = np.random.default_rng(521)
    xyz = rng.uniform(-3.0, 3.0, (40, 3))
    l = W.linspace_axis(4.0, n, half_width=0.4) + rng.uniform(-0.2, 0.2, n) * 0.8 / n
    axes = [np.array([0.1]), np.array([-0.2]), l]
    # a hint past which no axis counts as oversampled: the gradient on the map's own points
    plan = api.Plan(W.unit_species()[None], A_LAT, len(xyz), axes=axes, path="generic", radius_hint=1e6)
    x = torch.tensor(xyz, device="cuda:0")
    G = np.zeros(n, dtype=np.complex64)
    at = np.concatenate([rng.choice(n, 300, replace=False), [0, n - 1]])
    G[at] = (rng.normal(size=len(at)) + 1j * rng.normal(size=len(at))).astype(np.complex64)
    g = plan.vjp(x, torch.tensor(G, device="cuda:0")).cpu().numpy()
    plan.check()
    S = np.stack([np.full(len(at), 0.1), np.full(len(at), -0.2), l[at]], 1)
    f = oracle.amplitude(np.zeros((1, 3)), S, W.unit_species()[None], A_LAT)  # the form factor
    e = np.exp(2j * np.pi * (S @ xyz.T))
    ref = -2 * np.pi * np.einsum("md,mj->jd", S, np.imag((np.conj(G[at].astype(np.complex128)) * f)[:, None] * e))
    assert np.linalg.norm(g - ref) < 1e-5 * np.linalg.norm(ref)
