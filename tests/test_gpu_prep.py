"""The per-call position preparation (bounding box, centring, split phase) on
the sizes where its launches change (one CTA takes the box up to 4096 atoms,
partial boxes past it) and on coordinates at the ends of its fixed-point range,
through FP32 maps against the oracle.  Tolerance: the FP32 paths' 1e-4."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", [1, 33, 4096, 4097, 20011])
@pytest.mark.parametrize("offset", [(0.0, 0.0, 0.0), (-1000.75, 250.5, 3.25), (524286.0, -524289.0, 1.0e7)])
def test_sizes_and_offsets(n, offset):
    rng = np.random.default_rng(n)
    xyz = rng.uniform(-4.0, 4.0, (n, 3)) + np.array(offset)
    S = np.array([1.0, -2.0, 4.0]) + rng.uniform(-0.2, 0.2, (97, 3))
    plan = api.Plan(W.unit_species()[None], A_LAT, n, s_list=S, center=(1, -2, 4))
    A = plan.amplitude(torch.tensor(xyz, device="cuda:0")).cpu().numpy()
    plan.check()
    assert plan.info()["shift"] == [float(np.rint(0.5 * (xyz[:, d].min() + xyz[:, d].max()))) for d in range(3)]
    # phases of 1e6 cells cost the oracle digits too: compare with the crystal moved back, the offset's phase exact
    back = xyz - np.array(offset)
    ref = oracle.amplitude(back, S, W.unit_species()[None], A_LAT)
    ph = sum(np.modf(S[:, d] * np.floor(offset[d]))[0] + S[:, d] * (offset[d] - np.floor(offset[d])) for d in range(3))
    tol = 1e-4 if max(abs(o) for o in offset) < 2000 else 1e-3  # S rounds at 1e-16: 1e7 cells are 6e-9 rad off, xyz 1e-9
    assert _rel(A, ref * np.exp(2j * np.pi * ph)) < tol


def test_tiny_and_signed_coordinates():
    xyz = np.array([[5e-324, -0.0, 1e-13], [-1e-300, 0.5, -0.5], [1.5, -2.5, 2.0 ** -43], [0.25, 1 / 3, -1 / 7]])
    S = np.array([[0.3, -0.7, 4.2], [3.0, 2.0, -5.0], [11.5, 0.25, 7.75]])
    plan = api.Plan(W.unit_species()[None], A_LAT, 4, s_list=S)
    A = plan.amplitude(torch.tensor(xyz, device="cuda:0")).cpu().numpy()
    assert _rel(A, oracle.amplitude(xyz, S, W.unit_species()[None], A_LAT)) < 1e-5


def test_non_finite_atoms_are_reported_past_the_partial_boxes():
    from paper_1010_2641_gb300 import binding as B
    xyz = np.random.default_rng(3).uniform(-4.0, 4.0, (5000, 3))
    xyz[4321, 1] = np.inf
    plan = api.Plan(W.unit_species()[None], A_LAT, 5000, s_list=np.zeros((5, 3)) + 0.1)
    plan.amplitude(torch.tensor(xyz, device="cuda:0"))
    with pytest.raises(B.ScatterError) as e:
        plan.check()
    assert e.value.status == B.SCATTER_ERR_NUMERIC
