"""FP32 grids at the ends of what the factorised sum takes: axes longer than its
launch grid has column tiles for, and plans whose tables find no room, which keep
the sincos form.  Sampled points against the oracle; tolerance 1e-5, the FP32
sums'."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api
    from paper_1010_2641_gb300 import binding as B

A_LAT = W.LATTICE_A


def _t(v):
    return torch.tensor(v, device="cuda:0")


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("shape, uneven", [
    ((64, 1, 1000000), False), ((64, 1, 500000), True), ((1000000, 8, 8), False), ((3, 2000003, 2), True),
])
def test_long_axis(shape, uneven):
    rng = np.random.default_rng(511)
    xyz = rng.uniform(-3.0, 3.0, (100, 3))
    axes = [W.linspace_axis(x, n, half_width=0.4) if n > 1 else np.array([x]) for x, n in zip((0.0, 0.0, 4.0), shape)]
    if uneven:
        axes = [a + rng.uniform(-0.2, 0.2, len(a)) * 0.8 / len(a) for a in axes]
    plan = api.Plan(W.unit_species()[None], A_LAT, 100, axes=axes, path="generic")
    A = plan.amplitude(_t(xyz))
    plan.check()
    idx = np.concatenate([rng.choice(plan.n_s, 500, replace=False), [0, plan.n_s - 1]])
    i = np.unravel_index(idx, shape)
    S = np.stack([axes[d][i[d]] for d in range(3)], 1)
    got = A[torch.tensor(idx, device="cuda:0")].cpu().numpy()
    assert _rel(got, oracle.amplitude(xyz, S, W.unit_species()[None], A_LAT)) < 1e-5


def test_no_room_for_the_tables_keeps_the_sincos_form(monkeypatch):
    """Every device allocation of plan building in turn fails once: a plan is
    refused (OOM) or built without the table that found no room, and right."""
    c = W.fcc_sphere(radius_cells=9.0, seed=512)
    axes = [W.linspace_axis(x, n, step=0.05) for x, n in zip((0.0, 0.0, 4.0), (40, 35, 30))]
    make = lambda: api.Plan(c.coef, A_LAT, len(c.xyz), axes=axes, atom_species=c.species, path="generic")
    x = _t(c.xyz)
    whole = make()
    full = whole.amplitude(x).cpu().numpy()
    served = 0
    for n in range(1, 80):
        monkeypatch.setenv("SCATTER_FAULT", f"alloc:{n}")
        try:
            plan = make()
        except B.ScatterError as e:
            assert e.status == B.SCATTER_ERR_OOM
            continue
        finally:
            monkeypatch.delenv("SCATTER_FAULT")
        A = plan.amplitude(x).cpu().numpy()
        plan.check()
        assert _rel(A, full) < 1e-5
        if plan.info()["workspace_bytes"] == whole.info()["workspace_bytes"]:
            break  # past the last allocation
        served += 1
    else:
        pytest.fail("allocations without end")
    assert served >= 4  # the grid sum's tables
