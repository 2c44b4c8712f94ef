"""Tensor-core plans whose folded form finds no room keep the direct one: every
device allocation of plan building in turn fails once, and a plan is refused (OOM)
or built and right.  Tolerance 1e-4, the path's own."""
import numpy as np
import pytest

from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api
    from paper_1010_2641_gb300 import binding as B


@pytest.mark.parametrize("shape", [(40, 35, 30), (200, 1, 200)])
def test_no_room_for_the_folded_form(monkeypatch, shape):
    c = W.fcc_sphere(radius_cells=9.0, seed=551)
    axes = [W.linspace_axis(x, n, step=0.02) if n > 1 else np.array([x]) for x, n in zip((0.0, 0.0, 4.0), shape)]
    make = lambda: api.Plan(c.coef, W.LATTICE_A, len(c.xyz), axes=axes, atom_species=c.species, path="separable",
                            split_k=3)  # folded, without nodes
    x = torch.tensor(c.xyz, device="cuda:0")
    whole = make()
    full, direct = whole.amplitude(x).cpu().numpy(), whole.intensity(x).cpu().numpy()
    free = torch.cuda.mem_get_info()[0]
    served = 0
    for n in range(1, 80):
        monkeypatch.setenv("SCATTER_FAULT", f"alloc:{n}")
        try:
            plan = make()
        except B.ScatterError as e:
            assert e.status == B.SCATTER_ERR_OOM
            assert abs(torch.cuda.mem_get_info()[0] - free) <= 4 << 20
            continue
        finally:
            monkeypatch.delenv("SCATTER_FAULT")
        size = plan.info()["workspace_bytes"]  # a backward adds its own
        A = plan.amplitude(x).cpu().numpy()
        _, g = plan.backward(x, torch.tensor(A, device="cuda:0"), torch.tensor(np.abs(A) ** 2 * 0.9, device="cuda:0"))
        plan.check()
        assert np.linalg.norm(A - full) < 1e-4 * np.linalg.norm(full)
        assert np.all(np.isfinite(g.cpu().numpy()))
        if size == whole.info()["workspace_bytes"] and np.array_equal(A, full):
            plan.close()
            break  # past the last allocation
        # the direct form: what intensities take
        assert np.array_equal(plan.intensity(x).cpu().numpy(), direct)
        assert np.allclose(np.abs(A) ** 2, direct, rtol=1e-6, atol=0.0)
        plan.close()
        served += 1
    else:
        pytest.fail("allocations without end")
    assert served >= 5  # chunks of both, partials, records, offsets
