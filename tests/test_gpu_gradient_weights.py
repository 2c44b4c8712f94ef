"""A gradient is -2 pi w_j times a sum that does not depend on w_j, so a call with
occupancies w and one with ones give the same sum: each gradient is rounded once to
FP32, and their quotients by w differ by at most two such roundings (2 x 2^-24 of the
value, and 2^-40 for the double-float sums)."""
import numpy as np
import pytest

from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


@pytest.mark.parametrize("kind, shape, uneven, form", [
    ("list", 700, False, 1), ("patch", 30011, False, 1),
    ("generic", (16, 14, 12), False, 2), ("generic", (5, 4, 3), True, 1), ("generic", (80, 63, 48), False, 2),
    ("separable", (64, 40, 40), False, 3), ("separable", (33, 20, 21), True, 3),
])
def test_gradient_scales_with_the_occupancy(kind, shape, uneven, form):
    rng = np.random.default_rng(531)
    c = W.fcc_sphere(radius_cells=9.0, seed=532)
    n = len(c.xyz)
    kw = {}
    if kind in ("list", "patch"):
        kw["s_list"] = (W.ewald_slice(shape, rocking_deg=0.02, seed=533) if kind == "patch"
                        else np.array([0.0, 0.0, 4.0]) + rng.uniform(-0.3, 0.3, (shape, 3)))
    else:
        step = 0.002 if shape[0] == 80 else 0.05
        kw["axes"] = [W.linspace_axis(x, m, step=step) for x, m in zip((0.0, 0.0, 4.0), shape)]
        if uneven:
            kw["axes"] = [a + rng.uniform(-0.2, 0.2, len(a)) * step for a in kw["axes"]]
        kw["path"] = kind
    plan = api.Plan(c.coef, A_LAT, n, atom_species=c.species, **kw)
    G = torch.tensor((rng.normal(size=plan.n_s) + 1j * rng.normal(size=plan.n_s)).astype(np.complex64), device="cuda:0")
    x = torch.tensor(c.xyz, device="cuda:0")
    w = rng.uniform(0.5, 1.0, n).astype(np.float32)
    w[:4] = [2.0 ** -30, 3e-20, -0.7, 1e6]
    one = plan.vjp(x, G, torch.ones(n, device="cuda:0")).cpu().numpy().astype(np.float64)
    got = plan.vjp(x, G, torch.tensor(w, device="cuda:0")).cpu().numpy().astype(np.float64)
    plan.check()
    assert plan.info()["adjoint_form"] == form
    off = np.abs(got / w[:, None].astype(np.float64) - one)
    assert np.all(off <= (2.0 * 2.0 ** -24 + 2.0 ** -40) * np.abs(one))


def test_overflow_and_zero():
    xyz = np.array([[0.2, 0.1, 0.3], [0.4, -0.3, 0.25], [0.1, 0.7, -0.2]])
    S = np.array([[1.0, 2.0, 4.1], [0.3, -0.4, 3.9]])
    plan = api.Plan(W.unit_species()[None], A_LAT, 3, s_list=S)
    G = torch.tensor(np.array([1.0 + 2.0j, -0.5 + 1.0j], dtype=np.complex64) * np.float32(1e3), device="cuda:0")
    g = plan.vjp(torch.tensor(xyz, device="cuda:0"), G, torch.tensor([0.0, 3e37, 1.0], device="cuda:0")).cpu().numpy()
    assert np.all(g[0] == 0.0) and np.all(np.isinf(g[1])) and np.all(np.isfinite(g[2]))
