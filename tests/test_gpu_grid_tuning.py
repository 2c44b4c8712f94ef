"""Tuned FP32 grids: a cache entry serves plans of its launch shape only, and every
entry that is written is found again.  Maps against the oracle at the FP32 sums'
1e-5."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


def _axes(shape, uneven):
    rng = np.random.default_rng(541)
    axes = [W.linspace_axis(x, n, step=0.03) for x, n in zip((0.0, 0.0, 4.0), shape)]
    return [a + rng.uniform(-0.005, 0.005, len(a)) for a in axes] if uneven else axes


def test_entries_serve_their_own_shape(tmp_path):
    cache = tmp_path / "tune.jsonl"
    c = W.fcc_sphere(radius_cells=5.0, seed=542)
    # the same last axis and number of points throughout
    shapes = [((40, 10, 24), False), ((10, 40, 24), False), ((10, 40, 24), True), ((400, 1, 24), False)]
    for i, (shape, uneven) in enumerate(shapes):
        axes = _axes(shape, uneven)
        splits = []
        for _ in range(2):
            plan = api.Plan(c.coef, A_LAT, len(c.xyz), axes=axes, atom_species=c.species, path="generic", autotune=True,
                            tune_cache=str(cache))
            splits.append(plan.info()["split_k"])
            assert cache.read_text().count("\n") == i + 1
        assert splits[0] == splits[1]
        A = plan.amplitude(torch.tensor(c.xyz, device="cuda:0")).cpu().numpy()
        ref = oracle.amplitude(c.xyz, W.grid_points(axes), c.coef, A_LAT, species=c.species)
        assert np.linalg.norm(A - ref) < 1e-5 * np.linalg.norm(ref)


def test_many_chunks_are_found_again(tmp_path):
    cache = tmp_path / "tune.jsonl"
    n = 1000000
    axes = _axes((16, 16, 2), False)
    for _ in range(2):
        plan = api.Plan(W.unit_species()[None], A_LAT, n, axes=axes, path="generic", autotune=True, tune_cache=str(cache))
        assert plan.info()["split_k"] > 256
        assert cache.read_text().count("\n") == 1
