"""Plans that keep two node sets: crystals inside the smaller set's radius, between the
two and past both, in mixed order on one plan (eager, captured and replayed), are
summed by the first, the second set and the direct kernels.  A plan with the radius
hint of either set keeps that one alone, so which set served is read off the bits
of its map.  Against the oracle: FP32 2e-6, tensor cores 1e-4; gradients 1e-5 and 1e-4."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A
GID = dict(wavelength=W.WAVELENGTH_10KEV, alpha_i=W.GID_ALPHA_I, delta=W.GID_DELTA, beta=W.GID_BETA)
ORDER = ["small", "between", "past", "small", "past", "between", "between", "small", "small", "past", "past", "between"]


def _case(kind):
    """(crystal, axes, path, radii of the two sets, axes that count, gid)"""
    if kind == "gid":
        c, axes, path, f = W.truncated_pyramid(44, 16, 14), list(W.gid_axes(150, 150, 24)), "separable", (1.6, 2.3)
    else:
        cells, shape, step = (14.0, (80, 70, 50), 0.004) if kind == "generic" else (18.0, (128, 128, 64), 0.005)
        c, path, f = W.fcc_sphere(radius_cells=cells, seed=601), kind, (1.1, 1.3)
        axes = [W.linspace_axis(x, n, step=step) for x, n in zip((0.0, 0.0, 4.0), shape)]
    compact = np.cbrt(3 * len(c.xyz) / (16 * np.pi))
    return c, axes, path, [q * compact + 1.0 for q in f], 2 if kind == "gid" else 3


def _crystals(c, X, d):
    """The crystal with its two halves moved apart by whole cells along h, so that its largest |x'|
    comes to lie just inside the first radius, between the two and past the second.  The
    lattice stays in phase around the reflection."""
    x = c.xyz - np.rint(0.5 * (c.xyz.min(0) + c.xyz.max(0)))
    out = {}
    for name, lo, hi in (("small", 0.93 * X[0], X[0]), ("between", X[0], X[1]), ("past", X[1], 2.0 * X[1])):
        far = lambda k: np.abs(x[:, :d] + np.where(x[:, :1] > 0, k, -k) * np.eye(3)[0, :d]).max()
        k = next(k for k in range(100) if lo < far(k) < hi)
        out[name] = x + np.where(x[:, :1] > 0, k, -k) * np.eye(3)[0] + np.array([3.0, -2.0, 0.0 if d == 2 else 1.0])
    return out


def _plans(c, axes, path, X, **kw):
    make = lambda hint: api.Plan(c.coef, A_LAT, len(c.xyz), axes=axes, atom_species=c.species, path=path, radius_hint=hint,
                                 **kw)
    plan, one, two, bare = make(0.0), make(X[0]), make(X[1]), make(1e5)
    size = [p.info()["workspace_bytes"] - bare.info()["workspace_bytes"] for p in (plan, one, two)]
    assert size[1] > 0 and size[2] > 0 and abs(size[0] - size[1] - size[2]) < 256  # both sets
    return plan, {"small": one, "between": two, "past": bare}


@pytest.mark.parametrize("kind", ["generic", "separable", "gid"])
def test_maps(kind):
    c, axes, path, X, d = _case(kind)
    kw = {"gid": GID} if kind == "gid" else {}
    plan, own = _plans(c, axes, path, X, **kw)
    crystals = _crystals(c, X, d)
    want, size = {}, {}
    rng = np.random.default_rng(602)
    pts = W.grid_points(axes)
    idx = rng.choice(len(pts), 150, replace=False)
    for name, xyz in crystals.items():
        x = torch.tensor(xyz, device="cuda:0")
        want[name] = own[name].amplitude(x).clone()
        if name != "past":  # not the direct sum
            assert not torch.equal(want[name], own["past"].amplitude(x))
        got = want[name].cpu().numpy()
        ref = (oracle.dwba(xyz, pts[idx], c.coef, A_LAT, species=c.species, **GID) if kind == "gid"
               else oracle.amplitude(xyz, pts[idx], c.coef, A_LAT, species=c.species))
        scale = max(np.sqrt(np.mean(np.abs(got) ** 2)), np.sqrt(np.mean(np.abs(ref) ** 2)))
        assert np.sqrt(np.mean(np.abs(got[idx] - ref) ** 2)) < (2e-6 if kind == "generic" else 1e-4) * scale
    x = torch.tensor(crystals["small"], device="cuda:0")
    out = torch.empty(plan.n_s, dtype=torch.complex64, device="cuda:0")
    for name in ORDER:  # the same buffers: the second call captures, later ones replay
        x.copy_(torch.tensor(crystals[name], device="cuda:0"))
        out.fill_(complex(np.nan, np.nan))
        plan.amplitude(x, out=out)
        assert torch.equal(out, want[name]), name
        if kind == "generic":
            A = want[name]
            I = plan.intensity(x)
            assert torch.allclose(I, A.real ** 2 + A.imag ** 2, rtol=1e-6, atol=0.0)
        host = plan.amplitude_host(crystals[name])
        torch.cuda.synchronize()
        assert torch.equal(host.reshape(-1), want[name].cpu()), name
    plan.check()


@pytest.mark.parametrize("kind, tol", [("generic", 1e-5), ("separable", 1e-4)])
def test_gradients(kind, tol):
    c, axes, path, X, d = _case(kind)
    plan, own = _plans(c, axes, path, X)
    crystals = _crystals(c, X, d)
    rng = np.random.default_rng(603)
    A, I_obs, want = {}, {}, {}
    sel = rng.choice(len(c.xyz), 6, replace=False)
    for name, xyz in crystals.items():
        x = torch.tensor(xyz, device="cuda:0")
        A[name] = own["past"].amplitude(x).clone()
        I_obs[name] = (A[name].abs() ** 2 * torch.tensor(rng.uniform(0.7, 1.2, plan.n_s).astype(np.float32), device="cuda:0"))
        g = own[name].backward(x, A[name], I_obs[name])[1]
        direct = own["past"].backward(x, A[name], I_obs[name])[1]
        # a set has an adjoint of its own, or leaves the gradient to the map's own points
        want[name] = [g, direct]
        _, ref = oracle.loss_grad_atoms(xyz, W.grid_points(axes), A[name].cpu().numpy(), I_obs[name].cpu().numpy(), c.coef,
                                        A_LAT, sel, species=c.species)
        for v in (g, direct):
            assert np.linalg.norm(v.cpu().numpy()[sel] - ref) < tol * np.linalg.norm(ref)
    x = torch.tensor(crystals["small"], device="cuda:0")
    for name in ORDER:
        x.copy_(torch.tensor(crystals[name], device="cuda:0"))
        g = plan.backward(x, A[name], I_obs[name])[1]
        assert any(torch.equal(g, v) for v in want[name]), name
    plan.check()
    # the smaller set's gradient is in use
    x.copy_(torch.tensor(crystals["small"], device="cuda:0"))
    assert not torch.equal(plan.backward(x, A["small"], I_obs["small"])[1], want["small"][1])


def _shell(R, thickness):
    n = int(np.ceil(R)) + 1
    g = np.stack(np.meshgrid(*(np.arange(-n, n + 1),) * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.float64)
    g = np.concatenate([g + o for o in ([0, 0, 0], [0.5, 0.5, 0], [0.5, 0, 0.5], [0, 0.5, 0.5])])
    r = np.linalg.norm(g, axis=1)
    return g[(r <= R) & (r > R - thickness)]


def _lobes(R, q):
    b = _shell(q, q)
    s = np.rint((R - q) * np.array([0.8, 0.5, 0.33]) / np.linalg.norm([0.8, 0.5, 0.33]))
    return np.concatenate([b + s, b - s])


@pytest.mark.parametrize("kind, tol", [("list", 2e-6), ("generic", 2e-6), ("separable", 1e-4)])
@pytest.mark.parametrize("crystal", [lambda: _shell(18.0, 2.0), lambda: _lobes(22.0, 10.5)])
@pytest.mark.parametrize("part", [0.95, 0.999])
def test_atoms_at_the_radius(kind, tol, crystal, part):
    """Hollow and two-lobed crystals, all of whose atoms are far out, at 0.95 to 1.0 of the radius."""
    rng = np.random.default_rng(604)
    xyz = crystal()
    xyz = xyz + rng.normal(0.0, 0.004, xyz.shape)
    coef = W.unit_species()[None]
    far = np.linalg.norm(xyz, axis=1).max() if kind == "list" else np.abs(xyz).max()
    if kind == "list":
        kw = dict(s_list=W.ewald_slice(60001, rocking_deg=0.02, seed=605))
        S = kw["s_list"]
    else:
        shape, step = ((80, 70, 50), 0.002) if kind == "generic" else ((160, 160, 64), 0.003)
        kw = dict(axes=[W.linspace_axis(x, n, step=step) for x, n in zip((0.01, 0.0, 4.0), shape)], path=kind)
        S = W.grid_points(kw["axes"])
    plan = api.Plan(coef, A_LAT, len(xyz), radius_hint=far / part, **kw)
    bare = api.Plan(coef, A_LAT, len(xyz), **(dict(kw, split_k=1) if kind == "list" else dict(kw, radius_hint=1e5)))
    x = torch.tensor(xyz, device="cuda:0")
    A, B = plan.amplitude(x).cpu().numpy(), bare.amplitude(x).cpu().numpy()
    plan.check()
    assert not np.array_equal(A, B)  # clusters or nodes served
    idx = np.concatenate([rng.choice(len(S), 300, replace=False), np.argsort(np.abs(B))[-30:]])
    ref = oracle.amplitude(xyz, S[idx], coef, A_LAT)
    assert np.linalg.norm(A[idx] - ref) < tol * np.linalg.norm(ref)
    assert np.linalg.norm(A - B) < tol * np.linalg.norm(B)
