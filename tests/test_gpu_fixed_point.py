"""The fixed-point arithmetic of the moment engine, the self rules and the sums where its scales
could show in the results."""
import numpy as np
import pytest

from paper_2006_02545_gb300 import workloads as W
from .gpu_helpers import leaves_by_pair, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    from paper_2006_02545_gb300 import lcq
    c = lcq.Context(0)
    yield c
    c.close()


def one_patch(deg):
    s = W.ellipsoid(2, deg, axes=(1.0, 1.2, 0.9))
    n = W.n_nodes(deg)
    return W.Surface("one", s.deg[:1].copy(), s.node_off[:2].copy(),
                     np.ascontiguousarray(s.xyz[:, :n]), {})


def near_points(s, nt, seed=1):
    """Points 1e-3 to 0.3 off the patch, above its nodes."""
    rng = np.random.default_rng(seed)
    i = np.arange(nt) % s.n_points
    return np.ascontiguousarray(s.xyz[:, i] * (1.0 + 10.0 ** rng.uniform(-3, -0.5, nt)))


@pytest.mark.parametrize("deg", [3, 4, 6, 7, 8])
@pytest.mark.parametrize("far", [1e3, 1e9, 1e18])
def test_a_distant_target_leaves_the_others_alone(ctx, deg, far):
    """A target's corrections do not depend on the targets it shares the patch with: the
    allocation-free entry with its last target 2 away and far away gives the same rows of the
    others bit for bit; so does a generation (the far order at its cap, so that it is the same)."""
    import torch
    from paper_2006_02545_gb300 import lcq
    s, nt = one_patch(deg), 21
    x = near_points(s, nt)
    n = W.n_nodes(deg)
    y = torch.from_numpy(s.xyz).cuda()
    rows, vals = [], []
    for dist in (2.0, far):
        x[:, -1] = x[:, 0] * dist
        out = torch.zeros((nt, n), dtype=torch.complex128, device="cuda")
        st = lcq.adaptive_corrections_noalloc(deg, y, torch.from_numpy(x).cuda(), "CFIE", 2.0, 8, 1e-6,
                                              out, 1.0, -2j, max_depth=6)
        assert st in (0, 4)                       # the depth cap is reported
        rows.append(out.cpu().numpy())
        g = run_gpu(ctx, s, x, -np.ones(nt, np.int64), "CFIE", 2.0, 1e-12, eta=4 * far, alpha=1.0,
                    beta=-2j, eta1=4 * far, m_max=6, leaf_order=8, max_depth=5, eps_loosen=1e6)
        assert g["status"] in (0, 4) and g["q"][0] == 6
        vals.append(g["val"].reshape(nt, n))
    assert np.isfinite(rows[1]).all() and np.abs(rows[0]).max() > 0
    assert np.array_equal(rows[0][:-1], rows[1][:-1])
    assert np.array_equal(vals[0][:-1], vals[1][:-1])


def test_group_size_with_targets_far_beyond_the_patch():
    """The group size stays without effect on the results when adaptive targets lie well outside
    their patch's coordinate range (a large eta1)."""
    from paper_2006_02545_gb300 import lcq
    s = W.ellipsoid(2, 4, axes=(1.0, 1.5, 2.0))
    rng = np.random.default_rng(4)
    x = rng.standard_normal((3, 300))
    x *= 10.0 ** rng.uniform(0.35, 2.0, 300) / np.linalg.norm(x, axis=0)
    tn = -np.ones(300, np.int64)
    c = lcq.Context(0)
    try:
        runs, sizes = [], []
        for _ in range(6):
            g = run_gpu(c, s, x, tn, "CFIE", 1.0, 1e-8, 400.0, alpha=1.0, beta=-1j, eta1=400.0)
            assert g["status"] == 0
            sizes.append(int(c.counters()[5]))
            runs.append(g)
        assert len(set(sizes)) >= 2, sizes
        for g in runs[1:]:
            assert np.array_equal(g["val"], runs[0]["val"])
            assert np.array_equal(g["leaves"], runs[0]["leaves"])
    finally:
        c.close()


def coarse_patch(deg):
    """A patch of a torus far too coarse for its degree: its nodes take the FP64 recurrences."""
    s = W.torus(3, 3, deg)
    n = W.n_nodes(deg)
    return W.Surface("coarse", s.deg[:1].copy(), s.node_off[:2].copy(),
                     np.ascontiguousarray(s.xyz[:, :n]), {})


@pytest.mark.parametrize("deg,kind,precision,eps", [(6, "CFIE", "fp64", 1e-7), (8, "S", "fp64", 1e-7),
                                                    (10, "D", "fp64", 1e-6), (6, "Sp", "fp64", 1e-6),
                                                    (8, "CFIE", "mixed", 1e-7), (6, "D", "mixed", 1e-5)])
def test_coarse_patches(ctx, deg, kind, precision, eps):
    """Adaptive, smooth-rule and self integration on a chart that the fixed-point scales do not fit,
    against the oracle: leaf counts and the potential at the parity bars (the tiers of the mixed form
    keep FP64 values on such a chart, and their own rounding floors)."""
    s = coarse_patch(deg)
    rng = np.random.default_rng(deg)
    i = rng.integers(0, s.n_points, 9)
    x = s.xyz[:, i] + rng.standard_normal((3, 9)) * 0.2
    xs, ts = W.onsurface_targets(s)
    x = np.ascontiguousarray(np.concatenate([x, xs[:, :5]], axis=1))
    tn = np.concatenate([-np.ones(9, np.int64), ts[:5]])
    nrm = rng.standard_normal((3, 14)) if kind == "Sp" else None
    a, b = (1.0, -1j) if kind == "CFIE" else (1.0, 0.0)
    kw = dict(max_depth=7, eps_loosen=10.0)
    g = run_gpu(ctx, s, x, tn, kind, 1.0, eps, alpha=a, beta=b, precision=precision, tgt_normal=nrm, **kw)
    assert g["status"] in (0, 4)
    oc, uo = run_oracle(s, x, tn, kind, 1.0, eps, alpha=a, beta=b, sigma=g["sigma"], tgt_normal=nrm, **kw)
    assert np.array_equal(g["q"], oc.q)
    if precision == "fp64":
        assert all(p == q for p, q, _ in leaves_by_pair(g, oc))
    tol = 1e-10 if precision == "fp64" else eps
    assert np.linalg.norm(g["u"] - uo) <= tol * np.linalg.norm(uo)


@pytest.mark.parametrize("deg", [3, 6])
@pytest.mark.parametrize("kind", ["S", "D", "Sp"])
def test_low_frequency_imaginary_part(ctx, deg, kind):
    """The imaginary part at |k| r near zero, far below the real one, through generation, apply and
    adjoint with real densities: S ~ k against the oracle; D and S' ~ k^3, whose ratio at two wave
    numbers is the cube of theirs up to (k r)^2 < 1e-11."""
    import torch
    from paper_2006_02545_gb300 import lcq
    s = W.ellipsoid(1, deg, axes=(1.0, 1.2, 0.9))
    xs, ts = W.onsurface_targets(s)
    x = np.ascontiguousarray(np.concatenate([xs[:, ::3] * 1.05, xs], axis=1))
    tn = np.concatenate([-np.ones(xs[:, ::3].shape[1], np.int64), ts])
    nrm = np.random.default_rng(3).standard_normal(x.shape) if kind == "Sp" else None
    sig = np.random.default_rng(1).standard_normal(s.n_points) + 0j
    gt = np.random.default_rng(2).standard_normal(x.shape[1]) + 0j
    fn = {"S": lcq.apply_corrected_S, "D": lcq.apply_corrected_D, "Sp": lcq.apply_corrected_Sp}[kind]
    parts = []
    ks = (1e-12,) if kind == "S" else (1e-6, 1e-8)
    for k in ks:
        g = run_gpu(ctx, s, x, tn, kind, k, 1e-7, tgt_normal=nrm)
        assert g["status"] == 0
        u = fn(ctx, g["ds"], g["near"], g["corr"], torch.from_numpy(sig).cuda(), x.shape[1])
        z = lcq.apply_adjoint(ctx, g["ds"], g["near"], g["corr"], torch.from_numpy(gt).cuda())
        assert ctx.sync(60000) == 0
        parts.append((u.cpu().numpy().imag, z.cpu().numpy().imag))
    if kind == "S":
        oc, uo = run_oracle(s, x, tn, kind, ks[0], 1e-7, sigma=sig)
        u, z = parts[0]
        assert np.linalg.norm(u - uo.imag) <= 1e-10 * np.linalg.norm(uo.imag)
        # <g, A sigma> = <A^H g, sigma>, the imaginary part
        assert abs(gt.real @ u + z @ sig.real) <= 1e-10 * np.linalg.norm(u) * np.linalg.norm(gt)
    else:
        for a, b in zip(*parts):
            assert np.linalg.norm(a * (ks[1] / ks[0]) ** 3 - b) <= 1e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("deg", [3, 6])
def test_target_normal_of_length_zero(ctx, deg):
    """S' at a target whose normal is zero is not a number, in the corrections, the potential and the
    adjoint, and the other targets stay what they are without it."""
    import torch
    from paper_2006_02545_gb300 import lcq
    s = one_patch(deg)
    x = near_points(s, 6)
    tn = -np.ones(6, np.int64)
    nrm = np.random.default_rng(5).standard_normal((3, 6))
    ok = run_gpu(ctx, s, x, tn, "Sp", 2.0, 1e-6, tgt_normal=nrm)
    nrm[:, 2] = 0.0
    g = run_gpu(ctx, s, x, tn, "Sp", 2.0, 1e-6, tgt_normal=nrm)
    assert ok["status"] == 0 and g["status"] != 0
    v, w = g["val"].reshape(6, -1), ok["val"].reshape(6, -1)
    rest = [0, 1, 3, 4, 5]
    assert np.isnan(v[2]).all() and np.isnan(g["u"][2])
    assert np.array_equal(v[rest], w[rest]) and np.array_equal(g["u"][rest], ok["u"][rest])
    z = lcq.apply_adjoint(ctx, g["ds"], g["near"], g["corr"], torch.ones(6, dtype=torch.complex128).cuda())
    ctx.sync(60000)
    assert np.isnan(z.cpu().numpy()).all()


@pytest.mark.parametrize("deg", [3, 6])
@pytest.mark.parametrize("bad", [dict(beta=np.inf), dict(beta=complex(0, np.nan)), dict(alpha=np.inf)])
def test_constants_not_finite(ctx, deg, bad):
    """The allocation-free entry takes any constants; those that are not finite make every correction
    a NaN and the status says so."""
    import torch
    from paper_2006_02545_gb300 import lcq
    s = one_patch(deg)
    n = W.n_nodes(deg)
    x = torch.from_numpy(near_points(s, 5)).cuda()
    out = torch.zeros((5, n), dtype=torch.complex128, device="cuda")
    kw = dict(alpha=1.0, beta=0.0, max_depth=6)
    kw.update(bad)
    st = lcq.adaptive_corrections_noalloc(deg, torch.from_numpy(s.xyz).cuda(), x, "CFIE", 1.0, 8, 1e-6,
                                          out, **kw)
    assert st == 2                                    # LCQ_ERR_NONFINITE
    assert not torch.isfinite(torch.view_as_real(out)).all(-1).any()


@pytest.mark.parametrize("deg,kind", [(1, "S"), (2, "D"), (3, "CFIE")])
@pytest.mark.parametrize("scale", [1e-25, 1e25])
def test_surfaces_of_any_size(ctx, deg, kind, scale):
    """The smallest degrees in units far from 1: refinement (whose rounding floor comes from the
    kernel's envelope) and potential as the oracle's."""
    s = one_patch(deg)
    s.xyz[:] *= scale
    x = near_points(s, 9)
    tn = -np.ones(9, np.int64)
    k = 2.0 / scale
    a, b = (1.0, -1j * k) if kind == "CFIE" else (1.0, 0.0)
    kw = dict(max_depth=8, self_order=6)
    eps = 1e-9 / (1.0 if kind == "S" else scale)      # the tolerance is eps times a length
    g = run_gpu(ctx, s, x, tn, kind, k, eps, alpha=a, beta=b, leaf_order=6, **kw)
    oc, uo = run_oracle(s, x, tn, kind, k, eps, alpha=a, beta=b, sigma=g["sigma"], leaf_order=6, **kw)
    assert g["status"] in (0, 4)
    assert all(p == q for p, q, _ in leaves_by_pair(g, oc))
    assert np.linalg.norm(g["u"] - uo) <= 1e-10 * np.linalg.norm(uo)
