"""The moment engine, the far sum's parts and the self rules at the sizes where their tiles end:
one patch, 1 to 33 targets (tiles of 8, half a warp, a warp), leaf rules of 1 to 576 nodes
(pieces of 16 columns, rules beyond one piece of 128 nodes and beyond one chunk), every chunk
width (degrees up to 6 and above), self rules with more angles than the kept table; all against
the oracle with the bars of the parity tests."""
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


def one_patch(deg, axes=(1.0, 1.2, 0.9)):
    s = W.ellipsoid(1, deg, axes=axes)
    n = W.n_nodes(deg)
    return W.Surface("one", s.deg[:1].copy(), s.node_off[:2].copy(),
                     np.ascontiguousarray(s.xyz[:, :n]), {})


def check(g, oc, uo, tol=1e-10):
    """Structure, far order and refinement exactly, the applied potential at the FP64 bar.  (A
    pair's correction is a difference of moments that can cancel to nothing on a single smooth
    patch, so pairs are compared through the potential, which adds the smooth part back.)"""
    assert g["status"] == 0 and g["status_apply"] == 0
    assert np.array_equal(g["row_ptr"], oc.row_ptr) and np.array_equal(g["col"], oc.col)
    assert np.array_equal(g["q"], oc.q)
    if tol <= 1e-10:
        assert all(a == b for a, b, _ in leaves_by_pair(g, oc))
    assert np.linalg.norm(g["u"] - uo) <= tol * np.linalg.norm(uo)


# (degree, leaf rule, targets)
@pytest.mark.parametrize("deg,leaf,nt", [(1, 1, 1), (2, 3, 9), (3, 12, 8), (4, 16, 7), (4, 4, 33),
                                         (5, 24, 16), (6, 8, 17), (6, 11, 8), (7, 9, 15), (8, 12, 9),
                                         (10, 4, 3), (10, 8, 2)])
def test_tiles_and_pieces(ctx, deg, leaf, nt):
    s = one_patch(deg)
    x = W.radial_targets(s, nt, 11 * deg + leaf, 0.02, 0.5, True)
    tn = -np.ones(nt, np.int64)
    # a loose tolerance and a depth cap of 6 keep the small rules' trees short
    kw = dict(leaf_order=leaf, max_depth=6, eps_loosen=1e3)
    g = run_gpu(ctx, s, x, tn, "CFIE", 2.5, 1e-7, alpha=1.0, beta=-2.5j, **kw)
    g["status"] = 0 if g["status"] == 4 else g["status"]     # the depth cap is reported
    oc, uo = run_oracle(s, x, tn, "CFIE", 2.5, 1e-7, alpha=1.0, beta=-2.5j, sigma=g["sigma"], **kw)
    check(g, oc, uo)


@pytest.mark.parametrize("kind,k,precision", [("D", 1.5 + 0.7j, "fp64"), ("S", -3.0, "fp64"),
                                              ("Sp", 2.0, "fp64"), ("CFIE", 2.0, "mixed")])
def test_kernel_forms(ctx, kind, k, precision):
    """Complex k, negative k, S' and the two-float form through the engine and the far sum."""
    s = one_patch(5)
    x = W.radial_targets(s, 13, 5, 0.01, 1.5, True)
    tn = -np.ones(13, np.int64)
    nrm = np.random.default_rng(2).standard_normal((3, 13)) if kind == "Sp" else None
    a, b = (1.0, -1j * k) if kind == "CFIE" else (1.0, 0.0)
    g = run_gpu(ctx, s, x, tn, kind, k, 1e-8, alpha=a, beta=b, precision=precision, tgt_normal=nrm)
    oc, uo = run_oracle(s, x, tn, kind, k, 1e-8, alpha=a, beta=b, sigma=g["sigma"], tgt_normal=nrm)
    check(g, oc, uo, 1e-8 if precision == "mixed" else 1e-10)


@pytest.mark.parametrize("deg,order,axes", [(1, 6, (1.0, 1.2, 0.9)), (3, 24, (1.0, 1.0, 9.0)),
                                            (6, 11, (1.0, 2.0, 3.0)), (9, 7, (1.0, 1.2, 0.9))])
def test_self_rules(ctx, deg, order, axes):
    s = one_patch(deg, axes)
    x, tn = W.onsurface_targets(s)
    g = run_gpu(ctx, s, x, tn, "CFIE", 1.5, 1e-6, alpha=1.0, beta=-1.5j, self_order=order)
    oc, uo = run_oracle(s, x, tn, "CFIE", 1.5, 1e-6, alpha=1.0, beta=-1.5j, sigma=g["sigma"],
                        self_order=order)
    check(g, oc, uo)
