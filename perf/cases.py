"""The workloads by which this library's speed is judged: what a boundary-integral program
has it do, through its public entry points, from the smallest surface to a large one.

Operations (the "op" of a case):
  gen      near lists and correction weights of a surface, exported as a device CSR
  batch    the same for several independent surfaces of unlike degree, size, wave number and
           tolerance in one call
  plan     one captured regeneration after the nodes moved, and its CSR values
  field    near lists, corrections and the corrected potential at points off the surface
  apply    one corrected potential with the corrections at hand (an iterative solver's step)
  adjoint  one A^H g with the corrections at hand (the adjoint solve's step)
  grad     the corrected potential and its gradients by density and node coordinates

Surfaces are the library's synthetic ones (paper_2006_02545_gb300/workloads.py), turned by a
random rotation and scaled by up to a tenth (the wave number stays), both from the seed, so that
another seed is another scattering problem with another density and the same sparsity.
"""
import functools
import math

import numpy as np
import torch

from paper_2006_02545_gb300 import lcq
from paper_2006_02545_gb300 import workloads as W
from paper_2006_02545_gb300.autograd import corrected_potential

_APPLY = {"S": lcq.apply_corrected_S, "D": lcq.apply_corrected_D,
          "CFIE": lcq.apply_corrected_CFIE, "Sp": lcq.apply_corrected_Sp}


def listed():
    tau = 2.0 * math.pi
    return [
        # the smallest surface in use, 300 points: launches, host work and the longest walk
        _case("sphere20 S gen", "gen", "sphere", 1, 1, 4, "S", 1.0, 0.0, 1e-6, eta=1.25),
        # shape optimisation: a mid-size surface regenerated in place as its nodes move
        _case("ellipsoid320 CFIE plan", "plan", "ellipsoid", 4, 4, 6, "CFIE", math.pi, 0.0, 1e-7),
        # the ordinary set-up of a scattering solve in double precision, and in the mixed form
        _case("ellipsoid1280 CFIE gen", "gen", "ellipsoid", 8, 8, 6, "CFIE", tau, 0.0, 1e-9),
        _case("ellipsoid1280 CFIE mixed", "gen", "ellipsoid", 8, 8, 6, "CFIE", tau, 0.0, 1e-9,
              precision="mixed"),
        # low order on stretched patches: the twisted torus at order p = 4
        _case("stellarator2400 S gen", "gen", "stellarator", 20, 60, 3, "S", 1.0, 0.0, 5e-7),
        # a large surface at a high wave number
        _case("torus2916 CFIE gen", "gen", "torus", 27, 54, 6, "CFIE", 20.0, 0.0, 1e-9),
        # many unlike surfaces at once (degrees 3..8, odd sizes, two tolerances)
        _case("tori10 CFIE batch", "batch", "torus", 10, 10, 8, "CFIE", 20.0, 0.0, 1e-9,
              precision="mixed"),
        # a damped wave's double layer at points off the surface, high order, odd sizes
        _case("torus242 D field", "field", "torus", 11, 11, 8, "D", 7.3, 0.4, 1e-6, n_tgt=4099),
        # solver steps: one on a small sphere, one on the ordinary surface, one adjoint
        _case("sphere320 S apply", "apply", "sphere", 4, 4, 6, "S", 1.0, 0.0, 1e-8),
        _case("ellipsoid1280 CFIE apply", "apply", "ellipsoid", 8, 8, 6, "CFIE", tau, 0.0, 1e-9),
        _case("ellipsoid500 CFIE adjoint", "adjoint", "ellipsoid", 5, 5, 6, "CFIE", 4.0, 0.0,
              1e-7),
        # gradients by density and shape of the potential at 1000 exterior points
        _case("ellipsoid2000 S grad", "grad", "ellipsoid", 10, 10, 5, "S", 5.0, 0.0, 1e-8,
              n_tgt=1000),
    ]


def _case(name, op, shape, a, b, deg, kernel, k_re, k_im, eps, eta=-1.0, precision="fp64",
          n_tgt=0):
    c = dict(op=op, shape=shape, a=a, b=b, deg=deg, kernel=kernel, k_re=k_re, k_im=k_im, eps=eps,
             eta=eta, precision=precision, n_tgt=n_tgt)
    return dict(name=name, **c) if name else c


def draw(rng):
    """A case of the same ranges: surfaces of 20 to about 2500 patches of degree 1 to 8 and at
    most 36,000 points, k from 0.5 to 20, eps from 5e-3 to 5e-10, all kernels and forms."""
    op = rng.choice(["gen", "gen", "gen", "batch", "plan", "field", "apply", "apply", "adjoint",
                     "grad"])
    deg = rng.randint(3, 8) if rng.random() < 0.75 else rng.randint(1, 2)
    n = W.n_nodes(deg)
    if op == "batch":
        return _case("", "batch", "torus", rng.randint(2, 10), 10, 8,
                     rng.choice(["CFIE", "S", "D"]), 20.0, 0.0, 1e-9,
                     precision=rng.choice(["fp64", "mixed"]))
    most = {"gen": 36000, "plan": 9000, "field": 9000, "apply": 36000, "adjoint": 14000,
            "grad": 36000}[op]
    patches = math.exp(rng.uniform(math.log(20), math.log(max(24, min(2500, most // n)))))
    shape = rng.choice(["ellipsoid", "torus", "stellarator"])
    if op == "grad":
        shape = "ellipsoid"  # its exterior points need a body that is star-shaped
    if shape == "ellipsoid":
        a = b = max(1, int(math.sqrt(patches / 20.0)))
    else:
        # cells of unlike sides, the stretched ones among them
        asp = math.exp(rng.uniform(math.log(1.0), math.log(3.0)))
        a = max(3, int(math.sqrt(patches / 2.0 / asp)))
        b = max(3, int(patches / 2.0 / a))
    kernel = rng.choice(["S", "D", "CFIE"] if op == "grad" else ["S", "D", "CFIE", "CFIE", "Sp"])
    k_im = rng.choice([0.0, 0.0, 0.0, 0.3]) if op in ("gen", "field", "apply") else 0.0
    # wave numbers that the patches still resolve: a user refines a surface with k
    k = math.exp(rng.uniform(math.log(0.5), math.log(max(0.6, min(20.0, 1.2 * math.sqrt(patches))))))
    eps = math.exp(rng.uniform(math.log(5e-10), math.log(5e-3 if deg <= 4 else 1e-5)))
    prec = "mixed" if op in ("gen", "plan") and rng.random() < 0.3 else "fp64"
    nt = 0
    if op == "field":
        nt = int(math.exp(rng.uniform(math.log(100), math.log(8000))))
    elif op == "grad":
        nt = int(math.exp(rng.uniform(math.log(50), math.log(1000))))
    return _case("", op, shape, a, b, deg, kernel, k, k_im, eps, precision=prec, n_tgt=nt)


# ----------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _base(shape, a, b, deg):
    if shape == "sphere":
        return W.ellipsoid(a, deg)
    if shape == "ellipsoid":
        return W.ellipsoid(a, deg, axes=(1.0, 1.5, 2.5) if a >= 10 else (1.0, 2.0, 3.0))
    if shape == "torus":
        return W.torus(a, b, deg)
    return W.stellarator(a, b, deg)


@functools.lru_cache(maxsize=None)
def _ctx():
    """The process's library context (a program makes one and keeps it)."""
    return lcq.Context(0)


def _rng(seed):
    return np.random.default_rng(seed)


def _motion(rng, rigid=False):
    """A random rotation, times a scale between 0.9 and 1.1 unless rigid."""
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))
    if np.linalg.det(q) < 0:
        q[:, 0] = -q[:, 0]
    return q if rigid else q * rng.uniform(0.9, 1.1)


def _physics(case):
    k = complex(case["k_re"], case["k_im"])
    return k, 1.0, (-1j * k if case["kernel"] == "CFIE" else 0.0)


def _batch_parts(case):
    """Tori of unlike sizes: 8 to 400 patches, degrees 3..8, k 1..12, eps 1e-6 or 1e-9."""
    rng = _rng(1000 + case["a"])
    parts, phys = [], []
    for i in range(case["a"]):
        deg = 3 + i % 6
        nt = int(round(math.exp(rng.uniform(math.log(3.0), math.log(10.0)))))
        parts.append(_base("torus", nt, 2 * nt + i % 3 - 1, deg))
        k = float(rng.uniform(1.0, 12.0))
        phys.append((k, 1.0, -1j * k if case["kernel"] == "CFIE" else 0.0,
                     1e-6 if i % 2 else 1e-9))
    return parts, phys


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _harmonics(x, coef):
    """sum_l sum_m c_lm Y_lm for l = 0..2 (real, unnormalized), by degree l."""
    X, Y, Z = x
    one = np.ones_like(X)
    basis = [[one], [X, Y, Z], [X * Y, Y * Z, X * Z, X * X - Y * Y, 3.0 * Z * Z - 1.0]]
    out, i = [], 0
    for fs in basis:
        s = np.zeros_like(X, dtype=complex)
        for f in fs:
            s = s + coef[i] * f
            i += 1
        out.append(s)
    return out


def _sphere_inputs(case, seed):
    """Nodes of the rotated unit sphere, and a density of spherical harmonics up to degree 2."""
    rng = _rng(seed)
    xyz = _motion(rng, rigid=True) @ _base("sphere", case["a"], case["b"], case["deg"]).xyz
    coef = rng.standard_normal(9) + 1j * rng.standard_normal(9)
    return xyz, coef


def prepare(case, seed):
    ctx = _ctx()
    op, rng = case["op"], _rng(seed)
    st = dict(case=case, ctx=ctx)
    k, alpha, beta = _physics(case)
    dirs = W.test_directions(seed % 1000)
    st["prm"] = lcq.params(case["eps"], eta=case["eta"], test_dirs=dirs)
    if op == "batch":
        parts, phys = _batch_parts(case)
        shifts, moved = [], []
        for i, p in enumerate(parts):
            shifts.append((9.0 * (i % 4), 9.0 * (i // 4), 0.0))
            moved.append(W.Surface(p.name, p.deg, p.node_off, _motion(rng) @ p.xyz, p.meta))
        surf, st["patch_off"] = W.concat_surfaces(moved, shifts)
        st["phys"] = phys
        xyz = surf.xyz
    else:
        surf = _base(case["shape"], case["a"], case["b"], case["deg"])
        if case["shape"] == "sphere":
            xyz, coef = _sphere_inputs(case, seed)
        else:
            xyz = _motion(rng) @ surf.xyz
    xyz = np.ascontiguousarray(xyz)
    n = surf.n_points
    sig = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    if case["shape"] == "sphere":
        sig = sum(_harmonics(xyz, coef))
    st["sigma"] = _dev(sig)
    st["xyz"] = _dev(xyz)
    st["surf"] = lcq.DeviceSurface(surf.deg, surf.node_off, st["xyz"])
    if case["n_tgt"]:
        # points off the surface: node positions moved along the radius (field: to both sides)
        nt = case["n_tgt"]
        idx = rng.integers(0, n, nt)
        delta = rng.uniform(0.05, 0.5, nt) if op == "grad" else rng.uniform(-0.3, 0.6, nt)
        st["tx"] = _dev(xyz[:, idx] * (1.0 + delta))
        st["tn"] = torch.full((nt,), -1, dtype=torch.int64, device="cuda")
        if case["kernel"] == "Sp":
            st["nrm"] = _dev(rng.standard_normal((3, nt)))
    else:
        st["tx"] = _dev(xyz)
        st["tn"] = _dev(np.arange(n, dtype=np.int64))
    if op in ("apply", "adjoint", "plan"):
        near, corr = _generate(st)
        st["near"], st["corr"] = near, corr
        if op == "plan":
            st["val"] = torch.empty(max(near.nnz, 1), dtype=torch.complex128, device="cuda")
            st["plan"] = lcq.Plan(ctx, st["surf"], near, corr)
            # the nodes as they are after the step of the optimisation that comes next
            st["xyz"].mul_(1.0 + 0.01 * float(rng.uniform(0.5, 1.0)))
        st["g"] = _dev(rng.standard_normal(n) + 1j * rng.standard_normal(n))
    torch.cuda.synchronize()
    return st


# ----------------------------------------------------------------------------- one pass
def _generate(st):
    c, ctx = st["case"], st["ctx"]
    if c["op"] == "batch":
        near = lcq.build_near_lists_batched(ctx, st["surf"], st["patch_off"], st["tx"], st["tn"],
                                            st["prm"])
        return near, lcq.gen_corrections_batched(ctx, st["surf"], near, c["kernel"], st["phys"],
                                                 st["prm"], precision=c["precision"])
    k, alpha, beta = _physics(c)
    near = lcq.build_near_lists(ctx, st["surf"], st["tx"], st["tn"], st["prm"])
    if "nrm" in st:
        near.set_target_normals(st["nrm"])
    return near, lcq.gen_corrections(ctx, st["surf"], near, c["kernel"], k, st["prm"], alpha, beta,
                                     precision=c["precision"])


def run(st):
    c, ctx = st["case"], st["ctx"]
    op, nt = c["op"], int(st["tn"].shape[0])
    if op in ("gen", "batch"):
        near, corr = _generate(st)
        nnz = max(near.nnz, 1)
        out = (torch.empty(nt + 1, dtype=torch.int64, device="cuda"),
               torch.empty(nnz, dtype=torch.int32, device="cuda"),
               torch.empty(nnz, dtype=torch.complex128, device="cuda"))
        rp, col, val = corr.export(nt, out)
        corr.close()
        near.close()
        return {"row_ptr": rp, "col": col, "val": val}
    if op == "plan":
        st["plan"].launch()
        st["corr"].export(nt, (None, None, st["val"]))
        return {"val": st["val"]}
    if op == "field":
        near, corr = _generate(st)
        u = _APPLY[c["kernel"]](ctx, st["surf"], near, corr, st["sigma"], nt)
        corr.close()
        near.close()
        return {"u": u}
    if op == "apply":
        jump = {"D": 0.5, "CFIE": 0.5, "Sp": -0.5}.get(c["kernel"], 0.0)
        return {"u": _APPLY[c["kernel"]](ctx, st["surf"], st["near"], st["corr"], st["sigma"], nt,
                                         jump)}
    if op == "adjoint":
        return {"z": lcq.apply_adjoint(ctx, st["surf"], st["near"], st["corr"], st["g"], 0.5)}
    k, alpha, beta = _physics(c)
    xyz = st["xyz"].detach().requires_grad_(True)
    sig = st["sigma"].detach().requires_grad_(True)
    u = corrected_potential(ctx, st["surf"].deg, st["surf"].node_off, xyz, sig, st["tx"],
                            st["tn"], c["kernel"], k, st["prm"], alpha, beta)
    gy, gs = torch.autograd.grad((u.real ** 2 + u.imag ** 2).sum(), (xyz, sig))
    return {"u": u.detach(), "grad_xyz": gy, "grad_sigma": gs}


# ----------------------------------------------------------------------------- work
def _counts(case):
    """(surface points, basis size) of a case, summed over a batch's surfaces."""
    if case["op"] == "batch":
        return [(p.n_points, W.n_nodes(int(p.deg[0])), ph[3])
                for p, ph in zip(*_batch_parts(case))]
    s = _base(case["shape"], case["a"], case["b"], case["deg"])
    return [(s.n_points, W.n_nodes(case["deg"]), case["eps"])]


def work(case):
    """Bytes and operations of one pass.  Near entries per target: the nodes inside a disc of
    radius eta R around a patch of three equal sides, 2.42 eta^2 n.  Kernel evaluations per near
    pair: the nodes of the accepted leaves of a refinement that halves a triangle until it is as
    far from the target as it is large, 3 children a level over log4(1/eps) levels, on rules of
    as many nodes as digits ask for.  An evaluation is 23 operations, its contraction 4 a basis
    function; a far evaluation 31."""
    by = fl = 0.0
    for n, nb, eps in _counts(case):
        deg = int(round((math.sqrt(8.0 * nb + 1.0) - 3.0) / 2.0))
        eta = case["eta"] if case["eta"] > 0 else 2.75 if deg <= 3 else 2.0 if deg <= 7 else 1.25
        nt = case["n_tgt"] or n
        digits = max(1.0, -math.log10(eps))
        q = (0.5 * deg + 0.5 * digits) ** 2           # nodes of a smooth rule
        m = 2.42 * eta * eta * nb                     # near entries of a target
        ev = m / nb * 3.0 * digits / math.log10(4.0) * q * (23.0 + 4.0 * nb)
        over = n / nb * q                             # oversampled far sources
        gen = case["op"] in ("gen", "batch", "plan", "field", "grad")
        far = case["op"] in ("apply", "field", "adjoint", "grad")
        if gen:
            by += 24.0 * n + 24.0 * nt + nt * m * 20.0
            fl += nt * ev
        if far:
            by += nt * m * 20.0 + 32.0 * n + 16.0 * nt
            fl += nt * over * 31.0
        if case["op"] == "grad":
            by += 40.0 * n
            fl += nt * ev + nt * over * 62.0
    return {"bytes": by, "flops": fl}


# ----------------------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """On the unit sphere S_k Y_n = i k j_n(k) h_n(k) Y_n, so the single layer of a sum of
    spherical harmonics is known in closed form.  The other outputs are the weights of adaptive
    quadratures, whose recomputation in numpy takes minutes to hours."""
    if case["op"] != "apply" or case["shape"] != "sphere" or case["kernel"] != "S":
        return None
    xyz, coef = _sphere_inputs(case, seed)
    k = case["k_re"]
    s, c = math.sin(k), math.cos(k)
    j = [s / k, s / k ** 2 - c / k, (3.0 / k ** 2 - 1.0) * s / k - 3.0 * c / k ** 2]
    y = [-c / k, -c / k ** 2 - s / k, (1.0 - 3.0 / k ** 2) * c / k - 3.0 * s / k ** 2]
    u = sum(1j * k * j[n] * (j[n] + 1j * y[n]) * f for n, f in enumerate(_harmonics(xyz, coef)))
    return {"u": u}
