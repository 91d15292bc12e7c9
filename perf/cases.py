"""The calls that a fault or fracture simulation makes with this library, at the sizes of its
workloads: the product y = E x, the tangent solve, the block-Jacobi preconditioner, the
interface update and the assembly of the H-matrix.

  listed()            the named cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) mesh, operator and seeded inputs, as a program holds them before the call
  run(state)          one pass through the public entry points, and its outputs
  work(case)          bytes and operations one pass cannot do without
  exact(case, seed)   the outputs in plain FP64 torch, without the library
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_14397_gb300 import hmat, synth

LEAF, ETA = 64, 2.0
E_MOD, NU = 1.0, 0.25
DEV = "cuda"


def listed():
    return [
        # the smallest operator in use: a penny crack of 1,264 elements, where a product is launches and latency
        dict(name="product_penny_f32", kind="product", mesh="disk", grid=40, storage="f32", dtype="f32", nrhs=1, eps=1e-6),
        # the headline: one product of the 51,468-element disk fault, as every FP32 iteration applies it
        dict(name="product_fault_f32", kind="product", mesh="disk", grid=256, storage="f32", dtype="f32", nrhs=1, eps=1e-6),
        # the product of the plain FP64 solver (compensated FP64 vectors), on an unstructured triangle mesh
        dict(name="product_triangles_f64", kind="product", mesh="tri", grid=128, storage="f32", dtype="f64", nrhs=1, eps=1e-6),
        # six load cases at once (the six components of a far-field stress) in FP64: a ragged right-hand-side count
        dict(name="product_fault_f64_rhs6", kind="product", mesh="disk", grid=128, storage="f32", dtype="f64", nrhs=6, eps=1e-6),
        # a full pass of 16 right-hand sides on three intersecting fractures, FP32 factors
        dict(name="product_planes_f32_rhs16", kind="product", mesh="planes", grid=100, storage="f32", dtype="f32", nrhs=16, eps=1e-5),
        # the same with BF16 factors, the storage of the large three-fracture workload
        dict(name="product_planes_bf16_rhs16", kind="product", mesh="planes", grid=150, storage="bf16", dtype="f32", nrhs=16, eps=1e-5),
        # eight independent faults of 2,000 to 8,000 elements as one batch, BF16 factors
        dict(name="product_batch_bf16", kind="product", mesh="batch", grid=8, storage="bf16", dtype="f32", nrhs=1, eps=1e-6),
        # a tangent solve of a crack crossing a fault with interface stiffness k: BF16 corrections, FP64 refinement
        dict(name="solve_crack_mixed", kind="solve", mesh="crack", grid=160, storage="both", mode="mixed", precond="blockj", nrhs=1, eps=1e-6),
        # the smallest solve: the penny crack under traction, plain FP64
        dict(name="solve_penny_f64", kind="solve", mesh="disk", grid=40, storage="f32", mode="f64", precond="blockj", nrhs=1, eps=1e-6),
        # building and applying the block-Jacobi preconditioner, as each new stiffness k asks for it
        dict(name="precond_crack_blockj", kind="precond", mesh="crack", grid=160, storage="f32", precond="blockj", nrhs=1, eps=1e-6),
        # the interface law and its tangent at a million points of a softening joint, once per Newton iteration
        dict(name="interface_softening_1m", kind="interface", n=1000000, material="softening", tangent=True),
        # assembly of a new mesh's operator from its elements, and its first product
        dict(name="assemble_fault", kind="assemble", mesh="disk", grid=96, storage="f32", dtype="f64", nrhs=1, eps=1e-6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid_of(mesh, n):
    """The grid whose mesh has about n elements."""
    if mesh == "disk":
        return max(8, int(round(math.sqrt(n * 4 / math.pi))))
    if mesh == "tri":
        return max(8, int(round(math.sqrt(n * 2 / math.pi))))
    if mesh == "planes":
        return max(8, 2 * int(round(math.sqrt(n / 3) / 2)))
    if mesh == "crack":
        return max(8, 4 * int(round(math.sqrt(n * 4 / 5) / 4)))
    return max(2, min(8, n // 4000))  # batch: number of faults


def draw(rng):
    kind = rng.choice(["product"] * 6 + ["solve", "precond", "interface", "assemble"])
    if kind == "interface":
        return dict(kind=kind, n=_log(rng, 1000, 1000000), material=rng.choice(sorted(synth.INTERFACE_PARAMS)),
                    tangent=rng.random() < 0.8)
    mesh = rng.choice(["disk", "disk", "tri", "planes", "crack"] + (["batch"] if kind == "product" else []))
    top = {"product": 50000, "solve": 20000, "precond": 30000, "assemble": 7000}[kind]
    case = dict(kind=kind, mesh=mesh, grid=_grid_of(mesh, _log(rng, 1000, top)), eps=rng.choice([1e-5, 1e-6]))
    if kind in ("product", "assemble"):
        case.update(storage=rng.choice(["f32", "f32", "bf16"]) if kind == "product" else "f32",
                    dtype=rng.choice(["f32", "f64"]), nrhs=rng.choice([1, 1, 1, 2, 3, 4, 6, 8, 11, 16]))
    elif kind == "solve":
        mode = rng.choice(["f64", "mixed"])
        case.update(storage="both" if mode == "mixed" else "f32", mode=mode,
                    precond=rng.choice(["blockj", "blockj", "jacobi3"]), nrhs=rng.choice([1, 1, 2, 3]))
    else:
        case.update(storage="f32", precond=rng.choice(["blockj", "blockj", "jacobi3"]), nrhs=rng.choice([1, 1, 2, 5, 16]))
    return case


# ---------------------------------------------------------------- what a program holds before the call

def _meshes(case):
    """The elements of the case: one mesh, or the faults of a batch."""
    g = case["grid"]
    if case["mesh"] == "disk":
        return [synth.disk_mesh(g)]
    if case["mesh"] == "tri":
        return [synth.tri_disk_mesh(g)]
    if case["mesh"] == "planes":
        return [synth.config_three_planes(g)]
    if case["mesh"] == "crack":
        return [synth.config_crack_fault(h=4.0 / g)]
    return synth.config_faults_batch(n_faults=g, n_min=2000, n_max=8000)[0]


def _operator(case, els):
    trees = [hmat.ClusterTree(el, LEAF, ETA) for el in els]
    parts = [hmat.HMatrix(t, el, E_MOD, NU, case["eps"], case["storage"]) for t, el in zip(trees, els)]
    return parts[0] if len(parts) == 1 else hmat.HMatrix.batch(parts)


def _vectors(case, seed, ndof, dtype):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    shape = (ndof,) if case["nrhs"] == 1 else (case["nrhs"], ndof)
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float64).to(dtype)


def _stiffness(case, seed, n):
    """Interface stiffness per element, log-uniform over five decades about E / h."""
    h = {"crack": 4.0 / case["grid"]}.get(case["mesh"], 2.0 / case["grid"])
    return torch.from_numpy(synth.k_loguniform(n, int(seed) + 1, E_MOD, h)).to(DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "interface":
        states = [torch.from_numpy(a).to(DEV) for a in synth.interface_states(case["n"], int(seed))]
        return dict(case=case, states=states, params=synth.INTERFACE_PARAMS[case["material"]])
    els = _meshes(case)
    ndof = 3 * sum(el.N for el in els)
    state = dict(case=case)
    if kind == "assemble":
        dt = torch.float64 if case["dtype"] == "f64" else torch.float32
        state.update(el=els[0], x=_vectors(case, seed, ndof, dt))
        state["y"] = torch.empty_like(state["x"])
        return state
    state["H"] = _operator(case, els)
    if kind == "product":
        dt = torch.float64 if case["dtype"] == "f64" else torch.float32
        state["x"] = _vectors(case, seed, ndof, dt)
        state["y"] = torch.empty_like(state["x"])
    else:
        state["k"] = _stiffness(case, seed, ndof // 3)
        state["b"] = _vectors(case, seed, ndof, torch.float64)
        state["x"] = torch.empty_like(state["b"])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "product":
        state["H"].matvec(state["x"], state["y"])
        return state["y"]
    if kind == "solve":
        state["H"].solve(state["b"], state["x"], k=state["k"], tol=1e-8, precond=case["precond"], mode=case["mode"])
        return state["x"]
    if kind == "precond":
        state["H"].precond_apply(state["b"], state["x"], k=state["k"], precond=case["precond"])
        return state["x"]
    if kind == "interface":
        T1, dp1, chi1, cep, mode, _ = hmat.interface_update(state["params"], *state["states"], tangent=case["tangent"])
        return dict(T=T1, dp=dp1, chi=chi1, cep=cep, mode=mode)
    el = state["el"]
    tree = hmat.ClusterTree(el, LEAF, ETA)
    H = hmat.HMatrix(tree, el, E_MOD, NU, case["eps"], case["storage"])
    H.matvec(state["x"], state["y"])
    return state["y"]


# ---------------------------------------------------------------- what one pass cannot do without

def _product_work(info, case, vec_bytes):
    """Every stored near entry and factor entry once, x read and y written; a product and a sum per entry and RHS."""
    far = info["u_entries"] + info["v_entries"]
    fac = 2 if case["storage"] == "bf16" or case.get("mode") == "mixed" else 4
    nrhs = case["nrhs"]
    return dict(bytes=4 * info["near_entries"] + fac * far + 2 * vec_bytes * info["n_dof"] * nrhs,
                flops=2 * (info["near_entries"] + far) * nrhs)


def work(case):
    kind = case["kind"]
    if kind == "interface":
        # 12 doubles read; 9 (18 with the tangent) and the mode written; a few hundred operations of the return
        return dict(bytes=case["n"] * (96 + 72 + 4 + (72 if case["tangent"] else 0)), flops=400 * case["n"])
    els = _meshes(case)
    if kind == "precond":
        tree = hmat.ClusterTree(els[0], LEAF, ETA).export()
        rows = 3 * (tree["end"] - tree["begin"])[tree["left"] < 0].astype(np.float64)
        vec = 16 * 3 * els[0].N * case["nrhs"] + 8 * els[0].N
        if case["precond"] == "jacobi3":
            return dict(bytes=72 * els[0].N + vec, flops=els[0].N * (60 + 18 * case["nrhs"]))
        # every diagonal leaf block read, its inverse written
        return dict(bytes=float(8 * (rows**2).sum()) + vec, flops=float((2 * rows**3 + 2 * rows**2 * case["nrhs"]).sum()))
    H = _operator(case, els)
    info = H.info()
    if kind == "product":
        return _product_work(info, case, 8 if case["dtype"] == "f64" else 4)
    if kind == "solve":
        # one product for each iteration that the system takes
        s = prepare(case, 1)
        its = max(i["iters"] for i in s["H"].solve(s["b"], s["x"], k=s["k"], tol=1e-8, precond=case["precond"],
                                                   mode=case["mode"]))
        w = _product_work(info, case, 8)
        return dict(bytes=its * w["bytes"], flops=its * w["flops"])
    # assembly: the evaluated 3x3 blocks at about 400 operations each, every stored entry written once
    return dict(bytes=4 * (info["near_entries"] + info["u_entries"] + info["v_entries"]), flops=400 * info["coeff_blocks"])


# ---------------------------------------------------------------- the outputs in FP64 torch

def _edges(el):
    """Vertices of every element in its own (s1, s2) frame, counter-clockwise, (N, nv, 2)."""
    if int(np.asarray(el.shape)[0]) == 0:
        sg = np.array([[-1, -1], [1, -1], [1, 1], [-1, 1]], dtype=np.float64)
        return sg[None] * np.stack([el.a, el.b], axis=1)[:, None, :]
    v = el.tri.reshape(-1, 3, 3) - el.c[:, None, :]
    p = np.stack([np.einsum("nvk,nk->nv", v, el.s1), np.einsum("nvk,nk->nv", v, el.s2)], axis=2)
    e1, e2 = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]
    flip = e1[:, 0] * e2[:, 1] - e1[:, 1] * e2[:, 0] < 0
    p[flip] = p[flip][:, [0, 2, 1]]
    return p


def _dense_product(el, X):
    """X E^T (nrhs, 3N) with the dense matrix of influence blocks: tractions at the centroids from unit displacement
    discontinuities over the elements, phi = int 1/R by line integrals over the elements' edges (Stokes)."""
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(DEV)
    N = el.N
    c, fr = t(el.c), [t(el.s1), t(el.s2), t(el.n)]
    P = t(_edges(el))
    mu = E_MOD / (2 * (1 + NU))
    C = mu / (4 * math.pi * (1 - NU))
    Xs = X.double().reshape(-1, N, 3)
    Y = torch.empty_like(Xs)
    step = max(1, 6000000 // N)
    for r0 in range(0, N, step):
        r = slice(r0, min(N, r0 + step))
        d = [c[r, k, None] - c[None, :, k] for k in range(3)]
        x1, x2, z = (sum(d[k] * f[:, k] for k in range(3)) for f in fr)
        S = {k: 0.0 for k in ("11", "12", "13", "22", "23", "111", "112", "122", "222", "113", "123", "223")}
        for e in range(P.shape[1]):
            pa, pb = P[:, e], P[:, (e + 1) % P.shape[1]]
            L = (pb - pa).norm(dim=1)
            tx, ty = ((pb - pa) / L[:, None]).unbind(1)
            nx, ny = ty, -tx
            dx, dy = x1 - pa[:, 0], x2 - pa[:, 1]
            wa, hp = dx * tx + dy * ty, dx * nx + dy * ny
            wb = wa - L
            rho2 = hp * hp + z * z
            ra, rb = (rho2 + wa * wa).sqrt(), (rho2 + wb * wb).sqrt()
            ga, gb, ia, ib = wa / ra, wb / rb, 1 / (ra * ra), 1 / (rb * rb)
            k30 = torch.where(wa * wb > 0, (wa * wa - wb * wb) / (ra * rb * (wa * rb + wb * ra)), (ga - gb) / rho2)
            k31, k51 = 1 / rb - 1 / ra, (ib / rb - ia / ra) / 3
            k52 = k30 * (ga * ga + ga * gb + gb * gb) / 3
            k50 = k30 / 3 * (ia + ib + (ia + ib - rho2 * ia * ib) / (1 + ga * gb))
            h1, h2 = hp * nx, hp * ny
            i1, i2, i3 = h1 * k30 + tx * k31, h2 * k30 + ty * k31, z * k30
            j11 = 3 * (h1 * h1 * k50 + 2 * h1 * tx * k51 + tx * tx * k52) - k30
            j12 = 3 * (h1 * h2 * k50 + (h1 * ty + h2 * tx) * k51 + tx * ty * k52)
            j22 = 3 * (h2 * h2 * k50 + 2 * h2 * ty * k51 + ty * ty * k52) - k30
            j13, j23 = 3 * z * (h1 * k50 + tx * k51), 3 * z * (h2 * k50 + ty * k51)
            for key, v in (("11", nx * i1), ("12", nx * i2), ("13", nx * i3), ("22", ny * i2), ("23", ny * i3),
                           ("111", -nx * j11), ("112", -nx * j12), ("122", -nx * j22), ("222", -ny * j22),
                           ("113", -nx * j13), ("123", -nx * j23), ("223", -ny * j23)):
                S[key] = S[key] + v
        S["33"], S["133"] = -(S["11"] + S["22"]), -(S["111"] + S["122"])
        S["233"], S["333"] = -(S["112"] + S["222"]), -(S["113"] + S["223"])
        D = lambda *ix: S["".join(sorted(str(i + 1) for i in ix))]
        q = [[sum(f[r, k, None] * g[None, :, k] for k in range(3)) for g in fr] for f in fr]
        out = torch.zeros_like(Y[:, r])
        for m in range(3):
            sig = {}
            for k in range(3):
                for j in range(k, 3):
                    s = -z * D(m, k, j)
                    if k == j:
                        s = s + 2 * NU * D(2, m)
                    if k == m:
                        s = s + (1 - NU) * D(2, j)
                    if j == m:
                        s = s + (1 - NU) * D(2, k)
                    if m == 2:
                        s = s - (1 - 2 * NU) * D(k, j)
                    if k == 2:
                        s = s - NU * D(m, j)
                    if j == 2:
                        s = s - NU * D(m, k)
                    sig[k, j] = sig[j, k] = -C * s
            tr = [sum(sig[k, j] * q[2][j] for j in range(3)) for k in range(3)]
            for al in range(3):
                out[:, :, al] += (sum(q[al][k] * tr[k] for k in range(3)) @ Xs[:, :, m].T).T
        Y[:, r] = out
    return Y.reshape(X.shape)


def _dense_solve(el, k, b):
    """x of (E - diag(k)) x = b with the dense matrix."""
    n = 3 * el.N
    A = _dense_product(el, torch.eye(n, dtype=torch.float64, device=DEV)).T
    A = A - torch.diag(k.repeat_interleave(3))
    return torch.linalg.solve(A, b.reshape(-1, n).T).T.reshape(b.shape)


def _larger(a, b):
    return torch.where(a.real >= b.real, a, b)


def _interface(P, T, dp, chi, dd, dx=None):
    """Elastic predictor and plastic return of every point on complex numbers (the imaginary part of dd carries a
    derivative): T', delta^p and (chi_s, chi_t, w_dil) at the end of the step, and the mode."""
    Ks, Kn = P["Ks"], P["Kn"]
    cx = lambda a: a.to(torch.complex128)
    soft = lambda scale, x: torch.where(x.real / scale >= 1, 0 * x, 1 - x / scale) if scale > 0 else 0 * x
    fric = lambda s: (P["fp"] - P["fr"]) * soft(P["dc"], s) + P["fr"]
    dil = lambda s: P["psip"] * soft(P["dc"], s)
    coh = lambda s: P["cp"] * soft(P["wc"], s)
    ten = lambda s: P["sigp"] * soft(P["wc"], s)
    norm = lambda *a: sum(x * x for x in a).sqrt()
    chis, chit, wdil = (cx(a) for a in chi.unbind(1))
    damaged = (chit.real >= P["wc"]) if P["wc"] > 0 else torch.ones_like(chi[:, 0], dtype=torch.bool)
    p0, p1, p2 = (cx(a) for a in dp.unbind(1))
    pn = torch.where(damaged, cx(torch.minimum(dp[:, 2], P["alphaR"] * P["wc"] + chi[:, 2])), p2)
    t0, t1 = (cx(T[:, i]) + Ks * dd[:, i] for i in range(2))
    tn = cx(T[:, 2]) - Kn * (pn - p2) + Kn * dd[:, 2]
    tau = norm(t0, t1)
    s0, s1 = t0 / tau, t1 / tau

    def coulomb(x):
        a, b = p0 + x * s0, p1 + x * s1
        cs = _larger(chis, norm(a, b))
        psi = dil(cs)
        n = pn + x * psi
        ct = _larger(chit, norm(a, b, n))
        ta, tb = tau - Ks * x, tn - Kn * (psi * x)
        return ta + fric(cs) * tb - coh(ct), (ta * s0, ta * s1, tb, a, b, n, cs, ct, wdil + psi * x)

    def tensile(x):
        n = pn + x
        ct = _larger(chit, norm(p0, p1, n))
        return tn - Kn * x - ten(ct), (t0, t1, tn - Kn * x, p0, p1, n, chis, ct, wdil)

    a0, a1 = p0 + t0 / Ks, p1 + t1 / Ks
    acs = _larger(chis, norm(a0, a1))

    def apex(x):
        n = pn + x
        ct = _larger(chit, norm(a0, a1, n))
        return fric(acs) * (tn - Kn * x) - coh(ct), (0 * x, 0 * x, tn - Kn * x, a0, a1, n, acs, ct, wdil)

    f0, c0, st0 = (v.real for v in (fric(chis), coh(chit), ten(chit)))
    Fc = tau.real + f0 * tn.real - torch.where(damaged, 0 * c0, c0)
    plain = torch.where((Fc <= 0) & (tn.real - st0 <= 0), 0,
                        torch.where(tau.real - (c0 - f0 * st0) - ((1 + f0 * f0).sqrt() - f0) * (tn.real - st0) > 0, 1, 2))
    mode = torch.where(damaged, torch.where(tn.real > 0, 3, torch.where(Fc <= 0, 0, 1)), plain)
    mode = torch.where((mode == 1) & (coulomb(cx(tau.real / Ks))[0].real > 0), 4, mode)
    opened = (0 * tn, 0 * tn, 0 * tn, cx(dp[:, 0] + T[:, 0] / Ks) + dd[:, 0], cx(dp[:, 1] + T[:, 1] / Ks) + dd[:, 1],
              cx(dp[:, 2] + T[:, 2] / Kn) + dd[:, 2])
    opened += (_larger(chis, norm(*opened[3:5])), _larger(chit, norm(*opened[3:6])), wdil)
    res = [torch.where(mode == 3, a, b) for a, b in zip(opened, (t0, t1, tn, p0, p1, pn, chis, chit, wdil))]
    roots, keep = {}, mode.clone()
    for kind, g, hi in ((1, coulomb, tau.real / Ks), (2, tensile, tn.real / Kn), (4, apex, tn.real / Kn)):
        here = mode == kind
        if dx is None:  # bisection on the values
            lo, up = torch.zeros_like(hi), hi.clone()
            none = ~(g(cx(lo))[0].real > 0)
            for _ in range(110):
                mid = 0.5 * (lo + up)
                pos = g(cx(mid))[0].real > 0
                lo, up = torch.where(pos, mid, lo), torch.where(pos, up, mid)
            x = torch.where(none | ~here, torch.zeros_like(hi), 0.5 * (lo + up))
        else:
            x = dx[kind]
        roots[kind] = x
        xc = cx(x)
        slope = g(torch.complex(x, torch.full_like(x, 1e-30)))[0].imag / 1e-30 if not dd.imag.any() else None
        if slope is not None:
            roots["slope%d" % kind] = slope
        else:
            moved = -g(xc)[0].imag / dx["slope%d" % kind]
            xc = torch.complex(x, torch.where(x > 0, moved, torch.zeros_like(x)))
        out = g(xc)[1]
        if kind != 1:
            full = (out[7].real >= P["wc"]) if P["wc"] > 0 else torch.ones_like(here)
            out = [torch.where(full, a, b) for a, b in zip(opened, out)]
            keep = torch.where(here & full, 3, keep)
        res = [torch.where(here, a, b) for a, b in zip(out, res)]
    return res, keep.to(torch.int32), roots


def _exact_interface(case, state):
    P = state["params"]
    T, dp, chi, dd = state["states"]
    res, mode, roots = _interface(P, T, dp, chi, dd.to(torch.complex128))
    real = [a.real for a in res]
    cep = None
    if case["tangent"]:
        cep = torch.empty(T.shape[0], 3, 3, dtype=torch.float64, device=T.device)
        for j in range(3):
            step = torch.zeros_like(dd)
            step[:, j] = 1e-30
            r = _interface(P, T, dp, chi, torch.complex(dd, step), roots)[0]
            cep[:, :, j] = torch.stack([a.imag for a in r[:3]], dim=1) / 1e-30
    return dict(T=torch.stack(real[:3], 1), dp=torch.stack(real[3:6], 1), chi=torch.stack(real[6:], 1), cep=cep, mode=mode)


def exact(case, seed):
    kind = case["kind"]
    if kind == "interface":
        return _exact_interface(case, prepare(case, seed))
    if kind == "precond":
        return None  # its blocks are the library's own clusters
    els = _meshes(case)
    ndof = 3 * sum(el.N for el in els)
    if kind == "solve":
        if ndof > 6000:
            return None  # a dense LU of this size takes too long
        return _dense_solve(els[0], _stiffness(case, seed, ndof // 3), _vectors(case, seed, ndof, torch.float64))
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    x = _vectors(case, seed, ndof, dt)
    at, parts = 0, []
    for el in els:
        parts.append(_dense_product(el, x[..., at:at + 3 * el.N].contiguous()))
        at += 3 * el.N
    return torch.cat(parts, dim=-1)
