"""Timed cases of the framework: phi-function products and their parts, through the public entry points.

A case is a plain dict.  Its ``call`` is one of

  phiv     ``phiv(op, v, h, p, m)``: y_k = phi_k(hA) v, k = 0..p, one Krylov projection
  lincomb  ``phiv_lincomb(op, b, tau, m)``: sum_j tau^j phi_j(tau A) b_j (a stage of an exponential integrator)
  grad     ``Phi1GrayScott``: phi_1(hA(theta)) v and its gradient with respect to v, h and theta
  batch    ``Batch.run``: many phi products of uneven size in one launch
  matvec   ``matvec(op, x)``: the stencil alone (an integrator's Jacobian product)

and its operator ``op`` one of the three matrix-free stencils (advdiff2d, grayscott2d, adr3d).  The largest listed case
is the float64 product on the 256^3 grid, the smallest the stencil alone.
"""
import math

import torch

import paper_2410_14917_gb300 as lsa

DEV = "cuda"


def _phiv(name, op, nx, ny, nz, m, p, h, precision="fp64", variant="hcwy"):
    return dict(name=name, call="phiv", op=op, nx=nx, ny=ny, nz=nz, m=m, p=p, h=h, precision=precision, variant=variant)


def listed():
    return [
        # a stencil application on its own: the Jacobian products between an integrator's phi combinations
        dict(name="matvec_grayscott_512", call="matvec", op="grayscott2d", nx=512, ny=512, nz=1, m=1, p=0, h=1.0,
             precision="fp64", variant="hcwy"),
        # a small 2D problem, where latency and not throughput is what a user waits for
        _phiv("phiv_advdiff_64", "advdiff2d", 64, 64, 1, 30, 3, 1e-2),
        # a small grid that is no multiple of any tile, with the two-sweep Gauss-Seidel correction
        _phiv("phiv_advdiff_97x61_gsmgs", "advdiff2d", 97, 61, 1, 24, 1, 1e-2, variant="hgsmgs"),
        # the headline product: the Jacobian of a 2D reaction-diffusion system, three phi functions
        _phiv("phiv_grayscott_512", "grayscott2d", 512, 512, 1, 64, 2, 1.0),
        # the same with the basis in float32
        _phiv("phiv_grayscott_512_fp32", "grayscott2d", 512, 512, 1, 64, 2, 1.0, precision="fp32"),
        # a 3D problem of the size that fills the GPU, in both precisions of the basis
        _phiv("phiv_adr3d_256", "adr3d", 256, 256, 256, 40, 1, 5e-3),
        _phiv("phiv_adr3d_256_fp32", "adr3d", 256, 256, 256, 40, 1, 5e-3, precision="fp32"),
        # a ragged 3D box, float32 basis, truncated Neumann correction
        _phiv("phiv_adr3d_75x50x41_fp32", "adr3d", 75, 50, 41, 20, 1, 5e-3, precision="fp32", variant="hncwy"),
        # one stage of a fourth-order exponential integrator: four vectors, one augmented projection
        dict(name="lincomb_grayscott_512", call="lincomb", op="grayscott2d", nx=512, ny=512, nz=1, m=64, p=3, h=1.0,
             precision="fp64", variant="hcwy"),
        # forward and backward: the loss gradient with respect to the start vector, the step and the coefficients
        dict(name="grad_grayscott_256", call="grad", op="grayscott2d", nx=256, ny=256, nz=1, m=48, p=1, h=1.0,
             precision="fp64", variant="hcwy"),
        # many small problems of uneven size in one launch, in both precisions of the basis
        dict(name="batch_512", call="batch", op="advdiff2d", count=512, smin=32, smax=256, mmin=16, mmax=48, p=2, h=1e-2,
             precision="fp64", variant="hcwy"),
        dict(name="batch_512_fp32", call="batch", op="advdiff2d", count=512, smin=32, smax=256, mmin=16, mmax=48, p=2,
             h=1e-2, precision="fp32", variant="hcwy"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Sizes over the whole range, on their logarithm: 2D sides 24..640, 3D sides 16..224 (128 beside phiv), odd ones too."""
    call = rng.choice(["phiv", "phiv", "phiv", "phiv", "lincomb", "grad", "batch", "matvec"])
    precision = rng.choice(["fp64", "fp64", "fp32"])
    variant = rng.choice(["hcwy", "hcwy", "hcwy", "hncwy", "hgsmgs"])
    if call == "batch":
        smax = _log_int(rng, 48, 256)
        return dict(call=call, op="advdiff2d", count=_log_int(rng, 16, 384), smin=rng.randint(24, 40), smax=smax,
                    mmin=rng.randint(8, 20), mmax=rng.randint(24, 48), p=rng.randint(0, 3), h=1e-2, precision=precision,
                    variant=variant)
    op = "grayscott2d" if call == "grad" else rng.choice(["advdiff2d", "grayscott2d", "adr3d"])
    if call in ("lincomb", "grad"):
        precision = "fp64"
    if op == "adr3d":
        nx, ny, nz = (_log_int(rng, 16, 224 if call == "phiv" else 128) for _ in range(3))
    else:
        hi = 384 if call == "grad" else 640
        nx, ny, nz = _log_int(rng, 24, hi), _log_int(rng, 24, hi), 1
        if rng.random() < 0.4:                     # whole tiles, as most users choose them
            nx, ny = max(32, nx // 16 * 16), max(32, ny // 16 * 16)
    if call == "phiv" and op != "adr3d" and rng.random() < 0.12:   # the one-by-one orthogonalisation that the others are measured against
        variant = "mgs"
        nx, ny = min(nx, 256), min(ny, 256)
    m = 1 if call == "matvec" else rng.randint(12, 40 if op == "adr3d" or call == "grad" else 64)
    p = {"matvec": 0, "grad": 1}.get(call, rng.randint(0, 3))
    h = {"advdiff2d": 1e-2, "grayscott2d": 1.0, "adr3d": 5e-3}[op]
    return dict(call=call, op=op, nx=nx, ny=ny, nz=nz, m=m, p=p, h=h, precision=precision, variant=variant)


# ----------------------------------------------------------------------------
# inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, n, lo, hi):
    return torch.rand(n, dtype=torch.float64, device=DEV, generator=g).mul_(hi - lo).add_(lo)


GRAYSCOTT = dict(Du=2e-5, Dv=1e-5, F=0.04, k=0.06)
VEL2, VEL3 = (1.0, 0.5), (1.0, 1.0, 1.0)


def _problem(case, seed):
    """The operator's numbers and fields, and the vectors, of a case that has one operator."""
    g = _gen(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    npts = nx * ny * nz
    pr = dict(npts=npts, N=npts * (2 if case["op"] == "grayscott2d" else 1))
    if case["op"] == "advdiff2d":
        pr.update(dx=1.0 / max(nx, ny), diff=0.01)
    elif case["op"] == "grayscott2d":
        pr.update(dx=2.5 / max(nx, ny), u0=_uniform(g, npts, 0.0, 1.0), v0=_uniform(g, npts, 0.0, 1.0))
    else:
        pr.update(dx=1.0 / max(nx, ny, nz), diff=1e-3, r=_uniform(g, npts, -1.0, 0.0))
    if case["call"] == "lincomb":
        pr["b"] = _uniform(g, (case["p"] + 1) * pr["N"], -1.0, 1.0).view(case["p"] + 1, pr["N"])
    else:
        pr["v"] = _uniform(g, pr["N"], -1.0, 1.0)
    if case["call"] == "grad":
        pr["target"] = _uniform(g, pr["N"], -1.0, 1.0)
    return pr


def _operator(case, pr):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["op"] == "advdiff2d":
        return lsa.Operator.advdiff2d(nx, ny, pr["dx"], pr["diff"], VEL2)
    if case["op"] == "grayscott2d":
        return lsa.Operator.grayscott2d(nx, ny, pr["dx"], u0=pr["u0"], v0=pr["v0"], **GRAYSCOTT)
    return lsa.Operator.adr3d(nx, ny, nz, pr["dx"], pr["diff"], VEL3, pr["r"])


def _instances(case, seed):
    """Sides, diffusions and Krylov dimensions of a batch: the table is the case's own, the vectors are the seed's."""
    g = torch.Generator().manual_seed(case["count"] * 1000 + case["smax"])
    n = case["count"]
    sides = torch.randint(case["smin"], case["smax"] + 1, (n,), generator=g).tolist()
    sides = [max(32, s // 16 * 16) if i % 2 else s for i, s in enumerate(sides)]
    diffs = torch.exp(torch.rand(n, dtype=torch.float64, generator=g) * math.log(1e3) + math.log(1e-4)).tolist()
    ms = torch.randint(case["mmin"], case["mmax"] + 1, (n,), generator=g).tolist()
    total = sum(s * s for s in sides)
    v = _uniform(_gen(seed), total, -1.0, 1.0) if seed is not None else None
    return sides, diffs, ms, v


def prepare(case, seed):
    call, prec = case["call"], case["precision"]
    if call == "batch":
        sides, diffs, ms, v = _instances(case, seed)
        ops = [lsa.Operator.advdiff2d(s, s, 1.0 / s, d, VEL2) for s, d in zip(sides, diffs)]
        plan = lsa.Batch(ops, ms, case["h"], case["p"], variant=case["variant"], precision=prec)
        return dict(case=case, plan=plan, v=v, y=torch.empty(plan.y_elems, dtype=torch.float64, device=DEV))
    pr = _problem(case, seed)
    st = dict(case=case, op=_operator(case, pr), pr=pr)
    if call == "phiv":
        st["work"] = lsa.Workspace.for_call(st["op"], case["m"], case["p"], prec)
        st["y"] = torch.empty((case["p"] + 1, pr["N"]), dtype=torch.float64, device=DEV)
    elif call == "lincomb":
        st["work"] = lsa.Workspace.for_call(st["op"], case["m"], 0)
        st["u"] = torch.empty(pr["N"], dtype=torch.float64, device=DEV)
    elif call == "matvec":
        st["x"] = pr["v"].to(torch.float64 if prec == "fp64" else torch.float32)
        st["work"] = lsa.Workspace.for_call(st["op"], 1, 0, prec)
        st["y"] = torch.empty_like(st["x"])
    else:
        st["v"] = pr["v"].clone().requires_grad_()
        st["h"] = torch.tensor(case["h"], dtype=torch.float64, requires_grad=True)
        st["theta"] = torch.tensor([GRAYSCOTT[k] for k in ("Du", "Dv", "F", "k")], dtype=torch.float64, requires_grad=True)
    return st


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "phiv":
        y, _ = lsa.phiv(state["op"], state["pr"]["v"], case["h"], case["p"], case["m"], variant=case["variant"],
                        precision=case["precision"], y=state["y"], work=state["work"], stats=False)
        return y
    if call == "batch":
        return state["plan"].run(state["v"], state["y"])
    if call == "lincomb":
        u, _ = lsa.phiv_lincomb(state["op"], state["pr"]["b"], case["h"], case["m"], variant=case["variant"], u=state["u"],
                                work=state["work"], stats=False)
        return u
    if call == "matvec":
        return lsa.matvec(state["op"], state["x"], precision=case["precision"], y=state["y"], work=state["work"])
    v, h, theta = state["v"], state["h"], state["theta"]
    y = lsa.Phi1GrayScott.apply(v, h, theta, state["op"], case["m"], case["variant"])
    gv, gh, gt = torch.autograd.grad(y, (v, h, theta), y.detach() - state["pr"]["target"])
    return {"y": y.detach(), "grad_v": gv, "grad_h": gh, "grad_theta": gt}


# ----------------------------------------------------------------------------
# what a pass cannot do without: each input read and each output written once; the arithmetic of the projection

TAPS = {"advdiff2d": 5, "grayscott2d": 9, "adr3d": 8}


def _krylov_flops(N, m, taps, nout):
    # step j: subtract j - 1 columns, 2 (j - 1) + 3 inner products, the stencil; then v_{m+1} and the output combination
    per = sum(2 * (j - 1) + 2 * (2 * (j - 1) + 3) + 2 * taps for j in range(1, m + 1)) + 2 * m + 2 * m * nout
    return float(N) * per


def work(case):
    if case["call"] == "batch":
        sides, _, ms, _ = _instances(case, None)
        return {"bytes": sum(8.0 * s * s * (2 + case["p"]) for s in sides),
                "flops": sum(_krylov_flops(s * s, m, 5, case["p"] + 1) for s, m in zip(sides, ms))}
    npts = case["nx"] * case["ny"] * case["nz"]
    N = npts * (2 if case["op"] == "grayscott2d" else 1)
    fields = 8.0 * npts * {"advdiff2d": 0, "grayscott2d": 2, "adr3d": 1}[case["op"]]
    taps = TAPS[case["op"]]
    if case["call"] == "matvec":
        return {"bytes": (8.0 if case["precision"] == "fp64" else 4.0) * 2 * N + fields, "flops": 2.0 * taps * N}
    if case["call"] == "grad":
        # forward with three outputs, the transposed product, three products on twice the size
        m = case["m"]
        return {"bytes": 8.0 * 4 * N + fields,
                "flops": _krylov_flops(N, m, taps, 3) + _krylov_flops(N, m, taps, 1) + 3 * _krylov_flops(2 * N, m, taps + 1, 1)}
    vectors = case["p"] + 2
    nout = case["p"] + 1 if case["call"] == "phiv" else 1
    extra = 2 * case["p"] if case["call"] == "lincomb" else 0
    return {"bytes": 8.0 * vectors * N + fields, "flops": _krylov_flops(N, case["m"], taps + extra, nout)}


# ----------------------------------------------------------------------------
# the same results from plain torch in 64 bits

def _stencil(case, pr):
    nx, ny, nz, dx = case["nx"], case["ny"], case["nz"], pr["dx"]
    if case["op"] == "advdiff2d":
        return _advdiff(nx, ny, dx, pr["diff"])
    if case["op"] == "grayscott2d":
        return _grayscott(nx, ny, dx, pr["u0"], pr["v0"], GRAYSCOTT)
    eps, r = pr["diff"], pr["r"].view(nz, ny, nx)

    def mv(x):
        x = x.view(nz, ny, nx)
        out = r * x
        for ax in range(3):
            back, fwd = x.roll(1, ax), x.roll(-1, ax)
            out = out + (eps / dx ** 2) * (back + fwd - 2.0 * x) - (1.0 / dx) * (x - back)   # unit velocities, upwind
        return out.reshape(-1)
    return mv


def _advdiff(nx, ny, dx, diff):
    def mv(x):
        x = x.view(ny, nx)
        w, e, s, n = x.roll(1, 1), x.roll(-1, 1), x.roll(1, 0), x.roll(-1, 0)
        return ((diff / dx ** 2) * (w + e + s + n - 4.0 * x) - (0.5 / dx) * (VEL2[0] * (e - w) + VEL2[1] * (n - s))).reshape(-1)
    return mv


def _lap(x, dx):
    return (x.roll(1, 1) + x.roll(-1, 1) + x.roll(1, 0) + x.roll(-1, 0) - 4.0 * x) / dx ** 2


def _grayscott(nx, ny, dx, u0, v0, th, transpose=False):
    u0, v0 = u0.view(ny, nx), v0.view(ny, nx)
    a, b = v0 * v0, 2.0 * u0 * v0

    def mv(z):
        u, v = z.view(2, ny, nx)
        p, q = (-b * v, a * u) if not transpose else (a * v, -b * u)
        return torch.stack([th["Du"] * _lap(u, dx) - (a + th["F"]) * u + p,
                            th["Dv"] * _lap(v, dx) + (b - th["F"] - th["k"]) * v + q]).reshape(-1)
    return mv


def _krylov(mv, v, m):
    """Orthonormal basis (every vector orthogonalised twice) and Hessenberg matrix of K_m(A, v)."""
    N = v.numel()
    m = min(m, N)
    V = torch.empty((m, N), dtype=torch.float64, device=DEV)
    H = torch.zeros((m, m), dtype=torch.float64, device=DEV)
    beta = v.norm()
    V[0] = v / beta
    for j in range(m):
        w = mv(V[j])
        for _ in range(2):
            c = V[:j + 1] @ w
            w = w - V[:j + 1].T @ c
            H[:j + 1, j] += c
        if j + 1 < m:
            H[j + 1, j] = w.norm()
            V[j + 1] = w / H[j + 1, j]
    return beta, V, H


def _phis(mv, v, h, p, m):
    """(p+1, N): beta V phi_k(hH) e_1, the phi functions from one exponential of the augmented Hessenberg matrix."""
    beta, V, H = _krylov(mv, v, m)
    m = H.shape[0]
    big = torch.zeros((m + p + 1, m + p + 1), dtype=torch.float64, device=DEV)
    big[:m, :m] = h * H
    big[0, m] = 1.0
    for i in range(p):
        big[m + i, m + i + 1] = 1.0
    E = torch.linalg.matrix_exp(big.cpu()).to(DEV)
    C = torch.stack([E[:m, 0]] + [E[:m, m + k - 1] for k in range(1, p + 1)])
    return beta * (C @ V)


def exact(case, seed):
    call, h, m = case["call"], case["h"], case.get("m")
    if call == "batch":
        sides, diffs, ms, v = _instances(case, seed)
        out, at = [], 0
        for s, d, mm in zip(sides, diffs, ms):
            out.append(_phis(_advdiff(s, s, 1.0 / s, d), v[at:at + s * s], h, case["p"], mm).reshape(-1))
            at += s * s
        return torch.cat(out)
    pr = _problem(case, seed)
    mv = _stencil(case, pr)
    if call == "matvec":
        return mv(pr["v"].to(torch.float64 if case["precision"] == "fp64" else torch.float32).double())
    if call == "phiv":
        return _phis(mv, pr["v"], h, case["p"], m)
    N, nx, ny, dx = pr["N"], case["nx"], case["ny"], pr["dx"]
    if call == "lincomb":
        p, b = case["p"], pr["b"]

        def aug(z):                                # [A x + sum_k xi_k b_{p-k}; shift xi]
            x, xi = z[:N], z[N:]
            top = mv(x)
            for k in range(p):
                top = top + xi[k] * b[p - k]
            return torch.cat([top, xi[1:], torch.zeros(1 if p else 0, dtype=torch.float64, device=DEV)])
        start = torch.cat([b[0], torch.zeros(p, dtype=torch.float64, device=DEV)])
        if p:
            start[-1] = 1.0
        return _phis(aug, start, h, 0, m)[0, :N]
    # gradient of the loss whose cotangent is r = y - target
    phi = _phis(mv, pr["v"], h, 2, m)
    r = phi[1] - pr["target"]
    gv = _phis(_grayscott(nx, ny, dx, pr["u0"], pr["v0"], GRAYSCOTT, transpose=True), r, h, 1, m)[1]
    gh = torch.dot(r, phi[0] - phi[1]) / h

    def frechet(which):                            # [[A, dA/dtheta], [0, A]] on [0; v]
        def mvk(z):
            x, y = z[:N], z[N:]
            d = torch.zeros_like(y).view(2, ny, nx)
            if which in (0, 1):
                d[which] = _lap(y.view(2, ny, nx)[which], dx)
            else:
                d[1] = -y.view(2, ny, nx)[1]
            return torch.cat([mv(x) + d.reshape(-1), mv(y)])
        return torch.dot(r, _phis(mvk, torch.cat([torch.zeros_like(pr["v"]), pr["v"]]), h, 1, m)[1, :N])
    gt = torch.stack([frechet(0), frechet(1), -h * torch.dot(r, phi[1] - phi[2]), frechet(3)])
    return {"y": phi[1], "grad_v": gv, "grad_h": gh.cpu(), "grad_theta": gt.cpu()}
