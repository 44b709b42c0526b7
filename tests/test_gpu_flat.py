"""The flat two-phase Arnoldi kernel: operators and forms that the two-phase
tests do not reach (the augmented operator, the gradient's operators, shares
that end inside a chunk or are empty), and its fixed-point inner products on
vectors whose values span many binades."""
import os

import numpy as np
import pytest

import workloads as W
from tests.gpu_util import FP64_TOL, device_inputs, oracle_phiv, rel_errors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _forced(form, fn):
    kw = dict(LSA_TWO_PHASE=str(form), LSA_TMA="0", LSA_STREAM="0", LSA_CLUSTER="0")
    old = {k: os.environ.get(k) for k in kw}
    os.environ.update(kw)
    try:
        return fn()
    finally:
        for k, v in old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v


def _op(cfg):
    import paper_2410_14917_gb300 as lsa

    inp = W.make_inputs(cfg)
    v, fields = device_inputs(cfg, inp, torch)
    return lsa.Operator.from_workload(cfg, fields), v


# one point; a share of one point; odd columns (scalar loads); one and two chunks per share; one column
# per warp and eight
@pytest.mark.parametrize("nx,ny,m", [(1, 1, 1), (3, 43, 9), (127, 1, 8), (129, 31, 17), (200, 203, 33), (640, 511, 64)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_flat_edges_match_the_tile_form(nx, ny, m, precision):
    import paper_2410_14917_gb300 as lsa

    cfg = W.advdiff2d(nx, ny=ny, m=m, p=2, h=1e-3)
    op, v = _op(cfg)
    y0, s0 = _forced(0, lambda: lsa.phiv(op, v, cfg["h"], 2, m, precision=precision))
    y2, s2 = _forced(2, lambda: lsa.phiv(op, v, cfg["h"], 2, m, precision=precision))
    assert s2["arnoldi_kernel"] == 5 and s2["status"] == s0["status"] and s2["m_eff"] == s0["m_eff"]
    tol = 1e-12 if precision == "fp64" else 1e-5
    assert float((y2 - y0).norm()) <= tol * float(y0.norm())


@pytest.mark.parametrize("nx,ny,m", [(33, 21, 12), (96, 80, 40)])
@pytest.mark.parametrize("variant", ["hcwy", "hncwy", "hgsmgs"])
def test_flat_augmented_and_gradient_match_the_tile_form(nx, ny, m, variant):
    import paper_2410_14917_gb300 as lsa

    g = torch.Generator(device="cuda").manual_seed(11)
    u0, v0 = (torch.rand(nx * ny, dtype=torch.float64, device="cuda", generator=g) for _ in range(2))
    op = lsa.Operator.grayscott2d(nx, ny, dx=2.5 / nx, Du=2e-5, Dv=1e-5, F=0.04, k=0.06, u0=u0, v0=v0)
    b = torch.rand((4, op.N), dtype=torch.float64, device="cuda", generator=g) - 0.5
    out = {}
    for form in (0, 2):
        def both():
            u, _ = lsa.phiv_lincomb(op, b, 0.5, m, 2, variant=variant)
            y, _ = lsa.phiv(op, b[0].contiguous(), 0.5, 2, m, variant=variant)
            return u, lsa.phiv_vjp(op, b[0].contiguous(), 0.5, m, b[1].contiguous(), y, variant=variant)
        out[form] = _forced(form, both)
    (u0_, (gv0, gs0, _)), (u2, (gv2, gs2, _)) = out[0], out[2]
    assert float((u2 - u0_).norm()) <= 1e-12 * float(u0_.norm())
    assert float((gv2 - gv0).norm()) <= 1e-12 * float(gv0.norm())
    assert float((gs2 - gs0).abs().max()) <= 1e-11 * float(gs0.abs().max())


@pytest.mark.parametrize("kind", ["spike", "binades", "constant", "tiny", "huge", "one_sided"])
def test_fixed_point_products_keep_the_orthogonality(kind):
    """The basis of the flat kernel (its inner products in block fixed point)
    is as orthogonal as the float64 tile kernel's, and its phi products as
    close to the oracle, for start vectors that are hard on a common scale."""
    import paper_2410_14917_gb300 as lsa

    cfg = W.advdiff2d(96, ny=50, m=24, p=1)
    op, v = _op(cfg)
    rng = np.random.default_rng(5)
    x = v.cpu().numpy().copy()
    if kind == "spike":
        x = np.full_like(x, 1e-9)
        x[77] = 1.0
    elif kind == "binades":
        x *= 2.0 ** rng.integers(-40, 1, x.size)
    elif kind == "constant":
        x = 1.0 + 1e-6 * x
    elif kind == "tiny":
        x *= 1e-120
    elif kind == "huge":
        x *= 1e120
    else:
        x = np.abs(x) ** 6
    v = torch.from_numpy(x).cuda()
    loss, y = {}, {}
    for form in (0, 2):
        V, H, st = _forced(form, lambda: lsa.arnoldi(op, v, 24))
        k = st["m_eff"]
        G = V[:, :k].T @ V[:, :k]
        loss[form] = float((G - torch.eye(k, dtype=torch.float64, device="cuda")).norm())
        y[form], _ = _forced(form, lambda: lsa.phiv(op, v, cfg["h"], 1, 24))
    # both lose orthogonality by rounding alone: within the spread of two float64 orderings
    assert loss[2] <= 4.0 * loss[0] + 1e-14
    assert max(rel_errors(y[2] / float(v.norm()), (y[0] / float(v.norm())).cpu().numpy())) < FP64_TOL


@pytest.mark.parametrize("nx,ny,m", [(201, 203, 64), (37, 19, 20)])
def test_flat_without_room_for_the_limbs(nx, ny, m):
    """A workspace that ends before the fixed-point basis (the fixed one of
    phiv_noalloc, for the larger grid) converts the columns in place: the same
    products within rounding."""
    import paper_2410_14917_gb300 as lsa

    op, v = _op(W.advdiff2d(nx, ny=ny, m=m, p=1))
    ref, _ = _forced(2, lambda: lsa.phiv(op, v, 1e-2, 1, m))
    y, st = _forced(2, lambda: lsa.phiv_noalloc(op, v, 1e-2, 1, m))
    assert st["m_eff"] == m
    assert float((y - ref).norm()) <= 1e-12 * float(ref.norm())


@pytest.mark.parametrize("path", ["flat", "flat_in_place", "cluster", "batch"])
@pytest.mark.parametrize("bits", [-500, -505, 490])
def test_start_vectors_near_the_ends_of_the_range(path, bits):
    """v scaled by a power of two whose square is still a float64 gives the
    same products scaled: rounding is the same, and what underflows in the
    sums is 2^-1074 a value against squares above 2^-1010, so the two agree
    far below 1e-14."""
    import paper_2410_14917_gb300 as lsa

    n = 64 if path == "cluster" else 201
    cfg = W.advdiff2d(n, ny=n, m=20, p=1)
    op, v = _op(cfg)

    def call(x):
        if path == "batch":
            b = lsa.Batch([op], [20], 1e-2, 1)
            y = b.run(x).clone().view(2, -1)
            st, fin, _ = b.stats()
            assert st >= 0 and fin == 1
            b.close()
            return y
        if path == "cluster":
            y, st = lsa.phiv(op, x, 1e-2, 1, 20)
            assert st["arnoldi_kernel"] == 3
        elif path == "flat":
            y, st = _forced(2, lambda: lsa.phiv(op, x, 1e-2, 1, 20))
            assert st["arnoldi_kernel"] == 5
        else:
            w = lsa.Workspace.for_call(op, 20, 1)
            w.nbytes -= 256                  # ends inside the fixed-point basis
            y, st = _forced(2, lambda: lsa.phiv(op, x, 1e-2, 1, 20, work=w))
        assert st["m_eff"] == 20
        return y

    ref, y = call(v), call(v * 2.0**bits)
    assert float((y * 2.0**-bits - ref).norm()) <= 1e-14 * float(ref.norm())


@pytest.mark.parametrize("path", ["flat", "flat_in_place", "cluster"])
@pytest.mark.parametrize("background", [1e-2, 1e-4, 1e-7])
@pytest.mark.parametrize("peaks", [1, 40])
def test_peaks_over_a_background(path, background, peaks):
    """The integer sums keep every block's products to half a rounding unit of
    its vectors' norms (lsa_fix.cuh), so for peaks over a background beta is
    right to the roundings of some forty float64 additions and a square root
    (1e-15), and the basis loses orthogonality by rounding alone: as the
    float64 tile form, within the spread of two orders of its sums (4)."""
    import paper_2410_14917_gb300 as lsa

    m = 12
    cfg = W.advdiff2d(64, ny=64, m=m) if path == "cluster" else W.adr3d(128, m=m)
    op, v = _op(cfg)
    rng = np.random.default_rng(17)
    x = background * rng.uniform(-1.0, 1.0, v.numel())
    x[rng.integers(0, x.size, peaks)] = rng.uniform(0.5, 1.5, peaks)
    v = torch.from_numpy(x).cuda()

    def run(form):
        if form == 0 or path == "flat":
            return _forced(form, lambda: lsa.arnoldi(op, v, m))
        if path == "cluster":
            return lsa.arnoldi(op, v, m)
        w = lsa.Workspace.for_call(op, m, 0)
        w.nbytes -= 256                  # ends inside the fixed-point basis
        return _forced(2, lambda: lsa.arnoldi(op, v, m, work=w))

    loss = {}
    for form in (0, 2):
        V, H, st = run(form)
        assert st["m_eff"] == m and st["arnoldi_kernel"] == (0 if form == 0 else 3 if path == "cluster" else 5)
        V = V[:, :m].T.contiguous()
        G = V @ V.T - torch.eye(m, dtype=torch.float64, device="cuda")
        loss[form] = float((G - torch.diag(torch.diag(G))).norm())
        beta = np.sqrt(np.sum(np.square(x.astype(np.longdouble))))
        assert abs(st["beta"] / beta - 1) <= 1e-15, form
    assert loss[2] <= 4.0 * loss[0]


def test_least_workspace(monkeypatch):
    """lsa_workspace_least_bytes leaves out the fixed-point basis alone: calls
    take that much and no less, and Workspace.for_call falls back to it when
    the device has no room for the full one."""
    import paper_2410_14917_gb300 as lsa

    op, v = _op(W.advdiff2d(201, ny=203, m=20, p=1))
    full, least = (lsa.workspace_bytes(op, 20, 1, least=x) for x in (False, True))
    assert 8 * 20 * op.N <= full - least <= 8 * 20 * op.N * 1.05 + 65536
    assert lsa.workspace_bytes(op, 20, 1, "fp32", least=True) == lsa.workspace_bytes(op, 20, 1, "fp32")
    ref, _ = _forced(2, lambda: lsa.phiv(op, v, 1e-2, 1, 20))
    empty = torch.empty

    def short(n, *args, **kw):
        if kw.get("dtype") == torch.uint8 and n >= full:
            raise torch.OutOfMemoryError("no room")
        return empty(n, *args, **kw)

    monkeypatch.setattr(torch, "empty", short)
    w = lsa.Workspace.for_call(op, 20, 1)
    monkeypatch.undo()
    assert w.nbytes == least
    y, _ = _forced(2, lambda: lsa.phiv(op, v, 1e-2, 1, 20, work=w))
    assert float((y - ref).norm()) <= 1e-12 * float(ref.norm())
    w.nbytes -= 256
    with pytest.raises(lsa.LsaError):
        lsa.phiv(op, v, 1e-2, 1, 20, work=w)
