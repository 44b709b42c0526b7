"""The float32 3D two-phase kernel that spreads the tile passes' planes over all CTAs: every sum keeps the tile
passes' order, so the basis and H are the one-pass tile form's to the last bit -- on boxes smaller than a tile, of
whole and of ragged tiles, with one plane and many per rank, with more columns than one unit takes, and up to a
breakdown.  And the flat passes that stand in for the streaming kernel: its basis to the last bit, and H to the
rounding of the float64 sums over the CTAs, which alone are in another order."""
import os

import numpy as np
import pytest

import workloads as W
from tests.gpu_util import device_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOXES = [(1, 5, 7, 12), (16, 16, 4, 16), (17, 15, 9, 17), (33, 16, 64, 33), (48, 40, 41, 20), (130, 70, 11, 9),
         (4, 3, 4, 40)]


def arnoldi(op, v, m, variant, form, stream="0"):
    import paper_2410_14917_gb300 as lsa

    env = dict(LSA_TWO_PHASE=form, LSA_STREAM=stream, LSA_TMA="0")
    old = {k: os.environ.get(k) for k in env}
    os.environ.update(env)
    try:
        return lsa.arnoldi(op, v, m, variant=variant, precision="fp32")
    finally:
        for k, o in old.items():
            if o is None:
                os.environ.pop(k)
            else:
                os.environ[k] = o


@pytest.mark.parametrize("variant", ["hcwy", "hncwy", "hgsmgs"])
@pytest.mark.parametrize("box", BOXES, ids=["x".join(map(str, b[:3])) + f"_m{b[3]}" for b in BOXES])
def test_planes_in_parallel_repeat_the_tile_passes(box, variant):
    import paper_2410_14917_gb300 as lsa

    nx, ny, nz, m = box
    cfg = dict(W.adr3d(nx, m=m), ny=ny, nz=nz)
    v, fields = device_inputs(cfg, W.make_inputs(cfg), torch)
    op = lsa.Operator.from_workload(cfg, fields)
    V0, H0, st0 = arnoldi(op, v, m, variant, "0")
    V1, H1, st1 = arnoldi(op, v, m, variant, "1")
    k = st0["m_eff"]
    assert st1["m_eff"] == k and st1["breakdown"] == st0["breakdown"] and st1["grid_syncs"] == st0["grid_syncs"]
    assert torch.equal(V1[:, :k], V0[:, :k])
    assert np.array_equal(H1[: k + 1, :k].cpu().numpy(), H0[: k + 1, :k].cpu().numpy())


# one tile; fewer ranks than SMs and all of them, with 8, 4 and 2 warps to a block's columns; up to 63 columns
STRIPS = [(16, 16, 4, 12), (48, 32, 20, 20), (64, 64, 64, 38), (96, 96, 48, 24), (16, 16, 1, 16), (80, 48, 1, 33),
          (256, 240, 1, 64)]


@pytest.mark.parametrize("variant", ["hcwy", "hgsmgs"])
@pytest.mark.parametrize("box", STRIPS, ids=["x".join(map(str, b[:3])) + f"_m{b[3]}" for b in STRIPS])
def test_flat_passes_repeat_the_streaming_kernel(box, variant):
    import paper_2410_14917_gb300 as lsa

    nx, ny, nz, m = box
    cfg = dict(W.adr3d(nx, m=m), ny=ny, nz=nz) if nz > 1 else W.advdiff2d(nx, ny=ny, m=m)
    v, fields = device_inputs(cfg, W.make_inputs(cfg), torch)
    op = lsa.Operator.from_workload(cfg, fields)
    V0, H0, st0 = arnoldi(op, v, m, variant, "0", "1")
    V1, H1, st1 = arnoldi(op, v, m, variant, "0", "2")
    assert st0["arnoldi_kernel"] == st1["arnoldi_kernel"] == 2
    assert st1["m_eff"] == st0["m_eff"] == m and st1["grid_syncs"] == st0["grid_syncs"]
    assert torch.equal(V1, V0)
    H0, H1 = H0.cpu().numpy(), H1.cpu().numpy()
    assert np.abs(H1 - H0).max() <= 1e-13 * np.abs(H0).max()
