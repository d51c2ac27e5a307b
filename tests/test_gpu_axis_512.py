"""Axis transforms of 512 points: the TMA-staged launch shapes that hold 32
values per thread give, bit for bit, what the direct-load shapes (16 values
per thread) give, for wall sizes at the edges of the padded length and inner
extents that leave partial column tiles; the direct shape is held to the FP64
oracle at the repository's float32 tolerance."""
import numpy as np
import pytest

from oracle import fk
from paper_2608_28183_gb300 import synth
from tests.gpu_util import exact_input, rel_l2, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [("fk", "f32", 129, 131, 20), ("fk", "f16", 256, 130, 24), ("fk", "bf16", 200, 256, 40),
         ("pf", "f32", 255, 129, 64), ("pf", "f16", 130, 256, 64)]


@pytest.mark.parametrize("method,storage,nx,ny,nt", CASES)
def test_axis_512_launch_shapes_agree(method, storage, nx, ny, nt):
    from paper_2608_28183_gb300 import build, nlos
    build.build()
    g = synth.Geometry(nx, ny, nt, 200e-12, 2.0, 2.0)
    kw = dict(n_depths=13, depth_min_m=0.5, depth_max_m=1.5) if method == "pf" else {}
    plan = nlos.plan_for_capture(g, method, storage, separate_axes=True, **kw)
    dt = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[storage]
    H = synth.render(g, synth.Scene(points=np.array([(0.2, -0.3, 0.9, 1.0)])), peak=200.0, background=0.5,
                     seed=nx).counts
    x = to_device(H, dt)
    lib = nlos.load_library()
    names = [lib.nlos_plan_stage_name(plan.handle, i).decode() for i in range(len(plan.tiles))]
    axis = [i for i, n in enumerate(names)
            if any(k in n for k in ("_x_forward", "_y_forward", "_y_inverse", "_x_inverse"))]
    assert len(axis) == 4
    # one CTA per tile in the float32 depth sum: no atomic sums whose order could differ
    base = [0 if i in axis else 2 if names[i] == "pf_depth_sum" and storage == "f32" else t
            for i, t in enumerate(plan.tiles)]
    plan.tiles = base
    want = plan.reconstruct(x).clone()
    if method == "fk" and storage == "f32":
        ref = fk.fk_reconstruct(exact_input(H, dt), g.bin_width_s, g.wall_w_m, g.wall_h_m)
        assert rel_l2(want.cpu().numpy(), ref) <= 1e-5
    for i in axis:
        # the staged form of each column width (8, 4, 16); pairs of real
        # columns depend on the width, so each is held to its own direct form
        staged = 6 if names[i] == "fk_x_forward" else 3
        for width in range(3):
            out = []
            for tile in (width, width + staged):
                t = list(base)
                t[i] = tile
                plan.tiles = t
                assert plan.tiles[i] == tile
                out.append(plan.reconstruct(x).clone())
                assert plan.check_workspace() == 0
            assert torch.equal(out[0], out[1]), (names[i], width)
            if staged == 3:
                assert torch.equal(out[0], want), (names[i], width)
