"""Float32 f-k plans that take the inverse temporal transform last although
their time axis is no power of two, or their lateral stages are not fused both
ways: parity with the FP64 oracle at the repository's float32 tolerance, and
agreement with the separate-axis plan (temporal inverse inside the stage)."""
import numpy as np
import pytest

from oracle import fk
from paper_2608_28183_gb300 import synth
from tests.gpu_util import exact_input, rel_l2, same_peak, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (grid, stage names expected): the fused inverse needs a square padded grid
# of at least 128; V's L/2 columns exceed n by 1.0 to 1.7 times
CASES = [
    (synth.Geometry(96, 80, 300, 16e-12, 2.0, 1.7), ["fk_stolt", "fk_yx_inverse", "fk_z_inverse"]),
    (synth.Geometry(65, 128, 511, 16e-12, 1.0, 2.0), ["fk_stolt", "fk_yx_inverse", "fk_z_inverse"]),
    (synth.Geometry(48, 160, 336, 16e-12, 0.6, 2.0), ["fk_stolt", "fk_y_inverse", "fk_x_inverse", "fk_z_inverse"]),
    (synth.Geometry(260, 258, 24, 200e-12, 2.0, 2.0), ["fk_stolt", "fk_yx_inverse", "fk_z_inverse"]),
    (synth.Geometry(64, 40, 1300, 16e-12, 1.0, 0.7), ["fk_stolt", "fk_yx_inverse", "fk_z_inverse"]),
    # below the size rule, and growth above it: the temporal stage keeps its inverse
    (synth.Geometry(30, 30, 300, 16e-12, 1.0, 1.0), ["fk_stolt_z"]),
    (synth.Geometry(96, 80, 260, 16e-12, 2.0, 1.7), ["fk_stolt_z"]),
]


@pytest.mark.parametrize("output", ["magnitude", "complex"])
@pytest.mark.parametrize("geom,stages", CASES, ids=[f"{g.nx}x{g.ny}x{g.nt}" for g, _ in CASES])
def test_fk_temporal_inverse_last_any_time_axis(geom, stages, output):
    from paper_2608_28183_gb300 import build, nlos
    build.build()
    if output == "complex" and geom.nt == 1300:
        pytest.skip("one output is enough at the longest time axis")
    rng = np.random.default_rng(geom.nt)
    pts = [(rng.uniform(-0.3, 0.3) * geom.wall_w_m, rng.uniform(-0.3, 0.3) * geom.wall_h_m,
            rng.uniform(0.3, 0.8) * geom.nt * geom.bin_depth_m, 1.0) for _ in range(2)]
    H = synth.render(geom, synth.Scene(points=np.array(pts)), peak=200.0, background=0.5, seed=geom.nt).counts
    plan = nlos.plan_for_capture(geom, "fk", output=output)
    names = [nlos.load_library().nlos_plan_stage_name(plan.handle, i).decode() for i in range(len(plan.tiles))]
    assert [n for n in names if n in stages] == stages and ("fk_stolt" in names) == ("fk_stolt" in stages)
    x = to_device(H, torch.float32)
    ref = fk.fk_reconstruct(exact_input(H, torch.float32), geom.bin_width_s, geom.wall_w_m, geom.wall_h_m,
                            return_complex=output == "complex")
    sep = nlos.plan_for_capture(geom, "fk", output=output, separate_axes=True)
    for tile in ((0, 2, 3) if "fk_stolt" in names else (0,)):
        plan.tiles = [tile if n in ("fk_stolt", "fk_z_inverse") else t for n, t in zip(names, plan.tiles)]
        got = plan.reconstruct(x).cpu().numpy()
        assert plan.check_workspace() == 0
        assert rel_l2(got, ref) <= 1e-5
        if output == "magnitude":
            assert same_peak(got, ref)
    assert rel_l2(got, sep.reconstruct(x).cpu().numpy()) <= 1e-5
