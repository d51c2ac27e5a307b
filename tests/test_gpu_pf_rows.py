"""Phasor rows padded to four values inside a plan: every remainder of the
band's length, the plain stride kept where the padding would take a small
plan's buffers past 32 MiB, and a workspace of NaNs (the padding columns are
never read into a result)."""
import numpy as np
import pytest

from oracle import pf
from paper_2608_28183_gb300 import synth
from tests.gpu_util import exact_input, rel_l2, same_peak, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (band length F, wall, depths); 729 depths: 33.53 MB with F = 21 rows, 33.63 MB with 24
CASES = [(20, 0.44, 9), (21, 0.42, 9), (14, 0.62, 9), (19, 0.48, 9), (21, 0.42, 729)]


@pytest.mark.parametrize("F,wall,D", CASES)
def test_pf_row_padding(F, wall, D):
    from paper_2608_28183_gb300 import build, nlos
    build.build()
    g = synth.Geometry(20, 24, 128, 24e-12, wall, wall)
    plan = nlos.plan_for_capture(g, "pf", n_depths=D, depth_min_m=0.2, depth_max_m=0.4)
    oplan = pf.make_plan(g.nx, g.ny, g.nt, g.bin_width_s, wall, wall, D, 0.2, 0.4)
    assert plan.band[1] == F == len(oplan.band.freqs)
    if D == 729:
        assert plan.workspace_bytes <= (32 << 20)
    H = synth.render(g, synth.Scene(points=np.array([(0.05, -0.04, 0.3, 1.0), (-0.08, 0.02, 0.25, 0.6)])),
                     peak=300.0, background=0.5, seed=F).counts
    ref = pf.pf_reconstruct(exact_input(H, torch.float32), oplan)
    x = to_device(H, torch.float32)
    ws = torch.full(((plan.workspace_bytes + 3) // 4,), float("nan"), device="cuda")
    names = [nlos.load_library().nlos_plan_stage_name(plan.handle, i).decode() for i in range(len(plan.tiles))]
    stage = names.index("pf_depth_sum")
    for form in (0, 1, 2):
        plan.tiles = [form if i == stage else t for i, t in enumerate(plan.tiles)]
        got = plan.reconstruct(x, workspace=ws).cpu().numpy().astype(np.float64)
        assert rel_l2(got, ref) <= 1e-5
        assert same_peak(got, ref)
        ws.fill_(float("nan"))
    # compact phasors of the caller (band weights included) keep the plain stride
    P = pf.phasor_field(exact_input(H, torch.float32), oplan) * oplan.band.weights
    P = torch.from_numpy(np.ascontiguousarray(P, dtype=np.complex64)).cuda()
    assert rel_l2(plan.reconstruct_phasors(P).cpu().numpy().astype(np.float64), ref) <= 1e-5
