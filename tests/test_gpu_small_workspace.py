"""f-k plans whose faster stage structure needs a larger workspace: the smaller
form on request, and on a device that does not hold the larger one."""
import ctypes

import numpy as np
import pytest

from oracle import fk
from paper_2608_28183_gb300 import synth
from tests.gpu_util import exact_input, rel_l2, same_peak, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

G = synth.Geometry(96, 80, 300, 16e-12, 2.0, 1.7)
SMALL = ["fk_x_forward", "fk_y_forward", "fk_stolt_z", "fk_y_inverse", "fk_x_inverse"]


@pytest.fixture(scope="module")
def lib():
    from paper_2608_28183_gb300 import build, nlos
    build.build()
    return nlos.load_library()


def _names(lib, handle, n):
    return [lib.nlos_plan_stage_name(handle, i).decode() for i in range(n)]


def test_small_workspace_on_request(lib):
    from paper_2608_28183_gb300 import nlos
    plan = nlos.plan_for_capture(G, "fk")
    small = nlos.plan_for_capture(G, "fk", small_workspace=True)
    assert "fk_z_inverse" in _names(lib, plan.handle, len(plan.tiles))
    assert _names(lib, small.handle, len(small.tiles)) == SMALL
    assert small.workspace_bytes < plan.workspace_bytes <= 1.5 * small.workspace_bytes
    H = synth.point_capture(G, [(0.2, -0.1, 0.5, 1.0)], peak=200.0).counts
    ref = fk.fk_reconstruct(exact_input(H, torch.float32), G.bin_width_s, G.wall_w_m, G.wall_h_m)
    x = to_device(H, torch.float32)
    for p in (plan, small):
        got = p.reconstruct(x).cpu().numpy()
        assert rel_l2(got, ref) <= 1e-5 and same_peak(got, ref)
    # no choice to make: the flag changes nothing
    for g, st in ((synth.Geometry(64, 64, 256, 32e-12, 1.0, 1.0), "f32"), (G, "f16")):
        a, b = nlos.plan_for_capture(g, "fk", st), nlos.plan_for_capture(g, "fk", st, small_workspace=True)
        assert a.workspace_bytes == b.workspace_bytes and a.tiles == b.tiles


def test_plan_takes_the_small_form_when_the_device_is_full(lib):
    from paper_2608_28183_gb300 import nlos
    small = nlos.plan_for_capture(G, "fk", small_workspace=True)
    desc = nlos.desc_for_capture(G, "fk")
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]

    def create(k):
        h = ctypes.c_void_p()
        lib.nlos_debug_fail_allocation(k)
        st = lib.nlos_plan_create(ctypes.byref(desc), ctypes.byref(h))
        lib.nlos_debug_fail_allocation(0)
        ws = ctypes.c_size_t()
        if st == 0:
            assert lib.nlos_plan_query(h, None, ctypes.byref(ws), None, None) == 0
            assert lib.nlos_plan_destroy(h) == 0
        return st, ws.value

    n = 0
    while create(-(n + 1)) == (0, small.workspace_bytes):   # the (n + 1)-th allocation fails
        n += 1
        assert n < 64
    st, ws = create(-(n + 1))                                # there are only n: the plan as it is
    assert n >= 2 and st == 0 and ws > small.workspace_bytes
    assert create(n) == (2, 0)                               # an injected failure is reported as before
    torch.cuda.synchronize()
    assert abs(torch.cuda.mem_get_info()[0] - free0) < (64 << 20)
