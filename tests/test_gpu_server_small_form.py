"""The server under a budget that holds only the smaller form of a plan, and
plans that have no smaller form: refused after being built once."""
import ctypes

import pytest

from paper_2608_28183_gb300 import synth
from tests.gpu_util import to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    from paper_2608_28183_gb300 import build, nlos
    build.build()
    return nlos.load_library()


def test_budget_for_the_small_form_only(lib):
    from paper_2608_28183_gb300 import nlos
    g = synth.Geometry(96, 80, 300, 16e-12, 2.0, 1.7)
    large = nlos.plan_for_capture(g, "fk")
    small = nlos.plan_for_capture(g, "fk", small_workspace=True)
    small.autotune()             # the launch shapes the server's plan takes from the shared cache
    budget = small.resident_bytes + (1 << 20)          # its tables and its workspace
    assert budget < large.resident_bytes
    server = nlos.Server(memory_budget_bytes=budget, n_slots=2)
    desc = nlos.desc_for_capture(g, "fk")
    server.preload(desc)
    xs = [to_device(synth.point_capture(g, [(0.1 * k, 0.0, 0.5, 1.0)], peak=100.0).counts, torch.float32)
          for k in range(3)]
    outs = [small.empty_volume() for _ in xs]
    for t in [server.submit(desc, x, o) for x, o in zip(xs, outs)]:
        server.wait(t)
    for x, o in zip(xs, outs):
        assert torch.equal(o, small.reconstruct(x))
    m = server.memory()
    assert m["plan_bytes"] + m["workspace_bytes"] <= budget
    server.close()


@pytest.mark.parametrize("method,storage", [("pf", "f32"), ("fk", "f16"), ("fk", "f32")])
def test_refused_plans_without_a_small_form_are_built_once(lib, method, storage):
    from paper_2608_28183_gb300 import nlos
    g = synth.Geometry(64, 64, 256, 32e-12, 1.0, 1.0)
    kw = dict(n_depths=16, depth_min_m=0.4, depth_max_m=1.0) if method == "pf" else {}
    desc = nlos.desc_for_capture(g, method, storage, **kw)
    # the number of allocations that building the plan makes
    n = 0
    while True:
        h = ctypes.c_void_p()
        lib.nlos_debug_fail_allocation(n + 1)
        st = lib.nlos_plan_create_ex(ctypes.byref(desc), nlos.PLAN_NO_WORKSPACE, ctypes.byref(h))
        lib.nlos_debug_fail_allocation(0)
        if st == 0:
            break
        n += 1
    assert n >= 2 and lib.nlos_plan_destroy(h) == 0
    server = nlos.Server(memory_budget_bytes=4096, n_slots=1)
    lib.nlos_debug_fail_allocation(n + 1)               # the first allocation of a second build
    with pytest.raises(nlos.NlosError, match="exceed the budget"):
        server.preload(desc)
    lib.nlos_debug_fail_allocation(0)
    server.close()
