"""f-k layouts and launch shapes at the edges of their ranges, against the FP64
oracle at the repository's tolerances (float32 1e-5, f16 2e-3, bf16 3e-2):
every launch shape of the temporal stages up to length 8192, the temporal
stage that writes psi blocked by 8 columns, and blocked runs that end inside a
128-byte line, with the intermediate dropped from L2 and kept."""
import numpy as np
import pytest

from oracle import fk
from paper_2608_28183_gb300 import synth
from tests.gpu_util import exact_input, rel_l2, same_peak, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"f32": 1e-5, "f16": 2e-3, "bf16": 3e-2}


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_2608_28183_gb300 import build, nlos
    build.build()
    return nlos.load_library()


def _setup(lib, geom, storage, output="magnitude"):
    """(plan, stage names, device input, oracle volume)"""
    from paper_2608_28183_gb300 import nlos
    rng = np.random.default_rng(geom.nt + geom.ny)
    pts = [(rng.uniform(-0.3, 0.3) * geom.wall_w_m, rng.uniform(-0.3, 0.3) * geom.wall_h_m,
            rng.uniform(0.3, 0.8) * geom.nt * geom.bin_depth_m, 1.0) for _ in range(2)]
    H = synth.render(geom, synth.Scene(points=np.array(pts)), peak=200.0, background=0.5, seed=geom.nt).counts
    plan = nlos.plan_for_capture(geom, "fk", storage, output=output)
    names = [lib.nlos_plan_stage_name(plan.handle, i).decode() for i in range(len(plan.tiles))]
    dt = plan.input_dtype()
    ref = fk.fk_reconstruct(exact_input(H, dt), geom.bin_width_s, geom.wall_w_m, geom.wall_h_m,
                            return_complex=output == "complex")
    return plan, names, to_device(H, dt), ref


def _check(got, ref, storage):
    got = got.cpu().numpy()
    assert rel_l2(got, ref) <= TOL[storage]
    if storage != "bf16":
        assert same_peak(np.abs(got), np.abs(ref), rtol=1e-6 if storage == "f32" else 2e-3)


def _id(v):
    return f"{v.nx}x{v.ny}x{v.nt}" if hasattr(v, "nx") else None


# temporal lengths 32 to 8192 of float32 plans with the inverse temporal
# transform last, a time axis that is no power of two and one that is; at 4096
# and 8192 some shapes have one pencil per CTA, at 8192 the fused lateral
# inverse runs over 4096 columns
SPLIT = [
    synth.Geometry(260, 258, 24, 200e-12, 2.0, 2.0),      # 64
    synth.Geometry(260, 258, 16, 200e-12, 2.0, 2.0),      # 32 = 2 nt
    synth.Geometry(48, 160, 336, 16e-12, 0.6, 2.0),       # 1024
    synth.Geometry(40, 34, 600, 16e-12, 0.6, 0.5),        # 2048
    synth.Geometry(64, 40, 1300, 16e-12, 1.0, 0.7),       # 4096
    synth.Geometry(40, 34, 3002, 16e-12, 0.6, 0.5),       # 8192
    synth.Geometry(24, 20, 3002, 16e-12, 0.4, 0.3),       # 8192, separate lateral inverses
    synth.Geometry(34, 33, 4096, 16e-12, 0.5, 0.5),       # 8192 = 2 nt
]


@pytest.mark.parametrize("geom", SPLIT, ids=_id)
def test_split_temporal_stage_every_launch_shape(library, geom):
    plan, names, x, ref = _setup(library, geom, "f32")
    assert "fk_stolt" in names and "fk_z_inverse" in names
    for shape in range(4):
        plan.tiles = [shape if n in ("fk_stolt", "fk_z_inverse") else t for n, t in zip(names, plan.tiles)]
        _check(plan.reconstruct(x), ref, "f32")
    assert plan.check_workspace() == 0


def test_split_temporal_stage_complex_8192(library):
    geom = SPLIT[-3]
    plan, names, x, ref = _setup(library, geom, "f32", "complex")
    for shape in range(4):
        plan.tiles = [shape if n in ("fk_stolt", "fk_z_inverse") else t for n, t in zip(names, plan.tiles)]
        assert rel_l2(plan.reconstruct(x).cpu().numpy(), ref) <= 1e-5


# fused lateral stages around a temporal stage that keeps its inverse: 16-bit
# storage with nt no power of two, and float32 whose buffers would grow by
# more than half; length 1024 has the one-warp form as its fifth shape
BLOCKED = [(g, st, out)
           for g, storages in ((synth.Geometry(64, 64, 160, 24e-12, 1.0, 1.0), ("f16", "bf16")),
                               (synth.Geometry(64, 51, 336, 16e-12, 1.0, 0.8), ("f16", "bf16")),
                               (synth.Geometry(64, 64, 272, 16e-12, 1.0, 1.0), ("f32",)),
                               (synth.Geometry(128, 127, 144, 24e-12, 2.0, 2.0), ("f32",)))
           for st in storages for out in (("magnitude",) if st == "bf16" else ("magnitude", "complex"))]


@pytest.mark.parametrize("geom,storage,output", BLOCKED, ids=_id)
def test_blocked_output_of_the_whole_temporal_stage(library, geom, storage, output):
    plan, names, x, ref = _setup(library, geom, storage, output)
    assert [n for n in names if n != "volume_scale"] == ["fk_xy_forward", "fk_stolt_z", "fk_yx_inverse"]
    i = names.index("fk_stolt_z")
    for shape in range(5 if 256 < geom.nt <= 512 else 4):
        plan.tiles = [shape if k == i else t for k, t in enumerate(plan.tiles)]
        _check(plan.reconstruct(x), ref, storage)
    assert plan.check_workspace() == 0


# an odd number of wall rows: the forward's runs of 8 b values end inside a
# line, which the next item's run shares
ODD = [
    (synth.Geometry(100, 97, 256, 24e-12, 1.2, 1.2), "f32"),
    (synth.Geometry(100, 97, 256, 24e-12, 1.2, 1.2), "f16"),
    (synth.Geometry(66, 65, 160, 24e-12, 1.0, 1.0), "f16"),
    (synth.Geometry(130, 131, 64, 100e-12, 2.0, 2.0), "f32"),
]


@pytest.mark.parametrize("geom,storage", ODD, ids=_id)
def test_odd_wall_rows_with_and_without_l2_discard(library, geom, storage):
    plan, names, x, ref = _setup(library, geom, storage)
    chains = [n for n in names if n in ("fk_xy_forward", "fk_yx_inverse")]
    assert chains == ["fk_xy_forward", "fk_yx_inverse"]
    out = []
    for shape in range(4):                    # 0, 1: lines dropped after use; 2, 3: kept
        plan.tiles = [shape if n in chains else t for n, t in zip(names, plan.tiles)]
        ws = torch.full(((plan.workspace_bytes + 3) // 4,), float("nan"), device="cuda")
        out.append(plan.reconstruct(x, workspace=ws).clone())
        _check(out[-1], ref, storage)
    assert all(torch.equal(o, out[0]) for o in out[1:])
