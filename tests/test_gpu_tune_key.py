"""Autotuned launch shapes are shared by plans of the same stages only: one
entry per stage structure, transform lengths and output of a capture, whatever
was tuned first, and one for plans that differ in nothing the stages see."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CODE = """
from paper_2608_28183_gb300 import nlos, synth
small, fused = synth.Geometry(32, 32, 256, 32e-12, 1.0, 1.0), synth.Geometry(64, 64, 256, 32e-12, 1.0, 1.0)
wide = synth.Geometry(64, 64, 160, 24e-12, 1.0, 1.0)
pf = dict(n_depths=8, depth_min_m=0.4, depth_max_m=1.0)
PLANS = [(small, "fk", {}), (small, "fk", dict(pad_factor=1)), (small, "fk", dict(output="complex")),
         (fused, "fk", {}), (fused, "fk", dict(separate_axes=True)),
         (wide, "fk", {}), (wide, "fk", dict(small_workspace=True)), (wide, "fk", dict(separate_axes=True)),
         (small, "pf", pf), (small, "pf", dict(pf, output="complex"))]
for g, m, kw in PLANS:
    p = nlos.plan_for_capture(g, m, **kw)
    p.autotune()
    q = nlos.plan_for_capture(synth.Geometry(g.nx, g.ny, g.nt, g.bin_width_s, 1.0, 1.0), m, **kw)
    q.autotune()
    assert q.tiles == p.tiles
print(len(PLANS))
"""


def test_one_entry_per_stage_structure(tmp_path):
    from paper_2608_28183_gb300 import build
    build.build()
    cache = tmp_path / "tune.json"
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       env=dict(os.environ, NLOS_AUTOTUNE_CACHE=str(cache)))
    assert r.returncode == 0, r.stderr
    saved = json.loads(cache.read_text())
    assert len(saved) == int(r.stdout.split()[-1]), sorted(saved)
    assert "m0_s0_32x32x256_F0_D0" in saved and "m0_s0_64x64x256_F0_D0" in saved   # as shapes were always saved
