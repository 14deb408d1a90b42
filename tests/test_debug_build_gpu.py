"""The debug build of the library (-DFF_DEBUG: band ranks and grid coordinates of the band split, tile starts and rows of the
attention, positions of the exchange, rows of the plane buffer of the two-axis launch, load and store boxes of the two launches
with the second axis in registers are range-checked on the device, and a value out of range raises FF_ERR_INVALID_ARG in the status
word instead of being used) runs layers that reach every kernel with such checks: a second axis of 16 (W = 32 and 16) and of 32
(32x32x16, 16 heads), planes of 32 (32x32x16, three heads) and of 16 channels (16x16x128), head_dim 64, grids whose transform hands
on fp32, of few tiles and of more; no check may fire and the result must match the fp64 oracle like the release build's.  Run in a
child process, because the binding loads one variant of the library per process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, %r); sys.path.insert(0, %r)
import numpy as np
from paper_2604_22808_b200 import binding as B, configs as C, inputs as I
import harness as Hn
assert B._LIB_PATH.endswith("libfreqformer_debug.so")
for cfg, alloc in ((C.R64K, [1, 2, 4, 7, 2, 4]), (C.R_PAPER_REF, [1, 2, 4, 7]), (C.GEOM, [7, 2, 4]),
                   (C.GEOM32, [7, 2, 4]), (C.FOLD32, [7, 2, 4] + [0] * 13), (C.R128K.scaled("w16", batch=1), [1, 2, 4, 7, 2, 4]),
                   (C.RAGGED, [7, 2, 4]), (C.TILES, [1, 2, 0])):
    Q, K, V = Hn.host_inputs(cfg)
    weights = I.router_weights(cfg)
    ts = [cfg.timesteps[0]] * cfg.batch
    res = Hn.oracle_forward(cfg, Q, K, V, weights, I.summary_projection(cfg), ts, alloc=alloc)
    out, plan = Hn.gpu_forward(cfg, Q, K, V, weights, None, timesteps=ts, alloc=alloc)     # asserts device status 0
    assert plan.kernel_info()["forward_axis_in_registers"] == (cfg.name in ("64k_replica", "paper_ref_replica", "fold32", "w16"))
    Hn.assert_close(out[0], res[0]["out"], cfg.dtype, cfg.name)
    plan.destroy()
print("DEBUG_BUILD_OK")
"""


def test_debug_build_runs_clean_and_matches():
    from paper_2604_22808_b200 import build as ffbuild
    ffbuild.build(debug=True)
    env = dict(os.environ, FF_LIBRARY_VARIANT="debug")
    child = CHILD % (ROOT, os.path.join(ROOT, "tests"))
    child = child.replace("C.GEOM,", 'C._make("geom_16x16x128", 1, (16, 16, 128), 3, 128, "bf16", (1, 8), 8, 64, 8, 256, 16, 22, (500,)),')
    child = child.replace("C.GEOM32", 'C._make("geom_32x32x16", 1, (32, 32, 16), 3, 128, "bf16", (1, 8), 8, 64, 8, 256, 16, 21, (500,))')
    child = child.replace("C.FOLD32", 'C._make("fold32", 1, (32, 32, 16), 16, 128, "bf16", (1, 8), 8, 64, 8, 256, 16, 21, (500,))')
    child = child.replace("C.RAGGED", 'C.R64K.scaled("ragged", T=5, H=33, W=20, low_cut=(1, 4, 2), mid_cut=(3, 20, 12), heads=3)')
    child = child.replace("C.TILES", 'C.R64K.scaled("tiles", T=12, H=40, W=100, low_cut=(1, 4, 8), mid_cut=(7, 22, 50), heads=3)')
    r = subprocess.run([sys.executable, "-c", child], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "DEBUG_BUILD_OK" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
