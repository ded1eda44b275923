"""Device memory that the library keeps goes back to the process.

* g3_trim returns it;
* with less than an eighth of the device free, a freed near field is returned at once.
(Each in a process of its own; the second fills the device up to a tenth, untouched.)
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r"""
import gc, torch
import paper_2312_11219_gb300 as g3
from inputs import meshes
ctx = g3.Context(0)
F = g3.g3_freqs_bdf2(ctx, 128, 0.95, 0.05)
v, t = meshes.lshape(24)
T = g3.build_cluster_tree(ctx, v, t, 32, 1.0)
total = torch.cuda.mem_get_info()[1]
fill = None
if FILL:
    fill = torch.empty(torch.cuda.mem_get_info()[0] - total // 10, dtype=torch.uint8, device="cuda")
free0 = torch.cuda.mem_get_info()[0]
nf = g3.assemble_near(ctx, T, F, "slp")
size = nf.info()["bytes"]
assert size > 1 << 30
assert free0 - torch.cuda.mem_get_info()[0] >= size
del nf
gc.collect()
kept = free0 - torch.cuda.mem_get_info()[0]
if FILL:
    assert kept <= 64 << 20, kept
else:
    assert size <= kept <= total // 32, kept
    ctx.trim()
    assert free0 - torch.cuda.mem_get_info()[0] <= 64 << 20
y = g3.apply_gcq(ctx, T, g3.assemble_near(ctx, T, F, "slp"), None, torch.ones(128, t.shape[0], dtype=torch.complex64, device="cuda").t())
assert torch.isfinite(torch.view_as_real(y)).all()
print("ok")
"""


@pytest.mark.parametrize("fill", [False, True])
def test_kept_memory_is_returned(fill):
    r = subprocess.run([sys.executable, "-c", f"FILL = {fill}\n" + CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]
