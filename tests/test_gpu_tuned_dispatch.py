"""Calls without a shape while the tuning table names one: whatever kernel the
library then runs, results match the oracle in a workspace of that shape's size,
below, at and above the sizes where all tiles run at once."""
import json
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# a process of its own: the table is the process's
CODE = """
import sys
sys.path[:0] = [%(root)r, %(root)r + "/tests"]
import numpy as np, torch
import ka_inputs as ki, oracle
import paper_1709_07781_gb300 as ka
from gpu_util import Workspace, empty, stream, to_dev, to_host, word
shape = %(shape)r
assert ka.ka_autotune_load(%(path)r) == 0
for n in (1, 5000, 100003, 700001, 2098153, 3000001, 4194304, 4980737, 5300001):
    assert ka.ka_tile_for(ka.KA_KERNEL_COMPACT, n) == (0, shape)
    x = ki.uniform_u32(n & 0xFF, n)
    for off, live in ((0, None), (1, None), (3, n - n // 3)):
        ws = Workspace(ka, n, shape)
        buf = to_dev(np.concatenate([np.zeros(off, np.uint32), x]), pad=4)
        out, count = empty(n + 4), empty(1)
        d_n = None if live is None else to_dev(np.array([live], np.uint32))
        assert ka.ka_compact(buf.data_ptr() + 4 * off, n, d_n, ka.KA_PRED_MOD_NE0, 3, 1, out, count, ws.ptr, ws.nbytes,
                             None, stream()) == 0
        torch.cuda.synchronize()
        assert ws.status(ka) == 0
        y, k = oracle.compact(oracle.map_hash(x if live is None else x[:live]), "mod_ne0", 3)
        got = to_host(out)
        assert word(count) == k and np.array_equal(got[:k], y) and (got[k:] == 0xDEADBEEF).all(), (n, off, live)
"""


@pytest.mark.parametrize("shape", [(128, 4), (256, 4), (512, 8), (1024, 8), (256, 16), (512, 16), (768, 16)])
def test_a_shape_of_the_table(cuda_ok, tmp_path, shape):
    path = str(tmp_path / "tune.json")
    with open(path, "w") as fh:
        json.dump({"entries": [{"kernel": 0, "bucket": b, "block": shape[0], "ipt": shape[1], "us": 1.0}
                               for b in range(24)]}, fh)
    r = subprocess.run([sys.executable, "-c", CODE % {"root": ROOT, "shape": shape, "path": path}],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
