"""The tables of the sliced simulation, which a design can do without: an upload that has no memory for them goes on."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_batch_gpu import ctx, dp  # noqa: F401

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import zlib
import numpy as np
from paper_2608_03778_gb300 import dp, netgen
ctx = dp.dp_create(0, None)
try:
    d = dp.dp_design_load(ctx, netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4)), netgen.library_text())
except dp.DPError as e:
    print(e.name)
else:
    i = dp.dp_design_info(d)
    sp, tr = (a[:, 0].copy() for a in netgen.scenario_inputs(60, 5, 1))
    dp.dp_set_inputs(ctx, d, sp, tr)
    g, n = np.zeros(60, np.float32), [np.zeros(i.n_nets, np.uint32) for _ in range(2)]
    dp.dp_step(ctx, d, dp.config(grad_mode=2, sim_words=66), g)
    dp.dp_get_nets(ctx, d, toggles=n[0], ones=n[1])
    print(i.device_bytes, *(zlib.crc32(a.tobytes()) for a in (g, *n)))
"""


def test_no_memory_for_the_slices():
    """the N-th device allocation fails, N = 1, 2, ... until none of the upload's does: the tables' is the last one"""
    seen = []
    for n in range(20, 60):
        r = subprocess.run([sys.executable, "-c", CODE], env=dict(os.environ, DP_FAULT=f"alloc:{n}"), cwd=ROOT,
                           capture_output=True, text=True, timeout=300)
        assert r.returncode == 0 or "injected" in r.stderr, r.stderr[-2000:]
        seen.append(r.stdout.split())
        if r.returncode != 0:   # a first step's allocation: the upload is over
            break
    upload = [s for s in seen if s]
    assert upload[0] == ["DP_ENOMEM"]
    last = upload[-1]                      # without the tables
    full = subprocess.run([sys.executable, "-c", CODE], env={k: v for k, v in os.environ.items() if k != "DP_FAULT"},
                          cwd=ROOT, capture_output=True, text=True, timeout=300).stdout.split()
    assert len(last) == 4 and last[1:] == full[1:]
    assert int(last[0]) < int(full[0])

