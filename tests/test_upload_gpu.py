"""The tables of the sliced simulation, which a design can do without: an upload that has no memory for them goes on, and
what a long narrow netlist pads them to is bounded."""
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


@pytest.mark.parametrize("n", [40_000, 100_000])
def test_padding_of_a_chain_is_bounded(dp, ctx, n):  # noqa: F811
    lib = "cell BUF Z 0.7 A\ncell INV ZN 0.6 !A\nseq DFF D Q 0.8\n"
    lines = [f"net n{i} 1.0" for i in range(n + 1)] + ["input n0"]
    lines += [f"cell u{i} " + (f"INV A=n{i} ZN=n{i + 1}" if i % 3 else f"BUF A=n{i} Z=n{i + 1}") for i in range(n)]
    d = dp.dp_design_load(ctx, "\n".join(lines) + "\n", lib)
    try:
        info = dp.dp_design_info(d)
        assert info.n_levels == n
        # 64 MiB and 64 bytes a cell for the tables, 384 a level for the barriers, 200 for the rest
        assert info.device_bytes < (64 << 20) + n * (64 + 384 + 200)
        dp.dp_set_inputs(ctx, d, *(a[:, 0].copy() for a in netgen.scenario_inputs(1, 6, 1)))
        got = []
        for schedule in (0, 2):
            cfg = dp.config(schedule=schedule, sim_words=5)
            dp.dp_propagate(ctx, d, cfg)
            dp.dp_simulate(ctx, d, cfg)
            got.append([np.zeros(info.n_nets, np.uint32) for _ in range(2)])
            dp.dp_get_nets(ctx, d, toggles=got[-1][0], ones=got[-1][1])
        for a, b in zip(*got):
            np.testing.assert_array_equal(a, b)
    finally:
        dp.dp_design_free(d)
