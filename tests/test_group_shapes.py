"""Host logic of the scenario groups' shapes (no GPU needed): in every mode, whatever shape the environment may ask for
gives blocks of whole rows, so the passes' strides over a level's cells are never zero and no row is half a row.  A small
host program includes the kernels' own header, compiled by nvcc and run on the CPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
#include <cstdio>
#include "kernels.h"
int main() {
    for (int lanes = 1; lanes <= 32; lanes++)
        for (int v = 1; v <= 4; v *= 2)
            for (int threads = 32; threads <= 512; threads += 32) {
                const dp::GroupShape g{lanes, v, 16, threads};
                for (int tr = 0; tr <= 2; tr++) {
                    const dp::GroupShape r = dp::group_for(g, tr);
                    std::printf("%d %d %d %d %d %d %d %d\\n", lanes, v, threads, tr, (int)dp::group_ok(g), r.lanes, r.v,
                                r.threads);
                }
            }
    return 0;
}
"""


def test_every_accepted_shape_runs_in_whole_rows(tmp_path):
    if not shutil.which("nvcc"):
        pytest.skip("nvcc missing")
    src, exe = tmp_path / "groups.cu", tmp_path / "groups"
    src.write_text(PROGRAM)
    subprocess.run(["nvcc", "-std=c++17", "-I", os.path.join(ROOT, "paper_2608_03778_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True, capture_output=True)
    rows = [tuple(map(int, x.split())) for x in
            subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    seen = 0
    for lanes, v, threads, tr, ok, rl, rv, rt in rows:
        assert ok == (threads % lanes == 0)
        if not ok:
            continue
        seen += 1
        assert rt == threads and rt >= rl and rt % rl == 0               # whole rows, at least one
        assert v % rv == 0 and (rv <= 2 or tr != 2)                      # S stays a multiple of the scenarios a thread
        assert rl * rv == lanes * v or (tr == 2 and v == 4 and threads % (2 * lanes))
    assert seen > 100 and any(r[:4] == (32, 4, 32, 2) for r in rows)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", ["32,4,1,32", "32,4,2,96", "8,4,4,96"])
def test_lag_one_groups_of_four_scenarios_a_thread(monkeypatch, shape):
    """shapes whose doubled lanes would leave no whole row, or half a row over: the level launches' bits"""
    import numpy as np

    from paper_2608_03778_gb300 import dp, netgen
    from tests.test_batch_gpu import run_batch
    text, lib = netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4)), netgen.library_text()
    sp, tr = netgen.scenario_inputs(60, 7100, 36)
    c = dp.dp_create(0, None)
    got = []
    try:
        for name, value in (("DP_BATCH_SHAPE", "32,4"), ("DP_BATCH_GROUP", shape)):
            with monkeypatch.context() as m:
                m.setenv(name, value)
                d = dp.dp_design_load(c, text, lib)
                try:
                    got.append(run_batch(dp, c, d, sp, tr, dp.config(grad_mode=0, tr_mode=2)))
                finally:
                    dp.dp_design_free(d)
    finally:
        dp.dp_destroy(c)
    for k in got[0]:
        np.testing.assert_array_equal(got[1][k], got[0][k], err_msg=k)
