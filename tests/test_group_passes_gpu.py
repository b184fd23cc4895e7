"""The batched passes by scenario groups (one launch per pass) and the functions compiled into the cell
evaluation: the same bits as the level launches, and both against the oracle."""
import os

import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2608_03778_gb300 import netgen
from tests._netlists import custom_case
from tests.test_batch_gpu import check_lag1, check_scenarios, ctx, dp, run_batch  # noqa: F401

pytestmark = pytest.mark.gpu

# lanes, scenarios per thread, blocks of the cluster, threads: one row of lanes, idle lanes, several groups,
# one block and the largest cluster, more rows than a level has cells and fewer
SHAPES = ["8,1,16,512", "1,1,1,512", "2,2,4,64", "4,4,2,128", "32,1,8,256", "16,2,1,512"]


def runs(dp, ctx, text, lib, sp, tr, tr_mode):  # noqa: F811
    got = {}
    for name in ["level"] + SHAPES:
        os.environ["DP_BATCH_SHAPE" if name == "level" else "DP_BATCH_GROUP"] = "32,4" if name == "level" else name
        try:
            d = dp.dp_design_load(ctx, text, lib)
            try:
                got[name] = run_batch(dp, ctx, d, sp, tr, dp.config(grad_mode=0, tr_mode=tr_mode))
            finally:
                dp.dp_design_free(d)
        finally:
            os.environ.pop("DP_BATCH_SHAPE", None)
            os.environ.pop("DP_BATCH_GROUP", None)
    return got


@pytest.mark.parametrize("tr_mode", [0, 1, 2])
@pytest.mark.parametrize("S", [1, 7, 12, 33])
def test_groups_match_level_launches(dp, ctx, library_text, S, tr_mode):  # noqa: F811
    cases = [(netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4)), library_text),
             custom_case(np.random.default_rng(S), n_in=15, n_cells=300)]      # 0- to 4-input cells, any function
    for i, (text, lib) in enumerate(cases):
        o = Oracle(text, lib)
        sp, tr = netgen.scenario_inputs(o.n_start, 7000 + S, S)
        got = runs(dp, ctx, text, lib, sp, tr, tr_mode)
        for name in SHAPES:
            for k in got["level"]:
                np.testing.assert_array_equal(got[name][k], got["level"][k], err_msg=f"{name} {k} {i}")
        if tr_mode == 2:
            check_lag1(o, got["level"], sp, tr, range(min(S, 7)))
        else:
            check_scenarios(o, got["level"], sp, tr, dp.config(grad_mode=0, tr_mode=tr_mode), range(min(S, 7)))
