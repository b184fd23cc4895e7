"""The passes that a staged batch takes, as reported: the environment's choice, or the tuner's with its times."""
import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_batch_gpu import ctx, dp, run_batch  # noqa: F401

pytestmark = pytest.mark.gpu

SPEC = netgen.NetlistSpec(900, 20, 40, 9, 16, 4)


def stage(dp, ctx, d, S):  # noqa: F811
    dp.dp_set_inputs_batch(ctx, d, *(np.ascontiguousarray(a) for a in netgen.scenario_inputs(60, 77, S)), S)


@pytest.mark.parametrize("tr_mode", [0, 1, 2])
def test_passes_in_use(dp, ctx, library_text, monkeypatch, tr_mode):  # noqa: F811
    d = dp.dp_design_load(ctx, netgen.netlist_text(SPEC), library_text)
    try:
        levels = dp.dp_design_info(d).n_levels
        lag = tr_mode == 2
        for S, name, value, want in [
                (12, "DP_BATCH_SHAPE", "32,4,2", ("level", 1 if lag else 2, levels + 1, 0.0)),
                (13, "DP_BATCH_SHAPE", "32,4,2", ("level", 1, levels + 1, 0.0)),
                (12, "DP_BATCH_GROUP", "4,4,2,128", ("group", 2 if lag else 4, 1, 0.0)),
                (12, "DP_BATCH_FLOW", "4", ("dataflow", 2 if lag else 4, 2, 0.0))]:
            with monkeypatch.context() as m:
                m.setenv(name, value)
                stage(dp, ctx, d, S)
                assert dp.dp_batch_passes(d, tr_mode) == (want, want), (name, S)
        stage(dp, ctx, d, 64)
        got = dp.dp_batch_passes(d, tr_mode)
        for (kind, v, launches, ms), best in zip(got, dp.dp_batch_tuning(d)[2]):
            assert kind in ("level", "group", "dataflow") and 64 % v == 0
            assert launches == {"level": levels + 1, "group": 1, "dataflow": 2}[kind]
            assert 0 < ms <= best or (lag and kind != "dataflow" and ms == 0)
    finally:
        dp.dp_design_free(d)


@pytest.mark.parametrize("tr_mode", [0, 1, 2])
def test_refused_cooperative_launch(dp, ctx, library_text, monkeypatch, tr_mode):  # noqa: F811
    """A grid the device has no room for, which the runtime refuses before anything runs: the tuner leaves the dataflow
    passes out, a call that was to take them takes the others, and the results are the same bits."""
    d = dp.dp_design_load(ctx, netgen.netlist_text(SPEC), library_text)
    cfg = dp.config(grad_mode=0, tr_mode=tr_mode)
    sp, tr = netgen.scenario_inputs(60, 78, 64)
    try:
        want = run_batch(dp, ctx, d, sp, tr, cfg)
        for forced in (False, True):
            dp.dp_selftest_flow_grid(d, 100_000)
            with monkeypatch.context() as m:
                if forced:   # (set after the tuner has run: the launch itself is what is refused)
                    m.setenv("DP_BATCH_SHAPE", "32,4")
                    stage(dp, ctx, d, 64)
                    m.delenv("DP_BATCH_SHAPE")
                    m.setenv("DP_BATCH_FLOW", "1")
                got = run_batch(dp, ctx, d, sp, tr, cfg)
                assert all(p[0] != "dataflow" for p in dp.dp_batch_passes(d, tr_mode))
            for k in want:
                np.testing.assert_array_equal(got[k], want[k], err_msg=k)
            dp.dp_selftest_flow_grid(d, 0)
            got = run_batch(dp, ctx, d, sp, tr, cfg)
            for k in want:
                np.testing.assert_array_equal(got[k], want[k], err_msg=k)
    finally:
        dp.dp_design_free(d)


@pytest.mark.parametrize("tr_mode", [0, 2])
@pytest.mark.parametrize("S", [1, 6])
def test_no_room_for_the_clusters(dp, ctx, library_text, tr_mode, S):  # noqa: F811
    """A device without room for the groups' clusters (asked for a size that none has): level launches, in the tuner for
    one scenario, and where the lag-one mode goes by the rule; the same bits."""
    d = dp.dp_design_load(ctx, netgen.netlist_text(SPEC), library_text)
    cfg = dp.config(grad_mode=0, tr_mode=tr_mode)
    sp, tr = netgen.scenario_inputs(60, 79, S)
    try:
        want = run_batch(dp, ctx, d, sp, tr, cfg)
        dp.dp_selftest_flow_grid(d, 100_000)
        got = run_batch(dp, ctx, d, sp, tr, cfg)
        assert all(p[0] == "level" for p in dp.dp_batch_passes(d, tr_mode))
        for k in want:
            np.testing.assert_array_equal(got[k], want[k], err_msg=k)
    finally:
        dp.dp_design_free(d)
