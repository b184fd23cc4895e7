"""The dataflow forward and reverse passes (no barrier between levels) against the grid-wide
passes and the per-level launches: the same bits, at the sizes where their work splits change."""
import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_parity_gpu import ctx, dp, gpu_run  # noqa: F401

pytestmark = pytest.mark.gpu

KEYS = ["sp", "tr", "beta", "tr_hyb", "toggles", "grad_sp_in", "grad_tr_in", "grad_pincap", "grad_cload"]

# levels wider than the 38,912 cells the grid holds at once, with fanouts far above the eight edges a
# thread preloads; a narrow deep netlist; one level; more startpoints than the grid holds
SPECS = [netgen.NetlistSpec(130_000, 300, 200, 3, 64, 5), netgen.NetlistSpec(1_500, 9, 8, 200, 32, 6),
         netgen.NetlistSpec(2_500, 2_000, 500, 1, 16, 7), netgen.NetlistSpec(4_000, 45_000, 5_000, 9, 8, 8)]


@pytest.mark.parametrize("spec", SPECS, ids=lambda s: f"{s.n_cells}x{s.depth}")
def test_dataflow_matches_barriers_and_launches(dp, ctx, library_text, spec):  # noqa: F811
    text = netgen.netlist_text(spec)
    sp, tr = netgen.scenario_inputs(spec.n_start, 50)
    for grad_mode, tr_mode, use_step in [(0, 0, False), (1, 1, True)]:
        runs = [gpu_run(dp, ctx, text, library_text, sp[:, 0], tr[:, 0],
                        dp.config(grad_mode=grad_mode, tr_mode=tr_mode, schedule=s, sim_words=16), use_step, True)
                for s in (0, 3, 2, 1)]
        for other in runs[1:]:
            for k in KEYS:
                np.testing.assert_array_equal(runs[0][k], other[k], err_msg=k)


def test_dataflow_after_a_wait_that_gave_up(dp, ctx, library_text):  # noqa: F811
    """A timed-out wait may leave pairs of two passes behind; the next pass must not take one for its own."""
    spec = netgen.NetlistSpec(20_000, 300, 700, 12, 16, 9)
    text = netgen.netlist_text(spec)
    sp, tr = netgen.scenario_inputs(spec.n_start, 51, 2)
    d = dp.dp_design_load(ctx, text, library_text)
    try:
        nn = dp.dp_design_info(d).n_nets
        got = []
        for schedule in (3, 2):
            cfg = dp.config(schedule=schedule)
            for s in (0, 1):
                dp.dp_set_inputs(ctx, d, sp[:, s].copy(), tr[:, s].copy())
                with pytest.raises(dp.DPError):
                    dp.dp_selftest_wait(ctx, 0.01)
                dp.dp_propagate(ctx, d, cfg)
                out = np.zeros(nn, np.float32)
                dp.dp_get_nets(ctx, d, out)
                got.append(out)
        np.testing.assert_array_equal(got[0], got[2])
        np.testing.assert_array_equal(got[1], got[3])
        assert not np.array_equal(got[0], got[1])
    finally:
        dp.dp_design_free(d)


# word counts around the sliced simulation's runs (a run of N cycles adds N - 1), one wave of blocks and
# several, startpoint words around the generator's blocks of sixteen
@pytest.mark.parametrize("T", [2, 3, 4, 5, 15, 16, 17, 31, 32, 64, 65, 127, 250, 400])
def test_sliced_simulation_matches_the_others(dp, ctx, library_text, T):  # noqa: F811
    from tests._netlists import custom_case
    rng = np.random.default_rng(T)
    cases = [(netgen.netlist_text(netgen.NetlistSpec(3_000, 40, 60, 11, 16, 12)), library_text),
             (netgen.netlist_text(netgen.NetlistSpec(9_000, 400, 100, 3, 16, 13)), library_text)]   # 3 rounds a level
    if T in (5, 64, 65):
        cases.append(custom_case(rng, n_in=30, n_cells=2_500))   # 0- to 4-input cells, constants
    for text, lib in cases:
        d = dp.dp_design_load(ctx, text, lib)
        try:
            i = dp.dp_design_info(d)
            sp = rng.uniform(0, 1, i.n_start).astype(np.float32)
            sp[0] = 1.0                                          # a threshold of 2^16: the general chains
            tr = (rng.uniform(0, 1, i.n_start) * 2 * np.minimum(sp, 1 - sp)).astype(np.float32)
            dp.dp_set_inputs(ctx, d, sp, tr)
            got = []
            for schedule in (0, 2, 1):
                cfg = dp.config(schedule=schedule, sim_words=T, seed=T)
                dp.dp_propagate(ctx, d, cfg)
                dp.dp_simulate(ctx, d, cfg)
                tg, on = np.zeros(i.n_nets, np.uint32), np.zeros(i.n_nets, np.uint32)
                dp.dp_get_nets(ctx, d, None, None, None, None, tg, on)
                got.append((tg, on))
            for other in got[1:]:
                np.testing.assert_array_equal(got[0][0], other[0])
                np.testing.assert_array_equal(got[0][1], other[1])
        finally:
            dp.dp_design_free(d)


# one candidate, around one block's sort of 8,192 on both sides, every cell; host and device arrays
@pytest.mark.parametrize("k", [1, 2, 1000, 8191, 8192, 8193, 12_000])
@pytest.mark.parametrize("on_device", [0, 1])
def test_top_k_is_the_full_order(dp, ctx, library_text, k, on_device):  # noqa: F811
    import torch
    spec = netgen.NetlistSpec(12_000, 100, 300, 9, 16, 14)
    sp, tr = netgen.scenario_inputs(spec.n_start, 60)
    d = dp.dp_design_load(ctx, netgen.netlist_text(spec), library_text)
    try:
        cfg = dp.config(grad_mode=0)
        dp.dp_set_inputs(ctx, d, sp[:, 0].copy(), tr[:, 0].copy())
        dp.dp_propagate(ctx, d, cfg)
        dp.dp_backward(ctx, d, cfg)
        s, top, ts = np.zeros(12_000, np.float32), np.zeros(k, np.int32), np.zeros(k, np.float32)
        a = [torch.from_numpy(x).cuda() for x in (s, top, ts)] if on_device else [s, top, ts]
        dp.dp_sizing_scores(ctx, d, cfg, 0, a[0], k, a[1], a[2], on_device)
        s, top, ts = (x.cpu().numpy() if on_device else x for x in a)
    finally:
        dp.dp_design_free(d)
    want = np.lexsort((np.arange(len(s)), -s))[:k]
    np.testing.assert_array_equal(top, want.astype(np.int32))
    np.testing.assert_array_equal(ts, s[want])
