"""Inputs whose stored probabilities have a sign: -0.0, which the host's range check takes, and what a device caller may
bring unchecked.  The sign's bit is the ready tag of the passes without level barriers, so both parities of the pass are
run, against the passes with barriers: the same bits, and no wait that gives up."""
import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_parity_gpu import ctx, dp  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

VALUES = {"minus zero": -0.0, "below": -1e-3, "above": 1.001, "nan": -np.nan, "inf": np.inf}


def results(dp, ctx, d, info, sp, tr, cfg, device):  # noqa: F811
    if device:
        dp.dp_set_inputs(ctx, d, torch.from_numpy(sp).cuda(), torch.from_numpy(tr).cuda(), on_device=1)
    else:
        dp.dp_set_inputs(ctx, d, sp, tr)
    dp.dp_propagate(ctx, d, cfg)
    out = [np.zeros(n, np.float32) for n in (info.n_start, info.n_start, info.n_cells, info.n_nets)]
    dp.dp_backward(ctx, d, cfg, *out)
    nets = [np.zeros(info.n_nets, np.float32) for _ in range(2)]
    dp.dp_get_nets(ctx, d, *nets)
    return out + nets


@pytest.mark.parametrize("spec", [(1_500, 9, 8, 200), (20_000, 300, 700, 12), (130_000, 300, 200, 3)])
def test_signed_inputs_match_the_barrier_passes(dp, ctx, library_text, spec):  # noqa: F811
    text = netgen.netlist_text(netgen.NetlistSpec(*spec, 32, 6))
    d = dp.dp_design_load(ctx, text, library_text)
    try:
        info = dp.dp_design_info(d)
        sp, tr = (a[:, 0].copy() for a in netgen.scenario_inputs(info.n_start, 60, 1))
        for what, value in VALUES.items():
            sp[::3] = value
            for device in (False, True) if what == "minus zero" else (True,):
                for tr_mode in (0, 1):
                    want = results(dp, ctx, d, info, sp, tr, dp.config(schedule=2, grad_mode=0, tr_mode=tr_mode), device)
                    for schedule in (3, 3, 0, 0):   # a pass of either parity
                        cfg = dp.config(schedule=schedule, grad_mode=0, tr_mode=tr_mode)
                        for a, b in zip(results(dp, ctx, d, info, sp, tr, cfg, device), want):
                            np.testing.assert_array_equal(a, b, err_msg=f"{what} schedule {schedule} tr_mode {tr_mode}")
    finally:
        dp.dp_design_free(d)
