"""The batched passes without level barriers: the same bits as the level launches, whatever ran on the design's
buffers before, in a CUDA graph and with NaN inputs."""
import os

import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2608_03778_gb300 import netgen
from tests._netlists import custom_case
from tests.test_batch_gpu import check_lag1, check_scenarios, ctx, dp, run_batch  # noqa: F401

pytestmark = pytest.mark.gpu


class forced:
    """the batched passes of a block by level launches, or by dataflow with v scenarios per thread"""

    def __init__(self, how):
        self.env = ("DP_BATCH_SHAPE", "32,4") if how == "level" else ("DP_BATCH_FLOW", str(how))

    def __enter__(self):
        os.environ[self.env[0]] = self.env[1]

    def __exit__(self, *exc):
        os.environ.pop(self.env[0], None)


def run(dp, ctx, text, lib, how, sp, tr, tr_mode):  # noqa: F811
    with forced(how):
        d = dp.dp_design_load(ctx, text, lib)
        try:
            return run_batch(dp, ctx, d, sp, tr, dp.config(grad_mode=0, tr_mode=tr_mode))
        finally:
            dp.dp_design_free(d)


def same(a, b, msg):
    for k in b:
        np.testing.assert_array_equal(a[k], b[k], err_msg=f"{msg} {k}")


def netlists(library_text, S):
    # fanouts beyond the edges in flight; 0- to 4-input cells of any function; a single level
    return [(netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4)), library_text),
            custom_case(np.random.default_rng(S), n_in=15, n_cells=300),
            (netgen.netlist_text(netgen.NetlistSpec(40, 8, 8, 1, 16, 3)), library_text)]


# one lane, a ragged chunk, whole chunks, a ragged last chunk of 64 and of 128 columns
@pytest.mark.parametrize("tr_mode", [0, 1, 2])
@pytest.mark.parametrize("S", [1, 33, 64, 130, 260])
def test_dataflow_matches_level_launches(dp, ctx, library_text, S, tr_mode):  # noqa: F811
    for i, (text, lib) in enumerate(netlists(library_text, S)):
        o = Oracle(text, lib)
        sp, tr = netgen.scenario_inputs(o.n_start, 8000 + S, S)
        ref = run(dp, ctx, text, lib, "level", sp, tr, tr_mode)
        for v in (1, 2, 4):
            if S % v == 0:
                same(run(dp, ctx, text, lib, v, sp, tr, tr_mode), ref, f"netlist {i} v {v}")
        if tr_mode == 2:
            check_lag1(o, ref, sp, tr, range(min(S, 3)))
        else:
            check_scenarios(o, ref, sp, tr, dp.config(grad_mode=0, tr_mode=tr_mode), range(min(S, 3)))


def test_dataflow_after_other_passes(dp, ctx, library_text):  # noqa: F811
    """tags and resting words of other passes, other S and other modes on the same buffers"""
    text = netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4))
    inputs = {S: netgen.scenario_inputs(60, 50 + S, S) for S in (96, 64, 32)}
    ref = {(S, m): run(dp, ctx, text, library_text, "level", *inputs[S], m) for S in inputs for m in (0, 2)}
    d = dp.dp_design_load(ctx, text, library_text)
    try:
        for i, (how, S, m) in enumerate([(2, 96, 0), (2, 96, 0), (1, 64, 0), (4, 96, 0), ("level", 64, 0), (2, 64, 0),
                                         ("level", 64, 2), (2, 64, 0), (1, 32, 0), ("level", 32, 0), (2, 96, 0),
                                         (2, 96, 2), (1, 64, 2), ("level", 96, 2), (1, 96, 2), (4, 96, 0)]):
            with forced(how):
                got = run_batch(dp, ctx, d, *inputs[S], dp.config(grad_mode=0, tr_mode=m))
            same(got, ref[S, m], f"step {i}")
    finally:
        dp.dp_design_free(d)


@pytest.mark.parametrize("tr_mode", [1, 2])
def test_dataflow_nan_inputs(dp, ctx, library_text, tr_mode):  # noqa: F811
    torch = pytest.importorskip("torch")
    text = netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4))
    sp, tr = netgen.scenario_inputs(60, 5, 64)
    sp[3, 5], sp[7, 9], sp[11, 40] = np.nan, np.inf, -np.inf
    tr[8, 12] = np.array([0xFFFFFFFF], np.uint32).view(np.float32)[0]
    x, t = torch.from_numpy(sp).cuda(), torch.from_numpy(tr).cuda()
    cfg = dp.config(grad_mode=0, tr_mode=tr_mode)
    got = {}
    for how in ("level", 1, 4):
        d = dp.dp_design_load(ctx, text, library_text)
        try:
            with forced(how):
                dp.dp_set_inputs_batch(ctx, d, x, t, 64, on_device=1)
                dp.dp_propagate(ctx, d, cfg)
                g, p = torch.empty_like(x), torch.empty(64, dtype=torch.float64, device="cuda")
                dp.dp_backward_weighted(ctx, d, cfg, None, 1, g, None, None, None, on_device=1)
                dp.dp_get_power(ctx, d, p, 0, on_device=1)
                torch.cuda.synchronize()
                got[how] = (np.isnan(p.cpu().numpy()), p.cpu().numpy(), g.cpu().numpy())
        finally:
            dp.dp_design_free(d)
    clean = np.ones(64, bool)
    clean[[5, 9, 12, 40]] = False
    for how in (1, 4):
        np.testing.assert_array_equal(got[how][0], got["level"][0])
        np.testing.assert_array_equal(got[how][1][clean], got["level"][1][clean])
        np.testing.assert_array_equal(got[how][2][:, clean], got["level"][2][:, clean])
        np.testing.assert_array_equal(np.isnan(got[how][2]), np.isnan(got["level"][2]))


def test_dataflow_in_a_graph(dp, library_text):  # noqa: F811
    """a captured pass replayed after passes of another kind and size on the same design"""
    torch = pytest.importorskip("torch")
    text = netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4))
    st = torch.cuda.Stream()
    c = dp.dp_create(0, st.cuda_stream)
    d = dp.dp_design_load(c, text, library_text)
    cfg = dp.config(grad_mode=0, tr_mode=0)
    try:
        with torch.cuda.stream(st):
            x, t = (torch.from_numpy(a).cuda() for a in netgen.scenario_inputs(60, 9, 96))
            y, u = x[:, :32].contiguous(), t[:, :32].contiguous()
            g, p = torch.empty_like(x), torch.empty(96, dtype=torch.float64, device="cuda")
            h = torch.empty_like(y)

            def step(a, b, grad):
                dp.dp_set_inputs_batch(c, d, a, b, a.shape[1], on_device=1)
                dp.dp_propagate(c, d, cfg)
                dp.dp_backward_weighted(c, d, cfg, None, 1, grad, None, None, None, on_device=1)

            with forced(4):
                step(x, t, g)
                st.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=st):
                    step(x, t, g)
                    dp.dp_get_power(c, d, p, 0, on_device=1)
            with forced("level"):
                step(x, t, g)
                dp.dp_get_power(c, d, p, 0, on_device=1)
                st.synchronize()
                ref = g.cpu().numpy(), p.cpu().numpy()
            for other in ("level", 1, 2):
                with forced(other):
                    step(y, u, h)
                for _ in range(3):
                    g.zero_()
                    graph.replay()
                    st.synchronize()
                    np.testing.assert_array_equal(g.cpu().numpy(), ref[0])
                    np.testing.assert_array_equal(p.cpu().numpy(), ref[1])
    finally:
        dp.dp_design_free(d)
        dp.dp_destroy(c)


def test_more_levels_than_the_dataflow_passes_take(dp, ctx):  # noqa: F811
    """a chain of inverters and buffers beyond their level bounds runs as before"""
    n = 8200
    lib = "cell BUF Z 0.7 A\ncell INV ZN 0.6 !A\nseq DFF D Q 0.8\n"
    lines = [f"net n{i} 1.0" for i in range(n + 1)] + ["input n0"]
    lines += [f"cell u{i} " + (f"INV A=n{i} ZN=n{i + 1}" if i % 3 else f"BUF A=n{i} Z=n{i + 1}") for i in range(n)]
    text = "\n".join(lines) + "\n"
    sp, tr = netgen.scenario_inputs(1, 3, 8)
    same(run(dp, ctx, text, lib, 1, sp, tr, 1), run(dp, ctx, text, lib, "level", sp, tr, 1), "chain")
