"""The step's sliced simulation beside its forward pass: the same results as the phases called one after the other, for
forward passes in one block and in one cluster, whole and ragged word counts, and repeated steps with changed inputs."""
import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_batch_gpu import ctx, dp  # noqa: F401

pytestmark = pytest.mark.gpu


def nets(dp, ctx, d, info):  # noqa: F811
    out = [np.zeros(info.n_nets, t) for t in (np.float32, np.float32, np.uint32, np.uint32)]
    dp.dp_get_nets(ctx, d, beta=out[0], tr_hyb=out[1], toggles=out[2], ones=out[3])
    return out


@pytest.mark.parametrize("spec", [(900, 60, 9), (6000, 400, 24), (16000, 1200, 40)])
@pytest.mark.parametrize("T", [3, 64, 250])
def test_step_equals_its_phases(dp, ctx, library_text, spec, T):  # noqa: F811
    cells, start, depth = spec
    text = netgen.netlist_text(netgen.NetlistSpec(cells, start // 3, start - start // 3, depth, 16, 7))
    d = dp.dp_design_load(ctx, text, library_text)
    try:
        info = dp.dp_design_info(d)
        cfg = dp.config(grad_mode=2, tr_mode=0, sim_words=T)
        for seed in (1, 2):
            sp, tr = (a[:, 0].copy() for a in netgen.scenario_inputs(info.n_start, seed, 1))
            got = {}
            for how in ("phases", "step"):
                g = [np.zeros(n, np.float32) for n in (info.n_start, info.n_start, info.n_cells)]
                dp.dp_set_inputs(ctx, d, sp, tr)
                if how == "step":
                    dp.dp_step(ctx, d, cfg, g[0], g[1], g[2])
                else:
                    dp.dp_propagate(ctx, d, cfg)
                    dp.dp_simulate(ctx, d, cfg)
                    dp.dp_backward(ctx, d, cfg, g[0], g[1], g[2])
                got[how] = g + nets(dp, ctx, d, info)
            for a, b in zip(got["phases"], got["step"]):
                np.testing.assert_array_equal(a, b)
            assert got["step"][5][info.n_start:].any()
    finally:
        dp.dp_design_free(d)


@pytest.mark.parametrize("spec", [(900, 60, 9), (16000, 1200, 40)])
def test_simulation_beside_the_pass_before(dp, library_text, spec):  # noqa: F811
    """dp_simulate right after dp_propagate, again, after other calls, under capture and after a change of stream: the
    counts are those of the step."""
    torch = pytest.importorskip("torch")
    cells, start, depth = spec
    text = netgen.netlist_text(netgen.NetlistSpec(cells, start // 3, start - start // 3, depth, 16, 7))
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    c = dp.dp_create(0, a.cuda_stream)
    d = dp.dp_design_load(c, text, library_text)
    try:
        info = dp.dp_design_info(d)
        cfg = dp.config(grad_mode=2, tr_mode=0, sim_words=64)
        inputs = [[x[:, 0].copy() for x in netgen.scenario_inputs(info.n_start, seed, 1)] for seed in (1, 2)]
        ref = []
        for i in inputs:
            dp.dp_set_inputs(c, d, *i)
            dp.dp_step(c, d, cfg, np.zeros(info.n_start, np.float32))
            ref.append(nets(dp, c, d, info))

        def check(k, what):
            for x, y in zip(nets(dp, c, d, info), ref[k]):
                np.testing.assert_array_equal(x, y, err_msg=what)

        for k in (0, 1, 0, 1):
            dp.dp_set_inputs(c, d, *inputs[k])
            dp.dp_propagate(c, d, cfg)
            dp.dp_simulate(c, d, cfg)
            check(k, "after propagate")
            dp.dp_simulate(c, d, cfg)
            check(k, "again")
            dp.dp_propagate(c, d, cfg)
            dp.dp_step(c, d, cfg, np.zeros(info.n_start, np.float32))
            dp.dp_simulate(c, d, cfg)
            check(k, "after a step")
        e, g = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        dp.dp_propagate(c, d, cfg)
        a.synchronize()
        with torch.cuda.graph(e, stream=a):
            dp.dp_propagate(c, d, cfg)
        with torch.cuda.stream(a):
            e.replay()
            dp.dp_simulate(c, d, cfg)   # the pass before was captured
        check(1, "after a captured pass")
        dp.dp_propagate(c, d, cfg)
        a.synchronize()
        with torch.cuda.graph(g, stream=a):
            dp.dp_propagate(c, d, cfg)
            dp.dp_simulate(c, d, cfg)
        for _ in range(3):
            with torch.cuda.stream(a):
                dp.dp_propagate(c, d, cfg)
                g.replay()
                dp.dp_simulate(c, d, cfg)
            check(1, "after a replay")
        dp.dp_set_stream(c, b.cuda_stream)
        dp.dp_propagate(c, d, cfg)
        dp.dp_simulate(c, d, cfg)
        check(1, "another stream")
    finally:
        dp.dp_design_free(d)
        dp.dp_destroy(c)
