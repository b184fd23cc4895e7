"""A simulation that starts beside the forward pass before it, where the user replays graphs with calls on the design in
between: what the stream's order says is what the simulation reads, and nobody reads its counts half written."""
import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_batch_gpu import dp  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SPECS = [(900, 60, 9), (16000, 1200, 40)]   # a forward pass in one block, and in one cluster


class Case:
    """a design on a stream of its own, two sets of inputs and the counts that each of them gives"""

    def __init__(self, dp, spec, library_text):  # noqa: F811
        cells, start, depth = spec
        self.dp, self.stream = dp, torch.cuda.Stream()
        self.c = dp.dp_create(0, self.stream.cuda_stream)
        text = netgen.netlist_text(netgen.NetlistSpec(cells, start // 3, start - start // 3, depth, 16, 7))
        self.d = dp.dp_design_load(self.c, text, library_text)
        self.info = dp.dp_design_info(self.d)
        self.cfg = dp.config(grad_mode=2, tr_mode=0, sim_words=64)
        self.inputs = [[x[:, 0].copy() for x in netgen.scenario_inputs(self.info.n_start, seed, 1)] for seed in (1, 2)]
        self.want = []
        for i in self.inputs:
            dp.dp_set_inputs(self.c, self.d, *i)
            dp.dp_step(self.c, self.d, self.cfg, np.zeros(self.info.n_start, np.float32))
            self.want.append(self.counts())

    def counts(self):
        out = [np.zeros(self.info.n_nets, np.uint32) for _ in range(2)]
        self.dp.dp_get_nets(self.c, self.d, toggles=out[0], ones=out[1])
        return out

    def check(self, k, what):
        for x, y in zip(self.counts(), self.want[k]):
            np.testing.assert_array_equal(x, y, err_msg=what)

    def close(self):
        self.dp.dp_design_free(self.d)
        self.dp.dp_destroy(self.c)


@pytest.mark.parametrize("spec", SPECS)
def test_replayed_inputs_reach_the_simulation(dp, library_text, spec):  # noqa: F811
    t = Case(dp, spec, library_text)
    try:
        sp, tr = (torch.from_numpy(a).cuda() for a in t.inputs[0])
        other = [torch.from_numpy(a).cuda() for a in t.inputs[1]]
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=t.stream):
            dp.dp_set_inputs(t.c, t.d, sp, tr, on_device=1)
            dp.dp_propagate(t.c, t.d, t.cfg)
        for _ in range(5):
            with torch.cuda.stream(t.stream):
                dp.dp_set_inputs(t.c, t.d, *t.inputs[0])
                dp.dp_propagate(t.c, t.d, t.cfg)
                sp.copy_(other[0])
                tr.copy_(other[1])
                g.replay()
                dp.dp_simulate(t.c, t.d, t.cfg)
            t.check(1, "after a replay with new inputs")
    finally:
        t.close()


@pytest.mark.parametrize("spec", SPECS)
def test_replayed_reads_come_before_the_simulation(dp, library_text, spec):  # noqa: F811
    t = Case(dp, spec, library_text)
    try:
        tg, on = (torch.zeros(t.info.n_nets, dtype=torch.int32, device="cuda") for _ in range(2))
        dp.dp_set_inputs(t.c, t.d, *t.inputs[0])
        dp.dp_propagate(t.c, t.d, t.cfg)
        dp.dp_simulate(t.c, t.d, t.cfg)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=t.stream):
            dp.dp_get_nets(t.c, t.d, toggles=tg, ones=on, on_device=1)
        now = 0
        for _ in range(4):
            with torch.cuda.stream(t.stream):
                dp.dp_set_inputs(t.c, t.d, *t.inputs[1 - now])
                dp.dp_propagate(t.c, t.d, t.cfg)
                g.replay()   # the counts of the simulation before
                dp.dp_simulate(t.c, t.d, t.cfg)
            t.stream.synchronize()
            for x, y in zip((tg, on), t.want[now]):
                np.testing.assert_array_equal(x.cpu().numpy().view(np.uint32), y)
            now = 1 - now
            t.check(now, "after the replay")
    finally:
        t.close()


@pytest.mark.parametrize("spec", SPECS)
def test_another_streams_capture_goes_on(dp, library_text, spec):  # noqa: F811
    """while another stream captures (torch's mode: global), the phases run on their own stream as before, and the
    capture stays whole"""
    t = Case(dp, spec, library_text)
    try:
        dp.dp_set_inputs(t.c, t.d, *t.inputs[0])
        dp.dp_propagate(t.c, t.d, t.cfg)
        dp.dp_simulate(t.c, t.d, t.cfg)   # whatever is made on first use
        x = torch.zeros(8, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            x.add_(1.0)
            dp.dp_propagate(t.c, t.d, t.cfg)
            dp.dp_simulate(t.c, t.d, t.cfg)
            x.add_(1.0)
        t.check(0, "beside a capture")
        g.replay()
        torch.cuda.synchronize()
        assert x.eq(2.0).all()
    finally:
        t.close()
