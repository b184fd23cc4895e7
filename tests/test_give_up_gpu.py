"""Passes without level barriers in which a wait gave up: what they leave behind is not taken for the next pass's own, in
direct calls and in replayed graphs, which no host code precedes.  The netlist is a chain that takes milliseconds, and two
wide levels behind it whose warps wait all that time; the error word is set before the pass, so those waits give up."""
import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_batch_gpu import dp, run_batch  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LIB = "cell INV ZN 0.6 !A\nseq DFF D Q 0.8\n"
CHAIN, A, B = 2500, 64, 96
MORE = {"small": 0, "cluster": 5000}   # cells of three more levels beside the chain's first: what takes the cluster


def chain_text(more):
    """B's cells 64 to 95 (a warp with nothing to wait for) read A's cells 32 to 63 (a warp that waits for the chain)"""
    first = 1 + CHAIN + A + B
    n = first + 3 * more
    lines = [f"net n{i} 1.0" for i in range(n)] + ["input n0"]
    lines += [f"cell c{i} INV A=n{i} ZN=n{i + 1}" for i in range(CHAIN)]
    lines += [f"cell a{i} INV A=n{CHAIN} ZN=n{CHAIN + 1 + i}" for i in range(A)]
    lines += [f"cell b{i} INV A=n{CHAIN + 1 + (i - 32) % A} ZN=n{CHAIN + 1 + A + i}" for i in range(B)]
    lines += [f"cell m{i} INV A=n{0 if i < more else first + i - more} ZN=n{first + i}" for i in range(3 * more)]
    return "\n".join(lines) + "\n"


@pytest.fixture()
def make(dp):  # noqa: F811
    made = []

    def load(size):
        st = torch.cuda.Stream()
        c = dp.dp_create(0, st.cuda_stream)
        made.append((c, dp.dp_design_load(c, chain_text(MORE[size]), LIB)))
        return *made[-1], st, dp.dp_design_info(made[-1][1])

    yield load
    for c, d in made:
        dp.dp_design_free(d)
        dp.dp_destroy(c)


def gave_up(dp, c):  # noqa: F811
    with pytest.raises(dp.DPError) as e:
        dp.dp_sync(c)
    assert "DP_ETIMEOUT" in str(e.value)


@pytest.mark.parametrize("broken", ["dataflow", "cluster"])
def test_replayed_pass_after_one_that_gave_up(dp, make, broken):  # noqa: F811
    """broken: which pass gives up, the one over the whole grid or the cluster's; the next is one over the whole grid"""
    c, d, st, info = make("cluster")
    assert info.cluster_threads > 0
    tr = np.full(1, 0.25, np.float32)
    cfg, other = dp.config(schedule=3, grad_mode=0, tr_mode=1), dp.config(schedule=0, grad_mode=0, tr_mode=1)
    inputs = [np.float32(x) for x in (0.1, 0.3, 0.45)]
    want = []
    for x in inputs:
        dp.dp_set_inputs(c, d, np.full(1, x, np.float32), tr)
        dp.dp_propagate(c, d, other)
        want.append(np.zeros(info.n_nets, np.float32))
        dp.dp_get_nets(c, d, want[-1])
    sp, trd, out = torch.zeros(1, device="cuda"), torch.from_numpy(tr).cuda(), torch.zeros(info.n_nets, device="cuda")
    torch.cuda.synchronize()
    graphs = {}
    for name, cf in (("dataflow", cfg), ("cluster", other)):
        graphs[name] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graphs[name], stream=st):
            dp.dp_set_inputs(c, d, sp, trd, on_device=1)
            dp.dp_propagate(c, d, cf)
            dp.dp_get_nets(c, d, out, on_device=1)

    def replay(name, k):
        with torch.cuda.stream(st):
            sp.fill_(float(inputs[k]))
            graphs[name].replay()

    for _ in range(2):   # a broken pass of either parity
        replay("dataflow", 0)
        dp.dp_sync(c)
        np.testing.assert_array_equal(out.cpu().numpy(), want[0])
        for _ in range(2):
            dp.dp_selftest_give_up(c)
            replay(broken, 1)
            gave_up(dp, c)
            assert (out.cpu().numpy() != want[1]).any()   # it did not finish
            replay("dataflow", 2)
            dp.dp_sync(c)
            np.testing.assert_array_equal(out.cpu().numpy(), want[2])
        # two in a row, the word still set for the second
        dp.dp_selftest_give_up(c)
        replay(broken, 1)
        replay("dataflow", 1)
        gave_up(dp, c)
        for k in (2, 1):
            replay("dataflow", k)
            dp.dp_sync(c)
            np.testing.assert_array_equal(out.cpu().numpy(), want[k])
        replay("dataflow", 0)


@pytest.mark.parametrize("when", ["forward", "reverse"])
@pytest.mark.parametrize("tr_mode", [1, 2])
@pytest.mark.parametrize("v", [1, 2])
def test_batched_pass_after_one_that_gave_up(dp, make, monkeypatch, when, tr_mode, v):  # noqa: F811
    c, d, st, info = make("small")
    cfg = dp.config(grad_mode=0, tr_mode=tr_mode)
    data = [netgen.scenario_inputs(1, 900 + k, 34) for k in range(3)]
    with monkeypatch.context() as m:
        m.setenv("DP_BATCH_SHAPE", "32,4")
        want = [run_batch(dp, c, d, *x, cfg) for x in data]
    monkeypatch.setenv("DP_BATCH_FLOW", str(v))
    g = np.zeros((1, 34), np.float32)
    for k in (0, 1, 2, 1):
        got = run_batch(dp, c, d, *data[k], cfg)
        for key in want[k]:
            np.testing.assert_array_equal(got[key], want[k][key], err_msg=key)
        dp.dp_set_inputs_batch(c, d, *(np.ascontiguousarray(a) for a in data[k - 1]), 34)
        if when == "forward":
            dp.dp_selftest_give_up(c)
        dp.dp_propagate(c, d, cfg)
        if when == "reverse":
            dp.dp_selftest_give_up(c)
        with pytest.raises(dp.DPError):
            dp.dp_backward(c, d, cfg, g)
        if tr_mode != 2:   # (a chain has the same lag-one gradients for all inputs)
            assert (g != want[k - 1]["grad_sp_in"]).any()   # the reverse pass did not finish
