"""A server whose environment asks for the dataflow passes: batches on new inputs and on the reference inputs take
turns, and every result is the one of a server without the variable."""
import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_serve_gpu import dp  # noqa: F401

pytestmark = pytest.mark.gpu


def serve(dp, text, lib):  # noqa: F811
    srv = dp.dp_server_create(dp.server_config(max_batch=8))
    out = []
    try:
        d = dp.dp_server_add_design(srv, text, lib)
        for turn in range(8):   # new, reference, new, new, reference: tags of either parity under the reference's
            for i in range(3):
                sp, tr = (a[:, 0].copy() for a in netgen.scenario_inputs(60, 500 + 10 * turn + i, 1))
                ref = turn % 5 in (1, 4)
                power, g = np.zeros(1), np.zeros(60, np.float32)
                kw = {} if ref else dict(sp=sp, tr=tr)
                t = dp.dp_server_submit(srv, dp.request(d, power, want_grad=1, grad_sp=g, **kw))
                dp.dp_server_wait(srv, t, 60.0)
                out.append((power.copy(), g.copy()))
    finally:
        dp.dp_server_destroy(srv)
    return out


def test_reference_batches_between_new_ones(dp, monkeypatch):  # noqa: F811
    text, lib = netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4)), netgen.library_text()
    want = serve(dp, text, lib)
    monkeypatch.setenv("DP_BATCH_FLOW", "1")
    for i, (a, b) in enumerate(zip(serve(dp, text, lib), want)):
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x, y, err_msg=f"request {i}")
