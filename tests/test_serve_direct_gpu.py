"""The server's transfers in one launch each (requests' buffers addressed by the device) against a copy per buffer: the
same bits for pinned, pageable and unaligned buffers, absent gradients and deltas, and a batch of one and of many."""
import os

import numpy as np
import pytest

from paper_2608_03778_gb300 import netgen
from tests.test_serve_gpu import dp  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def buffer(n, kind, value=None):
    """n floats: pageable, pinned, or a view one element into its allocation"""
    a = np.zeros(n + 1, np.float32)
    if kind == "pinned":
        a = torch.zeros(n + 1).pin_memory().numpy()
    a = a[1:] if kind == "unaligned" else a[:n]
    if value is not None:
        a[...] = value
    return a


def serve(dp, text, lib, jobs, copies, batch):  # noqa: F811
    if copies:
        os.environ["DP_SERVER_COPIES"] = "1"
    try:
        srv = dp.dp_server_create(dp.server_config(max_batch=batch))
    finally:
        os.environ.pop("DP_SERVER_COPIES", None)
    try:
        d = dp.dp_server_add_design(srv, text, lib)
        out = []
        for sp, tr, cells, caps, kind, want in jobs:
            power = np.zeros(1)
            g = [buffer(n, kind) if w else None for n, w in zip((sp.size, sp.size, 900), want)]
            keep = [buffer(a.size, kind, a) for a in (sp, tr)]
            kw = {} if cells is not None else dict(sp=keep[0], tr=keep[1])
            if cells is not None:
                kw = dict(cells=cells, pincap=buffer(caps.size, kind, caps))
            names = ("grad_sp", "grad_tr", "grad_pincap")
            if any(want):
                kw |= {"want_grad": 1} | {n: a for n, a in zip(names, g) if a is not None}
            out.append((dp.request(d, power, **kw), power, g, keep, kw))
        tickets = [dp.dp_server_submit(srv, o[0]) for o in out]
        for t in tickets:
            dp.dp_server_wait(srv, t, 60.0)
        return [[o[1].copy()] + [a.copy() for a in o[2] if a is not None] for o in out]
    finally:
        dp.dp_server_destroy(srv)


@pytest.mark.parametrize("n, batch", [(1, 1), (5, 4), (33, 16)])
def test_direct_transfers_give_the_same_bits(dp, n, batch):  # noqa: F811
    text, lib = netgen.netlist_text(netgen.NetlistSpec(900, 20, 40, 9, 16, 4)), netgen.library_text()
    rng = np.random.default_rng(n)
    jobs = []
    for i in range(n):
        sp, tr = (a[:, 0].copy() for a in netgen.scenario_inputs(60, 300 + i, 1))
        m = int(rng.integers(1, 1500))   # entries, with repeats: up to more than a row's threads
        delta = i % 3 == 2
        jobs.append((sp, tr, rng.integers(0, 900, m).astype(np.int32) if delta else None,
                     rng.choice(np.array([1.6, 3.2], np.float32), m) if delta else None,
                     ("pageable", "pinned", "unaligned")[i % 3 if not delta else i % 2],
                     [(1, 1, 1), (0, 0, 0), (1, 0, 0), (0, 1, 1)][i % 4]))
    a, b = (serve(dp, text, lib, jobs, copies, batch) for copies in (False, True))
    for i, (x, y) in enumerate(zip(a, b)):
        assert len(x) == len(y)
        for u, v in zip(x, y):
            np.testing.assert_array_equal(u, v, err_msg=f"request {i}")
        assert x[0][0] > 0
