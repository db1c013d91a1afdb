"""lk_serve's device queue on a context whose clusters still run descriptors
posted before (the host runtime over the fake device): the queue's state is
cleared at once, by a cluster with nothing to run or by copies, and nothing
that writes the arena stays behind when the call returns."""
import os
import time

import numpy as np
import pytest

from paper_2310_01212_gb300 import lk


@pytest.fixture
def stall(native_built):
    """Every descriptor of the fake device takes 0.2 s."""
    saved = os.environ.get("LK_FAKE_STALL_US")
    os.environ["LK_FAKE_STALL_US"] = "200000"
    yield 0.2
    if saved is None:
        os.environ.pop("LK_FAKE_STALL_US")
    else:
        os.environ["LK_FAKE_STALL_US"] = saved


def _arena():
    n = lk.lk_serve_queue_state_bytes(64) + (1 << 20)
    buf = np.full(n + 256, 0x5A, dtype=np.uint8)
    return buf, (buf.ctypes.data + 255) // 256 * 256, n


def _serve(c, count, timeout_s):
    buf, base, n = _arena()
    reqs = np.zeros(count, dtype=lk.REQUEST_DTYPE)
    reqs["op"], reqs["n"], reqs["in0"], reqs["out"] = lk.LK_OP_COPY_I32, 16, 0x10000, 0x10000
    rc, res = lk.lk_serve(c, reqs, n_producers=1, budget_bytes=1 << 30, arena=base, arena_bytes=n,
                          timeout_ns=int(timeout_s * 1e9), mode=lk.LK_SERVE_QUEUE, max_inflight=64)
    return rc, res, buf


def _busy(c, cluster, descriptors):
    return [lk.lk_submit(c, cluster, lk.LK_OP_NOP, 0) for _ in range(descriptors)]


def test_an_idle_cluster_clears_and_serves(stall):
    """Cluster 0 is busy for three seconds: cluster 1 serves within the timeout."""
    with lk.lk_init([1, 1], fake=True) as c:
        hs = _busy(c, 0, 15)
        rc, res, _ = _serve(c, 1, 2.5)
        assert rc == lk.LK_OK and res["status"][0] == lk.LK_OK
        assert res["t_complete_ns"][0] < 2.5e9
        for h in hs:
            assert lk.lk_wait(c, h) == lk.LK_OK


@pytest.mark.parametrize("sizes", [(2,), (1, 1)])
def test_every_cluster_busy(stall, sizes):
    """The call waits for the serving descriptors behind the earlier ones; a
    short timeout does not leave a clear behind."""
    with lk.lk_init(list(sizes), fake=True) as c:
        for k in range(len(sizes)):
            _busy(c, k, 4)
        rc, _, buf = _serve(c, 0, 0.1)
        assert rc == lk.LK_OK
        buf[:] = 0xA5                        # the arena is the caller's again
        assert lk.lk_sync(c) == lk.LK_OK
        time.sleep(2 * stall)
        assert np.all(buf == 0xA5)
