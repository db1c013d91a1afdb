"""Waits of finite lists, whose CTAs run up to eight descriptors ahead of the
slowest one of their cluster.  Only rank 0 sums histograms: read from host
memory by many clusters at once, they make it slow."""
import time

import numpy as np
import pytest

from gpu_util import host, need_gpu, to_dev
from paper_2310_01212_gb300 import lk, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_ready(native_built):
    return need_gpu()


APART = 4096          # histograms (4 MB) between where two clusters start to read


@pytest.fixture(scope="module")
def host_hists(torch_ready):
    hp = torch_ready.zeros(((1 << 20) + 256 * APART, 256), dtype=torch_ready.int32, pin_memory=True)
    hp[::APART, 5] = 3
    return hp


def test_a_histogram_waits_for_a_slow_rank_0(torch_ready, oracle_lib, host_hists):
    """Seven sums of 512 MB in each of 152 clusters, some 2.7 s.  The other CTA
    reaches the histogram behind them at once and waits for rank 0 to clear its
    output."""
    torch, hp = torch_ready, host_hists
    C, n = 152, 1 << 19
    x = synth.bytes_uniform(51, 0, 1 << 16)
    dx = to_dev(x)
    out = torch.full((C, 8, 256), -1, dtype=torch.int32, device="cuda")
    rows = []
    for c in range(C):
        rows += [(c, lk.LK_OP_COMBINE_HIST, n, hp.data_ptr() + c * APART * 1024, out[c, j].data_ptr()) for j in range(7)]
        rows.append((c, lk.LK_OP_HIST_U8, x.size, dx.data_ptr(), out[c, 7].data_ptr()))
    torch.cuda.current_stream().synchronize()
    lk.lk_run_finite([2] * C, [(op, m) for _, op, m, _, _ in rows], [c for c, *_ in rows], in0=[a for *_, a, _ in rows],
                     out=[o for *_, o in rows], threads_per_cta=64, ctas_per_sm=2)
    got = host(out).astype(np.int64)
    sums = np.zeros(256, np.int64)
    sums[5] = 3 * (n // APART)
    assert np.array_equal(got[:, :7], np.broadcast_to(sums, (C, 7, 256)))
    assert np.array_equal(got[:, 7], np.broadcast_to(oracle_lib.hist_u8(x), (C, 256)))


def test_a_cluster_stops_soon_after_one_of_its_ctas(torch_ready, host_hists):
    """One sum of 1 GB in each of 256 clusters, more than a second; the other CTA
    of the larger clusters waits for it eight descriptors on, and with no lease
    gives up after that second.  Rank 0 must not wait out a second of its own
    for it."""
    torch, hp = torch_ready, host_hists
    sizes, n = [2] * 48 + [1] * 208, 1 << 20
    out = torch.zeros((256, 256), dtype=torch.int32, device="cuda")
    torch.cuda.current_stream().synchronize()

    def go(nops, **kw):
        rows = [(c, lk.LK_OP_COMBINE_HIST, n, hp.data_ptr() + c * APART * 1024, out[c].data_ptr()) for c in range(256)]
        rows += [(c, lk.LK_OP_NOP, 0, 0, 0) for c in range(48) for _ in range(nops)]
        t = time.perf_counter()
        lk.lk_run_finite(sizes, [(op, m) for _, op, m, _, _ in rows], [c for c, *_ in rows],
                         in0=[a for *_, a, _ in rows], out=[o for *_, o in rows], threads_per_cta=64, ctas_per_sm=2, **kw)
        return time.perf_counter() - t

    alone = go(0)
    t = time.perf_counter()
    try:
        go(40, idle_lease_ns=1)
    except lk.LkError as e:
        took = time.perf_counter() - t
        assert e.code == lk.LK_EDEVICE
    else:
        pytest.skip("host memory is too fast here for rank 0 to be late")
    assert took < max(alone, go(0)) + 0.7
