"""Waits of finite lists, whose CTAs run up to eight descriptors ahead of the
slowest one of their cluster."""
import numpy as np
import pytest

from gpu_util import host, need_gpu, to_dev
from paper_2310_01212_gb300 import lk, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_ready(native_built):
    return need_gpu()


def test_a_histogram_waits_for_a_slow_rank_0(torch_ready, oracle_lib):
    """Only rank 0 sums histograms; here seven times 512 MB, from host memory and
    in 152 clusters at once, some 2.7 s.  The other CTA reaches the histogram
    behind them at once and waits for rank 0 to clear its output."""
    torch = torch_ready
    C, n, apart = 152, 1 << 19, 4096                     # histograms each; clusters read 4 MB apart
    hp = torch.zeros((n + C * apart, 256), dtype=torch.int32, pin_memory=True)
    hp[::apart, 5] = 3
    x = synth.bytes_uniform(51, 0, 1 << 16)
    dx = to_dev(x)
    out = torch.full((C, 8, 256), -1, dtype=torch.int32, device="cuda")
    rows = []
    for c in range(C):
        rows += [(c, lk.LK_OP_COMBINE_HIST, n, hp.data_ptr() + c * apart * 1024, out[c, j].data_ptr()) for j in range(7)]
        rows.append((c, lk.LK_OP_HIST_U8, x.size, dx.data_ptr(), out[c, 7].data_ptr()))
    torch.cuda.current_stream().synchronize()
    lk.lk_run_finite([2] * C, [(op, m) for _, op, m, _, _ in rows], [c for c, *_ in rows], in0=[a for *_, a, _ in rows],
                     out=[o for *_, o in rows], threads_per_cta=64, ctas_per_sm=2)
    got = host(out).astype(np.int64)
    sums = np.zeros(256, np.int64)
    sums[5] = 3 * (n // apart)
    assert np.array_equal(got[:, :7], np.broadcast_to(sums, (C, 7, 256)))
    assert np.array_equal(got[:, 7], np.broadcast_to(oracle_lib.hist_u8(x), (C, 256)))
