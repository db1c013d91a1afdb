"""The last CTA to arrive combines a sum or a split histogram with one warp,
whose lanes all read what other CTAs wrote: every descriptor has other
partials (whole numbers, so the sums are exact), and the slots and the batch's
combine state are used again and again, so a stale word shows."""
import numpy as np
import pytest

from gpu_util import host, need_gpu
from paper_2310_01212_gb300 import lk

pytestmark = pytest.mark.gpu

COUNT = 400


@pytest.fixture(scope="module")
def rows(native_built):
    """Row i holds i + 1 everywhere (as float32) or i % 256 (as bytes)."""
    torch = need_gpu()
    n = 9728
    f = (torch.arange(COUNT, device="cuda", dtype=torch.float32)[:, None] + 1).repeat(1, n).contiguous()
    b = (torch.arange(COUNT, device="cuda") % 256).to(torch.uint8)[:, None].repeat(1, n).contiguous()
    return torch, n, f, b


def _check_sums(out, n):
    assert np.array_equal(host(out)[:, 0], np.float32(n) * np.arange(1, COUNT + 1, dtype=np.float32))


@pytest.mark.parametrize("threads", [256, 1024])
@pytest.mark.parametrize("sizes", [[152], [38] * 4])
@pytest.mark.parametrize("finite", [False, True])
def test_sums_back_to_back(rows, finite, sizes, threads):
    torch, n, f, _ = rows
    out = torch.full((COUNT, 4), float("nan"), device="cuda")
    torch.cuda.current_stream().synchronize()
    ins, outs = [f[i].data_ptr() for i in range(COUNT)], [out[i].data_ptr() for i in range(COUNT)]
    if finite:
        lk.lk_run_finite(sizes, [(lk.LK_OP_SUM_F32, n)] * COUNT, [i % len(sizes) for i in range(COUNT)], in0=ins,
                         out=outs, threads_per_cta=threads)
    else:
        with lk.lk_init(sizes, idle_lease_ns=5_000_000_000, threads_per_cta=threads) as c:
            hs = [lk.lk_submit(c, i % len(sizes), lk.LK_OP_SUM_F32, n, (ins[i],), outs[i]) for i in range(COUNT)]
            for h in hs:
                assert lk.lk_wait(c, h) == lk.LK_OK, lk.lk_device_error(c)
    _check_sums(out, n)


@pytest.mark.parametrize("threads", [64, 256, 1024])
def test_split_items_of_batches(rows, threads):
    torch, n, f, b = rows
    out = torch.full((COUNT, 4), float("nan"), device="cuda")
    bins = torch.full((COUNT, 256), -1, dtype=torch.int32, device="cuda")
    sums = lk.batch_items([(lk.LK_OP_SUM_F32, n, (f[i],), out[i], 8) for i in range(COUNT)])
    hists = [lk.batch_items([(lk.LK_OP_HIST_U8, n, (b[i],), bins[i], 5) for i in range(k, min(k + 200, COUNT))])
             for k in range(0, COUNT, 200)]
    torch.cuda.current_stream().synchronize()
    with lk.lk_init([152], idle_lease_ns=5_000_000_000, threads_per_cta=threads) as c:
        for _ in range(3):
            for items in [sums] + hists:
                assert lk.lk_wait(c, lk.lk_submit_batch(c, 0, items)) == lk.LK_OK, lk.lk_device_error(c)
    _check_sums(out, n)
    want = np.zeros((COUNT, 256), np.int64)
    want[np.arange(COUNT), np.arange(COUNT) % 256] = n
    assert np.array_equal(host(bins).astype(np.int64), want)
