"""Batches at the block sizes and residencies whose units run differently
(claimed ahead up to 256 threads, tiles on and off the tensor cores): mixed
items with tile counts around the claim-ahead size of each, whole and split,
on few CTAs, in the bounds-checking build."""
import numpy as np
import pytest

from gpu_util import gemm_ok, host, need_gpu, sum_ok, to_dev
from paper_2310_01212_gb300 import lk, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,per_sm,flags", [(64, 1, 0), (256, 1, 0), (256, 1, lk.LK_INIT_GEMM_FFMA), (256, 2, 0),
                                                  (64, 2, 0), (512, 1, 0), (768, 1, 0), (1024, 1, 0)])
def test_mixed_items(native_built, oracle_lib, threads, per_sm, flags):
    torch = need_gpu()
    rows, checks = [], []
    for i, tiles in enumerate([1, 2, 3, 4, 5, 15, 16, 17, 33]):
        parts = (1, 3)[i % 2]
        A = synth.normal_f32(71, 2 * i, tiles * 4096).reshape(tiles, 64, 64)
        B = synth.normal_f32(71, 2 * i + 1, tiles * 4096).reshape(tiles, 64, 64)
        x = synth.bytes_uniform(72, i, 8192 * tiles + 5)
        f = synth.normal_f32(73, i, 2048 * tiles + 3)
        oc = torch.full((tiles, 64, 64), float("nan"), device="cuda")
        oh = torch.full((256,), -1, dtype=torch.int32, device="cuda")
        os_ = torch.full((4,), float("nan"), device="cuda")
        rows += [(lk.LK_OP_GEMM64_F32, tiles, (to_dev(A), to_dev(B)), oc, parts),
                 (lk.LK_OP_HIST_U8, x.size, (to_dev(x),), oh, parts), (lk.LK_OP_SUM_F32, f.size, (to_dev(f),), os_, parts)]
        checks.append((A, B, x, f, oc, oh, os_))
    items = lk.batch_items(rows)
    torch.cuda.current_stream().synchronize()
    with lk.lk_init([5], bounds=True, idle_lease_ns=5_000_000_000, threads_per_cta=threads, ctas_per_sm=per_sm,
                    flags=flags) as c:
        for _ in range(2):
            assert lk.lk_wait(c, lk.lk_submit_batch(c, 0, items)) == lk.LK_OK, lk.lk_device_error(c)
    for A, B, x, f, oc, oh, os_ in checks:
        assert gemm_ok(host(oc), A, B, oracle_lib), A.shape
        assert np.array_equal(host(oh).astype(np.int64), oracle_lib.hist_u8(x)), x.size
        assert sum_ok(host(os_)[0], f, oracle_lib), f.size
    assert lk.lk_bounds_violations() == (0, 0)
