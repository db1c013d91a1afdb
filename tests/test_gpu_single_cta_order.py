"""A cluster of one CTA runs its work strictly in order: what a descriptor
wrote, the next one may read or overwrite."""
import numpy as np
import pytest

from gpu_util import gemm_ok, host, need_gpu, to_dev
from paper_2310_01212_gb300 import lk, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_ready(native_built):
    return need_gpu()


@pytest.mark.parametrize("per_sm,threads", [(1, 64), (1, 256), (2, 256), (1, 512)])
@pytest.mark.parametrize("finite", [False, True])
def test_a_sum_precedes_the_next_descriptor(torch_ready, finite, per_sm, threads):
    """Sums into one word, each copied out by the next descriptor; and sums
    whose word the next descriptor overwrites."""
    torch = torch_ready
    rounds, n = 300, 20_004
    x = (torch.arange(rounds, device="cuda", dtype=torch.float32)[:, None] + 1).repeat(1, n).contiguous()
    word = torch.zeros(4, device="cuda")                                  # read by the copy after it
    seen = torch.full((rounds, 4), float("nan"), device="cuda")
    over = torch.full((rounds, 4), float("nan"), device="cuda")           # overwritten by the copy after it
    mark = torch.tensor([7, 8, 9, 10], dtype=torch.int32, device="cuda")
    rows = []
    for i in range(rounds):
        rows.append((lk.LK_OP_SUM_F32, n, x[i], word))
        rows.append((lk.LK_OP_COPY_I32, 4, word, seen[i]))
        rows.append((lk.LK_OP_SUM_F32, n, x[i], over[i]))
        rows.append((lk.LK_OP_COPY_I32, 4, mark, over[i]))
    ptr = [(op, m, a.data_ptr(), o.data_ptr()) for op, m, a, o in rows]
    torch.cuda.current_stream().synchronize()
    if finite:
        lk.lk_run_finite([1], [(op, m) for op, m, *_ in ptr], [0] * len(ptr), in0=[a for *_, a, _ in ptr],
                         out=[o for *_, o in ptr], ctas_per_sm=per_sm, threads_per_cta=threads)
    else:
        with lk.lk_init([1], idle_lease_ns=5_000_000_000, ctas_per_sm=per_sm, threads_per_cta=threads,
                        ring_depth=2048) as c:
            hs = [lk.lk_submit(c, 0, op, m, (a,), o) for op, m, a, o in ptr]
            assert all(h is not None for h in hs)
            assert lk.lk_wait(c, hs[-1]) == lk.LK_OK, lk.lk_device_error(c)
    assert np.array_equal(host(seen)[:, 0], np.float32(n) * np.arange(1, rounds + 1, dtype=np.float32))
    assert np.array_equal(host(over).view(np.int32), np.tile(np.array([7, 8, 9, 10], np.int32), (rounds, 1)))


@pytest.mark.parametrize("per_sm,threads", [(1, 64), (1, 256), (2, 256), (1, 1024)])
def test_a_batch_keeps_the_callers_order(torch_ready, per_sm, threads):
    """A small item, then a larger one that reads what it wrote, and a small
    one, then a larger one into the same place."""
    torch = torch_ready
    rounds, n = 40, 1000
    x = torch.arange(rounds * n, device="cuda", dtype=torch.int32).view(rounds, n)
    f = (torch.arange(rounds, device="cuda", dtype=torch.float32)[:, None] + 1).repeat(1, n).contiguous()
    y = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    z = torch.full((rounds, n), -1, dtype=torch.int32, device="cuda")
    w = torch.full((rounds, 4), float("nan"), device="cuda")
    rows = []
    for i in range(rounds):
        rows.append((lk.LK_OP_COPY_I32, n, (x[i],), y))
        rows.append((lk.LK_OP_ADD_I32, n, (x[i], y), z[i]))
        rows.append((lk.LK_OP_COPY_I32, 4, (x[i],), w[i]))
        rows.append((lk.LK_OP_SUM_F32, n, (f[i],), w[i]))
    items = lk.batch_items(rows)
    torch.cuda.current_stream().synchronize()
    with lk.lk_init([1], idle_lease_ns=5_000_000_000, ctas_per_sm=per_sm, threads_per_cta=threads) as c:
        assert lk.lk_wait(c, lk.lk_submit_batch(c, 0, items)) == lk.LK_OK, lk.lk_device_error(c)
    assert np.array_equal(host(z), 2 * host(x))
    assert np.array_equal(host(w)[:, 0], np.float32(n) * np.arange(1, rounds + 1, dtype=np.float32))


@pytest.mark.parametrize("per_sm,threads,flags", [(1, 256, 0), (1, 256, lk.LK_INIT_GEMM_FFMA), (2, 256, 0), (1, 512, 0)])
@pytest.mark.parametrize("finite", [False, True])
def test_gemm_reads_what_the_descriptor_before_wrote(torch_ready, oracle_lib, finite, per_sm, threads, flags):
    """Tiles that an add stored with ordinary writes, read by bulk copies."""
    torch = torch_ready
    rounds, tiles = 40, 3
    A = synth.normal_f32(61, 0, rounds * tiles * 4096).reshape(rounds, tiles, 64, 64)
    B = synth.normal_f32(61, 1, tiles * 4096).reshape(tiles, 64, 64)
    dA, dB = to_dev(A), to_dev(B)
    zero = torch.zeros((tiles, 64, 64), dtype=torch.int32, device="cuda")
    buf = torch.full((tiles, 64, 64), float("nan"), device="cuda")
    C = torch.full((rounds, tiles, 64, 64), float("nan"), device="cuda")
    rows = []
    for i in range(rounds):
        rows.append((lk.LK_OP_ADD_I32, tiles * 4096, dA[i].data_ptr(), zero.data_ptr(), buf.data_ptr()))   # the same bits
        rows.append((lk.LK_OP_GEMM64_F32, tiles, buf.data_ptr(), dB.data_ptr(), C[i].data_ptr()))
    torch.cuda.current_stream().synchronize()
    if finite:
        lk.lk_run_finite([1], [r[:2] for r in rows], [0] * len(rows), in0=[r[2] for r in rows], in1=[r[3] for r in rows],
                         out=[r[4] for r in rows], ctas_per_sm=per_sm, threads_per_cta=threads, flags=flags)
    else:
        with lk.lk_init([1], idle_lease_ns=5_000_000_000, ctas_per_sm=per_sm, threads_per_cta=threads, flags=flags) as c:
            hs = [lk.lk_submit(c, 0, op, m, (a, b), o) for op, m, a, b, o in rows]
            assert lk.lk_wait(c, hs[-1]) == lk.LK_OK, lk.lk_device_error(c)
    got = host(C)
    for i in range(rounds):
        assert gemm_ok(got[i], A[i], B, oracle_lib), i
