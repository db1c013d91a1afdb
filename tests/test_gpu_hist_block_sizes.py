"""Histograms at the block sizes whose warps do not divide the rings' memory
evenly (9 to 12 and 17 to 28 warps), and their neighbours: shares around the
small-share cut, a stage and a ring, in live contexts (the bounds-checking
build), finite lists and ordinary launches.  Counts are exact."""
import numpy as np
import pytest

from gpu_util import host, need_gpu, to_dev
from paper_2310_01212_gb300 import lk, synth

pytestmark = pytest.mark.gpu

THREADS = [288, 320, 384, 416, 544, 640, 704, 768, 896, 992]


@pytest.fixture(scope="module")
def torch_ready(native_built):
    return need_gpu()


def _cases(torch, threads, extra):
    warps = threads // 32
    stage = 32768 // -(-warps // 4) // 64 * 16            # bytes of one stage: whole 16-byte vectors
    total = 4 * stage * warps
    sizes = [16 * 1024 - 1, 16 * 1024, warps * stage - 16, warps * stage + 16, total - 16, total + 17,
             3 * total + 16 * 129 + 7] + extra
    cases = [(x, to_dev(x), torch.full((256,), -1, dtype=torch.int32, device="cuda"))
             for x in (synth.bytes_uniform(41, i, n) for i, n in enumerate(sizes))]
    torch.cuda.current_stream().synchronize()
    return cases


def _check(cases, oracle_lib):
    for x, _, out in cases:
        assert np.array_equal(host(out).astype(np.int64), oracle_lib.hist_u8(x)), x.size


@pytest.mark.parametrize("threads", THREADS)
def test_live(torch_ready, oracle_lib, threads):
    cases = _cases(torch_ready, threads, [])
    with lk.lk_init([1], bounds=True, idle_lease_ns=5_000_000_000, threads_per_cta=threads) as c:
        hs = [lk.lk_submit(c, 0, lk.LK_OP_HIST_U8, x.size, (dx,), out) for x, dx, out in cases]
        for h in hs:
            assert lk.lk_wait(c, h) == lk.LK_OK, lk.lk_device_error(c)
    _check(cases, oracle_lib)
    assert lk.lk_bounds_violations() == (0, 0)


@pytest.mark.parametrize("threads", THREADS)
def test_finite(torch_ready, oracle_lib, threads):
    cases = _cases(torch_ready, threads, [5_000_011])
    lk.lk_run_finite([3], [(lk.LK_OP_HIST_U8, x.size) for x, _, _ in cases], [0] * len(cases),
                     in0=[dx for _, dx, _ in cases], out=[out for *_, out in cases], threads_per_cta=threads)
    _check(cases, oracle_lib)


@pytest.mark.parametrize("threads", THREADS)
def test_ordinary_launch(torch_ready, oracle_lib, threads):
    cases = _cases(torch_ready, threads, [5_000_011])
    for x, dx, out in cases:
        rc = lk.lk_launch_noalloc(lk.LK_OP_HIST_U8, x.size, (dx,), out, ctas=5, threads=threads,
                                  stream=torch_ready.cuda.current_stream().cuda_stream)
        assert rc == lk.LK_OK
    _check(cases, oracle_lib)
