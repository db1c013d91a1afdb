"""Tiles on the FFMA paths, bit for bit: every output is its 64 products in k
order with one fused multiply-add each, whichever path and split runs them
(the packed groups, the whole CTA on one tile, row blocks, other block
sizes)."""
import numpy as np
import pytest

from gpu_util import host, need_gpu, to_dev
from paper_2310_01212_gb300 import lk, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,per_sm,threads,flags", [(1, 1, 256, lk.LK_INIT_GEMM_FFMA), (3, 1, 256, lk.LK_INIT_GEMM_FFMA),
                                                    (1, 2, 256, 0), (3, 2, 256, 0), (3, 2, 64, 0), (3, 1, 64, 0),
                                                    (3, 1, 512, 0), (3, 1, 1024, 0)])
def test_bits(native_built, oracle_lib, S, per_sm, threads, flags):
    torch = need_gpu()
    cases = []
    for i, t in enumerate([1, 2, 3, 4, 5, 6, 7, 12, 17]):
        A = synth.normal_f32(81, 2 * i, t * 4096).reshape(t, 64, 64)
        B = synth.normal_f32(81, 2 * i + 1, t * 4096).reshape(t, 64, 64)
        cases.append((A, B, to_dev(A), to_dev(B), torch.full((t, 64, 64), float("nan"), device="cuda")))
    torch.cuda.current_stream().synchronize()
    with lk.lk_init([S], idle_lease_ns=5_000_000_000, ctas_per_sm=per_sm, threads_per_cta=threads, flags=flags) as c:
        hs = [lk.lk_submit(c, 0, lk.LK_OP_GEMM64_F32, A.shape[0], (dA, dB), dC) for A, B, dA, dB, dC in cases]
        for h in hs:
            assert lk.lk_wait(c, h) == lk.LK_OK, lk.lk_device_error(c)
    for A, B, _, _, dC in cases:
        assert np.array_equal(host(dC).view(np.uint32), oracle_lib.gemm64_fmaf(A, B).view(np.uint32)), A.shape
