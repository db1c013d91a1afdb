"""The histogram's counter table and per-warp rings, and the tensor-core GEMM's
stages and operand buffers, at the sizes where they can go wrong: around the
small-share cut, one granule more or less than a stage or a ring, every number
of rings before and after the table (the block size sets it), and tile counts
around the wrap of the stages and buffers.  The bounds-checking build runs
them, so every region is checked too.  Histograms are exact; GEMM elements
stay within 1e-4 sum|a b| of binary64.

Also the histogram's clearing of its output, which waits only for earlier
descriptors that touch it: other writers of the same buffer, neighbours that
end where it starts, and more than a relay ring of them in flight."""
import numpy as np
import pytest

from gpu_util import gemm_ok, host, need_gpu, sum_ok, to_dev
from paper_2310_01212_gb300 import lk, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_ready(native_built):
    return need_gpu()


@pytest.mark.parametrize("threads", [64, 96, 160, 256, 1024])
def test_hist_share_edges(torch_ready, oracle_lib, threads):
    torch = torch_ready
    ring = (32768 // -(-(threads // 32) // 4)) // 64 * 64      # bytes of one warp's ring
    total = ring * (threads // 32)
    sizes = [16 * 1024 - 16, 16 * 1024 - 1, 16 * 1024, 16 * 1024 + 1, total // 4 + 16, total - 16, total + 17,
             3 * total + 16 * 129 + 7]
    cases = [(x, to_dev(x), torch.full((256,), -1, dtype=torch.int32, device="cuda"))
             for x in (synth.bytes_uniform(31, i, n) for i, n in enumerate(sizes))]
    torch.cuda.current_stream().synchronize()
    with lk.lk_init([1], bounds=True, idle_lease_ns=5_000_000_000, threads_per_cta=threads) as c:
        hs = [lk.lk_submit(c, 0, lk.LK_OP_HIST_U8, x.size, (dx,), out) for x, dx, out in cases]
        for h in hs:
            assert lk.lk_wait(c, h) == lk.LK_OK, lk.lk_device_error(c)
    for x, _, out in cases:
        assert np.array_equal(host(out).astype(np.int64), oracle_lib.hist_u8(x)), x.size
    assert lk.lk_bounds_violations() == (0, 0)


# the tensor cores (one CTA per SM), the packed FFMA path, and it with two CTAs per SM
@pytest.mark.parametrize("S,per_sm,flags", [(1, 1, 0), (2, 1, 0), (1, 1, lk.LK_INIT_GEMM_FFMA), (2, 1, lk.LK_INIT_GEMM_FFMA),
                                            (1, 2, 0), (2, 2, 0)])
def test_gemm_tile_counts(torch_ready, oracle_lib, S, per_sm, flags):
    """Every number of tiles around the wrap of the stages, buffers and groups.
    The k-order check allows one element in a thousand: binary64 rounds the sum
    once before float32 does, which differs from one rounding for 2^-29 of them
    a step at most."""
    torch = torch_ready
    cases = []
    for i, t in enumerate(list(range(1, 11)) + [17]):
        A = synth.normal_f32(32, 2 * i, t * 4096).reshape(t, 64, 64)
        B = synth.normal_f32(32, 2 * i + 1, t * 4096).reshape(t, 64, 64)
        cases.append((A, B, to_dev(A), to_dev(B), torch.full((t, 64, 64), float("nan"), device="cuda")))
    torch.cuda.current_stream().synchronize()
    with lk.lk_init([S], bounds=True, idle_lease_ns=5_000_000_000, ctas_per_sm=per_sm, flags=flags) as c:
        hs = [lk.lk_submit(c, 0, lk.LK_OP_GEMM64_F32, A.shape[0], (dA, dB), dC) for A, B, dA, dB, dC in cases]
        for h in hs:
            assert lk.lk_wait(c, h) == lk.LK_OK, lk.lk_device_error(c)
    for A, B, _, _, dC in cases:
        assert gemm_ok(host(dC), A, B, oracle_lib), A.shape
        if (flags or per_sm == 2) and A.shape[0] >= S:   # fused multiply-adds in k order, bit for bit
            want = np.zeros(A.shape, np.float64)
            for k in range(64):   # a product of two floats is exact in binary64; its sum with a float rounds once there
                want = (A[:, :, k:k + 1].astype(np.float64) * B[:, k:k + 1, :].astype(np.float64)
                        + want).astype(np.float32).astype(np.float64)
            assert np.mean(host(dC) != want.astype(np.float32)) < 1e-3, A.shape   # double rounding, rarely
    assert lk.lk_bounds_violations() == (0, 0)


@pytest.mark.parametrize("finite", [False, True])
@pytest.mark.parametrize("per_sm", [1, 2])
def test_hist_clear_after_earlier_writers(torch_ready, oracle_lib, finite, per_sm):
    torch = torch_ready
    S, rounds = 9, 12
    xs = [synth.bytes_uniform(33, i, 200_000 + 977 * i) for i in range(rounds)]
    a = synth.int32_uniform(33, 99, 1024, -(1 << 20), 1 << 20)
    dxs, da = [to_dev(x) for x in xs], to_dev(a)
    buf = torch.zeros(1024, dtype=torch.int32, device="cuda")       # histograms go to words 256..511
    apart = torch.full((rounds, 256), -1, dtype=torch.int32, device="cuda")
    rows = []
    for i in range(rounds):
        rows.append((lk.LK_OP_ADD_I32, 512, (da, da), buf.data_ptr()))                    # covers the output
        rows.append((lk.LK_OP_HIST_U8, xs[i].size, (dxs[i],), buf.data_ptr() + 1024))
        rows.append((lk.LK_OP_COPY_I32, 256, (da,), buf.data_ptr()))                      # ends where it starts
        rows.append((lk.LK_OP_HIST_U8, xs[i].size, (dxs[i],), apart[i]))
    torch.cuda.current_stream().synchronize()
    if finite:
        lk.lk_run_finite([S], [(op, n) for op, n, _, _ in rows], [0] * len(rows), in0=[ins[0] for _, _, ins, _ in rows],
                         in1=[ins[1] if len(ins) > 1 else None for _, _, ins, _ in rows], out=[o for *_, o in rows],
                         ctas_per_sm=per_sm)
    else:
        with lk.lk_init([S], idle_lease_ns=5_000_000_000, ctas_per_sm=per_sm) as c:
            hs = [lk.lk_submit(c, 0, op, n, ins, out) for op, n, ins, out in rows]
            for h in hs:
                assert lk.lk_wait(c, h) == lk.LK_OK, lk.lk_device_error(c)
    assert np.array_equal(host(buf)[256:512].astype(np.int64), oracle_lib.hist_u8(xs[-1]))
    for i in range(rounds):
        assert np.array_equal(host(apart)[i].astype(np.int64), oracle_lib.hist_u8(xs[i])), i


def test_batch_units_around_the_claim_ahead_size(torch_ready, oracle_lib):
    """Units just below and above the size up to which a CTA claims its next
    unit beside the current one, split and whole, on few CTAs (many units
    each), in the bounds-checking build."""
    torch = torch_ready
    k = 512 * 1024
    rows, checks = [], []
    sizes = [16, 4096 + 3, k - 16, k, k + 16, 2 * k + 7]
    for rep in range(3):
        for i, nb in enumerate(sizes):
            x = synth.bytes_uniform(34, 10 * rep + i, nb)
            f = synth.normal_f32(35, 10 * rep + i, nb // 4)
            a = synth.int32_uniform(36, 10 * rep + i, nb // 8, -(1 << 20), 1 << 20)
            parts = (1, 2, 5)[rep]
            oh = torch.full((256,), -1, dtype=torch.int32, device="cuda")
            os_ = torch.full((4,), float("nan"), device="cuda")
            oa = torch.full((a.size,), -1, dtype=torch.int32, device="cuda")
            da = to_dev(a)
            rows += [(lk.LK_OP_HIST_U8, x.size, (to_dev(x),), oh, parts), (lk.LK_OP_SUM_F32, f.size, (to_dev(f),), os_, parts),
                     (lk.LK_OP_ADD_I32, a.size, (da, da), oa, parts)]
            checks += [(oh, x), (os_, f), (oa, a)]
    items = lk.batch_items(rows)
    torch.cuda.current_stream().synchronize()
    with lk.lk_init([5], bounds=True, idle_lease_ns=5_000_000_000) as c:
        for _ in range(3):                                   # the combine state returns to zero
            h = lk.lk_submit_batch(c, 0, items)
            assert lk.lk_wait(c, h) == lk.LK_OK, lk.lk_device_error(c)
    for out, ref in checks:
        if ref.dtype == np.uint8:
            assert np.array_equal(host(out).astype(np.int64), oracle_lib.hist_u8(ref)), ref.size
        elif ref.dtype == np.float32:
            assert sum_ok(host(out)[0], ref, oracle_lib), ref.size
        else:
            assert np.array_equal(host(out), oracle_lib.add_i32(ref, ref)), ref.size
    assert lk.lk_bounds_violations() == (0, 0)


@pytest.mark.parametrize("graph", [False, True])
def test_noalloc_launches_follow_one_another(torch_ready, oracle_lib, graph):
    """Dependent launches back to back on one stream, each reading what the one
    before wrote, with every body and a launch of another kernel between them;
    as they are and replayed from a captured graph."""
    torch = torch_ready
    n = 300_007
    a = synth.int32_uniform(37, 0, n, 0, 255)
    da = to_dev(a)
    y, z, w = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3))
    h = torch.zeros(256, dtype=torch.int32, device="cuda")
    s = torch.zeros(4, device="cuda")
    f = torch.zeros(n, device="cuda")

    def go(op, m, ins, out, ctas):
        rc = lk.lk_launch_noalloc(op, m, ins, out, ctas=ctas, stream=torch.cuda.current_stream().cuda_stream)
        assert rc == lk.LK_OK, rc

    def chain():
        go(lk.LK_OP_COPY_I32, n, (da,), y, 152)
        for _ in range(4):
            go(lk.LK_OP_ADD_I32, n, (y, da), z, 37)
            go(lk.LK_OP_NOP, 0, (), None, 4)
            go(lk.LK_OP_COPY_I32, n, (z,), y, 300)
        go(lk.LK_OP_HIST_U8, 4 * n, (y,), h, 152)
        torch.add(y, 1, out=w)
        f.copy_(w)
        go(lk.LK_OP_SUM_F32, n, (f,), s, 152)
        go(lk.LK_OP_COPY_I32, n, (w,), z, 19)

    go(lk.LK_OP_NOP, 0, (), None, 1)          # the scratch is set up before any capture
    if graph:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            chain()
        torch.cuda.current_stream().wait_stream(side)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            chain()
        for _ in range(3):
            z.zero_()
            g.replay()
    else:
        for _ in range(20):
            chain()
    want = 5 * a
    assert np.array_equal(host(y), want)
    assert np.array_equal(host(z), want + 1)
    assert np.array_equal(host(h).astype(np.int64), oracle_lib.hist_u8(want.astype("<i4").view(np.uint8)))
    assert float(host(s)[0]) == pytest.approx(float((want + 1).sum()), rel=1e-4)
