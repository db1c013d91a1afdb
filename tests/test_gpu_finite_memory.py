"""A long finite list gives its host memory back when the call returns."""
import pytest

from gpu_util import need_gpu
from paper_2310_01212_gb300 import lk

pytestmark = pytest.mark.gpu


def _resident_mb():
    with open("/proc/self/status") as f:
        return next(int(line.split()[1]) for line in f if line.startswith("VmRSS")) >> 10


def test_a_long_list_leaves_no_host_memory_behind(native_built):
    need_gpu()
    lk.lk_run_finite([1] * 16, [(lk.LK_OP_NOP, 0)] * 16, list(range(16)))    # the kernels are loaded
    count = (1 << 18) - 1                     # one ring of 2^18 slots a cluster: 256 MB
    descs, clusters = [(lk.LK_OP_NOP, 0)] * count, [0] * count
    before = _resident_mb()
    ms, log = lk.lk_run_finite([1] * 16, descs, clusters, log_cap=64, exec_log_cap=4)
    assert ms > 0 and log[log["cluster"] == 0]["seq"].max() == count
    assert _resident_mb() - before < 64
