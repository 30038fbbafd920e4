"""Which kernel takes a call, and what the host side does where a query of the runtime fails (no GPU: tests/fake_cudart.cpp)."""
import pytest

from paper_2412_14468_b200 import binding as ha
from tests._fake import BATCH, Fake


def test_a_failing_occupancy_query_leaves_no_error_behind(tmp_path):
    """The kernels that take the call instead are launched, and the call says so."""
    f = Fake(tmp_path)
    f.lib.fake_fail_queries(1)
    calls = [lambda: f.score_topk(64, 4, 8, 8000), lambda: f.score_topk(8, 4, 8, 140000), lambda: f.score_topk(20, 4, 8, 9000, page=16),
             lambda: f.step(1, 4, 8, 32768, 1024), lambda: f.step(4, 4, 8, 20000, 2000), lambda: f.step(64, 4, 8, 32768, 1024)]
    for i, call in enumerate(calls):
        assert call() == ha.HA_OK, i
        assert f.lib.cudaGetLastError() == 0, i
        kernels = [k for k, *_ in f.launches()]
        assert kernels and not {BATCH, "fused_step_kernel", "gather_cluster_kernel"} & set(kernels), kernels
