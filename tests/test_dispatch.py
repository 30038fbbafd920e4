"""Which kernel takes a call, and what the host side does where a query of the runtime fails (no GPU: tests/fake_cudart.cpp)."""
import pytest

from paper_2412_14468_b200 import binding as ha
from tests._fake import BATCH, RESIDENT, SEVERAL_UNITS_PER_CLUSTER, Fake


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


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return Fake(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("page", [0, 16])
@pytest.mark.parametrize("B,H,n,cs", SEVERAL_UNITS_PER_CLUSTER)
def test_the_call_order_tests_reach_clusters_of_several_units(fake, B, H, n, cs, page):
    assert fake.score_topk(B, 1, H, n, page=page, k_max=16) == ha.HA_OK
    (kernel, args, ctas, cluster, _), = fake.launches()
    assert kernel == BATCH and args == [1, cs, int(page > 0)] and cluster == cs and ctas <= RESIDENT[cs] * cs
