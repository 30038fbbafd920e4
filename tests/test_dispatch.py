"""Which kernel takes a call, and what the host side does where a query of the runtime fails (no GPU: tests/fake_cudart.cpp)."""
import pytest

from paper_2412_14468_b200 import binding as ha
from tests._fake import BATCH, BATCH_CASES, NEXT_TO_BATCH_CASES, PER_HEAD_BATCH_CASES, RESIDENT, SEVERAL_UNITS_PER_CLUSTER, Fake, batches, budgets, ragged


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
    (kernel, args, ctas, cluster, *_), = fake.launches()
    assert kernel == BATCH and args == [1, cs, int(page > 0)] and cluster == cs and ctas <= RESIDENT[cs] * cs


@pytest.mark.parametrize("case", BATCH_CASES, ids=lambda c: f"{c[0]}-{c[1]}-{len(c[2])}x{max(c[2])}")
def test_cases_of_clusters_of_several_units(fake, case):
    """The GPU test of these calls reaches the cluster size, the number of batches and the staging that it is there for."""
    G, Hkv, lens, pages, cs, n_batches, staged = case
    for page in pages:
        assert fake.score_topk(len(lens), G, Hkv, max(lens), page=page, k_max=max(max(budgets(lens)) + 137, 1)) == ha.HA_OK
        (kernel, args, ctas, cluster, _, is_staged), = fake.launches()
        assert kernel == BATCH and args == [G, cs, int(page > 0)] and cluster == cs
        assert ctas == cs * min(RESIDENT[cs], len(lens) * Hkv)
        assert bool(is_staged) == (page > 0 and (page > 16 if staged is None else staged))
        assert batches(Hkv, lens, cs, ctas // cs, page, is_staged) == n_batches


@pytest.mark.parametrize("case", NEXT_TO_BATCH_CASES, ids=lambda c: f"{c[0]}-{c[1]}-{len(c[2])}x{max(c[2])}")
def test_cases_beside_clusters_of_several_units(fake, case):
    G, Hkv, lens, pages = case
    for page in pages:
        assert fake.score_topk(len(lens), G, Hkv, max(lens), page=page) == ha.HA_OK
        assert BATCH not in [k for k, *_ in fake.launches()], page


@pytest.mark.parametrize("B,Hkv,G,longest,cs", PER_HEAD_BATCH_CASES)
def test_cases_of_lists_per_query_head_on_clusters_of_several_units(fake, B, Hkv, G, longest, cs):
    assert fake.score_topk(B, G, Hkv, longest, page=16, per_head=True, k_max=max(budgets(ragged(B, longest)))) == ha.HA_OK
    (kernel, args, ctas, cluster, *_), = fake.launches()
    assert kernel == BATCH and args == [1, cs, 1] and cluster == cs and ctas == cs * min(RESIDENT[cs], B * Hkv * G)


@pytest.mark.parametrize("B,Hkv,n,per_head,longest_list", [(64, 8, 8192, False, 768), (64, 8, 8192, True, 768), (15, 8, 16000, True, 1024)])
def test_long_lists_stay_with_clusters_of_one_unit(fake, B, Hkv, n, per_head, longest_list):
    for k_max in (longest_list, longest_list + 1):
        assert fake.score_topk(B, 4, Hkv, n, page=16, per_head=per_head, k_max=k_max) == ha.HA_OK
    assert [k for k, *_ in fake.launches()] == [BATCH, "score_select_cluster_kernel"]


@pytest.mark.parametrize("page", [0, 16, 64])
@pytest.mark.parametrize("G", [1, 2, 4, 8])
def test_up_to_32768_tokens_the_kernel_does_not_depend_on_how_the_budget_is_given(fake, G, page):
    """Sequences of one length take the same kernel with one budget for all and with one budget each."""
    for B in (3, 16, 23, 28, 29, 37, 46, 47, 48, 58, 64, 74, 100, 128, 200):
        for n in (1200, 4000, 8000, 9000, 16000, 17000, 24000, 30000, 32768):
            for budgets in (True, False):
                assert fake.score_topk(B, G, 8, n, array=budgets, page=page) == ha.HA_OK
            one, other = fake.launches()
            assert one == other, (B, n)


@pytest.mark.parametrize("B,Hkv,G,n,cs", [(16, 8, 4, 2100, 4), (30, 8, 2, 9000, 2), (40, 4, 4, 2100, 4), (14, 8, 1, 30000, 4),
                                          (10, 8, 1, 30000, 8)])
def test_cases_of_clusters_that_are_launched_with_a_cap_on_ctas_per_sm(fake, B, Hkv, G, n, cs):
    """One-unit clusters with fewer than six CTAs per SM ask for the shared memory of a whole share of the SM."""
    assert fake.score_topk(B, G, Hkv, n) == ha.HA_OK
    (kernel, args, ctas, cluster, smem, _), = fake.launches()
    assert kernel == "score_select_cluster_kernel" and cluster == cs == args[1] and ctas == cs * B * Hkv
    assert smem > 30 * 1024 and 227 * 1024 // (smem + 1024) == -(-ctas // 148) < 6
