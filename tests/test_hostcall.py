"""The native argument marshalling rejects what it cannot pass on, before anything reaches CUDA."""
import pytest
import torch

from paper_2412_14468_b200 import binding as ha
from paper_2412_14468_b200 import build as ha_build


@pytest.fixture(scope="module", autouse=True)
def built():
    ha_build.build()


@pytest.mark.parametrize("bad", [None, 3, "x", torch.zeros(1, 8, 4, 128), torch.zeros(1, 8, 4, 128, dtype=torch.bfloat16)])
def test_keys_have_to_be_bf16_on_the_device(bad):
    with pytest.raises(TypeError):
        ha.ha_encode(None, 1, bad, torch.zeros(1, 8, 4, dtype=torch.int32))
    with pytest.raises(TypeError):
        ha.ha_dense_decode(ha.make_shape(1, 32, 8, 0.1), torch.zeros(1), bad, bad, torch.zeros(1), 4, torch.zeros(1), torch.zeros(1))


def test_shape_has_to_be_a_structure_and_numbers_numbers():
    t = torch.zeros(1, 8, 8, dtype=torch.int32)
    good = dict(q_codes=t, k_codes=t, seq_lens=t, k_per_seq=None, k_uniform=1, k_max=1, idx=t, count=t, stream=0)
    with pytest.raises(TypeError):
        ha.ha_score_topk_sum(object(), **good)
    with pytest.raises(TypeError):
        ha.ha_score_topk_sum(ha.make_shape(1, 32, 8, 0.1), **dict(good, k_max=1.5))
    with pytest.raises(ha.HashAttnError) as e:      # all arguments arrive: the C entry refuses the head counts
        ha.ha_score_topk_sum(ha.make_shape(1, 32, 5, 0.1), **good)
    assert e.value.status in (ha.HA_ERR_INVALID_ARG, ha.HA_ERR_UNSUPPORTED)


def test_host_step_wants_contiguous_host_buffers():
    t = torch.zeros(2, 2)
    with pytest.raises(TypeError):
        ha.SparseDecodeHostStep(ha.make_shape(1, 32, 8, 0.1), None, None, t.t(), t, t, t, t, t, t, None, 1, 1, 1, t, t, t, t, stream=0)


@pytest.mark.parametrize("change", [None, "torch", "python"])
def test_the_extension_is_rebuilt_for_another_torch_or_python(monkeypatch, change):
    built_again = []
    monkeypatch.setattr(ha_build, "_build_hostcall", lambda: built_again.append(True))
    if change == "torch":
        monkeypatch.setattr(torch, "__version__", torch.__version__ + ".other")
    elif change == "python":
        monkeypatch.setattr(ha_build.sys, "version", "3.99")
    ha_build.build()
    assert bool(built_again) == (change is not None)
