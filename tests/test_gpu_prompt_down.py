"""The two forms of the prompt path's down projection, around the line between
them (48 tokens a work item, and half as many items as SMs) and past it on both
sides at any length: few and full items, items of one and two per expert, few
experts, and rows past the row buffer in either form."""
import pytest

from test_gpu_parity import layer_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["llama3_8b_batched", "gpt2m_gelu_bf16"])
@pytest.mark.parametrize("E,T,k", [(160, 300, 25), (160, 300, 26), (75, 300, 20), (77, 300, 20), (76, 260, 76), (160, 1500, 1),
                                   (12, 1100, 12), (9, 1900, 3), (256, 257, 256), (100, 1100, 100)])
def test_down_forms(pp, name, E, T, k):
    layer_parity(pp, name, T, float(k), "topk", d=264, E=E)
