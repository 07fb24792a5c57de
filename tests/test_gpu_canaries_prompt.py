"""Guard bands (test_gpu_canaries.py) around the outputs of prompts of more than
256 tokens, in both forms of the down projection, and of 2 to 4 tokens of wide
layers that go on with the union phases."""
import pytest

from test_gpu_canaries import layer_case, run_guarded_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,T,d,E,rule,p", [("llama3_8b_batched", 257, 200, 40, "min_prefix", 0.7), ("llama3_8b_batched", 385, 264, 90, "topk", 60.0),
                                               ("gpt2m_gelu_bf16", 1031, 1000, 33, "min_prefix", 0.9),
                                               ("llama3_8b_batched", 3, 4104, 200, "min_prefix", 0.97),
                                               ("llama3_8b_batched", 4, 4096, 224, "topk", 16.0)])
def test_guarded(pp, name, T, d, E, rule, p):
    w, L = layer_case(name, T, d, E)
    run_guarded_layer(pp, w, L, T, p, rule)
