"""The layer with at most 64 rows per expert, whose forward-shaped products run with the weights' columns as the rows of the MMA: at
and beside 32 and 64 tokens (and at 128), widths that end inside a tile, several tiles per CTA, biases, empty slots.  Against the oracle."""
import pytest
import torch

from paper_2202_09368_b200 import inputs as IN

from _parity import run_and_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,d,dff,E,router,gelu,bias", [
    (1, 64, 128, 4, "expert", "erf", False), (31, 72, 264, 4, "expert", "erf", True), (32, 136, 1032, 40, "expert", "tanh", False),
    (33, 64, 136, 8, "expert", "erf", True), (64, 72, 520, 40, "expert", "erf", False), (65, 128, 264, 4, "expert", "tanh", True),
    (128, 64, 392, 48, "expert", "erf", False), (96, 64, 264, 8, "token", "erf", True), (16, 8, 8, 16, "expert", "erf", False)])
def test_layer_with_few_rows_per_expert(k, d, dff, E, router, gelu, bias):
    n = k * E
    li = IN.make_layer_inputs(n, d, dff, E, torch.bfloat16, seed=k, expert_skew=1.0 if router == "token" else 0.0)
    biases = (IN.normal_tensor((E, dff), 0.5, k, IN.TID_AUX, torch.bfloat16), IN.normal_tensor((E, d), 0.5, k + 1, IN.TID_AUX, torch.bfloat16)) if bias else None
    run_and_check(n, d, dff, E, 1.0, torch.bfloat16, li, gelu=gelu, router=router, biases=biases)
