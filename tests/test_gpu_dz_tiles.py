"""The layer at sizes where the tiles of dZ = (dX_e . W2) * GeLU'(Z) meet their edges: many tiles per CTA pair with a last column
tile of eight columns, rows that end inside a warp's share, one tile per pair, single CTAs, tiles of empty slots that are
passed over.  Against the oracle, like every parity case."""
import pytest
import torch

from paper_2202_09368_b200 import inputs as IN

from _parity import run_and_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,dff,E,c,router,gelu", [(6000, 64, 1032, 40, 2.0, "expert", "erf"), (2600, 72, 520, 40, 2.0, "expert", "tanh"),
                                                     (512, 128, 264, 4, 2.0, "expert", "erf"), (970, 64, 392, 20, 2.0, "expert", "erf"),
                                                     (3000, 64, 648, 24, 3.0, "token", "erf")])
def test_layer_at_the_edges_of_the_dz_tiles(n, d, dff, E, c, router, gelu):
    li = IN.make_layer_inputs(n, d, dff, E, torch.bfloat16, seed=n, expert_skew=1.0 if router == "token" else 0.0)
    run_and_check(n, d, dff, E, c, torch.bfloat16, li, gelu=gelu, router=router)
