"""Edges of the kernels' own splits -- tiles, pairs of tiles, steps, blocks of tokens -- against the oracle, at sizes that
straddle them."""
import numpy as np
import pytest

from oracle import pquant_oracle as O
from paper_2602_22592_b200 import inputs as I
from test_gpu_forward import check_forward, run_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,K,E", [
    (1, 32, 2), (17, 288, 4),        # one token; one past a block of 16, one past a step of 256 elements
    (2369, 64, 5), (4737, 32, 9),    # one past 148 and past 2 x 148 blocks of tokens (one and two CTAs per SM); 8 / 16 experts
    (8209, 32, 16),                  # one past the 512 blocks of tokens that the scan takes in one go
])
def test_router_and_routing_tables(T, K, E):
    # indices, permutation and tables exact, gates and probabilities to the rounding of an fp32 softmax (check_forward)
    c = I.make_linear_case(T, K, 32, 16, E, seed=T + E, with_grad=False)
    check_forward(c, run_forward(c, False), O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"]))
    assert len(np.unique(O.router(c["X"], c["Wr"])["idx"])) >= min(T, 2)
