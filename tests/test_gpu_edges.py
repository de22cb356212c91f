"""Edges of the kernels' own splits -- tiles, pairs of tiles, steps, blocks of tokens -- against the oracle, at sizes that
straddle them."""
import numpy as np
import pytest

from oracle import pquant_oracle as O
from paper_2602_22592_b200 import inputs as I
from test_gpu_backward import check_backward, run_fwd_bwd
from test_gpu_ffn import test_ffn_decoupled_forward_matches_oracle as check_ffn
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


@pytest.mark.parametrize("T,K,N,r,E,vector", [
    (1, 32, 32, 8, 1, False), (257, 288, 544, 72, 2, True),   # a lone tile of every kind; second tile of a pair with one row, r past 64
    (513, 544, 288, 128, 16, False),                          # experts that share tiles and pairs of tiles, most with few tokens
    (640, 4128, 96, 0, 0, False),                             # no HP branch: no dH tile to wait for; 17 column tiles, one feature tile
    (300, 64, 4128, 40, 1, True),                             # the longest contraction is dX's
])
def test_training_step_on_pairs_of_tiles(T, K, N, r, E, vector):
    # forward and every gradient, the tolerances of check_forward and check_backward
    c = I.make_linear_case(T, K, N, r, E, seed=T, scale_vector=vector, alpha=1.5, beta=0.5)
    f = O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    g = O.linear_backward(c["dY"], c["X"], f, c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    L = run_fwd_bwd(c, vector)
    check_forward(c, L, f)
    check_backward(c, L, f, g, vector)


@pytest.mark.parametrize("F1", [1056, 2080, 4128, 8224])
def test_ffn_rows_of_one_to_eight_warps(F1):
    # one past what one, two and four warps hold of a row in registers, and past what eight do; an odd number of rows.  Codes
    # and scales exact on the hidden activation the GPU made
    check_ffn(131, 96, F1, 16)


def test_forward_of_long_rows_uses_the_general_tile():
    # K = 32768: a sum of the 1-bit product no longer fits the short conversion to float; rows of equal signs reach |sum| ~ 128 K
    c = I.make_linear_case(40, 32768, 32, 8, 1, seed=3, with_grad=False)
    c["X"][:] = I.bf16_values(np.abs(c["X"]) + 4.0)
    c["W"][:16] = np.abs(c["W"][:16]) + 0.01
    f = O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    check_forward(c, run_forward(c, False), f)
