"""The small-batch kernel where a CTA has several items and ends several sequences, where one position is cut into many pieces, and
where a sampled segment touches a row's outer vectors, against the oracle by the rules of tests/parity.py (GPU)."""
import pytest
import torch

import oracle
from test_gpu_phase import check, inputs

pytestmark = pytest.mark.gpu


# all positions of 32 sequences (more items than SMs, by far), a single position, pieces of 512 vectors and more, rows at every alignment
@pytest.mark.parametrize("B,gamma,V,dtype,sigma_d", [(32, 16, 1024, "bf16", 0.1), (32, 16, 1001, "bf16", 0.1), (1, 1, 152064, "bf16", 1.0), (1, 1, 100277, "f32", 1.0),
                                                     (20, 5, 40000, "bf16", 0.3), (7, 9, 50257, "bf16", 0.1), (31, 3, 8211, "f32", 3.0), (3, 64, 4096, "f32", 0.05)])
def test_items_and_ends(B, gamma, V, dtype, sigma_d, bv_options):
    bv_options("kernel", 4)
    check(inputs(B, gamma, V, dtype, V + B, sigma_d), (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY), 4)


@pytest.mark.parametrize("V,dtype", [(4099, "bf16"), (2053, "f32")])
@pytest.mark.parametrize("kernel", [4, 5])
def test_samples_from_the_outer_vectors_of_a_row(V, dtype, kernel, bv_options):
    # nearly all of the target's mass on the first or the last tokens, none of the draft's: the sampled token lies in a vector that the
    # row shares with its neighbour, at every alignment that 12 sequences of 4 and 5 rows have
    bv_options("kernel", kernel)
    inp = inputs(12, 4, V, dtype, V, 0.5)
    t, d, x = inp["target_logits"], inp["draft_logits"], inp["draft_tokens"]
    for b in range(12):
        edge = slice(0, 3) if b % 2 else slice(V - 3, V)
        t[b, :, edge] += 30.0
        d[b, :, edge] = -20.0
        x[b] = 7 + torch.arange(4)
    check(inp, (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY), kernel)
