"""Rows masked with finite values so large that a float holds them, times log2(e) / T, only to within 2^6 and more, against the
oracle (GPU)."""
import numpy as np
import pytest
import torch

import oracle
import test_gpu_sampler
from paper_2403_10444_b200 import specdec, workloads as wl
from parity import run_oracle, run_cuda, compare, assert_parity
from test_gpu_specdec import oracle_loop

pytestmark = pytest.mark.gpu
MASKS = [-1e9, -1e10, -1e20]


def masked(x, value, every):
    """All but each `every`-th of the last quarter of a row's elements: what sweeps a row from its start sees masks alone."""
    V = x.shape[-1]
    out = torch.arange(V) < V - V // 4
    out |= torch.arange(V) % every != 0
    x[..., out] = value
    return torch.nonzero(~out).flatten()


@pytest.mark.parametrize("value", MASKS)
@pytest.mark.parametrize("T", [0.8, 1.0, 2.0])
@pytest.mark.parametrize("dtype,V", [("bf16", 16384), ("f32", 4096), ("bf16", 4099)])
@pytest.mark.parametrize("kernel", [1, 2, 3, 4, 5])
def test_masked_rows(kernel, dtype, V, T, value, bv_options):
    if V % 8 and kernel in (1, 2):
        pytest.skip("these kernels take rows of whole 16-byte vectors")
    bv_options("kernel", kernel)
    inp = wl.make_inputs(wl.Workload("m", 6, 3, V, dtype, T, V, 2.0, 0.0, 0, 0.0, 0.5), "cpu")
    kept = masked(inp["target_logits"], value, 7)
    masked(inp["draft_logits"], value, 7)
    inp["draft_tokens"][:] = kept[torch.randint(0, len(kept), (6, 3), generator=torch.Generator().manual_seed(2))].to(torch.int32)
    for algo in (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY):
        ref = run_oracle(algo, inp)
        assert (ref.out_len > 0).all()
        for diag in (True, False):
            out = run_cuda(algo, inp, diagnostics=diag)
            assert_parity(compare(algo, ref, out[0], out[1], out[2] if diag else None, inp), diag)


@pytest.mark.parametrize("value", MASKS)
@pytest.mark.parametrize("T", [0.8, 1.0, 2.0])
@pytest.mark.parametrize("dtype,V", [("bf16", 65536), ("bf16", 1024), ("f32", 8192)])
def test_sampler(dtype, V, T, value):
    g = torch.Generator().manual_seed(5)
    z = torch.randn((40, V), generator=g) * 2.0
    z = z.bfloat16() if dtype == "bf16" else z
    masked(z, value, 5)
    test_gpu_sampler.check(z, torch.rand((40,), generator=g), T)


@pytest.mark.parametrize("value", MASKS)
@pytest.mark.parametrize("dtype,V", [("bf16", 2048), ("f32", 512)])
def test_decoding_loop(dtype, V, value):
    B, gamma, N = 6, 3, 3
    tt, dt = wl.markov_models(V, dtype, 3, 2.0, 0.5, 1.1, "cpu")
    kept = masked(tt, value, 5)
    masked(dt, value, 5)
    ud, uv = wl.loop_uniforms(N, B, gamma, 4, "cpu")
    first = kept[:B].to(torch.int32)
    for algo, oalgo in (("block_lse", oracle.BLOCK_VERIFY), ("token", oracle.TOKEN_VERIFY)):
        want = oracle_loop(tt, dt, first, ud, uv, gamma, 0.8, oalgo, algo == "block_lse")
        out = specdec.run(tt.cuda(), dt.cuda(), first.cuda(), ud.cuda(), uv.cuda(), gamma, 0.8, algo)
        got = [out["tokens"][b, : out["lengths"][b]].tolist() for b in range(B)]
        # (a draw within 1e-6 of the edge of its cell, 200 of them, sends a sequence its own way; none does here)
        assert got == want, algo


# (the scaled value and the integer that a float has for it lie 312, -328, 512 and 328 apart)
@pytest.mark.parametrize("value,T", [(-1e10, 1.3), (-1e10, 1.0), (-3e10, 1.3), (1e10, 1.0)])
@pytest.mark.parametrize("V", [4096, 4099])
@pytest.mark.parametrize("kernel", [1, 2, 3, 4, 5])
def test_a_row_without_a_normaliser_is_a_data_fault(kernel, V, value, T, bv_options):
    if V % 8 and kernel in (1, 2):
        pytest.skip("these kernels take rows of whole 16-byte vectors")
    bv_options("kernel", kernel)
    inp = wl.make_inputs(wl.Workload("m", 8, 3, V, "bf16", T, V, 2.0, 0.0, 0, 0.0, 0.5), "cpu")
    for b in range(8):
        (inp["target_logits"] if b < 4 else inp["draft_logits"])[b, b % 3] = value        # (flat)
    for algo in (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY):
        out = run_cuda(algo, inp, diagnostics=False)
        ref = run_oracle(algo, inp)
        for b in range(8):
            # (Algorithm 1 may end before it gets to the row)
            assert out[1][b] == -1 or (algo == oracle.TOKEN_VERIFY and out[1][b] == ref.out_len[b] <= b % 3), (algo, b)


@pytest.mark.parametrize("value,T", [(-1e10, 1.3), (-1e10, 1.0), (-3e10, 1.3), (1e10, 1.0)])
@pytest.mark.parametrize("V", [1024, 65536])
def test_nothing_is_drawn_from_a_row_without_a_normaliser(V, value, T):
    import paper_2403_10444_b200 as bv
    z = torch.randn((6, V), generator=torch.Generator().manual_seed(1)).bfloat16()
    z[1::2] = value
    tok, lse = bv.bv_sample_draft(z.cuda(), torch.full((6,), 0.3, device="cuda"), T)
    assert (tok[1::2] == -1).all() and torch.isnan(lse[1::2]).all()
    assert (tok[0::2] >= 0).all() and torch.isfinite(lse[0::2]).all()
