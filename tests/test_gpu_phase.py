"""The phase kernel at the edges of its work units, at every alignment of the rows, and where its second round runs, and the
small-batch kernel at every alignment, against the oracle by the rules of tests/parity.py (GPU)."""
import pytest
import torch

import oracle
from paper_2403_10444_b200 import workloads as wl
from parity import run_oracle, run_cuda, compare, assert_parity

pytestmark = pytest.mark.gpu


def check(inp, algos, kernel=5):
    import paper_2403_10444_b200 as bv
    for algo in algos:
        ref = run_oracle(algo, inp)
        for diag in (True, False):
            out = run_cuda(algo, inp, diagnostics=diag)
            assert bv.bv_last_kernel() == kernel and bv.bv_stream_status() == 0
            assert_parity(compare(algo, ref, out[0], out[1], out[2] if diag else None, inp), diag)


def inputs(B, gamma, V, dtype, seed, sigma_d=0.5):
    return wl.make_inputs(wl.Workload("ph", B, gamma, V, dtype, 0.9, seed, 2.0, 0.0, 0, 0.0, sigma_d), "cpu")


# a unit is 64 vectors: 512 bf16 or 256 fp32 logits; rows one short of, at and one beyond whole units and vectors
@pytest.mark.parametrize("dtype,V", [("bf16", v) for v in (1, 7, 8, 9, 505, 511, 512, 513, 519, 520, 1023, 1025, 8191, 50257)] +
                         [("f32", v) for v in (1, 3, 4, 5, 253, 255, 256, 257, 1021, 1023, 20003)])
@pytest.mark.parametrize("B,gamma,kernel", [(1, 1, 5), (3, 40, 5), (50, 5, 5), (1, 1, 4), (3, 40, 4), (25, 5, 4)])
def test_rows_around_whole_units(dtype, V, B, gamma, kernel, bv_options):
    bv_options("kernel", kernel)
    check(inputs(B, gamma, V, dtype, V + B), (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY), kernel)


@pytest.mark.parametrize("dtype,V,gamma", [("bf16", 152065, 1), ("f32", 152064, 33), ("f32", 152065, 20)])
def test_rows_in_more_than_32_pieces(dtype, V, gamma, bv_options):
    # (a fold in which all lanes of a warp look at one row)
    import test_gpu_lse
    bv_options("kernel", 5)
    inp = inputs(1, gamma, V, dtype, gamma)
    check(inp, (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY))
    if V % 4 == 0:
        test_gpu_lse.run_case(inp, test_gpu_lse.own_lse(inp))


@pytest.mark.parametrize("V,B,gamma", [(4096, 768, 1), (64, 768, 3), (1003, 2000, 2), (16, 769, 2), (5089, 1533, 2)])
def test_as_many_sequences_as_it_takes_and_more(V, B, gamma, bv_options):
    # 768 sequences a launch; rows at any alignment go through it in parts beyond that, others through the flow kernel
    import paper_2403_10444_b200 as bv
    inp = inputs(B, gamma, V, "bf16", B)
    for algo in (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY):
        ref = run_oracle(algo, inp)
        for diag in (True, False):
            out = run_cuda(algo, inp, diagnostics=diag)
            assert bv.bv_last_launch_count() == ((B + 767) // 768 if V % 8 else 1) and bv.bv_stream_status() == 0
            assert_parity(compare(algo, ref, out[0], out[1], out[2] if diag else None, inp), diag)


@pytest.mark.parametrize("kernel", [4, 5])
@pytest.mark.parametrize("dtype,V", [("bf16", 4104), ("bf16", 3001), ("f32", 4100)])
def test_tensors_that_start_inside_a_vector(dtype, V, kernel, bv_options):
    # the first and the last row's outer vectors reach beyond the tensors
    import paper_2403_10444_b200 as bv
    bv_options("kernel", kernel)
    inp = inputs(5, 3, V, dtype, V)
    t, d = inp["target_logits"], inp["draft_logits"]
    for ot, od in ((1, 0), (0, 3), (3, 2)):
        dev = {k: v.cuda() if torch.is_tensor(v) else v for k, v in inp.items()}
        for k, src, off in (("target_logits", t, ot), ("draft_logits", d, od)):
            flat = torch.full((src.numel() + off,), float("nan"), dtype=src.dtype, device="cuda")
            flat[off:] = src.flatten().cuda()
            dev[k] = flat[off:].view(src.shape)
        for algo, fn in ((oracle.BLOCK_VERIFY, bv.bv_verify), (oracle.TOKEN_VERIFY, bv.tv_verify)):
            ref = run_oracle(algo, inp)
            out = fn(dev["target_logits"], dev["draft_logits"], dev["draft_tokens"], dev["uniforms"], inp["temperature"])
            assert bv.bv_last_kernel() == kernel
            assert_parity(compare(algo, ref, out[0], out[1], None, inp), False)


@pytest.mark.parametrize("V", [4096, 4099])
def test_candidates_below_an_empty_residual(V, bv_options):
    # P_2 == Q_2 and p_2 = 1: position 2 passes unless its residual is empty, which it is, and the candidates below it
    # get a round of their own.  (A last position that cannot pass, so that tau is not gamma.)
    bv_options("kernel", 5)
    inp = inputs(60, 4, V, "bf16", 9, sigma_d=1.0)
    t, d, x = inp["target_logits"], inp["draft_logits"], inp["draft_tokens"]
    t[:, :3] = d[:, :3]
    for b in range(60):
        t[b, 2, int(x[b, 2])] = -float("inf") if b % 2 else t[b, 2, int(x[b, 2])]      # (odd ones: a residual after all)
        t[b, 3, int(x[b, 3])] = -float("inf")
    check(inp, (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY))


@pytest.mark.parametrize("V,kernel", [(4096, 5), (4097, 5), (4097, 4)])
def test_faults_are_per_sequence(V, kernel, bv_options):
    bv_options("kernel", kernel)
    inp = inputs(12, 3, V, "f32", 3)
    t, d, x = inp["target_logits"], inp["draft_logits"], inp["draft_tokens"]
    t[1, 0, 3] = float("nan")
    x[2, 1] = V
    d[3, 0, int(x[3, 0])] = -float("inf")
    t[4, 1, :] = -float("inf")
    t[5, 2, 7] = float("inf")
    x[6, 0] = -1
    t[7, :, : V // 2] = -float("inf")
    ref = run_oracle(oracle.BLOCK_VERIFY, inp)
    ot, ol = run_cuda(oracle.BLOCK_VERIFY, inp, diagnostics=False)[:2]
    assert (ol[1:7] == -1).all() and (ot[1:7] == -1).all()
    assert (ol.cpu().numpy() == ref.out_len).all() and (ot.cpu().numpy() == ref.out_tokens).all()
    ref = run_oracle(oracle.TOKEN_VERIFY, inp)
    ot, ol = run_cuda(oracle.TOKEN_VERIFY, inp, diagnostics=False)[:2]
    assert (ol.cpu().numpy() == ref.out_len).all() and (ot.cpu().numpy() == ref.out_tokens).all()


@pytest.mark.parametrize("dtype,V", [("bf16", 8), ("bf16", 504), ("bf16", 520), ("bf16", 8200), ("f32", 4), ("f32", 260), ("f32", 20000)])
@pytest.mark.parametrize("B,gamma", [(1, 1), (7, 34), (50, 5)])
def test_the_other_entry_points_around_whole_units(dtype, V, B, gamma, bv_options):
    # Algorithm 4, supplied normalisers and probabilities, forced onto the phase kernel
    import paper_2403_10444_b200 as bv
    import test_gpu_lse
    import test_gpu_probs
    bv_options("kernel", 5)
    inp = inputs(B, gamma, V, dtype, V + B)
    check(inp, (oracle.GREEDY_BLOCK_VERIFY,))
    for algo in (oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY):
        test_gpu_lse.run_case(inp, test_gpu_lse.own_lse(inp), algo)
        assert bv.bv_last_kernel() == 5 and bv.bv_stream_status() == 0
    pin = test_gpu_probs.probs_inputs(wl.Workload("ph", B, gamma, V, dtype, 0.9, V + B, 2.0, 0.0, 0, 0.0, 0.5))
    for algo in ("block", "token"):
        test_gpu_probs.run_case(algo, pin, "phase kernel probs V=%d B=%d gamma=%d %s %s" % (V, B, gamma, dtype, algo))
        assert bv.bv_last_kernel() == 5 and bv.bv_stream_status() == 0


@pytest.mark.parametrize("algo", [oracle.BLOCK_VERIFY, oracle.TOKEN_VERIFY])
def test_supplied_normalisers_that_are_not_finite(algo, bv_options):
    import test_gpu_lse
    bv_options("kernel", 5)
    inp = inputs(12, 4, 4096, "bf16", 8)
    lse = test_gpu_lse.own_lse(inp)
    lse[2, 0], lse[3, 0], lse[4, 0], lse[5, 3] = float("nan"), float("inf"), -float("inf"), float("nan")
    ref = test_gpu_lse.run_case(inp, lse, algo)
    assert (ref.out_len[2:5] == -1).all() and (ref.out_len[[0, 1, 6]] > 0).all()


@pytest.mark.parametrize("V", [4096, 4099])
def test_a_wait_that_runs_out_is_reported_and_the_next_call_works(V, bv_options):
    import paper_2403_10444_b200 as bv
    bv_options("kernel", 5)
    inp = inputs(3, 2, V, "bf16", 1)
    a = [inp[k].cuda() for k in ("target_logits", "draft_logits", "draft_tokens", "uniforms")] + [inp["temperature"]]
    want = bv.bv_verify(*a)
    bv_options("wait_limit", 2000)
    bv_options("never_signal", 1)
    bv.bv_verify(*a)
    assert bv.bv_stream_status() == -4
    bv_options("never_signal", 0)
    bv_options("wait_limit", 0)
    got = bv.bv_verify(*a)
    assert bv.bv_stream_status() == 0
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("probs", [False, True])
@pytest.mark.parametrize("V", [4096, 4099])
def test_the_wait_for_the_second_sweeps_runs_out_too(V, probs, bv_options):
    # never_signal: 1 on probabilities, which have no first sweep, and 2 leave only the second sweeps unreported
    import paper_2403_10444_b200 as bv
    if probs and V % 8:
        pytest.skip("probabilities come in rows of whole 16-byte vectors")
    bv_options("kernel", 5)
    inp = inputs(3, 2, V, "bf16", 1)
    a = [inp[k].cuda() for k in ("target_logits", "draft_logits", "draft_tokens", "uniforms")]
    if probs:
        a[0], a[1] = a[0].float().softmax(-1).bfloat16(), a[1].float().softmax(-1).bfloat16()
    call = (lambda: bv.bv_verify_probs(*a)) if probs else (lambda: bv.bv_verify(*a, inp["temperature"]))
    want = call()
    assert bv.bv_stream_status() == 0
    bv_options("wait_limit", 2000)
    bv_options("never_signal", 1 if probs else 2)
    call()
    assert bv.bv_stream_status() == -4
    bv_options("never_signal", 0)
    bv_options("wait_limit", 0)
    got = call()
    assert bv.bv_stream_status() == 0
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
